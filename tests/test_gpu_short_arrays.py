"""A caller's device array that ends before the state does is refused on the
host, by set-up and by read-back, and the grid goes on with the state it had."""
import ctypes
import math

import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

SHORT = 1 << 20  # bytes of the short array; the states below take 16 MB and more


@pytest.fixture
def short_array(cuda_device):
    import torch
    torch.zeros(1, device=cuda_device)  # the device's context is current
    cu = ctypes.CDLL("libcuda.so.1")
    p = ctypes.c_uint64()
    assert cu.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(SHORT)) == 0
    yield p.value
    torch.cuda.synchronize()
    assert cu.cuMemFree_v2(p) == 0


@pytest.mark.parametrize("eq,rfft,precision", [("nls", 0, "fp32"), ("sg", 0, "fp32"), ("sg", 1, "fp64"),
                                               ("ns", 0, "fp32"), ("ns", 1, "fp64")])
def test_short_device_arrays_are_refused(lib, cuda_device, short_array, eq, rfft, precision):
    n = 2048 if precision == "fp32" else 1024
    kw = dict(lx=2 * math.pi, ly=2 * math.pi, dt=1e-3)
    if eq != "nls":
        kw["rfft"] = rfft
    rng = np.random.default_rng(1)
    x = S.nls_gaussian(n)[None] if eq == "nls" else rng.standard_normal((1, n, n))
    g = lib.Grid(eq, n, precision, batch=2, **kw)
    g.set_state(np.concatenate([x, 2 * x]))
    before = g.get_state()
    first = before[0] if eq == "sg" else before
    calls = [lambda: lib.pss_set_state(g.h, short_array, None, lib.PSS_DEVICE),
             lambda: lib.pss_get_state(g.h, short_array, None, lib.PSS_DEVICE),
             lambda: lib.pss_set_field(g.h, 1, short_array, None, lib.PSS_DEVICE),
             lambda: lib.pss_get_field(g.h, 1, short_array, None, lib.PSS_DEVICE)]
    for call in calls:
        with pytest.raises(lib.PssError) as e:
            call()
        assert e.value.code == lib.PSS_E_CUDA
    after = g.get_state()
    assert np.array_equal(after[0] if eq == "sg" else after, first)
    g.step(1)
    g.sync()
    g.close()
