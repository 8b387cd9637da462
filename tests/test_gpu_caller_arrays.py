"""Caller arrays on the device that are aligned for their elements only (a
slice one element into an allocation): set-up and read-back go through a copy
where the kernels read wider, and the standalone transform asks for no bulk
prefetch; the results are those of aligned arrays, bit for bit."""
import math

import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu


def _shifted(x):
    """The same values one element into a larger allocation."""
    import torch
    buf = torch.zeros(x.numel() + 1, dtype=x.dtype, device=x.device)
    buf[1:] = x.reshape(-1)
    return buf[1:].reshape(x.shape)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("eq,rfft", [("nls", 0), ("sg", 0), ("sg", 1), ("ns", 0), ("ns", 1)])
def test_set_and_get_state(lib, cuda_device, eq, rfft, precision):
    import torch
    n, batch = 128, 2
    real = torch.float32 if precision == "fp32" else torch.float64
    kw = dict(lx=2 * math.pi, ly=2 * math.pi, dt=1e-3)
    if eq == "nls":
        x = torch.tensor(S.nls_gaussian(n, batch=batch), device=cuda_device)
        x = x.to(torch.complex64 if precision == "fp32" else torch.complex128)
    else:
        w = S.ns_power_law(n, batch=batch) if eq == "ns" else S.sg_gaussian(n, batch=batch)[0]
        x = torch.tensor(w, device=cuda_device, dtype=real)
        kw["rfft"] = rfft
    v = 0.1 * x if eq == "sg" else None
    out = []
    for move in (lambda t: t, _shifted):
        g = lib.Grid(eq, n, precision, batch=batch, **kw)
        a, b = move(x), None if v is None else move(v)
        torch.cuda.synchronize()
        g.set_state(a, b)
        g.step(3)
        ra, rb = move(torch.zeros_like(x)), move(torch.zeros_like(x)) if eq == "sg" else None
        torch.cuda.synchronize()
        g.get_state_device(ra, rb)
        out.append([t.cpu().numpy() for t in (ra, rb) if t is not None])
        g.close()
    assert all(np.array_equal(p, q) for p, q in zip(*out))
    assert np.any(out[0][0])


@pytest.mark.parametrize("nx,ny", [(512, 64), (2048, 16)])
def test_fft2d(lib, cuda_device, nx, ny):
    import torch
    g = torch.Generator(device=cuda_device).manual_seed(nx)
    x = torch.randn((400, ny, nx), generator=g, dtype=torch.complex64, device=cuda_device)
    a, b = x.clone(), _shifted(x)
    for t in (a, b):
        lib.pss_fft2d(t.data_ptr(), nx, ny, 400, lib.PSS_FP32, -1, torch.cuda.current_stream().cuda_stream)
    assert torch.equal(torch.view_as_real(a), torch.view_as_real(b.contiguous()))
