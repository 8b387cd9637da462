"""FP64 stepping over many steps with short lines: rounding errors of the
transforms must not repeat.  Against the same scheme in wider arithmetic; errors
that are independent from pass to pass add in quadrature, one rounding per
butterfly level: eps sqrt(passes * levels), four transforms per step."""
import math

import numpy as np
import pytest

import synthetic as S
from gpu_util import EPS

pytestmark = pytest.mark.gpu

L, DT = 20 * math.pi, 1e-3


def _reference(p0, n, steps):
    """NLS split steps in extended precision."""
    ld, cld = np.longdouble, np.clongdouble
    k = (ld(math.pi) + ld(1.2246467991473532e-16)) * 2 / ld(L) * np.fft.fftfreq(n, 1.0 / n).astype(ld)
    k2 = (k ** 2)[None] + (k ** 2)[:, None]
    dt = ld(DT)

    def turn(a):
        return np.cos(a) - 1j * np.sin(a)

    h = np.fft.fft2(p0.astype(cld)) * turn(k2 * dt / 2)
    for i in range(steps):
        q = np.fft.ifft2(h)
        q = q * turn((q.real ** 2 + q.imag ** 2) * dt)
        h = np.fft.fft2(q) * turn(k2 * (dt if i + 1 < steps else dt / 2))
    return np.fft.ifft2(h)


@pytest.mark.parametrize("n,steps", [(32, 100), (64, 200), (512, 10)])
def test_nls_rounding_does_not_accumulate(lib, cuda_device, n, steps):
    p0 = S.nls_gaussian(n)
    ref = _reference(p0, n, steps)
    g = lib.Grid("nls", n, "fp64", lx=L, ly=L, dt=DT)
    g.set_state(p0[None])
    g.step(steps)
    d = g.get_state()[0] - ref
    err = float(np.sqrt((np.abs(d) ** 2).sum() / (np.abs(ref) ** 2).sum()))
    assert err <= EPS["fp64"] * math.sqrt(4 * steps * math.log2(n)), err


@pytest.mark.parametrize("nx,ny", [(16, 16), (16, 64), (32, 32), (64, 64), (64, 1024), (128, 1024), (512, 512)])
def test_transform_error(lib, cuda_device, nx, ny):
    # as above for one 2D transform: one rounding per butterfly level
    import torch
    rng = np.random.default_rng(nx + ny)
    a = rng.standard_normal((2, ny, nx)) + 1j * rng.standard_normal((2, ny, nx))
    s = torch.cuda.current_stream().cuda_stream
    for direction, ref in ((-1, np.fft.fft2(a.astype(np.clongdouble))), (1, np.fft.ifft2(a.astype(np.clongdouble)))):
        t = torch.tensor(a, device=cuda_device)
        lib.pss_fft2d(t.data_ptr(), nx, ny, 2, lib.PSS_FP64, direction, s)
        d = t.cpu().numpy() - ref
        err = float(np.sqrt((np.abs(d) ** 2).sum() / (np.abs(ref) ** 2).sum()))
        assert err <= EPS["fp64"] * math.sqrt(math.log2(nx * ny)), err
