"""Short FP64 lines (up to 512 points) run with fewer points per thread, again
fewer in small fields (at most 2^16 points): both sides of that line, the
shortest lengths, and batches that do not fill a CTA, against the oracle (FP32
beside it)."""
import math

import numpy as np
import pytest

import synthetic as S
from gpu_util import EPS, check

pytestmark = pytest.mark.gpu

SHAPES = [(16, 16, 1), (32, 16, 3), (16, 32, 2), (64, 1024, 1), (64, 2048, 1), (1024, 64, 1), (2048, 64, 1),
          (128, 512, 1), (128, 1024, 1), (1024, 128, 1), (256, 256, 3), (256, 512, 1), (512, 256, 1), (512, 16, 3)]


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nx,ny,batch", SHAPES)
def test_fft2d_short_lines(lib, orc, cuda_device, precision, nx, ny, batch):
    import torch
    rng = np.random.default_rng(nx * 31 + ny + batch)
    a = rng.standard_normal((batch, ny, nx)) + 1j * rng.standard_normal((batch, ny, nx))
    a = a.astype(np.complex64 if precision == "fp32" else np.complex128)
    t = torch.tensor(a, device=cuda_device)
    prec = lib.PSS_FP32 if precision == "fp32" else lib.PSS_FP64
    s = torch.cuda.current_stream().cuda_stream
    lib.pss_fft2d(t.data_ptr(), nx, ny, batch, prec, -1, s)
    tol = 4 * EPS[precision] * math.log2(nx * ny)  # eps log2(size), as for the other lengths
    check(t.cpu().numpy(), np.stack([orc.fft2d(x.astype(np.complex128)) for x in a]), tol)
    lib.pss_fft2d(t.data_ptr(), nx, ny, batch, prec, +1, s)
    check(t.cpu().numpy(), a, 2 * tol)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [64, 128, 256])
def test_sg_half_spectra_short_lines(lib, orc, cuda_device, precision, n):
    # the half-spectrum row pass transforms rows of n/2 points
    dt, steps, Ls = 1e-3, 10, 10 * math.pi
    u0, v0 = S.sg_gaussian(n, batch=3)
    g = lib.Grid("sg", n, precision, batch=3, lx=Ls, ly=Ls, x0=-Ls / 2, y0=-Ls / 2, dt=dt, rfft=1)
    g.set_state(u0, v0)
    g.step(steps)
    got = g.get_state()[0]
    for b in (0, 2):
        un, um = orc.sg_init(u0[b], v0[b], Ls, Ls, dt)
        un, um = orc.sg_run(un, um, Ls, Ls, dt, steps)
        check(got[b], orc.sg_fields(un, um)[0], 2e-5 if precision == "fp32" else 1e-10)
