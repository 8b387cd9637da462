"""Accuracy of read-back alone: the state read back against the exact inverse
transform of the spectra that a checkpoint holds, on half spectra and on full
ones.  Both take the transforms of whole rows, then of whole columns, and the
real part, which drops half of the error variance of each stage; half spectra
extend each row by another row's conjugate, so that at worst their row stage
keeps its whole variance: (r + c / 2) / (r / 2 + c / 2) <= 1.5 for r <= c, a
factor of sqrt(1.5) in the error.  Transforming half the columns first, or
half-length rows, lies above that."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

L = 10 * math.pi
BATCH = 3


def _rel(a, b):
    d = (a.astype(b.dtype) - b).ravel()
    return float(np.sqrt((d * d).sum() / (b * b).sum()))


@pytest.mark.parametrize("eq", ["sg", "ns"])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nx,ny", [(64, 64), (256, 128), (256, 256), (128, 512)])
def test_half_spectra_read_back_as_accurately_as_full_ones(lib, cuda_device, nx, ny, precision, eq):
    rng = np.random.default_rng(nx + 3 * ny)
    real, cplx = (np.float32, np.complex64) if precision == "fp32" else (np.float64, np.complex128)
    wide = np.complex128 if precision == "fp32" else np.clongdouble
    w0 = rng.standard_normal((BATCH, ny, nx)).astype(real)
    err = []
    for rfft in (0, 1):
        g = lib.Grid(eq, (nx, ny), precision, batch=BATCH, lx=L, ly=L, dt=1e-3, rfft=rfft)
        g.set_state(w0)
        got = g.get_state()
        got = got[0] if eq == "sg" else got
        n = BATCH * ny * nx
        hat = g.checkpoint()[: n * np.dtype(cplx).itemsize].view(cplx).reshape(BATCH, ny, nx)
        err.append(_rel(got, np.real(np.fft.ifft2(hat.astype(wide)))))
        g.close()
    assert err[1] <= math.sqrt(1.5) * err[0], err
