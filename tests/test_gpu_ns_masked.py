"""A dealiased Navier-Stokes grid that restores a checkpoint with non-zero modes
above the 2/3 cut (a grid without dealiasing wrote it): the first Jacobian is
that of the whole restored field.  One update from the restored state, against
the oracle's Jacobian in FP64; setting a state afterwards goes back to a field
without such modes."""
import math

import numpy as np
import pytest

from gpu_util import EPS, rel_l2

pytestmark = pytest.mark.gpu

L, NU, DT = 2 * math.pi, 1e-3, 1e-2


def _k(n):
    return np.fft.fftfreq(n, 1.0 / n)


def _one_update(orc, w_hat, keep):
    ny, nx = w_hat.shape
    j = np.fft.fft2(orc.ns_jacobian(w_hat, L, L)) * keep
    a = 0.5 * DT * NU * (_k(nx)[None] ** 2 + _k(ny)[:, None] ** 2)
    return ((1 - a) * w_hat - DT * j) / (1 + a)


@pytest.mark.parametrize("rfft", [0, 1])
@pytest.mark.parametrize("precision,nx,ny", [("fp32", 128, 64), ("fp64", 128, 64), ("fp32", 4096, 16)])
def test_restored_masked_modes_enter_the_jacobian(lib, orc, cuda_device, precision, nx, ny, rfft):
    rng = np.random.default_rng(nx + ny)
    keep = ((3 * np.abs(_k(nx)) < nx)[None] & (3 * np.abs(_k(ny)) < ny)[:, None]).astype(float)
    # real fields; a twentieth of the amplitude sits above the cut
    f = np.fft.fft2(rng.standard_normal((2, ny, nx))) / (1 + _k(nx)[None] ** 2 + _k(ny)[:, None] ** 2)
    edge = (np.abs(_k(nx))[None] == nx // 3 + 2) & (np.abs(_k(ny))[:, None] <= 3)
    f = f * keep + np.fft.fft2(rng.standard_normal((2, ny, nx))) * edge * 0.05
    w0 = np.real(np.fft.ifft2(f))
    kw = dict(batch=2, lx=L, ly=L, dt=DT, nu=NU, rfft=rfft, max_iter=1)
    a = lib.Grid("ns", (nx, ny), precision, dealias=0, **kw)
    a.set_state(w0)
    b = lib.Grid("ns", (nx, ny), precision, dealias=1, **kw)
    b.set_state(0.1 * w0)
    b.restore(a.checkpoint())

    def step_and_compare(w_hat):
        b.step(1)
        with pytest.raises(lib.PssError) as e:  # one update is all max_iter allows
            b.sync()
        assert e.value.code == lib.PSS_E_NOT_CONVERGED
        got = np.fft.fft2(b.get_state().astype(np.float64)) * keep
        for g, w in zip(got, w_hat):
            ref = _one_update(orc, w, keep) * keep
            # the change of the state, with the rounding of a state of its size
            tol = 8 * EPS[precision] * math.log2(nx * ny) * np.linalg.norm(ref) / np.linalg.norm(ref - w * keep)
            assert tol < 0.1 and rel_l2(g - w * keep, ref - w * keep) <= tol

    step_and_compare(np.fft.fft2(w0))
    b.set_state(w0)  # masks: the field without those modes
    step_and_compare(np.fft.fft2(w0) * keep)
