"""Sine-Gordon Hamiltonian on half spectra at the shortest rows: at nx = 16 a
row of the half spectrum is as long as one of the full spectrum."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

L, DT = 10 * math.pi, 1e-3


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nx,ny", [(16, 16), (16, 128), (32, 16)])
def test_hamiltonian_of_short_rows(lib, orc, cuda_device, nx, ny, precision):
    # a quadratic form of the state, summed in FP64: its relative error is twice
    # the state's, at most 2 eps log2(points) (steps + 1) with eps = 2^-24 or 2^-53
    steps = 3
    rng = np.random.default_rng(nx + ny)
    u0 = rng.standard_normal((2, ny, nx)).astype(np.float32).astype(np.float64)
    eps = 2.0 ** (-24 if precision == "fp32" else -53)
    tol = 2 * eps * math.log2(nx * ny) * (steps + 1)
    got = []
    for rfft in (0, 1):
        g = lib.Grid("sg", (nx, ny), precision, batch=2, lx=L, ly=L, dt=DT, rfft=rfft)
        g.set_state(u0)
        g.step(steps)
        got.append(g.conserved()[:, 0])
        g.close()
    ref = []
    for b in range(2):
        un, um = orc.sg_init(u0[b], np.zeros_like(u0[b]), L, L, DT)
        un, um = orc.sg_run(un, um, L, L, DT, steps)
        ref.append(orc.sg_hamiltonian(un, um, L, L, DT))
    assert np.allclose(got[1], ref, rtol=tol, atol=0.0), (got, ref)
    assert np.allclose(got[0], ref, rtol=tol, atol=0.0), (got, ref)
