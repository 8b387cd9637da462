"""Navier-Stokes convergence test on column tiles of less than a warp: the
squared difference of the iterates is summed over the threads that exist.  The
tolerance is set just above and just below the norm of the second update (from
the oracle), so that a sum off by more than the margin changes the number of
updates."""
import math

import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

L, NU, DT = 2 * math.pi, 1e-3, 2e-2
MARGIN = 1.3


def _field(nx, ny):
    X, Y = np.meshgrid(S.grid_coords(nx, 0.0, L), S.grid_coords(ny, 0.0, L), indexing="xy")
    return np.sin(3 * X) * np.cos(2 * Y) + 0.5 * np.cos(X + Y) + 0.2 * np.sin(2 * X - 3 * Y)


def _second_norm(orc, w0, scheme):
    """The norm of the second update: the tolerance at which two updates become enough."""
    def updates(tol):
        return int(orc.ns_run(orc.ns_init(w0, True), L, L, NU, DT, 1, tol=tol, scheme=scheme)[1][0])

    lo, hi = 1e-14, 1.0
    while updates(hi) < 2:
        hi /= 10
    assert updates(hi) == 2 and updates(lo) > 2
    while hi / lo > 1.01:
        mid = math.sqrt(lo * hi)
        lo, hi = (lo, mid) if updates(mid) <= 2 else (mid, hi)
    return math.sqrt(lo * hi)


@pytest.mark.parametrize("scheme", ["cn", "midpoint"])
@pytest.mark.parametrize("precision,nx,ny", [("fp32", 64, 16), ("fp32", 64, 32), ("fp32", 64, 64), ("fp32", 64, 128),
                                             ("fp64", 64, 16), ("fp64", 64, 32), ("fp64", 4096, 32)])
def test_updates_at_the_edge_of_the_tolerance(lib, orc, cuda_device, precision, nx, ny, scheme):
    w0 = _field(nx, ny)
    norm = _second_norm(orc, w0, scheme)
    for tol, expected in ((norm * MARGIN, 2), (norm / MARGIN, 3)):
        g = lib.Grid("ns", (nx, ny), precision, batch=2, lx=L, ly=L, dt=DT, nu=NU, tol=tol, scheme=scheme)
        g.set_state(np.stack([w0, w0]))
        g.step(1)
        assert g.stats()[1] == 2 * expected
        g.close()
