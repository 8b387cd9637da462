"""Navier-Stokes fields of one call step on their own: fields of a batch that
take different, odd and even, numbers of updates per step, over several steps,
give the bits and the update counts of their solo runs, in the captured loop
(two updates per body) and launched kernel by kernel (one).  In the midpoint
scheme a field that ends its step within a body waits for the next one."""
import math

import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

L, NU, DT, STEPS = 2 * math.pi, 1e-3, 1e-2, 7


def _fields(nx, ny):
    X, Y = np.meshgrid(S.grid_coords(nx, 0.0, L), S.grid_coords(ny, 0.0, L), indexing="xy")
    a = np.sin(X) * np.sin(Y)  # J = 0: two updates per step
    b = np.sin(3 * X) * np.cos(2 * Y) + 0.5 * np.cos(X + Y) + 0.2 * np.sin(2 * X - 3 * Y)
    return np.stack([a, 0.01 * b, 0.1 * b, b, 4 * b])


@pytest.mark.parametrize("scheme", ["cn", "midpoint"])
@pytest.mark.parametrize("precision,nx,ny,rfft", [("fp32", 128, 128, 0), ("fp32", 128, 128, 1),
                                                  ("fp64", 128, 128, 0), ("fp64", 128, 128, 1)])
def test_mixed_update_counts_equal_solo_runs(lib, cuda_device, monkeypatch, precision, nx, ny, rfft, scheme):
    w0 = _fields(nx, ny)

    def run(w, calls):
        g = lib.Grid("ns", (nx, ny), precision, batch=len(w), lx=L, ly=L, dt=DT, nu=NU, rfft=rfft, scheme=scheme)
        g.set_state(w)
        for n in calls:
            g.step(n)
        out = g.get_state(), g.stats()[1]
        g.close()
        return out

    solo = [run(w0[i:i + 1], [STEPS]) for i in range(len(w0))]
    counts = [c for _, c in solo]
    assert len(set(counts)) >= 3 and any(c % 2 for c in counts), counts
    for graphs in ("1", "0"):
        monkeypatch.setenv("PSS_GRAPHS", graphs)
        for calls in ([STEPS], [1, 2, STEPS - 3]):
            state, updates = run(w0, calls)
            assert updates == sum(counts)
            for i, (alone, _) in enumerate(solo):
                assert np.array_equal(state[i], alone[0]), (graphs, calls, i)
