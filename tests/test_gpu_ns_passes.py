"""Navier-Stokes FP32 passes by shape: rows of up to 2048 points run one
transform at a time with C1 parked in shared memory, longer ones hold both
arrays; small grids on half spectra share a column tile among groups of
threads."""
import math

import numpy as np
import pytest

import synthetic as S
from gpu_util import check

pytestmark = pytest.mark.gpu

L, NU = 2 * math.pi, 1e-3


def _field(nx, ny):
    X, Y = np.meshgrid(S.grid_coords(nx, 0.0, L), S.grid_coords(ny, 0.0, L), indexing="xy")
    return np.sin(3 * X) * np.cos(2 * Y) + 0.5 * np.cos(X + Y) + 0.2 * np.sin(2 * X - 3 * Y)


@pytest.mark.parametrize("rfft,dealias", [(0, 1), (1, 1), (0, 0), (1, 0)])
@pytest.mark.parametrize("nx,ny", [(16, 64), (64, 16), (256, 32), (512, 32), (2048, 16), (4096, 16)])
def test_row_lengths_match_oracle(lib, orc, cuda_device, nx, ny, rfft, dealias):
    dt, steps = 2.5e-3, 4
    w0 = _field(nx, ny)
    ref, _, ok = orc.ns_run(orc.ns_init(w0, bool(dealias)), L, L, NU, dt, steps, dealias=bool(dealias))
    assert ok
    g = lib.Grid("ns", (nx, ny), "fp32", batch=3, lx=L, ly=L, dt=dt, nu=NU, dealias=dealias, rfft=rfft)
    g.set_state(np.stack([w0, 0.5 * w0, w0]))
    g.step(steps)
    got = g.get_state()
    check(got[0], orc.ns_field(ref), 1e-5)
    assert np.array_equal(got[0], got[2])


@pytest.mark.parametrize("scheme", ["cn", "midpoint"])
@pytest.mark.parametrize("nx,ny,batch", [(128, 128, 3), (256, 256, 1), (512, 256, 2), (64, 512, 1), (512, 512, 8),
                                         (1024, 1024, 1), (32, 2048, 1)])
def test_shared_column_tiles_are_bitwise_equal(lib, cuda_device, monkeypatch, nx, ny, batch, scheme):
    # four or two groups per tile (as many as run at once) against one
    w0 = np.stack([_field(nx, ny) * (1 + b) for b in range(batch)])
    out = []
    for fan in ("1", "0"):
        monkeypatch.setenv("PSS_COL_FAN", fan)
        g = lib.Grid("ns", (nx, ny), "fp32", batch=batch, lx=L, ly=L, dt=2.5e-3, nu=NU, rfft=1, scheme=scheme)
        g.set_state(w0)
        g.step(4)
        out.append((g.get_state(), g.stats()[1]))
        g.close()
    assert out[0][1] == out[1][1]
    assert np.array_equal(out[0][0].view(np.uint32), out[1][0].view(np.uint32))
