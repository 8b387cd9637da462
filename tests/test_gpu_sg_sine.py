"""Sine-Gordon FP32 passes: threads whose values all lie within pi/4 run the
sine polynomial without the argument reduction.  Fields below, across and above
that line, with both layouts, against the oracle."""
import math

import numpy as np
import pytest

import synthetic as S
from gpu_util import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rfft", [0, 1])
@pytest.mark.parametrize("amp", [0.7, 0.785, 0.8, 3.0])
@pytest.mark.parametrize("n", [64, 512])
def test_sine_range_matches_oracle(lib, orc, cuda_device, n, amp, rfft):
    L, dt, steps = 10 * math.pi, 1e-3, 10
    x = S.grid_coords(n, -L / 2, L)
    X, Y = np.meshgrid(x, x, indexing="xy")
    u0 = amp * np.exp(-(X * X + Y * Y) / 4)
    un, um = orc.sg_init(u0, np.zeros_like(u0), L, L, dt)
    un, um = orc.sg_run(un, um, L, L, dt, steps)
    g = lib.Grid("sg", n, "fp32", lx=L, ly=L, x0=-L / 2, y0=-L / 2, dt=dt, rfft=rfft)
    g.set_state(u0[None])
    g.step(steps)
    check(g.get_state()[0][0], orc.sg_fields(un, um)[0], 2e-5)
