"""Accuracy of the sine-Gordon start-up: d^0 (read from a checkpoint) against its
formula in wider arithmetic, at small, mixed and large amplitudes, with and
without an initial velocity, on both layouts."""
import math

import numpy as np
import pytest

from gpu_util import EPS, rel_l2

pytestmark = pytest.mark.gpu

L, DT = 10 * math.pi, 1e-3


def _fields(nx, ny, amp, real):
    rng = np.random.default_rng(nx + ny)
    x = -L / 2 + np.arange(nx) * L / nx
    y = (-L / 2 + np.arange(ny) * L / ny)[:, None]
    u0 = amp * np.exp(-(x * x + y * y) / 4) + 1e-3 * rng.standard_normal((ny, nx))
    v0 = 0.3 * np.exp(-(x * x + (y - 1) ** 2) / 3) + 1e-3 * rng.standard_normal((ny, nx))
    return u0.astype(real), v0.astype(real)


@pytest.mark.parametrize("rfft", [0, 1])
@pytest.mark.parametrize("velocity", [False, True])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nx,ny,amp", [(64, 64, 0.5), (64, 64, 3.0), (256, 128, 0.79), (128, 512, 40.0)])
def test_start_up_increment(lib, cuda_device, nx, ny, amp, precision, velocity, rfft):
    real, cplx = (np.float32, np.complex64) if precision == "fp32" else (np.float64, np.complex128)
    wide = np.float64 if precision == "fp32" else np.longdouble
    u0, v0 = _fields(nx, ny, amp, real)
    g = lib.Grid("sg", (nx, ny), precision, lx=L, ly=L, dt=DT, rfft=rfft)
    g.set_state(u0[None], v0[None] if velocity else None)
    n = nx * ny * np.dtype(cplx).itemsize
    hat = g.checkpoint()[: 2 * n].view(cplx).reshape(2, ny, nx).astype(np.complex128 if precision == "fp32" else np.clongdouble)
    # the sum's own terms: exact transforms of sin u0 and v0, the stored transform of u0
    h = wide(DT) * wide(DT) / 2
    pi = wide(math.pi) + wide(1.2246467991473532e-16)
    k2 = ((2 * pi / wide(L) * np.fft.fftfreq(nx, 1.0 / nx).astype(wide)) ** 2)[None] \
        + ((2 * pi / wide(L) * np.fft.fftfreq(ny, 1.0 / ny).astype(wide)) ** 2)[:, None]
    s = np.fft.fft2(h * np.sin(u0.astype(wide)))
    v = np.fft.fft2(wide(DT) * v0.astype(wide)) if velocity else 0 * s
    ref = v + s + h * k2 * hat[0]
    # each transform is off by at most eps log2(points) of its size (the sine and
    # the sum round once each): bound the error by those of the terms together
    size = np.linalg.norm(s) + (np.linalg.norm(v) if velocity else 0.0)
    tol = EPS[precision] * (math.log2(nx * ny) * float(size) + float(np.linalg.norm(ref))) / float(np.linalg.norm(ref))
    assert rel_l2(hat[1], ref) <= tol


@pytest.mark.parametrize("rfft", [0, 1])
def test_start_up_sine_is_rounded_once(lib, cuda_device, rfft):
    # d^0 of fields that differ in u0 only through sin: constant fields, where
    # only the mean mode is there and no |k|^2 term: d(0,0) = nx ny (dt^2/2) sin u
    n = 16
    rng = np.random.default_rng(5)
    u = np.concatenate([rng.uniform(-0.785, 0.785, 300), rng.uniform(-60, 60, 100), 10.0 ** rng.uniform(-6, 0, 100),
                        [0.0, 0.785, -0.785, 0.7851, 1e5, -3e6]]).astype(np.float32)
    g = lib.Grid("sg", n, "fp32", batch=len(u), lx=L, ly=L, dt=DT, rfft=rfft)
    g.set_state(np.broadcast_to(u[:, None, None], (len(u), n, n)).copy())
    size = len(u) * n * n * 8
    d = g.checkpoint()[size: 2 * size].view(np.complex64).reshape(len(u), n, n)[:, 0, 0].real.astype(np.float64)
    # powers of two scale exactly; sums of 256 equal values round 8 times at
    # most up the tree, none of them for a value of the mean's own precision
    ref = n * n * (0.5 * DT * DT) * np.sin(u.astype(np.float64)).astype(np.float32).astype(np.float64)
    assert np.all(np.abs(d - ref) <= 2.0 ** -23 * np.abs(ref))
