"""What is measured: whole solves, as a user's program runs them.

A pass sets the initial state of a grid from device arrays, advances it, reads the state back into device
arrays (and, where a program watches them, the conserved quantities): ``pss_set_state``, ``pss_step_n`` (or
``pss_step_n_batch`` over several grids), ``pss_conserved_quantities``, ``pss_get_state``.  One kind of case
is the standalone transform ``pss_fft2d``.  The grid, its plan and its buffers are made once, as a program
keeps them.

Equations, boxes, time steps and initial laws are those of the repository's workloads (``synthetic.py``,
``bench.py``, the tests); sizes run over the lengths those use, square and not, with odd batch sizes.
"""
from __future__ import annotations

import math

import torch

import paper_1206_3215_gb300 as P

PI = math.pi
CARD_L2 = 129e6  # bytes; a state that fits stays there between the passes of a step

# box and time step of each equation's workload
BOX = {"nls": 20 * PI, "sg": 10 * PI, "ns": 2 * PI}
DT = {"nls": 1e-3, "sg": 1e-3, "ns": 2.5e-4}
NU, TOL = 1e-3, 1e-10


def _solve(name, eq, nx, ny, batch, precision, steps, rfft=0, scheme="cn", dealias=1, invariants=False):
    c = {"kind": "solve", "eq": eq, "nx": nx, "ny": ny, "batch": batch, "precision": precision, "steps": steps,
         "rfft": rfft, "scheme": scheme, "dealias": dealias, "invariants": invariants}
    return {"name": name, **c} if name else c


def _fft(name, nx, ny, batch, precision, direction):
    c = {"kind": "fft2d", "nx": nx, "ny": ny, "batch": batch, "precision": precision, "direction": direction}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest workload: one 64^2 field in double, 200 steps, mass and energy watched (launches count)
        _solve("nls-f64-64", "nls", 64, 64, 1, "fp64", 200, invariants=True),
        # one round of a serving pool of small Schroedinger solves: eight 256^2 fields, 50 steps
        _solve("nls-f32-256-b8", "nls", 256, 256, 8, "fp32", 50),
        # the benchmark's batch: 32 fields of 1024^2 in single precision
        _solve("nls-f32-1024-b32", "nls", 1024, 1024, 32, "fp32", 50, invariants=True),
        # the same equation on the fine grid
        _solve("nls-f32-4096-b2", "nls", 4096, 4096, 2, "fp32", 20),
        # the double-precision path a single-precision run is compared with
        _solve("nls-f64-1024-b3", "nls", 1024, 1024, 3, "fp64", 10),
        # a serving round of sine-Gordon solves, half spectra
        _solve("sg-f32-512-b8", "sg", 512, 512, 8, "fp32", 50, rfft=1),
        # the sine-Gordon workload: 2048^2 in single precision, half spectra, Hamiltonian watched
        _solve("sg-f32-2048-b8", "sg", 2048, 2048, 8, "fp32", 50, rfft=1, invariants=True),
        # a small Navier-Stokes solve on the default full spectra, implicit midpoint, not square
        _solve("ns-f32-512x256-b5-mid", "ns", 512, 256, 5, "fp32", 20, scheme="midpoint"),
        # the Navier-Stokes workload: one 4096^2 field, half spectra
        _solve("ns-f32-4096", "ns", 4096, 4096, 1, "fp32", 10, rfft=1),
        # the paper's double-precision Navier-Stokes runs (no dealiasing, full spectra)
        _solve("ns-f64-256-paper", "ns", 256, 256, 1, "fp64", 20, dealias=0, invariants=True),
        # a server's round: pools of several equations and sizes advanced by one call, each on its own stream
        {"name": "serve-round", "kind": "round", "pools": "nls:128:8 sg:256:8 ns:512:8 ns:1024:4 nls:1024:4",
         "precision": "fp32", "steps": 20},
        # the standalone transform, long rows and a ragged batch
        _fft("fft2d-f32-4096x512-b5", 4096, 512, 5, "fp32", -1),
    ]


def _lengths(rng, cap, lo=6, hi=13):
    """nx, ny (powers of two, square about half the time), batch with nx ny batch <= cap."""
    while True:
        ex = rng.randint(lo, hi)
        ey = ex if rng.random() < 0.5 else rng.randint(lo, hi)
        nx, ny = 1 << ex, 1 << ey
        if nx * ny > cap:
            continue
        most = min(32, cap // (nx * ny))
        return nx, ny, int(round(math.exp(rng.uniform(0.0, math.log(most))))) if most > 1 else 1


def draw(rng):
    kind = rng.choice(["nls", "nls", "sg", "sg", "ns", "ns", "fft2d", "round"])
    double = rng.random() < 0.3
    precision = "fp64" if double else "fp32"
    if kind == "fft2d":
        nx, ny, batch = _lengths(rng, 1 << (21 if double else 25))
        return _fft(None, nx, ny, batch, precision, rng.choice([-1, 1]))
    if kind == "round":
        pools = []
        for _ in range(rng.randint(2, 5)):
            n = 1 << rng.randint(7, 10)
            pools.append(f"{rng.choice(['nls', 'sg', 'ns'])}:{n}:{min(8, (1 << 22) // (n * n))}")
        return {"kind": "round", "pools": " ".join(pools), "precision": "fp32", "steps": rng.randint(10, 30)}
    cap = 1 << (21 if double else 25)
    if kind == "ns":
        cap //= 2
    nx, ny, batch = _lengths(rng, cap)
    work = nx * ny * batch
    most = max(5, min(100, cap * (10 if kind == "ns" else 20) // work))
    steps = int(round(math.exp(rng.uniform(math.log(5), math.log(most)))))
    return _solve(None, kind, nx, ny, batch, precision, steps,
                  rfft=0 if kind == "nls" else int(rng.random() < 0.7),
                  scheme=rng.choice(["cn", "midpoint"]) if kind == "ns" else "cn",
                  dealias=int(rng.random() < 0.8) if kind == "ns" else 1, invariants=rng.random() < 0.3)


# ---- inputs ------------------------------------------------------------------


def _real(precision):
    return torch.float32 if precision == "fp32" else torch.float64


def _axes(nx, ny, length):
    x = -length / 2 + torch.arange(nx, dtype=torch.float64, device="cuda") * (length / nx)
    y = -length / 2 + torch.arange(ny, dtype=torch.float64, device="cuda") * (length / ny)
    return x[None, :], y[:, None]


def _wave(nx, ny, length, odd=False):
    """kx [1][nx], ky [ny][1]; odd: zero at the Nyquist index, as an odd derivative has it."""
    ks = []
    for n in (nx, ny):
        m = torch.arange(n, dtype=torch.float64, device="cuda")
        k = 2 * PI / length * torch.where(m < n // 2, m, m - n)
        if odd:
            k[n // 2] = 0.0
        ks.append(k)
    return ks[0][None, :], ks[1][:, None]


def _initial(eq, nx, ny, batch, precision, seed):
    """The workload's initial field, drawn from the seed, in the run's precision."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    L, shape = BOX[eq], (batch, ny, nx)

    def noise():
        return torch.randn(shape, generator=g, dtype=torch.float64, device="cuda")

    x, y = _axes(nx, ny, L)
    if eq == "nls":  # exp(-(x^2 + y^2)) + 1e-3 complex Gaussian
        s = 1e-3 * math.sqrt(0.5)
        f = torch.complex(torch.exp(-(x * x + y * y)) + s * noise(), s * noise())
        return f.to(torch.complex64 if precision == "fp32" else torch.complex128).contiguous()
    if eq == "sg":  # 0.5 exp(-(x^2 + y^2) / 4) + 1e-3 Gaussian, at rest
        return (0.5 * torch.exp(-(x * x + y * y) / 4) + 1e-3 * noise()).to(_real(precision)).contiguous()
    # vorticity with amplitudes |k|^-3, zero mean, unit rms
    kx, ky = _wave(nx, ny, L)
    k = torch.sqrt(kx * kx + ky * ky)
    amp = torch.where(k > 0, k, torch.ones_like(k)) ** -3.0
    amp[0, 0] = 0.0
    w = torch.empty(shape, dtype=_real(precision), device="cuda")
    for b in range(batch):
        z = torch.complex(torch.randn((ny, nx), generator=g, dtype=torch.float64, device="cuda"),
                          torch.randn((ny, nx), generator=g, dtype=torch.float64, device="cuda"))
        f = torch.fft.ifft2(amp * z).real
        f = f - f.mean()
        w[b] = (f / torch.sqrt((f * f).mean())).to(w.dtype)
    return w


def _fft_input(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((case["batch"], case["ny"], case["nx"]), generator=g, device="cuda",
                       dtype=torch.complex64 if case["precision"] == "fp32" else torch.complex128)


def _pools(case):
    """The grids of a round, as solves (half spectra where the server uses them)."""
    for text in case["pools"].split():
        eq, n, slots = text.split(":")
        yield _solve(None, eq, int(n), int(n), int(slots), case["precision"], case["steps"], rfft=0 if eq == "nls" else 1)


class _Run:
    """A grid with its input and output arrays."""

    def __init__(self, case, seed):
        eq, L = case["eq"], BOX[case["eq"]]
        self.case = case
        self.a = _initial(eq, case["nx"], case["ny"], case["batch"], case["precision"], seed)
        self.out = torch.empty_like(self.a)
        self.prev = torch.empty_like(self.a) if eq == "sg" else None
        kw = dict(x0=-L / 2, y0=-L / 2, lx=L, ly=L, dt=DT[eq])
        if eq != "nls":
            kw["rfft"] = case["rfft"]
        if eq == "ns":
            kw.update(nu=NU, tol=TOL, scheme=case["scheme"], dealias=case["dealias"])
        self.grid = P.Grid(eq, (case["nx"], case["ny"]), case["precision"], batch=case["batch"], **kw)

    def read(self):
        outs = {"state": self.out}
        if self.prev is not None:
            outs["previous"] = self.prev
        if self.case["invariants"]:
            outs["invariants"] = self.grid.conserved()
        self.grid.get_state_device(self.out, self.prev)
        return outs


def prepare(case, seed):
    if case["kind"] == "fft2d":
        state = {"case": case, "in": _fft_input(case, seed)}
        state["out"] = torch.empty_like(state["in"])
    elif case["kind"] == "round":
        state = {"case": case, "runs": [_Run(c, seed + 17 * i) for i, c in enumerate(_pools(case))]}
    else:
        state = {"case": case, "runs": [_Run(case, seed)]}
    torch.cuda.synchronize()  # the inputs are complete before another stream reads them
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "fft2d":  # in place, on a copy of the input, on torch's stream
        out = state["out"]
        out.copy_(state["in"])
        P.pss_fft2d(out.data_ptr(), case["nx"], case["ny"], case["batch"],
                    P.PSS_FP32 if case["precision"] == "fp32" else P.PSS_FP64, case["direction"],
                    torch.cuda.current_stream().cuda_stream)
        return out
    runs = state["runs"]
    for r in runs:
        r.grid.set_state(r.a)
    if case["kind"] == "round":
        P.pss_step_n_batch([r.grid.h for r in runs], [case["steps"]] * len(runs))
        return [r.read() for r in runs]
    runs[0].grid.step(case["steps"])
    return runs[0].read()


# ---- what a pass cannot do without --------------------------------------------


def _solve_work(case):
    """A solve reads the initial state and writes the final one.  A time step needs the transforms of its
    equation along both axes, with everything pointwise fused into them: a state too large for the L2 cache
    is then read and written once per axis (NLS: psi; SG: the transformed field per axis, and both time
    levels once; NS: per evaluation of the Jacobian the two packed derivative fields in, the Jacobian out, the
    vorticity at both levels).  Flops: 5 n log2 n per complex transform of n points, half for a real one,
    and the pointwise arithmetic."""
    nx, ny, eq = case["nx"], case["ny"], case["eq"]
    pts = nx * ny * case["batch"]
    cplx = 8 if case["precision"] == "fp32" else 16
    half = 2 if case["rfft"] else 1
    lg = math.log2(nx * ny)
    if eq == "nls":
        io, state, per_step = 2 * cplx * pts, cplx * pts, 4 * cplx * pts
        flops = case["steps"] * pts * (2 * 5 * lg + 30)
    elif eq == "sg":  # real fields: u in, u and its predecessor out
        io, state, per_step = 3 * (cplx // 2) * pts, 3 * cplx * pts // half, 8 * cplx * pts // half
        flops = case["steps"] * pts * (5 * lg + 30)
    else:  # two evaluations of the Jacobian per step: at the old level and once more
        kept = 4 / 9 if case["dealias"] else 1.0  # modes the 2/3 rule keeps; it prunes one axis of a pass
        line = 2 / 3 if case["dealias"] else 1.0
        w = cplx * pts / half * line
        io, state, per_step = (cplx // 2) * 2 * pts, 2 * cplx * pts + 3 * w, 2 * (4 * cplx * pts * line + 2 * w + 4 * w)
        flops = case["steps"] * pts * 2 * (2.5 * 5 * lg * (1 + line) / 2 + 30 * kept)
    moved = case["steps"] * per_step if state > CARD_L2 else 0
    return {"bytes": io + moved, "flops": flops}


def work(case):
    if case["kind"] == "fft2d":
        pts = case["nx"] * case["ny"] * case["batch"]
        size = (8 if case["precision"] == "fp32" else 16) * pts
        # read and written once; a field too large for the cache once per axis
        field = size / case["batch"]
        return {"bytes": size * (4 if field > CARD_L2 else 2), "flops": 5 * pts * math.log2(case["nx"] * case["ny"])}
    if case["kind"] == "round":
        ws = [_solve_work(c) for c in _pools(case)]
        return {"bytes": sum(w["bytes"] for w in ws), "flops": sum(w["flops"] for w in ws)}
    return _solve_work(case)


# ---- the same solves in 64 bits, plain torch -------------------------------------


def _exact_nls(case, a):
    L, dt = BOX["nls"], DT["nls"]
    kx, ky = _wave(case["nx"], case["ny"], L)
    k2 = kx * kx + ky * ky
    half = torch.polar(torch.ones_like(k2), -k2 * dt / 2)
    full = torch.polar(torch.ones_like(k2), -k2 * dt)
    out, inv = torch.empty_like(a), []
    for b in range(a.shape[0]):
        h = torch.fft.fft2(a[b]) * half
        for i in range(case["steps"]):
            p = torch.fft.ifft2(h)
            p = p * torch.polar(torch.ones_like(p.real), -(p.real ** 2 + p.imag ** 2) * dt)
            h = torch.fft.fft2(p) * (full if i + 1 < case["steps"] else half)
        p = torch.fft.ifft2(h)
        out[b] = p
        dA, n = L * L / k2.numel(), k2.numel()
        d = p.real ** 2 + p.imag ** 2
        inv.append([float(d.sum()) * dA, dA * (0.5 * float((k2 * (h.real ** 2 + h.imag ** 2)).sum()) / n
                                               + 0.25 * float((d * d).sum()))])
    return {"state": out, "invariants": inv}


def _exact_sg(case, a):
    L, dt = BOX["sg"], DT["sg"]
    nx, ny = case["nx"], case["ny"]
    kx, ky = _wave(nx, ny, L)
    k2 = (kx * kx + ky * ky)[:, : nx // 2 + 1].contiguous()
    q = dt * dt * k2
    out, prev, inv = torch.empty_like(a), torch.empty_like(a), []
    for b in range(a.shape[0]):
        u = a[b]
        h = torch.fft.rfft2(u)
        hm = h - 0.5 * dt * dt * (k2 * h + torch.fft.rfft2(torch.sin(u)))  # at rest: backward Taylor step
        for _ in range(case["steps"]):
            s = torch.fft.rfft2(torch.sin(torch.fft.irfft2(h, s=(ny, nx))))
            h, hm = ((2 - 0.5 * q) * h - dt * dt * s) / (1 + 0.25 * q) - hm, h
        u, um = torch.fft.irfft2(h, s=(ny, nx)), torch.fft.irfft2(hm, s=(ny, nx))
        out[b], prev[b] = u, um
        dA, n = L * L / (nx * ny), nx * ny
        mid = 0.5 * (h + hm)
        g = k2 * (mid.real ** 2 + mid.imag ** 2)
        grad = float(2 * g.sum() - g[:, 0].sum() - g[:, -1].sum()) / n
        pot = float(((u - um) ** 2 / (2 * dt * dt) + 2 * torch.sin(0.25 * (u + um)) ** 2).sum())
        inv.append([dA * (pot + 0.5 * grad)])
    return {"state": out, "previous": prev, "invariants": inv}


def _exact_ns(case, a):
    L, dt = BOX["ns"], DT["ns"]
    nx, ny = case["nx"], case["ny"]
    cut = slice(0, nx // 2 + 1)
    kx, ky = _wave(nx, ny, L)
    k2 = (kx * kx + ky * ky)[:, cut].contiguous()
    kx, ky = _wave(nx, ny, L, odd=True)
    ikx, iky = 1j * kx[:, cut], 1j * ky
    inv_k2 = torch.where(k2 > 0, 1 / torch.where(k2 > 0, k2, torch.ones_like(k2)), torch.zeros_like(k2))
    if case["dealias"]:
        keep = [3 * (m if m < n // 2 else n - m) < n for n in (nx, ny) for m in range(n)]
        keep = torch.tensor(keep, dtype=torch.float64, device="cuda")
        mask = keep[:nx][None, cut] * keep[nx:][:, None]
    else:
        mask = torch.ones_like(k2)
    # Parseval over the half spectrum: every column but the first and the last stands for two
    weight = torch.full((1, nx // 2 + 1), 2.0, dtype=torch.float64, device="cuda")
    weight[0, 0] = weight[0, -1] = 1.0
    scale = L * L / float(nx * ny) ** 2
    al = 0.5 * dt * NU * k2

    def jac(w):
        psi = w * inv_k2

        def phys(f):
            return torch.fft.irfft2(f, s=(ny, nx))

        j = phys(iky * psi) * phys(ikx * w) - phys(ikx * psi) * phys(iky * w)
        return torch.fft.rfft2(j) * mask

    out, inv = torch.empty_like(a), []
    for b in range(a.shape[0]):
        w = torch.fft.rfft2(a[b]) * mask
        for _ in range(case["steps"]):
            jn, wk = jac(w), w
            for k in range(100):
                if k == 0:
                    j2 = 2 * jn
                else:
                    j2 = 2 * jac(0.5 * (wk + w)) if case["scheme"] == "midpoint" else jac(wk) + jn
                new = ((1 - al) * w - 0.5 * dt * j2) / (1 + al)
                d = new - wk
                norm = scale * float((weight * (d.real ** 2 + d.imag ** 2)).sum())
                wk = new
                if norm < TOL:
                    break
            w = wk
        out[b] = torch.fft.irfft2(w, s=(ny, nx))
        e = weight * (w.real ** 2 + w.imag ** 2)
        inv.append([L * L / (nx * ny) * float(w[0, 0].real), 0.5 * scale * float(e.sum()),
                    0.5 * scale * float((e * inv_k2).sum())])
    return {"state": out, "invariants": inv}


def _exact_solve(case, seed):
    a = _initial(case["eq"], case["nx"], case["ny"], case["batch"], case["precision"], seed)
    a = a.to(torch.complex128 if case["eq"] == "nls" else torch.float64)
    outs = {"nls": _exact_nls, "sg": _exact_sg, "ns": _exact_ns}[case["eq"]](case, a)
    inv = outs.pop("invariants")
    if case["invariants"]:
        outs["invariants"] = torch.tensor(inv, dtype=torch.float64)
    return outs


def exact(case, seed):
    if case["kind"] == "fft2d":
        x = _fft_input(case, seed).to(torch.complex128)
        return torch.fft.fft2(x) if case["direction"] < 0 else torch.fft.ifft2(x)
    if case["kind"] == "round":
        return [_exact_solve(c, seed + 17 * i) for i, c in enumerate(_pools(case))]
    return _exact_solve(case, seed)
