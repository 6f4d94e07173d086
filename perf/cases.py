"""Timing cases of the solver: whole solves through the public entry points.

One pass of a case is what a user's program does with a problem that it has
set up: set_initial (u0 on the device), nsteps time steps from t = 0 (the
Richardson start-up, then Adams steps), and the read-out of u on the grid.
The set-up itself (the Problem with its tables, V(x, t), the pulse) is in
prepare().

A case is a dict of plain values:
  kind       "periodic" (1D, 2D, 3D), "free" (the same with modes on the
             contour) or "uneven" (1D periodic members of several sizes
             stepped together by Batch)
  shape      "512x512"; for "uneven" one size per member, "256,512"
  batch      instances; for "uneven" one count per member, "77,71"
  precision  "fp64" or "mixed"
  order, dt, nsteps
  V          "wells" (static), "factor" (f(t) V0(x)), "shared_table" (a moving
             well sampled at the scheme's times, one table for the batch)
  A0         amplitude of the sin^2 pulse along axis 0 (0: no field)
  ratio      free space: nu / n per axis; H, n_r: contour offset and panels

Outputs are u of every instance: complex128 for FP64 solves; a mixed solve
carries six to seven digits (FP32 transforms and history), so its user keeps
complex64.
"""
from __future__ import annotations

import math
from fractions import Fraction

import numpy as np
import torch

from paper_2001_06113_gb300 import Batch, Problem

OMEGA = 10.0
ON_CHIP_INSTANCE = 480e3      # bytes of state and history that one SM can hold (registers and shared memory)
ON_CHIP_ALL = 126e6           # bytes that stay in the L2 from step to step


def _case(name, kind, shape, batch, precision, nsteps, dt, order=8, V="wells", A0=2.0, ratio=0, H=0.0, n_r=1):
    return {"name": name, "kind": kind, "shape": shape, "batch": batch, "precision": precision, "nsteps": nsteps,
            "dt": dt, "order": order, "V": V, "A0": A0, "ratio": ratio, "H": H, "n_r": n_r}


def listed():
    return [
        # one small 1D problem, time-dependent potential, T = 1: the smallest call, all latency
        _case("1d_128_fp64", "periodic", "128", "1", "fp64", 100, 1e-2, V="factor", A0=0.0),
        # a sweep over initial states in one moving well (Example 1 of the paper), part of its 3200 steps
        _case("1d_512_mixed_x2048", "periodic", "512", "2048", "mixed", 300, 2.0 * math.pi / 15.0 / 3200,
              V="shared_table", A0=0.0),
        # an uneven batch of 512 members, 256 to 16384 points
        _case("1d_uneven_mixed_x512", "uneven", "256,512,1024,2048,4096,8192,16384", "77,71,75,69,73,69,78", "mixed",
              200, 1e-3),
        # a large 1D grid on its own, as a request of the serving loop brings it
        _case("1d_65536_mixed", "periodic", "65536", "1", "mixed", 300, 5e-4),
        # a small non-square 2D problem on its own, as a request of the serving loop brings it
        _case("2d_128x256_mixed", "periodic", "128x256", "1", "mixed", 400, 1e-3),
        # the headline workload: 64 instances of 512^2 in mixed precision, part of its 2000 steps
        _case("2d_512_mixed_x64", "periodic", "512x512", "64", "mixed", 300, 1e-3),
        # the same problem in the paper's precision
        _case("2d_512_fp64_x4", "periodic", "512x512", "4", "fp64", 100, 1e-3),
        # 3D wells
        _case("3d_128_mixed_x5", "periodic", "128x128x128", "5", "mixed", 120, 1e-3),
        # 1D free space, no refined panels (Example 3 of the paper)
        _case("free1d_128_fp64", "free", "128", "1", "fp64", 200, 1e-3, ratio=8, H=4.5, n_r=0),
        # the 2D free-space workload in FP64 and with FP32 transforms, part of its 2000 steps
        _case("free2d_256_fp64", "free", "256x256", "1", "fp64", 60, 5e-4, ratio=8, H=2.178),
        _case("free2d_256_mixed", "free", "256x256", "1", "mixed", 200, 5e-4, ratio=8, H=0.84),
        # 3D free space with FP32 transforms
        _case("free3d_64_mixed", "free", "64x64x64", "1", "mixed", 40, 1e-3, ratio=4, H=0.56),
    ]


def _pow2(rng, lo, hi):
    return 2 ** rng.randint(lo, hi)


def draw(rng):
    """One more case of the listed ranges: sizes by their logarithm, odd batches, every order and precision."""
    family = rng.choice(["1d", "1d", "uneven", "2d", "2d", "3d", "free1d", "free2d", "free3d"])
    precision = rng.choice(["mixed", "mixed", "fp64"])
    order = rng.choice([8, 8, 8, 6, 4])
    A0 = round(rng.uniform(0.5, 3.0), 3)
    dt = float("%.3g" % math.exp(rng.uniform(math.log(2e-4), math.log(2e-3))))

    def count(points, most):        # instances: log-uniform up to `most` points in all, any whole number
        return max(1, int(round(math.exp(rng.uniform(0.0, math.log(max(1.0, most / points)))))))

    if family == "1d":
        n = _pow2(rng, 6, 17)
        V = rng.choice(["wells", "factor", "shared_table"]) if n <= 4096 else "wells"
        return _case("", "periodic", str(n), str(count(n, 2 ** 20 if precision == "mixed" else 2 ** 18)), precision,
                     rng.randint(60, 300), dt, order, V, A0)
    if family == "uneven":
        sizes = sorted(rng.sample([2 ** p for p in range(8, 15)], rng.randint(2, 5)))
        return _case("", "uneven", ",".join(map(str, sizes)), ",".join(str(count(n, 2 ** 18)) for n in sizes), "mixed",
                     rng.randint(60, 200), dt, order, "wells", A0)
    if family == "2d":
        n0, n1 = _pow2(rng, 6, 10), _pow2(rng, 6, 10)
        return _case("", "periodic", "%dx%d" % (n0, n1), str(count(n0 * n1, 2 ** 23 if precision == "mixed" else 2 ** 19)),
                     precision, rng.randint(50, 300 if n0 * n1 <= 2 ** 18 else 100), dt, order,
                     rng.choice(["wells", "factor"]), A0)
    if family == "3d":
        n = [_pow2(rng, 4, 7) for _ in range(3)]
        p = n[0] * n[1] * n[2]
        return _case("", "periodic", "x".join(map(str, n)), str(count(p, 2 ** 22 if precision == "mixed" else 2 ** 19)),
                     precision, rng.randint(30, 100), dt, order, "wells", A0)
    d = {"free1d": 1, "free2d": 2, "free3d": 3}[family]
    n_r = rng.choice([0, 1, 2]) if d == 1 else 1
    # contour offset for eps = 1e-10 (FP64 sums) or 1e-4 (FP32 sums), ||V|| about 20, phi_max about 0.1
    gain = math.log(1e-10 / (21.0 * 2.0 ** -52)) if precision == "fp64" else math.log(1e-4 / (21.0 * 2.0 ** -23))
    H = round(gain / (2.0 * d * 1.1), 3)
    if d == 1:
        n, ratio = _pow2(rng, 5, 9), rng.choice([4, 8])
        return _case("", "free", str(n), str(count(n, 2 ** 13)), precision, rng.randint(60, 200), dt, order, "wells", A0,
                     ratio, H, n_r)
    if d == 2:
        n = [_pow2(rng, 5, 8), _pow2(rng, 5, 7)]
        rng.shuffle(n)
        return _case("", "free", "%dx%d" % tuple(n), str(count(n[0] * n[1], 2 ** 15)), precision, rng.randint(30, 100),
                     dt, order, "wells", A0, rng.choice([4, 8]), H, n_r)
    n = [_pow2(rng, 5, 6) if precision == "mixed" else 32 for _ in range(3)]
    return _case("", "free", "x".join(map(str, n)), "1", precision, rng.randint(16, 40), dt, order, "wells", A0, 4, H, n_r)


# ------------------------------------------------------------------ problem data
def _ints(text, sep):
    return [int(v) for v in text.split(sep)]


def _members(case):
    """[(shape, batch)] of a case: one entry, or one per member of an uneven batch."""
    if case["kind"] == "uneven":
        return [((n,), b) for n, b in zip(_ints(case["shape"], ","), _ints(case["batch"], ","))]
    return [(tuple(_ints(case["shape"], "x")), int(case["batch"]))]


def _grid(case, n):
    j = torch.arange(n, dtype=torch.float64, device="cuda")
    return -1.0 + 2.0 * j / n if case["kind"] == "free" else -math.pi + 2.0 * math.pi * j / n


def _outer(lines):
    """[B, n_a] per axis -> [B, n_0, .., n_{d-1}], the product."""
    out = lines[0]
    for g in lines[1:]:
        out = out.unsqueeze(-1) * g.reshape(g.shape[0], *([1] * (out.dim() - 1)), g.shape[1])
    return out


def _gaussians(case, shape, centres, sigmas):
    """exp(-|x - c|^2 / 2 s^2) of B instances on the grid, summed over the lattice images when periodic."""
    images = (0,) if case["kind"] == "free" else range(-3, 4)
    c = torch.from_numpy(centres).cuda()
    s = torch.from_numpy(sigmas).cuda()[:, None]
    lines = []
    for a, n in enumerate(shape):
        x = _grid(case, n)[None, :]
        lines.append(sum(torch.exp(-(x - c[:, a, None] - 2.0 * math.pi * m) ** 2 / (2.0 * s * s)) for m in images))
    return _outer(lines)


def _window(case, shape):
    """The smooth compact window of the free-space data; 1 when periodic."""
    if case["kind"] != "free":
        return 1.0
    r2 = 0.0
    for a, n in enumerate(shape):
        x = _grid(case, n).reshape([1] * a + [n] + [1] * (len(shape) - a - 1))
        r2 = r2 + x * x / 0.95 ** 2
    return torch.where(r2 < 1.0, torch.exp(1.0 - 1.0 / (1.0 - r2).clamp_min(1e-9)), torch.zeros_like(r2))


def _normalised(u, length):
    h = math.prod(length / n for n in u.shape[1:])
    norm = torch.sqrt((u.abs() ** 2).reshape(u.shape[0], -1).sum(1) * h)
    return u / norm.reshape(-1, *([1] * (u.dim() - 1)))


def _ground_state(depth, width, K=96):
    """Fourier coefficients of the static periodic Gaussian well's ground state."""
    k = np.arange(-K, K + 1)
    m = k[:, None] - k[None, :]
    ham = -depth * width / math.sqrt(2.0 * math.pi) * np.exp(-0.5 * width * width * m * m) + np.diag(k.astype(float) ** 2)
    return k, np.linalg.eigh(ham)[1][:, 0] / math.sqrt(2.0 * math.pi)


WELL_DEPTH, WELL_WIDTH = 300.0, 0.2


def _data(case, seed, member):
    """(u0 [B, ...], V(t) -> [B or 1, ...], V0 or None) of one member, on the GPU."""
    shape, B = _members(case)[member]
    rng = np.random.default_rng([int(seed), member, 41])
    d, free = len(shape), case["kind"] == "free"
    if case["V"] == "shared_table":         # ground state of the well, displaced and kicked; the well moves
        x = _grid(case, shape[0])
        k, coef = _ground_state(WELL_DEPTH, WELL_WIDTH)
        speed = float(rng.uniform(15.0, 45.0))
        shift = torch.from_numpy(rng.integers(-12, 13, size=B) * (2.0 * math.pi / 512)).cuda()[:, None]
        kick = torch.from_numpy(rng.integers(-6, 7, size=B).astype(np.float64)).cuda()[:, None]
        ph = torch.exp(1j * torch.outer(x, torch.from_numpy(k.astype(np.float64)).cuda()).to(torch.complex128))
        c = torch.from_numpy(coef.astype(np.complex128)).cuda()
        kk = torch.from_numpy(k.astype(np.float64)).cuda()[None, :]
        u0 = (c[None, :] * torch.exp(-1j * kk * shift)) @ ph.T * torch.exp(1j * kick * x[None, :])

        def table(t):
            return -WELL_DEPTH * sum(torch.exp(-(x - speed * t - 2.0 * math.pi * m) ** 2 / (2.0 * WELL_WIDTH ** 2))
                                     for m in range(-3, 4))[None, :]

        return u0, table, None
    lo_u, hi_u, box = (0.08, 0.15, 0.4) if free else (0.2, 0.4, 1.5)
    lo_v, hi_v = (0.08, 0.15) if free else (0.3, 0.6)
    win = _window(case, shape)
    u0 = 0.0
    for _ in range(3):
        phase = torch.from_numpy(np.exp(2j * math.pi * rng.random(B))).cuda().reshape(-1, *([1] * d))
        u0 = u0 + phase * _gaussians(case, shape, rng.uniform(-box, box, (B, d)), rng.uniform(lo_u, hi_u, B))
    u0 = _normalised(u0 * win, 2.0 if free else 2.0 * math.pi)
    if d == 1 and not free:                 # four cosine modes
        x = _grid(case, shape[0])
        V0 = sum(torch.from_numpy(rng.uniform(-10.0, 10.0, (B, 1))).cuda() * torch.cos(m * x)[None, :]
                 for m in range(1, 5))
    else:                                   # four attractive wells
        V0 = 0.0
        for _ in range(4):
            depth = torch.from_numpy(rng.uniform(5.0, 20.0, B)).cuda().reshape(-1, *([1] * d))
            V0 = V0 - depth * _gaussians(case, shape, rng.uniform(-box, box, (B, d)), rng.uniform(lo_v, hi_v, B))
        V0 = V0 * win
    return u0.contiguous(), (lambda t: _factor(case, t) * V0), V0.contiguous()


def _factor(case, t):
    return 1.0 + 0.5 * np.sin(2.0 * t) if case["V"] == "factor" else 1.0


def _pulse(case, d):
    return case["A0"], OMEGA, case["nsteps"] * case["dt"], [1.0] + [0.0] * (d - 1)


# ------------------------------------------------------------------ the measured pass
def prepare(case, seed):
    stream = torch.cuda.Stream() if case["kind"] == "uneven" else None
    probs, u0s, outs = [], [], []
    for i, (shape, B) in enumerate(_members(case)):
        u0, Vt, V0 = _data(case, seed, i)
        kw = {}
        if case["kind"] == "free":
            kw = dict(bc="free", nu=[case["ratio"] * n for n in shape], H=case["H"], n_r=case["n_r"])
        if case["kind"] == "uneven" and shape[0] >= 16384:
            kw = dict(layout_1d="passes")
        torch.cuda.synchronize()
        p = Problem(shape, case["dt"], case["nsteps"], order=case["order"], batch=B, precision=case["precision"],
                    potential="shared_table" if V0 is None else "separable", stream=stream, **kw)
        if V0 is None:
            p.set_potential_table(torch.cat([Vt(float(t)) for t in p.potential_times()]))
        else:
            fine = np.arange(8 * case["nsteps"] + 1) * case["dt"] / 8.0
            f = _factor(case, fine) if case["V"] == "factor" else None
            for b in range(B):
                p.set_potential(V0[b], f, instance=b)
        if case["A0"]:
            p.set_pulse(*_pulse(case, len(shape)))
        torch.cuda.synchronize()
        probs.append(p)
        u0s.append(u0)
        outs.append(torch.empty_like(u0))
    batch = None
    if case["kind"] == "uneven":
        batch = Batch(probs, stream=stream)
        batch.set_mode("streams")
    return {"probs": probs, "u0": u0s, "out": outs, "batch": batch, "stream": stream, "nsteps": case["nsteps"],
            "mixed": case["precision"] == "mixed"}


def run(state):
    def keep(u):
        return u.to(torch.complex64) if state["mixed"] else u

    if state["batch"] is None:
        p = state["probs"][0]
        p.set_initial_batch(state["u0"][0])
        p.step(state["nsteps"])
        return [keep(p.read_u(out=state["out"][0]))]
    caller, side = torch.cuda.current_stream(), state["stream"]
    side.wait_stream(caller)
    with torch.cuda.stream(side):
        for p, u0 in zip(state["probs"], state["u0"]):
            p.set_initial_batch(u0)
        state["batch"].step(state["nsteps"])
        got = [keep(p.read_u(out=out)) for p, out in zip(state["probs"], state["out"])]
    caller.wait_stream(side)
    return got


# ------------------------------------------------------------------ work
def _fft_flops(n):
    return 5.0 * n * math.log2(n)


def work(case):
    """u0, V and u once; and, where the state and the history of a step stay
    neither on an SM per instance nor in the L2, their traffic per step.
    Flops: the transforms (5 n log2 n), 10 per mode and history term, 20 per
    grid point of the implicit solve, of every sub-step (start-up: L chains of
    1, 2, 4, .. trapezoid steps, one history term each)."""
    bytes_, flops = 0.0, 0.0
    order, lags = case["order"], case["order"] - 1
    start = min(case["nsteps"], order - 1)
    sub = start * (2 ** (order // 2) - 1)
    main = case["nsteps"] - start
    state_b, ring_b = 16.0, 8.0 if case["precision"] == "mixed" else 16.0
    steps = []
    for shape, B in _members(case):
        X = math.prod(shape)
        if case["kind"] == "free":
            nu = [case["ratio"] * n for n in shape]
            N = [v - 10 + (10 if case["n_r"] == 0 else 20 * case["n_r"]) for v in nu]      # 2 NE + 2 p + NC
            modes = math.prod(N)
            transform = 0.0
            for a, n in enumerate(shape):   # lines along axis a: the axes after it on the grid, those before in modes
                lines = math.prod(N[:a]) * math.prod(shape[a + 1:])
                transform += lines * (2 * case["ratio"] * _fft_flops(n) + 2 * 6.0 * nu[a] + 8.0 * (N[a] - nu[a] + 26) * n)
        else:
            modes, transform = X, sum(X / n * _fft_flops(n) for n in shape)
        bytes_ += B * X * (16.0 + 16.0) + (1 if case["V"] == "shared_table" else B) * X * 8.0
        flops += B * (sub * (2 * transform + 16.0 * modes + 20.0 * X) + main * (2 * transform + 10.0 * lags * modes + 20.0 * X))
        per_step = modes * (2 * state_b + lags * ring_b) + X * 8.0
        steps.append((B, per_step, modes * (state_b + lags * ring_b), modes * (2 * state_b + 2 * ring_b) + X * 8.0))
    resident = sum(B * held for B, _, held, _ in steps if held > ON_CHIP_INSTANCE)
    if resident > ON_CHIP_ALL:
        bytes_ += sum(B * (main * p + sub * t) for B, p, held, t in steps if held > ON_CHIP_INSTANCE)
    return {"bytes": bytes_, "flops": flops}


# ------------------------------------------------------------------ the scheme in 64 bits
def _adams(order):
    """Implicit Adams weights: the integrals over [0, 1] of the Lagrange polynomials on 0, 1, .., order - 1."""
    mu = []
    for j in range(order):
        c, den = [Fraction(1)], Fraction(1)
        for m in range(order):
            if m != j:
                c = [a - m * b for a, b in zip([Fraction(0)] + c, c + [Fraction(0)])]
                den *= j - m
        mu.append(float(sum(v / (p + 1) for p, v in enumerate(c)) / den))
    return mu


def _phi(case, t):
    """Integral of A0 sin^2(pi s / T) sin(omega s) from 0 to t."""
    W = 2.0 * math.pi / (case["nsteps"] * case["dt"])

    def part(a):
        return 0.0 if a == 0.0 else 2.0 * math.sin(0.5 * a * t) ** 2 / a

    return 0.5 * case["A0"] * (part(OMEGA) - 0.5 * (part(OMEGA + W) + part(OMEGA - W)))


# Alpert's one-sided endpoint correction, p = 8, kappa = 7 (sum w x^m = B_{m+1}(7) / (m + 1), m < 16)
ALPERT_X = (0.09811761953716494, 0.5030225801568811, 1.1773437618437677, 2.0403429473991146, 3.0033918526940644,
            3.9995199797444103, 4.999921139726787, 5.9999984429959)
ALPERT_W = (0.25018432855612355, 0.551110758587803, 0.7837008206663483, 0.9269830825297909, 0.9875980230216356,
            1.0001904301204154, 1.0002243493491265, 1.0000082071687568)


def _contour(n, ratio, H, n_r, q=10, kappa=7):
    """Nodes and weights of the contour rule of one axis."""
    NE = ratio * n // 2 - 2 * kappa + 1
    h = math.pi * n / 2.0 / (NE + 2 * kappa - 1)
    tau = np.concatenate([np.array(ALPERT_X) * h, kappa * h + h * np.arange(NE)]) + H
    w3 = np.concatenate([h * np.array(ALPERT_W), np.full(NE, h)])
    z3 = tau - 1j * H
    pos = [0.0] + [H / 2.0 ** (n_r - k) for k in range(1, n_r + 1)]
    edges = [-e for e in reversed(pos[1:])] + pos if n_r else [-H, H]
    xg, wg = np.polynomial.legendre.leggauss(q)
    zc = np.concatenate([(1 - 1j) * (0.5 * (b - a) * xg + 0.5 * (a + b)) for a, b in zip(edges[:-1], edges[1:])])
    wc = np.concatenate([(1 - 1j) * 0.5 * (b - a) * wg for a, b in zip(edges[:-1], edges[1:])])
    return np.concatenate([-z3[::-1], zc, z3]), np.concatenate([w3[::-1], wc, w3])


def _basis(case, shape):
    """(forward, inverse, mode nodes per axis): the transform pair of a case, axes 1.. of [B, ...]."""
    axes = tuple(range(1, len(shape) + 1))
    if case["kind"] != "free":
        k = [torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda") for n in shape]
        return (lambda f: torch.fft.fftn(f, dim=axes, norm="forward"), lambda f: torch.fft.ifftn(f, dim=axes, norm="forward"), k)
    zs, Fs, Gs = [], [], []
    for n in shape:
        z, w = _contour(n, case["ratio"], case["H"], case["n_r"])
        x = -1.0 + 2.0 * np.arange(n) / n
        zs.append(torch.from_numpy(z).cuda())
        Fs.append(torch.from_numpy(2.0 / n * np.exp(-1j * np.outer(z, x))).cuda())
        Gs.append(torch.from_numpy(np.exp(1j * np.outer(x, z)) * (w / (2.0 * math.pi))[None, :]).cuda())

    def apply(mats, f, order):
        for a in order:
            f = torch.movedim(torch.tensordot(mats[a], f, dims=([1], [a + 1])), 0, a + 1)
        return f.contiguous()

    d = len(shape)
    return (lambda f: apply(Fs, f, range(d - 1, -1, -1)), lambda f: apply(Gs, f, range(d)), zs)


def _solve(case, seed, member):
    shape, _ = _members(case)[member]
    u, V, _ = _data(case, seed, member)
    fwd, inv, nodes = _basis(case, shape)
    d, order, dt, free = len(shape), case["order"], case["dt"], case["kind"] == "free"
    mu, L = _adams(order), order // 2

    def phase(t0, t1):          # e^{-i k^2 (t1 - t0) + i k dphi}, the product over the axes
        out = None
        for a, k in enumerate(nodes):
            dphi = _phi(case, t1) - _phi(case, t0) if a == 0 and case["A0"] else 0.0
            e = torch.exp(1j * (-k * k * (t1 - t0) + k * dphi))
            out = e if out is None else out.unsqueeze(-1) * e
        return out[None]

    def implicit(W, h, m0, t):  # u and (Vu)^ of the implicit step, the new mode state
        g = inv(W) / (1.0 + 1j * m0 * h * V(t))
        R = fwd(V(t) * g)
        return g, R, W - 1j * m0 * h * R

    uh = fwd(u)
    hist = [fwd(V(0.0) * u)]                # (Vu)^ of the last steps, newest first
    steps = [phase(0.0, dt)]                # one-step phases, newest first
    for n in range(1, case["nsteps"] + 1):
        t0, t = (n - 1) * dt, n * dt
        P = phase(t0, t)
        steps = [P] + steps[: order - 2]
        if n <= order - 1:
            tab = []
            for c in range(L):
                m, a, r, g = 2 ** c, uh, hist[0], None
                for s in range(m):
                    h = dt / m
                    g, r, a = implicit(phase(t0 + s * h, t0 + (s + 1) * h) * (a - 0.5j * h * r), h, 0.5, t0 + (s + 1) * h)
                tab.append((a, g))
            for lev in range(1, L):
                f = 4.0 ** lev
                tab = [tuple((f * y - x) / (f - 1.0) for x, y in zip(tab[c], tab[c + 1])) for c in range(len(tab) - 1)]
            uh, g = tab[0]
            if not free:
                g = inv(uh)
            R = fwd(V(t) * g)
        else:
            S = mu[order - 1] * hist[order - 2]
            for j in range(order - 2, 0, -1):
                S = mu[j] * hist[j - 1] + steps[j] * S
            g, R, uh = implicit(P * (uh - 1j * dt * S), dt, mu[0], t)
        hist = [R] + hist[: order - 2]
    return g


def exact(case, seed):
    return [_solve(case, seed, i) for i in range(len(_members(case)))]
