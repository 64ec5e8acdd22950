"""The calls of this library whose time counts, each through the package's public entry points.

A case is a dict of plain values; its "kind" says what the program around it does:

  steps     a channel with a fixed chart advanced by `steps` LBM steps, then the wall force and the fields
            (periodic flow, body force): the plain use of CurvedLattice
  cycle     one cycle of a channel whose wall moves (inflow, outflow, moving top wall): chart change, face
            velocities, 10 steps, mass, wall force, fields
  coupled   the fluid side of a coupled loop on a small lattice: per step a chart change, the wall's velocity,
            one step, the force and the mass read back; the fields at the end
  interp    Taylor-Green flow under a moving periodic chart: per step one LBM step and one interpolating chart change
  batch     uneven channels advanced together (CurvedBatch), then every channel's fields
  adjoint   gradient of the wall force with respect to the geometry (forward and backward)
  gradient  lattice derivatives of the six metric components
  d2q9      the two-dimensional lattice

Sizes are those of the benchmark (256^3, 128 x 256 x 128, 4096 x 1024, the 64-channel batch, the 64 x 128 x 64
adjoint channel), of the tests (16 x 32 x 16, 64 x 128 x 64, the 91 x 77 x 93 channel of the batch) and of the
studies (Taylor-Green, piston).  Inputs are made on the GPU from the seed: deformations of the top wall by a few
Fourier modes of bounded slope, a parabolic flow with a smooth perturbation.

Fields come back at the precision the lattice stores its populations in (FP64 only from FP64 storage).

The second half of the file is the method once more in plain torch, FP64, written from the equations (`exact`).
"""
import math
import random

import numpy as np
import torch

DEVICE = "cuda" if torch.cuda.is_available() else "cpu"
F64 = torch.float64
FIELD = {"fp32": torch.float32, "fp64": torch.float64, "fp16": torch.float16, "bf16": torch.bfloat16}
PERIODIC, WALL, INFLOW, OUTFLOW = 0, 1, 2, 3


def listed():
    return [
        # the smallest lattice in use (validation runs, the smoke run): launches and latency
        dict(name="channel 16x32x16 fp32", kind="steps", n0=16, n1=32, n2=16, storage="fp32", steps=20),
        # a coupled run's fluid solver: small lattice, the host reads the force every step
        dict(name="coupled 32x32x64 fp32", kind="coupled", n0=32, n1=32, n2=64, storage="fp32", steps=5),
        # a channel of odd extents (any size a user's geometry gives)
        dict(name="channel 91x77x93 fp32", kind="steps", n0=91, n1=77, n2=93, storage="fp32", steps=10),
        # FP64 storage: validation and convergence studies
        dict(name="channel 64x128x64 fp64", kind="steps", n0=64, n1=128, n2=64, storage="fp64", steps=10),
        # the Taylor-Green study's loop (all periodic, chart moving every step)
        dict(name="moving box 256x256x16 fp32", kind="interp", n0=256, n1=256, n2=16, storage="fp32", steps=4),
        # data generation: 64 uneven channels
        dict(name="batch of 64 fp32", kind="batch", nb=64, lo=32, hi=96, steps=10),
        # shape optimisation: gradient over 40 steps, checkpoints every 20
        dict(name="adjoint 64x128x64 fp32", kind="adjoint", n0=64, n1=128, n2=64, steps=40, every=20),
        # geometry from the metric alone
        dict(name="gradient 128x256x128 order 4", kind="gradient", n0=128, n1=256, n2=128, order=4),
        # the 2-D variant at its benchmark size
        dict(name="d2q9 4096x1024 fp32", kind="d2q9", n0=4096, n1=1024, storage="fp32", steps=20),
        # the dynamic channel, chart in FP64
        dict(name="cycle 128x256x128 fp32", kind="cycle", n0=128, n1=256, n2=128, storage="fp32", mixed=False),
        # the same with 16-bit populations (larger problems in the same memory), chart derivatives in FP32
        dict(name="cycle 128x256x128 fp16", kind="cycle", n0=128, n1=256, n2=128, storage="fp16", mixed=True),
        # the largest: the benchmark's default workload
        dict(name="cycle 256x256x256 fp32", kind="cycle", n0=256, n1=256, n2=256, storage="fp32", mixed=True),
    ]


def _size(rng, lo, hi):
    """An extent spread over the logarithm of lo..hi; a third of them odd, a third multiples of 16."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    how = rng.randrange(3)
    if how == 0:
        v = int(v) // 2 * 2 + 1
    elif how == 1:
        v = round(v / 16) * 16
    return max(lo, min(hi, int(v)))


def draw(rng: random.Random):
    kind = rng.choice(["steps", "steps", "steps", "cycle", "cycle", "coupled", "interp", "batch", "adjoint", "gradient",
                       "d2q9"])
    if kind == "steps":
        storage = rng.choice(["fp32", "fp32", "fp16", "bf16", "fp64"])
        hi = 128 if storage == "fp64" else 256
        return dict(kind=kind, n0=_size(rng, 16, 320 if storage != "fp64" else hi), n1=_size(rng, 16, hi),
                    n2=_size(rng, 12, hi), storage=storage, steps=rng.randint(4, 12))
    if kind == "cycle":
        storage = rng.choice(["fp32", "fp32", "fp16", "bf16"])
        return dict(kind=kind, n0=_size(rng, 32, 256), n1=_size(rng, 48, 256), n2=_size(rng, 32, 192), storage=storage,
                    mixed=rng.random() < 0.5)
    if kind == "coupled":
        return dict(kind=kind, n0=_size(rng, 16, 64), n1=_size(rng, 16, 64), n2=_size(rng, 16, 96),
                    storage=rng.choice(["fp32", "fp64"]), steps=rng.randint(3, 8))
    if kind == "interp":
        return dict(kind=kind, n0=_size(rng, 32, 256), n1=_size(rng, 32, 256), n2=_size(rng, 4, 32),
                    storage=rng.choice(["fp32", "fp64"]), steps=rng.randint(2, 5))
    if kind == "batch":
        lo = rng.randint(16, 40)
        return dict(kind=kind, nb=rng.randint(4, 48), lo=lo, hi=lo + rng.randint(8, 48), steps=rng.randint(5, 12))
    if kind == "adjoint":
        return dict(kind=kind, n0=_size(rng, 16, 64), n1=_size(rng, 32, 128), n2=_size(rng, 16, 64),
                    steps=rng.randint(10, 45), every=rng.choice([10, 20]))
    if kind == "gradient":
        return dict(kind=kind, n0=_size(rng, 24, 192), n1=_size(rng, 24, 256), n2=_size(rng, 16, 128),
                    order=rng.choice([2, 4]))
    return dict(kind=kind, n0=_size(rng, 64, 4096), n1=_size(rng, 32, 1024), storage=rng.choice(["fp32", "fp32", "fp64"]),
                steps=rng.randint(10, 25))


# ---------------------------------------------------------------------------
# what one pass cannot do without
# ---------------------------------------------------------------------------
_SB = {"fp32": 4, "fp64": 8, "fp16": 2, "bf16": 2}
# arithmetic of one node: a step in three dimensions, in two, a chart change
_STEP_FLOP, _STEP2_FLOP, _CHART_FLOP = 900.0, 300.0, 700.0


def work(case):
    k = case["kind"]
    if k == "d2q9":
        N, r, steps = case["n0"] * case["n1"], _SB[case["storage"]], case["steps"]
        per = (2 * 9 + 2 * 6 + 10) * r
        return dict(bytes=N * (steps * per + (9 + 6 + 1) * r + 3 * 8), flops=N * steps * _STEP2_FLOP)
    if k == "batch":
        N = sum(a * b * c for a, b, c in _batch_sizes(case, 0))
        return dict(bytes=N * (case["steps"] * 332.0 + 120 + 32), flops=N * case["steps"] * _STEP_FLOP)
    N = case["n0"] * case["n1"] * case["n2"]
    if k == "gradient":
        return dict(bytes=N * 8.0 * (6 + 18), flops=N * 6.0 * (24 + (22 if case["order"] == 4 else 0)))
    s = _SB[case.get("storage", "fp32")]
    r = 8 if case.get("storage") == "fp64" else 4
    state = 19 * s + 10 * r                      # populations and forcing history of a node
    step = 2 * state + 25 * r                    # read, written, and the geometry read
    read = state + 10 * r + 4 * 8                # the fields: state, sqrt(g), Jacobian in; rho, u out
    # chart change: state in and out, old sqrt(g), new geometry out, the Jacobian old in and new out, the chart in
    chart = 2 * state + r + 25 * r + 2 * 9 * r + (6 * 8 + 27 * 4 if case.get("mixed") else 33 * 8)
    if k == "steps":
        return dict(bytes=N * (case["steps"] * step + read), flops=N * case["steps"] * _STEP_FLOP)
    if k == "cycle":
        return dict(bytes=N * (10 * step + chart + state + r + read), flops=N * (10 * _STEP_FLOP + _CHART_FLOP))
    if k == "coupled":
        return dict(bytes=N * (case["steps"] * (step + chart + state + r) + read),
                    flops=N * case["steps"] * (_STEP_FLOP + _CHART_FLOP))
    if k == "interp":
        return dict(bytes=N * (case["steps"] * (step + chart + 3 * 8) + read),
                    flops=N * case["steps"] * (_STEP_FLOP + _CHART_FLOP + 8 * 2 * 29))
    # adjoint, per step: the forward step twice (once to recompute), then the backward one: forward state and
    # geometry in, adjoint state in and out, the geometry's adjoint in and out
    back = state + 25 * r + 2 * state + 2 * 25 * r
    return dict(bytes=N * (case["steps"] * (2 * step + back) + 33 * 8 * 2), flops=N * case["steps"] * 4 * _STEP_FLOP)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _modes(rng, count, kmax, lmax):
    return [(rng.randint(1, kmax), rng.randint(0, lmax), rng.gauss(0.0, 1.0), rng.uniform(0.0, 2.0 * math.pi))
            for _ in range(count)]


def _deformation(n, modes, amp, slope, taper):
    """Displacement d(x0, x1) of the top wall [n1, n0] and its derivatives (d, d0, d1, d00, d01, d11): a sum of
    Fourier modes scaled to the smaller of amp (fraction of the height) and the given largest slope; with `taper`
    it vanishes at both ends of axis 1."""
    x = torch.arange(n[0], dtype=F64, device=DEVICE)[None, :]
    y = torch.arange(n[1], dtype=F64, device=DEVICE)[:, None]
    L = n[1] - 1 if taper else n[1]
    z = torch.zeros(n[1], n[0], dtype=F64, device=DEVICE)
    D, D0, D1, D00, D01, D11 = (z.clone() for _ in range(6))
    for k, l, c, phi in modes:
        ky, kx = 2.0 * math.pi * k / L, 2.0 * math.pi * l / n[0]
        th = ky * y + kx * x + phi
        co, si = c * torch.cos(th), c * torch.sin(th)
        D += co
        D0 -= kx * si
        D1 -= ky * si
        D00 -= kx * kx * co
        D01 -= kx * ky * co
        D11 -= ky * ky * co
    if taper:
        w = math.pi / L
        S, S1, S2 = torch.sin(w * y) ** 2, w * torch.sin(2 * w * y), 2 * w * w * torch.cos(2 * w * y)
        D, D0, D1, D00, D01, D11 = (D * S, D0 * S, D1 * S + D * S1, D00 * S, D01 * S + D0 * S1,
                                    D11 * S + 2 * D1 * S1 + D * S2)
    H = n[2] - 1
    a = min(amp * H / float(D.abs().max()), slope / float((D0 ** 2 + D1 ** 2).sqrt().max()))
    return [a * v for v in (D, D0, D1, D00, D01, D11)]


def _channel_chart(n, dfm, a=1.0):
    """(g6 [6, N], dg18 [18, N], J9 [9, N]) of the chart h^2 = x2 (1 + a d / H), h^0 = x0, h^1 = x1."""
    H = n[2] - 1
    N = n[0] * n[1] * n[2]
    z = torch.arange(n[2], dtype=F64, device=DEVICE)[:, None, None]
    d, d0, d1, d00, d01, d11 = ((a / H) * v[None] for v in dfm)
    J = [z * d0, z * d1, (1.0 + d).expand(n[2], -1, -1)]             # the row d h^2 / d x^i
    Hs = {(0, 0): z * d00, (0, 1): z * d01, (1, 1): z * d11, (0, 2): d0, (1, 2): d1}

    def hess(i, k):
        return Hs.get((min(i, k), max(i, k)))

    g6 = torch.empty(6, n[2], n[1], n[0], dtype=F64, device=DEVICE)
    dg18 = torch.zeros(18, n[2], n[1], n[0], dtype=F64, device=DEVICE)
    J9 = torch.zeros(9, n[2], n[1], n[0], dtype=F64, device=DEVICE)
    J9[0], J9[4] = 1.0, 1.0
    for i in range(3):
        J9[6 + i] = J[i]
    for m, (i, j) in enumerate(_sym(3)):
        g6[m] = J[i] * J[j] + (1.0 if i == j and i < 2 else 0.0)
        for k in range(3):
            if hess(k, i) is not None:
                dg18[6 * k + m] += hess(k, i) * J[j]
            if hess(k, j) is not None:
                dg18[6 * k + m] += hess(k, j) * J[i]
    return g6.view(6, N), dg18.view(18, N), J9.view(9, N)


def _sym(d):
    return [(i, j) for i in range(d) for j in range(i, d)]


def _flow(n, umax, rng):
    """A parabolic flow along axis 1 with a smooth perturbation: rho [N], u [3, N]."""
    z = torch.arange(n[2], dtype=F64, device=DEVICE)[:, None, None] / (n[2] - 1)
    ph = [rng.uniform(0.0, 2.0 * math.pi) for _ in range(3)]
    b = sum(torch.sin(2.0 * math.pi * torch.arange(n[a], dtype=F64, device=DEVICE) / n[a] + ph[a]).view(
        [-1 if 2 - a == k else 1 for k in range(3)]) for a in range(3))
    u = torch.zeros(3, n[2], n[1], n[0], dtype=F64, device=DEVICE)
    u[1] = 4.0 * umax * z * (1.0 - z) * (1.0 + 0.01 * b)
    return (1.0 + 1e-3 * b).reshape(-1).contiguous(), u.view(3, -1)


def _channel(case, seed):
    """A periodic channel with walls across axis 2 and a deformed top wall, driven along axis 1."""
    rng = random.Random(seed)
    n = (case["n0"], case["n1"], case["n2"])
    tau = rng.uniform(0.65, 0.9)
    umax, H = 0.05, n[2] - 1
    nu = (tau - 0.5) / 3.0
    dfm = _deformation(n, _modes(rng, 4, 2, 1), 0.06, 0.2, False)
    rho, u = _flow(n, umax, rng)
    return dict(n=n, bc=(PERIODIC, PERIODIC, WALL), tau=tau, fext=(0.0, 8.0 * nu * umax / H ** 2, 0.0), dfm=dfm,
                chart=_channel_chart(n, dfm), rho=rho, u=u)


def _dynamic(case, seed):
    """A channel with inflow, outflow and a moving top wall: charts at three times, the velocity of the inflow
    face and of the top wall at each."""
    rng = random.Random(seed)
    n = (case["n0"], case["n1"], case["n2"])
    tau, H = 0.6, n[2] - 1
    umax = min(0.05, 100.0 * (tau - 0.5) / 3.0 / H)
    dfm = _deformation(n, _modes(rng, 8, 3, 2), 0.08, 0.2, True)
    z = torch.arange(n[2], dtype=F64, device=DEVICE) / H
    inflow = torch.zeros(3, n[2], n[0], dtype=F64, device=DEVICE)
    inflow[1] = (4.0 * umax * z * (1.0 - z))[:, None]
    times = []
    for t in (500.0, 510.0, 520.0):
        a, rate = math.sin(math.pi * t / 2000.0) ** 2, math.pi / 2000.0 * math.sin(2.0 * math.pi * t / 2000.0)
        wall = torch.zeros(3, n[1], n[0], dtype=F64, device=DEVICE)
        wall[2] = rate * dfm[0] / (1.0 + a * dfm[0] / H)              # contravariant: J^-1 v
        times.append((_channel_chart(n, dfm, a), wall.view(3, -1)))
    rho, u = _flow(n, umax, rng)
    return dict(n=n, lo=(PERIODIC, INFLOW, WALL), hi=(PERIODIC, OUTFLOW, WALL), tau=tau, inflow=inflow.view(3, -1),
                times=times, rho=rho, u=u)


def _piston(case, seed):
    """A box whose deformed top wall is pressed down a little every step, then back."""
    rng = random.Random(seed)
    n = (case["n0"], case["n1"], case["n2"])
    H = n[2] - 1
    dfm = _deformation(n, _modes(rng, 3, 2, 1), 0.05, 0.15, False)
    times = []
    for t in range(4):
        a, rate = 0.5 + 0.002 * t, 0.002 if t < 3 else 0.0
        wall = torch.zeros(3, n[1], n[0], dtype=F64, device=DEVICE)
        wall[2] = rate * dfm[0] / (1.0 + a * dfm[0] / H)
        times.append((_channel_chart(n, dfm, a), wall.view(3, -1)))
    rho, u = _flow(n, 0.03, rng)
    return dict(n=n, bc=(PERIODIC, PERIODIC, WALL), tau=0.8, times=times, rho=rho, u=u)


def _box_chart(n, t, eta, ph, eps=0.1):
    """The periodic moving chart x_c^a = x^a - eps (L/2pi) cos(2 pi x^a / L - eta t + ph_a) of axes 0 and 1."""
    N = n[0] * n[1] * n[2]
    J9 = torch.zeros(9, n[2], n[1], n[0], dtype=F64, device=DEVICE)
    g6, dg18 = J9.new_zeros((6, *J9.shape[1:])), J9.new_zeros((18, *J9.shape[1:]))
    J9[8] = 1.0
    g6[5] = 1.0
    for a in (0, 1):
        k = 2.0 * math.pi / n[a]
        th = (k * torch.arange(n[a], dtype=F64, device=DEVICE) - eta * t + ph[a]).view([-1, 1] if a else [-1])
        j, h, m = 1.0 + eps * torch.sin(th), eps * k * torch.cos(th), 3 * a
        J9[4 * a] = j
        g6[m] = j * j
        dg18[6 * a + m] = 2.0 * j * h
    return g6.view(6, N), dg18.view(18, N), J9.view(9, N)


def _box_psi(n, t0, t1, eta, ph, eps=0.1):
    """Old lattice coordinates at time t0 of the nodes' points at time t1 [3, N] (Newton's method per axis)."""
    out = []
    for a in range(3):
        r = torch.arange(n[a], dtype=F64, device=DEVICE)
        x = r.clone()
        if a < 2:
            k = 2.0 * math.pi / n[a]
            xc = r - eps / k * torch.cos(k * r - eta * t1 + ph[a])
            for _ in range(12):
                x = x - (x - eps / k * torch.cos(k * x - eta * t0 + ph[a]) - xc) / (1.0 + eps * torch.sin(k * x - eta * t0 + ph[a]))
        out.append(x.view([-1 if 2 - a == q else 1 for q in range(3)]).expand(n[2], n[1], n[0]))
    return torch.stack(out).reshape(3, -1).contiguous()


def _box(case, seed):
    rng = random.Random(seed)
    n = (case["n0"], case["n1"], case["n2"])
    ph = [rng.uniform(0.0, 2.0 * math.pi) for _ in range(2)]
    eta, v0 = 0.05 * 32.0 / max(n[0], n[1]), 0.04
    charts = [_box_chart(n, float(t), eta, ph) for t in range(4)]
    psis = [_box_psi(n, float((t - 1) % 4), float(t), eta, ph) for t in range(4)]
    x = [2.0 * math.pi / n[a] * torch.arange(n[a], dtype=F64, device=DEVICE).view([-1 if 2 - a == q else 1 for q in range(3)])
         for a in range(3)]
    th = rng.uniform(0.0, 2.0 * math.pi)
    v = torch.zeros(3, n[2], n[1], n[0], dtype=F64, device=DEVICE)
    v[0] = v0 * torch.sin(x[0] + th) * torch.cos(x[1])
    v[1] = -v0 * torch.cos(x[0] + th) * torch.sin(x[1])
    rho = (1.0 - 0.75 * v0 * v0 * (torch.cos(2 * (x[0] + th)) + torch.cos(2 * x[1])) + 0.0 * x[2]).reshape(-1).contiguous()
    J9 = charts[0][2].view(9, n[2], n[1], n[0])
    u = torch.stack([v[0] / J9[0], v[1] / J9[4], v[2]]).view(3, -1).contiguous()
    return dict(n=n, tau=0.74, charts=charts, psis=psis, rho=rho, u=u)


def _batch_sizes(case, seed):
    """Sides of the channels: drawn once for a case, the same for every seed (a program's set of geometries)."""
    rng = random.Random(1000 * case["lo"] + case["hi"])
    return [tuple(rng.randint(case["lo"], case["hi"]) for _ in range(3)) for _ in range(case["nb"])]


def _batch(case, seed):
    return [_channel(dict(n0=s[0], n1=s[1], n2=s[2]), 4000 * (seed + 1) + i)
            for i, s in enumerate(_batch_sizes(case, seed))]


def _plane(case, seed):
    """A two-dimensional channel: periodic along axis 0, walls across axis 1, the top wall displaced."""
    rng = random.Random(seed)
    n = (case["n0"], case["n1"])
    H, N = n[1] - 1, n[0] * n[1]
    x = torch.arange(n[0], dtype=F64, device=DEVICE)
    k, ph = 2.0 * math.pi / n[0], rng.uniform(0.0, 2.0 * math.pi)
    amp = min(0.06 * H, 0.2 / k)
    d, dd, ddd = (amp * torch.cos(k * x + ph) / H, -amp * k * torch.sin(k * x + ph) / H, -amp * k * k * torch.cos(k * x + ph) / H)
    y = torch.arange(n[1], dtype=F64, device=DEVICE)[:, None]
    one = torch.ones(n[1], n[0], dtype=F64, device=DEVICE)
    Ja, Jb = y * dd, one * (1.0 + d)                                  # d h^1 / d x^0, d x^1
    J4 = torch.stack([one, 0 * one, Ja, Jb]).view(4, N)
    g3 = torch.stack([1.0 + Ja * Ja, Ja * Jb, Jb * Jb]).view(3, N)
    hxx, hxy = y * ddd, one * dd
    dg6 = torch.stack([2 * hxx * Ja, hxx * Jb + Ja * hxy, 2 * hxy * Jb, 2 * hxy * Ja, hxy * Jb, 0 * one]).view(6, N)
    tau, umax = 0.8, 0.05
    b = torch.sin(k * x + rng.uniform(0.0, 6.0))
    u = torch.zeros(2, n[1], n[0], dtype=F64, device=DEVICE)
    u[0] = 4.0 * umax * (y / H) * (1.0 - y / H) * (1.0 + 0.01 * b)
    rho = (1.0 + 1e-3 * b + 0.0 * y).reshape(-1).contiguous()
    return dict(n=n, tau=tau, fext=(8.0 * (tau - 0.5) / 3.0 * umax / H ** 2, 0.0), chart=(g3, dg6, J4), rho=rho,
                u=u.view(2, -1))


# ---------------------------------------------------------------------------
# the program around the calls
# ---------------------------------------------------------------------------
def prepare(case, seed):
    from paper_1803_07822_gb300.lattice import CurvedBatch, CurvedLattice, CurvedLattice2D
    k = case["kind"]
    if k == "batch":
        ws = _batch(case, seed)
        b = CurvedBatch([dict(n=w["n"], bc_lo=w["bc"], tau=w["tau"], fext=w["fext"]) for w in ws])
        for i, w in enumerate(ws):
            b[i].set_metric(*w["chart"][:2])
            b[i].set_jacobian(w["chart"][2])
            b[i].init_equilibrium(w["rho"], w["u"])
        b.tune(3)
        return dict(case=case, batch=b)
    if k == "d2q9":
        w = _plane(case, seed)
        lat = CurvedLattice2D(w["n"], (PERIODIC, WALL), tau=w["tau"], fext=w["fext"], storage=case["storage"])
        lat.set_metric(*w["chart"][:2])
        lat.set_jacobian(w["chart"][2])
        lat.init_equilibrium(w["rho"], w["u"])
        return dict(case=case, lat=lat)
    if k == "steps":
        w = _channel(case, seed)
        lat = CurvedLattice(w["n"], w["bc"], tau=w["tau"], fext=w["fext"], storage=case["storage"])
        lat.set_metric(*w["chart"][:2])
        lat.set_jacobian(w["chart"][2])
        lat.init_equilibrium(w["rho"], w["u"])
        return dict(case=case, lat=lat)
    if k == "gradient":
        w = _channel(case, seed)
        lat = CurvedLattice(w["n"], w["bc"], tau=w["tau"])
        return dict(case=case, lat=lat, g6=w["chart"][0])
    if k == "adjoint":
        w = _channel(case, seed)
        lat = CurvedLattice(w["n"], w["bc"], tau=w["tau"], fext=w["fext"], storage="fp32")
        return dict(case=case, lat=lat, leaves=[t.requires_grad_(True) for t in w["chart"]])
    if k == "interp":
        w = _box(case, seed)
        lat = CurvedLattice(w["n"], tau=w["tau"], storage=case["storage"])
        lat.set_metric(*w["charts"][0][:2])
        lat.set_jacobian(w["charts"][0][2])
        lat.init_equilibrium(w["rho"], w["u"])
        return dict(case=case, lat=lat, charts=w["charts"], psis=w["psis"], at=0)
    if k == "coupled":
        w = _piston(case, seed)
        lat = CurvedLattice(w["n"], w["bc"], tau=w["tau"], storage=case["storage"])
    else:
        w = _dynamic(case, seed)
        lat = CurvedLattice(w["n"], w["lo"], w["hi"], tau=w["tau"], storage=case["storage"])
    times = w["times"]
    lat.set_metric(*times[0][0][:2])
    lat.set_jacobian(times[0][0][2])
    lat.set_boundary_velocity(2, 1, times[0][1])
    if k == "cycle":
        lat.set_boundary_velocity(1, 0, w["inflow"])
        if case["mixed"]:
            times = [((c[0], c[1].float(), c[2].float()), v) for c, v in times]
    lat.init_equilibrium(w["rho"], w["u"])
    return dict(case=case, lat=lat, times=times, inflow=w.get("inflow"), at=0)


def _fields(lat, storage):
    rho, v = lat.moments(cartesian=True, host=False)
    return rho.to(FIELD[storage]), v.to(FIELD[storage])


def _vector(F, storage):
    return np.asarray(F, dtype=np.float64 if storage == "fp64" else np.float32)


def _order(i):
    """Charts 0, 1, 2, 1, 0, ... of the wall's motion to and fro."""
    return (0, 1, 2, 1)[i % 4]


def run(state):
    case = state["case"]
    k = case["kind"]
    storage = case.get("storage", "fp32")
    if k == "batch":
        b = state["batch"]
        b.step(case["steps"])
        from paper_1803_07822_gb300._abi import call
        rho = torch.empty(b.nodes, dtype=F64, device=b.device)
        u = torch.empty(3 * b.nodes, dtype=F64, device=b.device)
        o = 0
        for c in b.channels:  # every channel's fields into one array (the binding's moments() allocates per channel)
            call("cslbm_get_moments", c.ctx, rho.data_ptr() + 8 * o, u.data_ptr() + 24 * o, 1, 1)
            o += c.N
        return dict(rho=rho.float(), u=u.float())
    lat = state["lat"]
    if k == "steps":
        lat.step(case["steps"])
        F = lat.wall_force(2, 1)
        rho, v = _fields(lat, storage)
        return dict(rho=rho, v=v, force=_vector(F, storage))
    if k == "cycle":
        state["at"] += 1
        (g6, dg18, J9), wall = state["times"][_order(state["at"])]
        if case["mixed"]:
            lat.update_metric_mixed(g6, dg18, J9)
        else:
            lat.update_metric(g6, dg18, J9)
        lat.set_boundary_velocity(1, 0, state["inflow"])
        lat.set_boundary_velocity(2, 1, wall)
        lat.step(10)
        mass = lat.total_mass()
        F = lat.wall_force(2, 1)
        rho, v = _fields(lat, storage)
        return dict(rho=rho, v=v, force=_vector(F, storage), mass=mass)
    if k == "coupled":
        forces, masses = [], []
        for _ in range(case["steps"]):
            state["at"] += 1
            (g6, dg18, J9), wall = state["times"][(0, 1, 2, 3, 2, 1)[state["at"] % 6]]
            lat.update_metric(g6, dg18, J9)
            lat.set_boundary_velocity(2, 1, wall)
            lat.step(1)
            forces.append(lat.wall_force(2, 1))
            masses.append(lat.total_mass())
        rho, v = _fields(lat, storage)
        return dict(rho=rho, v=v, forces=_vector(forces, storage), masses=_vector(masses, storage))
    if k == "interp":
        for _ in range(case["steps"]):
            state["at"] += 1
            i = state["at"] % 4
            lat.step(1)
            lat.update_metric_interp(*state["charts"][i], state["psis"][i])
        rho, v = _fields(lat, storage)
        return dict(rho=rho, v=v)
    if k == "gradient":
        return lat.lattice_gradient(state["g6"], case["order"])
    if k == "adjoint":
        from paper_1803_07822_gb300.adjoint import wall_force_objective
        J = wall_force_objective(lat, *state["leaves"], case["steps"], case["every"], axis=2, side=1, e3=(0.0, 1.0, 0.0))
        g = torch.autograd.grad(J, state["leaves"])
        return dict(value=J.detach().float(), g6=g[0].float(), dg18=g[1].float(), J9=g[2].float())
    # d2q9: the fields stay on the device (the binding's moments() copies them to the host)
    from paper_1803_07822_gb300._abi import call
    lat.step(case["steps"])
    F = lat.wall_force(1, 1)
    rho = torch.empty(lat.N, dtype=F64, device=lat.device)
    v = torch.empty((2, lat.N), dtype=F64, device=lat.device)
    call("cslbm2d_get_moments", lat.ctx, rho.data_ptr(), v.data_ptr(), 1, 1)
    return dict(rho=rho.to(FIELD[storage]), v=v.to(FIELD[storage]), force=_vector(F, storage))


# ---------------------------------------------------------------------------
# the method in plain torch, 64 bits (D2Q9 or D3Q19; populations [Q, N] as streamed, fields as lists of [N])
# ---------------------------------------------------------------------------
class Plain:
    def __init__(self, n, lo, hi, tau, fext=None):
        self.n, self.lo, self.hi, self.tau, self.d = n, lo, hi, tau, len(n)
        d, self.N = self.d, math.prod(n)
        self.fext = fext or (0.0,) * d
        unit = [tuple(s if b == a else 0 for b in range(d)) for a in range(d) for s in (1, -1)]
        diag = [tuple(s if q == a else (t if q == b else 0) for q in range(d))
                for a in range(d) for b in range(a + 1, d) for s in (1, -1) for t in (1, -1)]
        self.c = [(0,) * d] + unit + diag
        self.w = ([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4) if d == 2 else ([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
        self.Q = len(self.c)
        self.face_u = {}
        self.faces = self._faces()

    def grid(self, t):
        return t.reshape(*t.shape[:-1], *self.n[::-1])

    def dim(self, a):
        return -(a + 1)

    def coords(self):
        v = torch.arange(self.N, device=DEVICE)
        r = []
        for a in range(self.d):
            r.append(v % self.n[a])
            v = v // self.n[a]
        return r

    def index(self, r):
        v = torch.zeros_like(r[0])
        for a in reversed(range(self.d)):
            v = v * self.n[a] + r[a]
        return v

    def _faces(self):
        """[(rule, axis, side, nodes, inner nodes, index on the face)] of every node on a non-periodic face: the
        rule of highest rank (wall, inflow, outflow; then the lower axis, the low side)."""
        r = self.coords()
        rank = torch.zeros(self.N, dtype=torch.long, device=DEVICE)
        own = torch.full((self.N,), -1, dtype=torch.long, device=DEVICE)
        inner = list(r)
        for a in range(self.d):
            for s in (0, 1):
                rule = self.hi[a] if s else self.lo[a]
                if rule == PERIODIC:
                    continue
                on = r[a] == (self.n[a] - 1 if s else 0)
                inner[a] = torch.where(on, r[a] + (-1 if s else 1), inner[a])
                k = {WALL: 3, INFLOW: 2, OUTFLOW: 1}[rule]
                take = on & (rank < k)
                rank = torch.where(take, torch.full_like(rank, k), rank)
                own = torch.where(take, torch.full_like(own, 2 * a + s), own)
        vi = self.index(inner)
        out = []
        for k in range(2 * self.d):
            a, s = k // 2, k % 2
            nodes = (own == k).nonzero()[:, 0]
            if nodes.numel():
                fi, m = torch.zeros_like(nodes), 1
                for b in range(self.d):
                    if b != a:
                        fi = fi + m * r[b][nodes]
                        m *= self.n[b]
                out.append((self.hi[a] if s else self.lo[a], a, s, nodes, vi[nodes], fi))
        return out

    def set_metric(self, gs, dgs, J):
        d = self.d
        S = {ij: m for m, ij in enumerate(_sym(d))}
        sym = lambda m, i, j: m[S[(min(i, j), max(i, j))]]
        g = [[sym(gs, i, j) for j in range(d)] for i in range(d)]
        dg = [[[sym(dgs[len(S) * k:], i, j) for j in range(d)] for i in range(d)] for k in range(d)]
        det, inv = _inverse(g)
        self.sg, self.gi, self.J = det.sqrt(), inv, [[J[a * d + i] for i in range(d)] for a in range(d)]
        self.gam = [[[0.5 * sum(inv[i][l] * (dg[j][k][l] + dg[k][j][l] - dg[l][j][k]) for l in range(d)) for k in range(d)]
                     for j in range(d)] for i in range(d)]
        self.tr = [sum(self.gam[j][k][j] for j in range(d)) for k in range(d)]

    def hermite(self, a0, a1, a2, sg):
        d = self.d
        tr = sum(a2[i][i] for i in range(d)) / 3.0
        out = []
        for c, w in zip(self.c, self.w):
            v = a0 - 4.5 * tr
            for i in range(d):
                if c[i]:
                    v = v + 3.0 * c[i] * a1[i]
                for j in range(d):
                    if c[i] * c[j]:
                        v = v + 4.5 * (c[i] * c[j]) * a2[i][j]
            out.append(w * v / sg)
        return torch.stack(out)

    def feq(self, rho, j, gi, sg):
        d = self.d
        a2 = [[rho * (gi[a][b] - (1.0 if a == b else 0.0)) / 3.0 + j[a] * j[b] / rho for b in range(d)] for a in range(d)]
        return self.hermite(rho, j, a2, sg)

    def forcing(self, A, B, C):
        d = self.d
        b2 = [[C[a][b] - (A / 3.0 if a == b else 0.0) for b in range(d)] for a in range(d)]
        return self.hermite(A, B, b2, self.sg)

    def moments(self, f, sg, second=True):
        d = self.d
        tot = lambda of: sg * sum(of(c) * f[l] for l, c in enumerate(self.c) if of(c))
        rho, j = tot(lambda c: 1), [tot(lambda c: c[a]) for a in range(d)]
        Pi = [[tot(lambda c: c[a] * c[b]) for b in range(d)] for a in range(d)] if second else None
        return rho, j, Pi

    def fill(self, f):
        """The boundary rules, from the inner nodes."""
        if not self.faces:
            return f
        out = f.clone()
        at = lambda m, v: [[m[a][b][v] for b in range(self.d)] for a in range(self.d)]
        for rule, a, s, vw, vi, fi in self.faces:
            ratio = self.sg[vi] / self.sg[vw]
            if rule == OUTFLOW:
                out[:, vw] = f[:, vi] * ratio
                continue
            rho, j, _ = self.moments(f[:, vi], self.sg[vi], False)
            u = self.face_u.get((a, s))
            jw = [rho * (u[b][fi] if u is not None else 0.0) for b in range(self.d)]
            out[:, vw] = self.feq(rho, jw, at(self.gi, vw), self.sg[vw]) + ratio * (
                f[:, vi] - self.feq(rho, j, at(self.gi, vi), self.sg[vi]))
        return out

    def gradient(self, j):
        """D[k][i] = 3 sum_l w_l c_l^k j^i(x + c_l); one site beyond a face 2 j(face) - j(face - n)."""
        p = self.grid(torch.stack(j))
        for a in range(self.d):
            m = self.dim(a)
            lo, hi = p.narrow(m, 0, 1), p.narrow(m, self.n[a] - 1, 1)
            if self.lo[a] == PERIODIC:
                p = torch.cat([hi, p, lo], m)
            else:
                p = torch.cat([2 * lo - p.narrow(m, 1, 1), p, 2 * hi - p.narrow(m, self.n[a] - 2, 1)], m)
        D = [0.0] * self.d
        for c, w in zip(self.c, self.w):
            if not any(c):
                continue
            s = p
            for a in range(self.d):
                s = s.narrow(self.dim(a), 1 + c[a], self.n[a])
            for k in range(self.d):
                if c[k]:
                    D[k] = D[k] + 3.0 * w * c[k] * s
        return [[D[k][i].reshape(-1) for i in range(self.d)] for k in range(self.d)]

    def stress(self, rho, j, Pi):
        d, kv = self.d, 1.0 - 0.5 / self.tau
        out = [[None] * d for _ in range(d)]
        for a in range(d):
            for b in range(d):
                eq = rho * self.gi[a][b] / 3.0 + j[a] * j[b] / rho
                out[a][b] = eq + kv * (Pi[a][b] - eq)
        return out

    def forcing_moments(self, f):
        d, gam, tr, gi = self.d, self.gam, self.tr, self.gi
        rho, j, Pi = self.moments(f, self.sg)
        T, D = self.stress(rho, j, Pi), self.gradient(j)
        A = -2.0 * sum(tr[i] * j[i] for i in range(d))
        B = [self.fext[i] - 2.0 * sum(tr[k] * T[i][k] for k in range(d))
             - sum(gam[i][k][l] * T[k][l] for k in range(d) for l in range(d)) for i in range(d)]
        bar = [[D[k][i] - tr[k] * j[i] for i in range(d)] for k in range(d)]
        cov = [[D[k][i] + sum(gam[i][k][l] * j[l] for l in range(d)) for i in range(d)] for k in range(d)]
        db, dc = sum(bar[k][k] for k in range(d)), sum(cov[k][k] for k in range(d))
        C = [[None] * d for _ in range(d)]
        for a in range(d):
            for b in range(a, d):
                s = bar[b][a] + bar[a][b] - gi[a][b] * dc
                if a == b:
                    s = s + db
                C[a][b] = C[b][a] = (s - sum(gi[b][k] * cov[k][a] + gi[a][k] * cov[k][b] for k in range(d))) / 3.0
        return rho, j, (A, B, C)

    def init(self, rho=None, u=None):
        rho = torch.ones_like(self.sg) if rho is None else rho
        u = [torch.zeros_like(self.sg)] * self.d if u is None else u
        self.f = self.feq(rho, [rho * u[a] for a in range(self.d)], self.gi, self.sg)
        self.hist = self.forcing_moments(self.fill(self.f))[2]

    def step(self, count=1):
        for _ in range(count):
            self.f, self.hist = self.advance(self.f, self.hist)

    def advance(self, f, hist):
        f = self.fill(f)
        rho, j, new = self.forcing_moments(f)
        F = self.forcing(*new)
        post = f - (f - self.feq(rho, j, self.gi, self.sg)) / self.tau + F - 0.5 * self.forcing(*hist)
        post = self.grid(post)
        dims = [self.dim(a) for a in range(self.d)]
        pulled = torch.stack([torch.roll(post[l], c, dims) for l, c in enumerate(self.c)])
        # the second half of F(t) enters at the node that receives the population
        return pulled.reshape(self.Q, self.N) + 0.5 * F, new

    def _dphi(self, J_new, J_old):
        _, inv = _inverse(J_new)
        d = self.d
        return [[sum(inv[i][a] * J_old[a][k] for a in range(d)) for k in range(d)] for i in range(d)]

    def change(self, chart, psi=None):
        """The chart change: node by node, or with the old fields sampled at psi (trilinear)."""
        d = self.d
        rho, j, Pi = self.moments(self.fill(self.f), self.sg)
        A, B, C = self.hist
        old = self.J
        if psi is not None:
            s = self.sampler(psi)
            rho, A, j, B = s(rho), s(A), [s(x) for x in j], [s(x) for x in B]
            Pi, C, old = ([[s(x) for x in row] for row in m] for m in (Pi, C, old))
        self.set_metric(*chart)
        D = self._dphi(self.J, old)
        vec = lambda x: [sum(D[i][k] * x[k] for k in range(d)) for i in range(d)]
        ten = lambda x: [[sum(D[i][k] * x[k][l] * D[q][l] for k in range(d) for l in range(d)) for q in range(d)] for i in range(d)]
        j, Pi = vec(j), ten(Pi)
        self.hist = (A, vec(B), ten(C))
        a2 = [[Pi[a][b] - (rho / 3.0 if a == b else 0.0) for b in range(d)] for a in range(d)]
        self.f = self.hermite(rho, j, a2, self.sg)

    def sampler(self, psi):
        axes = []
        for a in range(self.d):
            n, p = self.n[a], psi[a]
            p = torch.remainder(p, n) if self.lo[a] == PERIODIC else p.clamp(0.0, n - 1.0)
            i0 = p.floor().long().clamp(max=n - 1)
            i1 = (i0 + 1) % n if self.lo[a] == PERIODIC else (i0 + 1).clamp(max=n - 1)
            t = p - i0
            axes.append(((i0, 1.0 - t), (i1, t)))
        terms = []
        for k in range(2 ** self.d):
            pick = [axes[a][(k >> a) & 1] for a in range(self.d)]
            terms.append((self.index([q[0] for q in pick]), math.prod([q[1] for q in pick[1:]], start=pick[0][1])))
        return lambda x: sum(w * x[i] for i, w in terms)

    def fields(self):
        rho, j, _ = self.moments(self.fill(self.f), self.sg, False)
        u = [x / rho for x in j]
        return rho, torch.stack([sum(self.J[a][i] * u[i] for i in range(self.d)) for a in range(self.d)])

    def mass(self):
        return (self.sg * self.fields()[0]).sum()

    def force(self, axis, side):
        d = self.d
        v = (self.coords()[axis] == (self.n[axis] - 1 if side else 0)).nonzero()[:, 0]
        rho, j, Pi = self.moments(self.fill(self.f), self.sg)
        T = self.stress(rho, j, Pi)
        s = 1.0 if side else -1.0
        return torch.stack([s * sum(self.J[a][i][v] * T[i][axis][v] * self.sg[v] for i in range(d)).sum() for a in range(d)])


def _inverse(m):
    """Determinant and inverse of a matrix of fields by cofactors."""
    if len(m) == 2:
        det = m[0][0] * m[1][1] - m[0][1] * m[1][0]
        return det, [[m[1][1] / det, -m[0][1] / det], [-m[1][0] / det, m[0][0] / det]]
    cof = lambda i, j: (m[(i + 1) % 3][(j + 1) % 3] * m[(i + 2) % 3][(j + 2) % 3]
                        - m[(i + 1) % 3][(j + 2) % 3] * m[(i + 2) % 3][(j + 1) % 3])
    co = [[cof(i, j) for j in range(3)] for i in range(3)]
    det = sum(m[0][j] * co[0][j] for j in range(3))
    return det, [[co[j][i] / det for j in range(3)] for i in range(3)]


def _exact_gradient(n, lo, f, order):
    """d_k f_c [3, ncomp, N] by the isotropic stencils: G_i f (order 2), G_i [f - L f / 6] (order 4), the field
    continued beyond a face by the polynomial of degree `order` through the nodes nearest it."""
    P = Plain(n, (PERIODIC,) * 3, (PERIODIC,) * 3, 1.0)
    p = f.view(-1, *n[::-1])
    for a in range(3):
        m = P.dim(a)
        if lo[a] == PERIODIC:
            p = torch.cat([p.narrow(m, n[a] - 2, 2), p, p.narrow(m, 0, 2)], m)
            continue
        ends = []
        for side in (0, 1):
            two = []
            for t in (1, 2):  # Lagrange weights of the nodes 0 .. order at -t
                w = [math.prod([(-t - q) / (k - q) for q in range(order + 1) if q != k]) for k in range(order + 1)]
                two.append(sum(w[k] * p.narrow(m, n[a] - 1 - k if side else k, 1) for k in range(order + 1)))
            ends.append(torch.cat(two if side else two[::-1], m))
        p = torch.cat([ends[0], p, ends[1]], m)

    def shifted(x, c, margin):
        for a in range(3):
            x = x.narrow(P.dim(a), margin + c[a], x.shape[P.dim(a)] - 2 * margin)
        return x

    F = shifted(p, (0, 0, 0), 1)
    if order == 4:
        F = F - sum(w * (shifted(p, c, 1) - F) for c, w in zip(P.c[1:], P.w[1:]))
    D = [sum(3.0 * w * c[k] * shifted(F, c, 1) for c, w in zip(P.c, P.w) if c[k]) for k in range(3)]
    return torch.stack([x.reshape(x.shape[0], -1) for x in D])


def exact(case, seed):
    k = case["kind"]
    with torch.set_grad_enabled(k == "adjoint"):
        return _exact(case, seed, k)


def _exact(case, seed, k):
    if k == "batch":
        rho, u = [], []
        for w in _batch(case, seed):
            P = Plain(w["n"], w["bc"], w["bc"], w["tau"], w["fext"])
            P.set_metric(*w["chart"])
            P.init(w["rho"], w["u"])
            P.step(case["steps"])
            r, v = P.fields()
            rho.append(r)
            u.append(v.reshape(-1))
        return dict(rho=torch.cat(rho), u=torch.cat(u))
    if k == "gradient":
        w = _channel(case, seed)
        return _exact_gradient(w["n"], w["bc"], w["chart"][0], case["order"])
    if k in ("steps", "d2q9"):
        w = _plane(case, seed) if k == "d2q9" else _channel(case, seed)
        bc = (PERIODIC, WALL) if k == "d2q9" else w["bc"]
        P = Plain(w["n"], bc, bc, w["tau"], w["fext"])
        P.set_metric(*w["chart"])
        P.init(w["rho"], w["u"])
        P.step(case["steps"])
        rho, v = P.fields()
        return dict(rho=rho, v=v, force=P.force(len(bc) - 1, 1))
    if k == "interp":
        w = _box(case, seed)
        P = Plain(w["n"], (PERIODIC,) * 3, (PERIODIC,) * 3, w["tau"])
        P.set_metric(*w["charts"][0])
        P.init(w["rho"], w["u"])
        for t in range(1, case["steps"] + 1):
            P.step()
            P.change(w["charts"][t % 4], w["psis"][t % 4])
        rho, v = P.fields()
        return dict(rho=rho, v=v)
    if k == "adjoint":
        from torch.utils.checkpoint import checkpoint
        w = _channel(case, seed)
        leaves = [t.requires_grad_(True) for t in w["chart"]]
        P = Plain(w["n"], w["bc"], w["bc"], w["tau"], w["fext"])
        P.set_metric(*leaves)
        P.init()

        def ahead(f, A, B, C):
            f, (A, B, C) = P.advance(f, (A, B.unbind(), [m.unbind() for m in C.unbind()]))
            return f, A, torch.stack(B), torch.stack([torch.stack(m) for m in C])

        A, B, C = P.hist
        s = (P.f, A, torch.stack(B), torch.stack([torch.stack(m) for m in C]))
        for _ in range(case["steps"]):
            s = checkpoint(ahead, *s, use_reentrant=False)
        P.f = s[0]
        J = P.force(2, 1)[1]
        g = torch.autograd.grad(J, leaves)
        return dict(value=J.detach(), g6=g[0], dg18=g[1], J9=g[2])
    w = _dynamic(case, seed) if k == "cycle" else _piston(case, seed)
    lo, hi = (w["lo"], w["hi"]) if k == "cycle" else (w["bc"], w["bc"])
    P = Plain(w["n"], lo, hi, w["tau"])
    P.set_metric(*w["times"][0][0])
    if k == "cycle":
        P.face_u[(1, 0)] = w["inflow"]
    P.face_u[(2, 1)] = w["times"][0][1]
    P.init(w["rho"], w["u"])
    forces, masses = [], []
    for t in range(1, (case["steps"] if k == "coupled" else 1) + 1):
        chart, wall = w["times"][(0, 1, 2, 3, 2, 1)[t % 6] if k == "coupled" else _order(t)]
        P.change(chart)
        P.face_u[(2, 1)] = wall
        P.step(1 if k == "coupled" else 10)
        forces.append(P.force(2, 1))
        masses.append(P.mass())
    rho, v = P.fields()
    if k == "coupled":
        return dict(rho=rho, v=v, forces=torch.stack(forces), masses=torch.stack(masses))
    return dict(rho=rho, v=v, force=forces[0], mass=masses[0])
