"""Performance cases of the entropic JKO library, run through its Python binding.

``listed()`` are the workloads a user runs: single steps, flows over the range of
grids, precisions and energies, the batch, the differentiable flow, the coupled
step, the heat kernel and the FFT kernel.  ``draw`` gives more cases of the same
ranges.  Inputs are seeded here (NumPy only), so that ``exact`` (plain 64-bit
torch, dense 1-D Gibbs factors) shares no code with the library.
"""
import math

import numpy as np
import torch

from paper_1502_06216_gb300 import jko

DEV = "cuda:0"


# ---- cases ---------------------------------------------------------------------------

def listed():
    return [
        # one step on the smallest grid of the test suite: an interactive caller, or a
        # service that advances one small crowd per request; launches and latency count
        dict(name="step-crowd-64-fp32", entry="step", energy="crowd", nx=64, ny=64,
             prec="FP32", gamma=2e-3, tau=0.02, steps=1, max_iter=200, tol=1e-6, pairs=2),
        # the plain crowd-motion workload in double precision, 20 steps to tol 1e-9
        dict(name="flow-crowd-64-fp64", entry="flow", energy="crowd", nx=64, ny=64,
             prec="FP64", gamma=2e-3, tau=0.02, steps=20, max_iter=200, tol=1e-9, pairs=60),
        # crowd motion at the size of the paper's figures (200 x 200), on a domain that is
        # neither square nor a multiple of anything: what a user's own geometry looks like
        dict(name="flow-crowd-201x149-fp32", entry="flow", energy="crowd", nx=201, ny=149,
             prec="FP32", gamma=1e-3, tau=0.02, steps=10, max_iter=200, tol=1e-6, pairs=60),
        # non-linear diffusion with obstacles: the plain FP32 diffusion workload
        dict(name="flow-porous-512-fp32", entry="flow", energy="porous", nx=512, ny=512,
             prec="FP32", gamma=5e-4, tau=5e-3, steps=10, max_iter=500, tol=1e-6, pairs=3),
        # the headline workload: 1024 x 1024 crowd on the tensor cores, BF16 image pairs
        dict(name="flow-crowd-1024-bf16", entry="flow", energy="crowd", nx=1024, ny=1024,
             prec="BF16", gamma=2e-4, tau=0.02, steps=6, max_iter=200, tol=1e-6, pairs=200),
        # the same flow in plain FP32, for users who need 1e-6 accuracy
        dict(name="flow-crowd-1024-fp32", entry="flow", energy="crowd", nx=1024, ny=1024,
             prec="FP32", gamma=2e-4, tau=0.02, steps=8, max_iter=200, tol=1e-6, pairs=60),
        # the largest grid of the precision workload, in TF32
        dict(name="flow-crowd-2048-tf32", entry="flow", energy="crowd", nx=2048, ny=2048,
             prec="TF32", gamma=2e-4, tau=0.02, steps=2, max_iter=200, tol=1e-6, pairs=200),
        # many independent flows of uneven sizes advanced together
        dict(name="batch-32-fp32", entry="batch", energy="mixed", flows=32, smallest=64,
             largest=512, prec="FP32", gamma=5e-4, gamma_max=4e-3, tau=0.02, steps=4,
             max_iter=200, tol=1e-6, pairs=20),
        # one optimiser step of potential recovery: forward, loss, gradients to w and p_0
        dict(name="diff-crowd-256-fp32", entry="diff", energy="crowd", nx=256, ny=256,
             prec="FP32", gamma=1e-3, tau=0.02, steps=10, max_iter=200, tol=1e-6, pairs=20),
        # Wasserstein attraction with congestion: the step with two couplings
        dict(name="flow-attraction-256-fp32", entry="flow", energy="attraction", nx=256, ny=256,
             prec="FP32", gamma=5e-3, tau=0.3, steps=5, max_iter=2000, tol=1e-6, pairs=40),
        # crowd motion in two rooms with the heat kernel, at the paper's 100 x 100
        dict(name="flow-heat-100-fp32", entry="flow", energy="heat", nx=100, ny=100,
             prec="FP32", gamma=5e-4, tau=0.02, steps=4, max_iter=300, tol=1e-6, pairs=20),
        # diffusion in double precision with the Gaussian by FFT, the fast form there
        dict(name="flow-porous-512-fp64-fft", entry="flow", energy="porous", nx=512, ny=512,
             prec="FP64", gamma=4e-3, tau=5e-3, fft=1, steps=5, max_iter=500, tol=1e-6, pairs=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes spread over the logarithm of their range, odd ones among
    them; precisions and energies as their forms take them."""
    kind = rng.choice(["step", "simt", "simt", "simt", "tc", "tc", "fft", "batch", "diff",
                       "coupled", "coupled", "heat"])
    base = dict(max_iter=200, tol=1e-6)
    if kind in ("step", "simt"):
        prec = rng.choice(["FP32", "FP32", "FP64"])
        energy = rng.choice(["crowd", "porous", "entropy", "exponents"])
        hi = 700 if prec == "FP32" else 128
        nx = _log_int(rng, 40, hi)
        ny = nx if rng.random() < 0.3 else max(33, int(nx * rng.uniform(0.6, 1.5)))
        steps = 1 if kind == "step" else rng.randint(2, 8)
        # gamma falls with the grid, as the workloads' does: the blur stays a few cells wide
        gamma = min(4e-3, max(5e-4, 0.2 / min(nx, ny))) * rng.uniform(0.7, 1.3)
        tau = 0.02 if energy == "crowd" else 5e-3
        if energy in ("entropy", "exponents"):     # sigma = 5, as the noise workload has it
            gamma = rng.uniform(1e-3, 2e-3)
            tau, steps, nx, ny = 5 * gamma, min(steps, 3), min(nx, 512), min(ny, 512)
        return dict(base, entry="step" if kind == "step" else "flow", energy=energy, nx=nx, ny=ny,
                    prec=prec, gamma=gamma, tau=tau, steps=steps,
                    tol=1e-6 if prec == "FP32" else 1e-9, pairs=20)
    if kind == "tc":
        prec = rng.choice(["BF16", "BF16X3", "TF32"])
        nx = 8 * _log_int(rng, 12, 128)
        ny = nx if rng.random() < 0.5 else 8 * max(8, int(nx / 8 * rng.uniform(0.6, 1.0)))
        return dict(base, entry="flow", energy=rng.choice(["crowd", "porous"]), nx=nx, ny=ny,
                    prec=prec, gamma=rng.uniform(5e-4, 2e-3), tau=5e-3,
                    steps=rng.randint(2, 4), pairs=200)
    if kind == "fft":
        prec = rng.choice(["FP32", "FP64"])
        nx = _log_int(rng, 64, 600)
        ny = max(64, int(nx * rng.uniform(0.7, 1.3)))
        return dict(base, entry="flow", energy="porous", nx=nx, ny=ny, prec=prec, fft=1,
                    gamma=rng.uniform(1e-3, 4e-3), tau=5e-3, steps=rng.randint(2, 5),
                    pairs=3)
    if kind == "batch":
        return dict(base, entry="batch", energy="mixed", flows=rng.randint(6, 32), smallest=48,
                    largest=_log_int(rng, 96, 384), prec=rng.choice(["FP32", "FP32", "BF16"]),
                    gamma=1e-3, gamma_max=4e-3, tau=0.02, steps=rng.randint(1, 3), pairs=20)
    if kind == "diff":
        nx = _log_int(rng, 48, 256)
        return dict(base, entry="diff", energy="crowd", nx=nx, ny=max(40, int(nx * rng.uniform(0.7, 1.0))),
                    prec="FP32", gamma=rng.uniform(1e-3, 3e-3), tau=0.02, steps=rng.randint(3, 10),
                    pairs=20)
    if kind == "coupled":
        energy = rng.choice(["attraction", "species", "pairwise"])
        nx = _log_int(rng, 48, 256)
        gamma = {"attraction": 5e-3, "species": 2e-3, "pairwise": 8e-3}[energy]
        return dict(base, entry="flow", energy=energy, nx=nx,
                    ny=nx if rng.random() < 0.5 else max(40, int(nx * rng.uniform(0.7, 1.0))),
                    prec="FP32", gamma=gamma, tau={"attraction": 0.3}.get(energy, 0.05),
                    steps=rng.randint(1, 4), max_iter=2000, pairs=50)
    nx = _log_int(rng, 36, 100)
    return dict(base, entry="flow", energy="heat", nx=nx, ny=max(32, int(nx * rng.uniform(0.7, 1.0))),
                prec=rng.choice(["FP32", "FP64"]), gamma=5e-4, tau=0.02, steps=rng.randint(1, 4),
                max_iter=300, pairs=20)


# ---- inputs --------------------------------------------------------------------------

def _mesh(nx, ny):
    return np.meshgrid((np.arange(nx) + 0.5) / nx, (np.arange(ny) + 0.5) / ny, indexing="xy")


def _disk(X, Y, cx, cy, r):
    q = ((X - cx) ** 2 + (Y - cy) ** 2 <= r * r).astype(np.float64)
    return q / q.sum()


def _bumps(rng, X, Y, n, smin, smax, lo, hi):
    f = np.zeros_like(X)
    for _ in range(n):
        a, s = rng.uniform(0.5, 1.0), rng.uniform(smin, smax)
        cx, cy = rng.uniform(lo, hi, 2)
        f += a * np.exp(-((X - cx) ** 2 + (Y - cy) ** 2) / (2 * s * s))
    return f


def _unit(f):
    return (f - f.min()) / (f.max() - f.min())


def _obstacles(rng, X, Y):
    m = np.zeros(X.shape, bool)
    for _ in range(3):
        cx, cy = rng.uniform(0.1, 0.9, 2)
        hx, hy = rng.uniform(0.08, 0.15, 2)
        m |= (np.abs(X - cx) <= hx) & (np.abs(Y - cy) <= hy)
    return m


def _problem(energy, nx, ny, rng):
    """Fields of one flow: q0, and as the energy has them w, kappa, m, alpha, m_field,
    mask, target, w2, species, pair_alpha, heat_L (float64 arrays of N entries)."""
    X, Y = _mesh(nx, ny)
    pb = dict(w=None, kappa=math.inf, m=0.0, alpha=None, m_field=None, mask=None)
    if energy == "crowd":
        # a disk of people walking to an exit, kappa a little above the start's density
        q = _disk(X, Y, rng.uniform(0.23, 0.3), rng.uniform(0.45, 0.55), rng.uniform(0.17, 0.21))
        tx, ty = rng.uniform(0.85, 0.92), rng.uniform(0.46, 0.54)
        pb.update(q0=q, w=(X - tx) ** 2 + (Y - ty) ** 2, kappa=rng.uniform(1.15, 1.35) * q.max())
    elif energy == "porous":
        alpha = 0.5 + 1.5 * _unit(_bumps(rng, X, Y, 8, 0.05, 0.2, 0.0, 1.0))
        mask = _obstacles(rng, X, Y)
        q = _bumps(rng, X, Y, 4, 0.03, 0.08, 0.15, 0.85)
        q = np.where(mask, 0.0, q + 1e-6)
        pb.update(q0=q / q.sum(), m=2.0, alpha=alpha, mask=mask)
    elif energy == "entropy":
        q = rng.uniform(0.5, 1.0, X.shape)
        pb.update(q0=q / q.sum(), m=1.0, alpha=0.5 + 0.5 * _unit(_bumps(rng, X, Y, 4, 0.1, 0.2, 0.0, 1.0)),
                  w=0.05 * _unit(_bumps(rng, X, Y, 4, 0.1, 0.2, 0.0, 1.0)))
    elif energy == "exponents":
        q = rng.uniform(0.0, 1.0, X.shape)
        d = np.minimum(np.minimum(X, 1 - X), np.minimum(Y, 1 - Y))
        pb.update(q0=q / q.sum(), alpha=np.ones(X.shape), m_field=1.0 + d / d.max())
    elif energy == "attraction":
        q = _disk(X, Y, rng.uniform(0.25, 0.3), rng.uniform(0.45, 0.55), 0.15)
        pb.update(q0=q, kappa=q.max(),
                  target=_disk(X, Y, rng.uniform(0.7, 0.75), rng.uniform(0.45, 0.55), 0.1))
    elif energy in ("species", "pairwise"):
        if energy == "species":
            c1, c2 = (rng.uniform(0.2, 0.25), 0.5), (rng.uniform(0.75, 0.8), 0.5)
            t1, t2 = (0.85, rng.uniform(0.45, 0.55)), (0.15, rng.uniform(0.45, 0.55))
        else:
            c1, c2 = (rng.uniform(0.3, 0.35), 0.38), (rng.uniform(0.65, 0.7), 0.62)
            t1, t2 = (0.35, rng.uniform(0.43, 0.47)), (0.65, rng.uniform(0.53, 0.57))
            pb.update(pair_alpha=1.0)
        q1, q2 = (0.5 * _disk(X, Y, c[0], c[1], 0.15) for c in (c1, c2))
        pb.update(q0=np.stack([q1, q2]), kappa=(q1 + q2).max(), species=2,
                  w=(X - t1[0]) ** 2 + (Y - t1[1]) ** 2, w2=(X - t2[0]) ** 2 + (Y - t2[1]) ** 2)
    elif energy == "heat":
        q = _disk(X, Y, rng.uniform(0.22, 0.28), rng.uniform(0.45, 0.55), 0.15)
        mask = (np.abs(X - 0.5) < 0.02) & (np.abs(Y - 0.5) >= 0.1)
        pb.update(q0=q, mask=mask, w=(X - 1.0) ** 2 + (Y - 0.5) ** 2, kappa=1.2 * q.max(),
                  heat_L=10)
    return {k: v.reshape(-1) if isinstance(v, np.ndarray) else v for k, v in pb.items()}


def _batch(case, seed):
    """The flows of a batch: crowd (even) and porous (odd), sizes of powers of two and
    ragged ones in between, gammas spread over their range."""
    shape = np.random.default_rng(case["flows"])     # sizes belong to the case, not the seed
    rng = np.random.default_rng(seed)
    out = []
    for f in range(case["flows"]):
        sizes = [n for n in (64, 100, 128, 256, 512) if case["smallest"] <= n <= case["largest"]]
        nx = int(shape.choice(sizes or [case["smallest"]]))
        g = float(math.exp(rng.uniform(math.log(case["gamma"]), math.log(case["gamma_max"]))))
        energy = "crowd" if f % 2 == 0 else "porous"
        n8 = nx // 8 * 8 if case["prec"] != "FP32" else nx
        out.append(dict(_problem(energy, n8, n8, rng), nx=n8, ny=n8, gamma=g,
                        tau=case["tau"] if energy == "crowd" else 5e-3))
    return out


class _Flow:
    """A batch flow's description, as ``jko.jko_batch_create`` takes it."""

    def __init__(self, pb, case):
        self.lx = self.ly = 1.0
        self.max_iter, self.tol = case["max_iter"], case["tol"]
        self.__dict__.update(pb)


def prepare(case, seed):
    prec = jko.Precision[case["prec"]]
    dt = torch.float64 if case["prec"] == "FP64" else torch.float32
    if case["entry"] == "batch":
        pbs = _batch(case, seed)
        b = jko.jko_batch_create([_Flow(pb, case) for pb in pbs], precision=prec)
        return dict(case=case, batch=b, p0s=[torch.tensor(pb["q0"], dtype=dt, device=DEV) for pb in pbs])
    pb = _problem(case["energy"], case["nx"], case["ny"], np.random.default_rng(seed))
    q0 = pb.pop("q0")
    h = jko.jko_create(case["nx"], case["ny"], case["gamma"], case["tau"], tol=case["tol"],
                       max_iter=case["max_iter"], precision=prec, fft=case.get("fft", 0), **pb)
    state = dict(case=case, handle=h, p0=torch.tensor(q0, dtype=dt, device=DEV))
    if case["entry"] == "diff":
        rng = np.random.default_rng(seed + 1)
        X, Y = _mesh(case["nx"], case["ny"])
        t = _disk(X, Y, rng.uniform(0.45, 0.55), rng.uniform(0.45, 0.55), 0.2)
        state.update(w=torch.tensor(pb["w"], dtype=dt, device=DEV),
                     target=torch.tensor(t.reshape(-1), dtype=dt, device=DEV))
    return state


def run(state):
    case = state["case"]
    if case["entry"] == "step":
        return [jko.jko_step(state["handle"], state["p0"])[0]]
    if case["entry"] == "flow":
        p, traj, _ = jko.jko_flow(state["handle"], state["p0"], case["steps"])
        return [p, traj]
    if case["entry"] == "batch":
        return jko.jko_batch_flow(state["batch"], state["p0s"], case["steps"])[0]
    p0 = state["p0"].clone().requires_grad_(True)
    w = state["w"].clone().requires_grad_(True)
    p = jko.jko_flow_autograd(p0, w, state["handle"], case["steps"])
    loss = ((p - state["target"]) ** 2).sum()
    gp, gw = torch.autograd.grad(loss, (p0, w))
    return [p.detach(), gp, gw]


def work(case):
    """The band-limited separable contraction (2 flops per tap whose Gaussian is a normal
    FP32 / FP64 number, and output) of a typical number of pairs; the images and fields
    read and the outputs written once.  Heat kernel: one 5-point stencil (10 flops) per
    degree of the expansion.  The reverse pass of a gradient counts as the forward."""
    size = 8 if case["prec"] == "FP64" else 4

    def one(nx, ny, gamma, steps):
        N = nx * ny
        if case["energy"] == "heat":
            deg = 24.0 * math.sqrt(gamma) * max(nx, ny)
            ap = 10.0 * N * deg
        elif case.get("fft"):
            ap = 10.0 * N * (math.log2(2 * nx) + math.log2(2 * ny))
        else:
            reach = math.sqrt((708.0 if size == 8 else 87.0) * gamma)
            ap = 2.0 * N * sum(min(2 * n - 1, 2 * reach * n + 1) for n in (nx, ny))
        images = {"attraction": 2, "species": 2, "pairwise": 3}.get(case["energy"], 1)
        state = 2 if case["energy"] in ("species", "pairwise") else 1
        return {"flops": 2.0 * ap * images * case["pairs"] * steps,
                "bytes": float(size * N * (state * (1 + steps) + 2))}

    if case["entry"] == "batch":
        got = [one(pb["nx"], pb["ny"], pb["gamma"], case["steps"]) for pb in _batch(case, 0)]
        return {k: sum(g[k] for g in got) for k in ("flops", "bytes")}
    got = one(case["nx"], case["ny"], case["gamma"], case["steps"])
    if case["entry"] == "diff":
        got = {k: 2 * v for k, v in got.items()}
    return got


# ---- 64-bit values --------------------------------------------------------------------

def _d(x):
    return None if x is None else torch.tensor(np.asarray(x), dtype=torch.float64, device=DEV)


def _gauss(n, gamma):
    x = (torch.arange(n, dtype=torch.float64, device=DEV) + 0.5) / n
    return torch.exp(-(x[:, None] - x[None, :]) ** 2 / gamma)


def _gibbs(pb, nx, ny, gamma):
    """xi as a function of an image of nx ny cells."""
    if not pb.get("heat_L"):
        Kx, Ky = _gauss(nx, gamma), _gauss(ny, gamma)
        return lambda v: (Ky @ (v.reshape(ny, nx) @ Kx)).reshape(-1)
    N, L = nx * ny, pb["heat_L"]
    free = np.flatnonzero(~pb["mask"])
    at = np.full(N, -1)
    at[free] = np.arange(free.size)
    grid = at.reshape(ny, nx)
    A = torch.zeros(free.size, free.size, dtype=torch.float64, device=DEV)
    for a, b, h in ((grid[:, :-1], grid[:, 1:], 1.0 / nx), (grid[:-1], grid[1:], 1.0 / ny)):
        ok = (a >= 0) & (b >= 0)
        i = torch.tensor(a[ok], device=DEV)
        j = torch.tensor(b[ok], device=DEV)
        c = torch.full((i.numel(),), gamma / L / h ** 2, dtype=torch.float64, device=DEV)
        for u, v in ((i, j), (j, i)):
            A.index_put_((u, v), -c, accumulate=True)
            A.index_put_((u, u), c, accumulate=True)
    A.diagonal().add_(1.0)
    inv = torch.linalg.inv(A)
    idx = torch.tensor(free, device=DEV)

    def xi(v):
        x = v[idx]
        for _ in range(L):
            x = inv @ x
        out = torch.zeros_like(v)
        out[idx] = x
        return out
    return xi


def _div(x, y):
    return torch.where(x != 0, x / torch.where(x != 0, y, torch.ones_like(y)), torch.zeros_like(x))


def _ratio_maker(pb, sigma, w=None):
    """a = Prox_{sigma f}(s) / s."""
    w = _d(pb["w"]) if w is None else w
    sw = 0.0 if w is None else sigma * w
    m, alpha, kappa = pb["m"], _d(pb["alpha"]), pb["kappa"]
    mask = None if pb["mask"] is None else torch.tensor(pb["mask"], device=DEV)
    mf = _d(pb["m_field"])

    def newton(l, c, f):
        # the root of the increasing convex g(y) = y + c e(y) - l from above
        y = l / (1 + c) if mf is not None else torch.minimum(l, torch.log(l.clamp_min(1e-3) / c) / (m - 1) + 1).maximum(l - 50)
        for _ in range(200):
            g, dg = f(y)
            dy = g / dg
            y = y - dy
            if float((dy.abs() / (1 + y.abs())).max()) < 1e-15:
                break
        return y

    def ratio(s):
        pos = s > 0
        ls = torch.log(torch.where(pos, s, torch.ones_like(s)))
        if mf is not None:
            m1 = mf - 1
            c = sigma * alpha * mf
            safe = m1.clamp_min(1e-300)
            l = ls - sw

            def f(y):
                e = torch.where(m1 > 1e-12, torch.expm1(m1 * y) / safe, y)
                return y + c * e - l, 1 + c * torch.exp(m1 * y)
            a = torch.exp(newton(l, c, f) - ls)
            a = torch.where(pos, a, torch.exp(c / m1.clamp_min(1e-3) - sw))
        elif m > 1:
            c = sigma * alpha * m / (m - 1)
            l = ls - sw

            def f(y):
                e = c * torch.exp((m - 1) * y)
                return y + e - l, 1 + (m - 1) * e
            a = torch.where(pos, torch.exp(newton(l, c, f) - ls), torch.exp(-sw * torch.ones_like(s)))
        elif m == 1:
            c = sigma * alpha
            a = torch.where(pos, torch.exp(-(c * ls + sw) / (1 + c)), torch.zeros_like(s))
        else:
            a = torch.exp(-sw) if w is not None else torch.ones_like(s)
        if math.isfinite(kappa):
            over = a * s > kappa
            a = torch.where(over, kappa / torch.where(over, s, torch.ones_like(s)), a)
        return a if mask is None else torch.where(mask, torch.zeros_like(a), a)
    return ratio


def _step1(xi, q, ratio, tol, most):
    a, b = torch.ones_like(q), None
    for k in range(most + 1):
        Y = xi(a)
        if k and (k == most or float((b * Y - q).detach().abs().sum()) <= tol):
            break
        b = q / Y if q.requires_grad else _div(q, Y)   # db/dq is 1 / Y at q = 0 too
        s = xi(b)
        a = ratio(s)
    return a * s


def _mean(u, v, t):
    ok = (u > 0) & (v > 0)
    one = torch.ones_like(u)
    g = torch.exp((torch.log(torch.where(ok, u, one)) + t * torch.log(torch.where(ok, v, one))) / (1 + t))
    return torch.where(ok, g, torch.zeros_like(u))


def _step_coupled(xi, q, pb, energy, sigma, tau, tol, most):
    N = pb["nx"] * pb["ny"]
    kappa, w1, w2 = pb["kappa"], _d(pb["w"]), _d(pb.get("w2"))
    if energy == "attraction":
        t, targets = tau, (q, _d(pb["target"]))
    else:
        t, targets = tau, (q[:N], q[N:])
    b = [torch.ones(N, dtype=torch.float64, device=DEV) for _ in range(3 if energy == "pairwise" else 2)]
    for k in range(most):
        s = [xi(x) for x in b]
        if energy == "attraction":
            p = torch.clamp(_mean(s[0], s[1], t), max=kappa)
            a = [_div(p, x) for x in s]
        elif energy == "species":
            u = [s[0] * torch.exp(-sigma * w1), s[1] * torch.exp(-sigma * w2)]
            c = torch.clamp(kappa / (u[0] + u[1]).clamp_min(1e-300), max=1.0)
            a = [_div(x * c, y) for x, y in zip(u, s)]
            p = torch.cat([u[0] * c, u[1] * c])
        else:
            p1 = torch.clamp(_mean(s[0], s[2], t) * torch.exp(-sigma / (1 + t) * w1), max=kappa)
            a = [_div(p1, s[0]), _div(targets[1], s[1]), _div(p1, s[2])]
        Y = [xi(x) for x in a]
        if energy == "pairwise":
            p = torch.cat([p1, b[1] * Y[1]])
            r = (b[0] * Y[0] - targets[0]).abs().sum() + (b[1] * Y[1] - b[2] * Y[2]).abs().sum()
        else:
            r = sum((b[m] * Y[m] - targets[m]).abs().sum() for m in range(2))
        if float(r) <= tol:
            break
        if energy == "pairwise":
            pp = torch.clamp(_mean(Y[1], Y[2], t) * torch.exp(-sigma / (1 + t) * w2), max=kappa)
            b = [_div(targets[0], Y[0]), _div(pp, Y[1]), _div(pp, Y[2])]
        else:
            b = [_div(targets[m], Y[m]) for m in range(2)]
    return p


def _flow(pb, case, q, steps, w=None):
    gamma, tau = pb["gamma"], pb["tau"]
    xi = _gibbs(pb, pb["nx"], pb["ny"], gamma)
    ratio = _ratio_maker(pb, tau / gamma, w)
    traj = []
    for _ in range(steps):
        if case["energy"] in ("attraction", "species", "pairwise"):
            p = _step_coupled(xi, q, pb, case["energy"], tau / gamma, tau, case["tol"], case["max_iter"])
        else:
            p = _step1(xi, q, ratio, case["tol"], case["max_iter"])
        q = p / p.sum()
        traj.append(q)
    return traj


def exact(case, seed):
    if case["entry"] == "batch":
        return [_flow(pb, case, _d(pb["q0"].astype(np.float32)), case["steps"])[-1] for pb in _batch(case, seed)]
    pb = dict(_problem(case["energy"], case["nx"], case["ny"], np.random.default_rng(seed)),
              nx=case["nx"], ny=case["ny"], gamma=case["gamma"], tau=case["tau"])
    q0 = _d(pb["q0"].astype(np.float64 if case["prec"] == "FP64" else np.float32))
    if case["entry"] == "diff":
        rng = np.random.default_rng(seed + 1)
        X, Y = _mesh(case["nx"], case["ny"])
        t = _d(_disk(X, Y, rng.uniform(0.45, 0.55), rng.uniform(0.45, 0.55), 0.2).reshape(-1).astype(np.float32))
        q0.requires_grad_(True)
        w = _d(pb["w"].astype(np.float32)).requires_grad_(True)
        p = _flow(pb, case, q0, case["steps"], w)[-1]
        gp, gw = torch.autograd.grad(((p - t) ** 2).sum(), (q0, w))
        return [p.detach(), gp, gw]
    traj = _flow(pb, case, q0, case["steps"])
    return [traj[-1]] if case["entry"] == "step" else [traj[-1], torch.stack(traj)]
