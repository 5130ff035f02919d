"""The solver's work in real use, case by case, for measurement.

Each case is one call (or a few steps) through the Python binding of
libwcns on seeded synthetic states: single grids in 1D, 2D and 3D, packed
batches of independent 1D and 2D problems, the right-hand side alone, and
the host-buffer path, in FP64 and in mixed precision.  ``exact`` evaluates
the same calls in plain float64 torch, written from the method's equations
(Wong, Angel, Barad & Kiris, arXiv 2102.05287).
"""
from __future__ import annotations

import math

import numpy as np
import torch

WATER_AIR = dict(gamma_g=1.4, gamma_l=4.4, pinf_l=6e8)
PAPER = dict(gamma_g=1.4, gamma_l=6.12, pinf_l=3.43e8)
FLOOR = 1e-6
# Floating operations per cell and direction of one right-hand side (every
# add, mul, min/max, division and square root one), by dimension.
FLOPS = {1: 2118, 2: 2432, 3: 2839}
TR, PER, SYM = "transmissive", "periodic", "symmetry"


def listed():
    return [
        # one step of the 200-cell water-air shock tube: the smallest call, launches and latency
        dict(name="tube_step_200", kind="tube", precision="fp64", nx=200, call="step", steps=1),
        # a stretch of the 1D smooth-interface convergence study at its finest grid
        dict(name="advect_4096_mixed", kind="advect", precision="mixed", nx=4096, call="advance", steps=20),
        # the same study in FP64 at a middle grid
        dict(name="advect_512", kind="advect", precision="fp64", nx=512, call="advance", steps=10),
        # a semi-discrete right-hand side for an outside integrator: odd sizes, every kind of wave and jump
        dict(name="rhs_2d_odd", kind="waves", precision="fp64", nx=253, ny=131, call="rhs", steps=1),
        # the headline simulation, one step on its full grid
        dict(name="bubble_2d_2048", kind="bubble", precision="fp64", nx=2048, ny=1024, call="advance", steps=1),
        # the same in mixed precision, a few replayed steps
        dict(name="bubble_2d_2048_mixed", kind="bubble", precision="mixed", nx=2048, ny=1024, call="advance", steps=3),
        # Mach 10 shock on a water cylinder at the paper's grid: strong shocks, limiters at work
        dict(name="cylinder_1152", kind="cylinder", precision="fp64", nx=1152, ny=768, call="advance", steps=1),
        # 3D bubble collapse, FP64, a size whose rows leave partial tiles
        dict(name="bubble_3d_120", kind="bubble3", precision="fp64", nx=120, ny=120, nz=120, call="step", steps=1),
        # 3D bubble collapse, mixed precision, large
        dict(name="bubble_3d_256_mixed", kind="bubble3", precision="mixed", nx=256, ny=256, nz=256, call="step", steps=1),
        # a parameter study: thousands of independent Riemann problems of uneven sizes
        dict(name="riemann_4096", kind="riemann", precision="fp64", nprob=4096, nmin=128, nmax=8192, call="batch", steps=1),
        # uneven 2D bubble problems packed together
        dict(name="batch_2d_256_mixed", kind="bubbles", precision="mixed", nprob=256, nmin=32, nmax=256, call="batch", steps=2),
        # a coupled host code: the state comes from and goes back to pinned host memory every step
        dict(name="bubble_2d_host_mixed", kind="bubble", precision="mixed", nx=1024, ny=512, call="host", steps=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tube", "advect", "waves", "bubble", "cylinder", "bubble3", "riemann", "bubbles"])
    prec = rng.choice(["fp64", "mixed"])
    c = dict(kind=kind, precision=prec)
    if kind in ("tube", "advect"):
        c.update(nx=_log(rng, 64, 8192), call=rng.choice(["step", "advance"]), steps=1)
        if c["call"] == "advance":
            c["steps"] = rng.randint(2, 16)
    elif kind in ("waves", "bubble", "cylinder"):
        c.update(nx=_log(rng, 48, 1600), ny=_log(rng, 32, 1000), steps=1)
        c["call"] = rng.choice(["rhs", "step", "advance"]) if kind == "waves" else rng.choice(["step", "advance", "host"])
    elif kind == "bubble3":
        top = 110 if prec == "fp64" else 200
        c.update(nx=_log(rng, 20, top), ny=_log(rng, 20, top), nz=_log(rng, 20, top), call="step", steps=1)
    elif kind == "riemann":
        c.update(nprob=_log(rng, 16, 3000), nmin=rng.choice([32, 100, 128]), nmax=_log(rng, 500, 6000), call="batch", steps=1)
    else:
        c.update(nprob=_log(rng, 8, 200), nmin=rng.choice([16, 32, 48]), nmax=_log(rng, 64, 220), call="batch", steps=1)
    return c


# ---------------------------------------------------------------------------
# Initial states, made on the GPU from the seed.
# ---------------------------------------------------------------------------
def _conservative(eos, a1r1, a2r2, vel, p, a1):
    """(nf, ...) conservative state from primitive fields (Section 2)."""
    rho = a1r1 + a2r2
    rhoe = p * (a1 / (eos["gamma_l"] - 1.0) + (1.0 - a1) / (eos["gamma_g"] - 1.0))
    rhoe = rhoe + a1 * (eos["gamma_l"] * eos["pinf_l"] / (eos["gamma_l"] - 1.0))
    ke = sum(v * v for v in vel)
    return torch.stack(torch.broadcast_tensors(a1r1, a2r2, *[rho * v for v in vel], rhoe + 0.5 * rho * ke, a1)).contiguous()


def _mixture(eos, a1):
    """(gamma_bar, pinf_bar) of a fixed-alpha mixture."""
    G = a1 / (eos["gamma_l"] - 1) + (1 - a1) / (eos["gamma_g"] - 1)
    gb = 1 + 1 / G
    return gb, a1 * eos["gamma_l"] * eos["pinf_l"] / (eos["gamma_l"] - 1) * (gb - 1) / gb


def _post_shock(rho0, p0, p1, gamma, pinf):
    """(density, velocity) behind a shock into a stiffened gas at rest."""
    a, b = p1 + pinf, p0 + pinf
    rho1 = rho0 * ((gamma + 1) * a + (gamma - 1) * b) / ((gamma - 1) * a + (gamma + 1) * b)
    m = np.sqrt((p1 - p0) / (1.0 / rho0 - 1.0 / rho1))
    return rho1, m * (1.0 / rho0 - 1.0 / rho1)


def _centres(n, lo, hi):
    return lo + (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * ((hi - lo) / n)


def _smooth(rng, X, L, modes=4):
    """A seeded smooth field in [-1, 1] of the coordinates X over lengths L."""
    f = 0.0
    for _ in range(modes):
        k = [rng.integers(1, 5) * rng.choice([-1, 1]) for _ in X]
        f = f + rng.uniform(0.3, 1.0) * torch.sin(sum(2 * math.pi * int(ki) * x / l for ki, x, l in zip(k, X, L)) + rng.uniform(0, 2 * math.pi))
    return f / modes


def _grid_problem(case, seed):
    """State and grid of a single-grid case: (W, n, lo, hi, bcs, eos)."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "tube":  # water-air shock tube: sharp interface, limiters active
        n, lo, hi, eos = (case["nx"],), (0.0,), (1.0,), WATER_AIR
        x = _centres(n[0], 0.0, 1.0)
        left = x < rng.uniform(0.6, 0.75)
        a1 = torch.where(left, 1 - FLOOR, FLOOR).double()
        p = torch.where(left, 1e9 * rng.uniform(0.5, 1.5), 1e5).double()
        W = _conservative(eos, a1 * 1000.0, (1 - a1) * rng.uniform(30.0, 60.0), [torch.zeros_like(x)], p, a1)
        return W, n, lo, hi, ((TR, TR),), eos
    if kind == "advect":  # smooth interface carried at constant velocity
        n, lo, hi, eos = (case["nx"],), (0.0,), (1.0,), WATER_AIR
        x = _centres(n[0], 0.0, 1.0)
        a1 = 0.5 + 0.25 * torch.sin(2 * math.pi * (x - rng.uniform(0, 1)))
        W = _conservative(eos, 1000.0 * a1, 1 - a1, [torch.full_like(x, rng.uniform(0.5, 2.0))], torch.full_like(x, 1e5), a1)
        return W, n, lo, hi, ((PER, PER),), eos
    if kind == "bubble3":  # high-pressure water around a perturbed air bubble, with weak waves in the water
        n, lo, hi, eos = (case["nx"], case["ny"], case["nz"]), (0.0,) * 3, (1.0,) * 3, WATER_AIR
        Z, Y, X = torch.meshgrid(*[_centres(m, 0.0, 1.0) for m in reversed(n)], indexing="ij")
        r = torch.sqrt((X - 0.5) ** 2 + (Y - 0.5) ** 2 + (Z - 0.5) ** 2) + 1e-3 * _smooth(rng, (X, Y, Z), (0.3,) * 3)
        a1 = 1 - (FLOOR + (1 - 2 * FLOOR) * 0.5 * (1 - torch.tanh((r - 0.25) * max(n))))
        p = torch.where(r < 0.25, 1e5, 1e8 * (1 + 0.05 * _smooth(rng, (X, Y, Z), (1.0,) * 3)))
        u = [rng.uniform(0.5, 3.0) * _smooth(rng, (X, Y, Z), (1.0,) * 3) for _ in range(3)]
        return _conservative(eos, a1 * 1000.0, 1 - a1, u, p, a1), n, lo, hi, ((TR, TR),) * 3, eos
    n = (case["nx"], case["ny"])
    if kind == "waves":  # strong smooth waves everywhere plus material and pressure jumps
        lo, hi, eos = (0.0, 0.0), (2.0, 1.0), WATER_AIR
        Y, X = torch.meshgrid(_centres(n[1], 0.0, 1.0), _centres(n[0], 0.0, 2.0), indexing="ij")
        f = lambda: _smooth(rng, (X, Y), (2.0, 1.0))  # noqa: E731
        a1 = 0.5 + 0.45 * f()
        rw, ra, p = 1000.0 + 50.0 * f(), 3.0 + 2.0 * f(), 2.5e6 * (1 + 0.9 * f())
        u = [200.0 * f(), 200.0 * f()]
        for j in range(2):
            m = (X if j else Y) > rng.uniform(0.3, 0.7)
            a1 = torch.where(m, rng.choice([FLOOR, 1 - FLOOR]), a1)
            p = torch.where(m, p * rng.uniform(1.0, 50.0), p)
        return _conservative(eos, a1 * rw, (1 - a1) * ra, u, p, a1), n, lo, hi, ((TR, TR), (SYM, TR)), eos
    if kind == "cylinder":  # Mach 10 shock about to strike a water cylinder
        L, eos = 1e-3, PAPER
        lo, hi = (0.0, -10 * L), (30 * L, 10 * L)
        Y, X = torch.meshgrid(_centres(n[1], lo[1], hi[1]), _centres(n[0], 0.0, hi[0]), indexing="ij")
        water = torch.hypot(X - 13 * L, Y - rng.uniform(-1, 1) * L) < 4 * L
        post = (X < rng.uniform(7.0, 8.5) * L) & ~water
        g = 1 + 0.02 * _smooth(rng, (X, Y), (30 * L, 20 * L))
        a1 = torch.where(water, 1 - 1e-8, 1e-8).double()
        a1r1 = torch.where(water, 1000.0, 1e-8).double()
        a2r2 = torch.where(water, 1e-8, torch.where(post, 6.8571, 1.2) * g)
        W = _conservative(eos, a1r1, a2r2, [torch.where(post, 2817.9, 0.0) * g, torch.zeros_like(X)], torch.where(post, 1.165e7, 1e5) * g, a1)
        return W, n, lo, hi, ((TR, TR), (TR, TR)), eos
    # bubble: an air bubble in water, hit by a planar shock; still water ahead of it
    lo, hi, eos = (0.0, 0.0), (2.0, 1.0), WATER_AIR
    Y, X = torch.meshgrid(_centres(n[1], 0.0, 1.0), _centres(n[0], 0.0, 2.0), indexing="ij")
    r = torch.hypot(X - 1.0, Y) + 1e-3 * _smooth(rng, (X, Y), (0.2, 0.2))
    a1 = 1 - (FLOOR + (1 - 2 * FLOOR) * 0.5 * (1 - torch.tanh((r - 0.2) * (n[0] / 2.0))))
    gb, pb = _mixture(eos, 1 - FLOOR)
    rho0 = (1 - FLOOR) * 1000.0 + FLOOR
    rho1, u1 = _post_shock(rho0, 1e5, 1.9e9, gb, pb)
    post = X < rng.uniform(0.55, 0.7)
    # weak waves behind the shock, as a driver upstream sends them
    g = 1 + 0.02 * _smooth(rng, (X, Y), (2.0, 1.0))
    comp = torch.where(post, rho1 / rho0, 1.0)
    W = _conservative(eos, a1 * 1000.0 * comp, (1 - a1) * comp, [torch.where(post, float(u1) * g, 0.0), torch.zeros_like(X)],
                      torch.where(post, 1.9e9 * g, 1e5), a1)
    return W, n, lo, hi, ((TR, TR), (SYM, TR)), eos


def _batch_problem(case, seed):
    """Packed state and sizes of a batch case: (W, sizes (nprob, ndim))."""
    rng = np.random.default_rng(seed)
    nd = 1 if case["kind"] == "riemann" else 2
    k = case["nprob"]
    # sizes are part of the case (the same for every seed), log-uniform
    szr = np.random.default_rng(1000 + k)
    sizes = np.exp(szr.uniform(math.log(case["nmin"]), math.log(case["nmax"]), size=(k, nd))).astype(np.int64)
    cells = sizes.prod(axis=1)
    off = np.concatenate([[0], np.cumsum(cells)])
    prob = torch.from_numpy(np.repeat(np.arange(k), cells)).cuda()
    dev = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()[prob]  # noqa: E731
    at = torch.arange(int(off[-1]), device="cuda") - dev(off[:-1])
    nx = dev(sizes[:, 0])
    x = ((at % nx).double() + 0.5) / nx
    ratio = np.exp(rng.uniform(math.log(10.0), math.log(1e4), size=k))
    rho_l, rho_g = rng.uniform(900.0, 1100.0, size=k), rng.uniform(1.0, 100.0, size=k)
    if nd == 1:  # two-phase Riemann problems
        left = x < dev(rng.uniform(0.3, 0.7, size=k))
        a1 = torch.where(left, 1 - FLOOR, FLOOR).double()
        p = torch.where(left, 1e5 * dev(ratio), 1e5)
        return _conservative(WATER_AIR, a1 * dev(rho_l), (1 - a1) * dev(rho_g), [torch.zeros_like(x)], p, a1), sizes
    ny = dev(sizes[:, 1])
    y = (torch.div(at, nx, rounding_mode="floor").double() + 0.5) / ny
    r = torch.hypot(x - dev(rng.uniform(0.4, 0.6, size=k)), y - dev(rng.uniform(0.4, 0.6, size=k)))
    h = 1.0 / torch.maximum(nx, ny)
    a1 = 1 - (FLOOR + (1 - 2 * FLOOR) * 0.5 * (1 - torch.tanh((r - dev(rng.uniform(0.1, 0.25, size=k))) / h)))
    gb, pb = _mixture(WATER_AIR, 1 - FLOOR)
    rho0 = (1 - FLOOR) * rho_l + FLOOR * rho_g
    rho1, u1 = _post_shock(rho0, 1e5, 1e5 * ratio, gb, pb)
    post = x < dev(rng.uniform(0.05, 0.3, size=k))
    comp = torch.where(post, dev(rho1 / rho0), 1.0)
    W = _conservative(WATER_AIR, a1 * dev(rho_l) * comp, (1 - a1) * dev(rho_g) * comp, [torch.where(post, dev(u1), 0.0), torch.zeros_like(x)],
                      torch.where(post, 1e5 * dev(ratio), 1e5), a1)
    return W, sizes


def _dt_fixed(case, seed):
    """The explicit step of the calls that take one: CFL about 0.3 for the states above."""
    h = max(case.get("nx", 1), case.get("ny", 1), case.get("nz", 1))
    nd = 3 if "nz" in case else 2 if "ny" in case else 1
    speed = {"tube": 5000.0, "advect": 5000.0, "waves": 20000.0, "bubble": 6000.0, "cylinder": 3e5, "bubble3": 4000.0}[case["kind"]]
    return 0.3 / (nd * speed * h) * (1 + 1e-3 * (seed % 7))


# ---------------------------------------------------------------------------
# The calls.
# ---------------------------------------------------------------------------
def prepare(case, seed):
    from paper_2102_05287_gb300.wcns import Batch, Solver

    s = dict(case=case, call=case["call"], steps=case["steps"])
    if case["call"] == "batch":
        W, sizes = _batch_problem(case, seed)
        k, nd = sizes.shape
        lo, hi = np.zeros((k, nd)), np.ones((k, nd))
        if nd == 1:
            s["batch"] = Batch(sizes[:, 0], lo[:, 0], hi[:, 0], TR, TR, precision=case["precision"], **WATER_AIR)
        else:
            s["batch"] = Batch.grids(sizes, lo, hi, ((TR, TR),) * 2, precision=case["precision"], **WATER_AIR)
        s["t"] = torch.zeros(k, dtype=torch.float64, device="cuda")
    else:
        W, n, lo, hi, bcs, eos = _grid_problem(case, seed)
        s["solver"] = Solver(n, lo, hi, bcs, precision=case["precision"], **eos)
        s["dt"] = _dt_fixed(case, seed)
    if case["call"] == "host":
        s["W"] = W.cpu().pin_memory()
    elif case["call"] == "rhs":
        s["W"], s["L"] = W, torch.empty_like(W)
    else:  # every pass starts from the same state, as the members of a study do
        s["W0"], s["W"] = W, torch.empty_like(W)
    return s


def run(s):
    call, W = s["call"], s["W"]
    if call == "rhs":
        return s["solver"].rhs(W, s["dt"], out=s["L"])
    if call == "host":
        return {"t": s["solver"].advance_steps_host(W, s["steps"], cfl=0.5), "W": W}
    W.copy_(s["W0"])
    if call == "batch":
        s["t"].zero_()
        return {"W": s["batch"].advance(W, s["steps"], cfl=0.5, t=s["t"]), "t": s["t"]}
    if call == "step":
        return s["solver"].rk3_step(W, s["dt"])
    return {"t": s["solver"].advance_steps(W, s["steps"], cfl=0.5), "W": W}


def _cells(case):
    if case["call"] == "batch":
        nd = 1 if case["kind"] == "riemann" else 2
        szr = np.random.default_rng(1000 + case["nprob"])
        sizes = np.exp(szr.uniform(math.log(case["nmin"]), math.log(case["nmax"]), size=(case["nprob"], nd))).astype(np.int64)
        return int(sizes.prod(axis=1).sum()), nd
    n = [case[k] for k in ("nx", "ny", "nz") if k in case]
    return int(np.prod(n)), len(n)


def work(case):
    cells, nd = _cells(case)
    rhs = case["steps"] * (1 if case["call"] == "rhs" else 3)
    return {"bytes": 2.0 * 8 * (nd + 4) * cells, "flops": float(rhs) * cells * nd * FLOPS[nd]}


# ---------------------------------------------------------------------------
# The same calls in plain float64 torch.
# ---------------------------------------------------------------------------
class _Exact:
    """Cells in one packed row; for each axis the position, count and stride
    of every cell, so that a stencil is a gather of remapped positions."""

    chunk = 1 << 21
    eps_ar, eps_a, eps_rc = 1e-10, 1e-10, 1e-8
    hs_ar, hs_a, hs_rc = 1e-11, 1e-11, 1e-9

    def __init__(self, eos, axes, dx, bcs, prob, nprob):
        self.nd = len(axes)
        self.r1, self.r2 = 1.0 / (eos["gamma_l"] - 1.0), 1.0 / (eos["gamma_g"] - 1.0)
        self.q1 = eos["gamma_l"] * eos["pinf_l"] * self.r1
        self.axes, self.dx, self.bcs, self.prob, self.nprob = axes, dx, bcs, prob, nprob

    def gam(self, a):
        return a * self.r1 + (1 - a) * self.r2

    def node(self, W):
        """Velocities, pressure, sound speed (Section 2)."""
        nd = self.nd
        rho = W[0] + W[1]
        v = [W[2 + j] / rho for j in range(nd)]
        rhoe = W[2 + nd] - 0.5 * sum(W[2 + j] * v[j] for j in range(nd))
        G, P = self.gam(W[3 + nd]), W[3 + nd] * self.q1
        p = (rhoe - P) / G
        return v, p, torch.sqrt(((G + 1) * p + P) / (G * rho))

    def stencil(self, W, d, off, sl):
        """W at position + off along axis d, for the cells of the slice."""
        pos, n, stride = (t[sl] if torch.is_tensor(t) else t for t in self.axes[d])
        q = pos + off
        lo, hi = self.bcs[d]
        nm = n - 1
        flip = None
        if lo == PER:
            src = q % n
        else:
            src = torch.minimum(torch.clamp(q, min=0), nm if torch.is_tensor(nm) else torch.full_like(q, nm))
            if lo == SYM:
                src = torch.where(q < 0, -1 - q, src)
                flip = q < 0
            if hi == SYM:
                src = torch.where(q > nm, 2 * n - 1 - q, src)
                flip = (q > nm) if flip is None else flip | (q > nm)
        at = torch.arange(W.shape[1], device=W.device)[sl] + (src - pos) * stride
        w = W[:, at]
        if flip is not None:
            w[2 + d] = torch.where(flip, -w[2 + d], w[2 + d])
        return w

    @staticmethod
    def wenois(a, b, c, d, e):
        """Incremental-stencil interpolation to i+1/2 from i-2 .. i+2 (Section 4.3)."""
        beta = lambda x, y: 13.0 / 12.0 * x * x + 0.25 * y * y  # noqa: E731
        s0, s1 = 0.5 * (c + d), 0.5 * (3 * c - b)
        s2, s3 = (3 * c + 6 * d - e) / 8, (3 * a - 10 * b + 15 * c) / 8
        eps = 1e-40
        tau = beta(e - 4 * d + 6 * c - 4 * b + a, e - 2 * d + 2 * b - a)
        r01 = tau / (beta(b - 2 * c + d, b - d) + eps)
        w0 = 15.0 / 32.0 * (1 + tau / ((c - d) ** 2 + eps) * r01)
        w1 = 5.0 / 32.0 * (1 + tau / ((b - c) ** 2 + eps) * r01)
        w2 = 10.0 / 32.0 * (1 + tau / (beta(c - 2 * d + e, 3 * c - 4 * d + e) + eps))
        w3 = 2.0 / 32.0 * (1 + tau / (beta(a - 2 * b + c, a - 4 * b + 3 * c) + eps))
        return (w0 * s0 + w1 * s1 + w2 * s2 + w3 * s3) / (w0 + w1 + w2 + w3)

    def hllc(self, d, WL, vL, pL, cL, WR, vR, pR, cR):
        nd = self.nd
        uL, uR = vL[d], vR[d]
        rL, rR = WL[0] + WL[1], WR[0] + WR[1]
        ub, cb = 0.5 * (uL + uR), 0.5 * (cL + cR)
        sL, sR = torch.minimum(ub - cb, uL - cL), torch.maximum(ub + cb, uR + cR)
        mL, mR = rL * (sL - uL), rR * (sR - uR)
        ss = (pR - pL + mL * uL - mR * uR) / (mL - mR)
        out = []
        for W, v, p, rho, u, sK, sw in ((WL, vL, pL, rL, uL, sL, sL.clamp(max=0)), (WR, vR, pR, rR, uR, sR, sR.clamp(min=0))):
            x = (ss - u) / (sK - ss)  # chi - 1
            G = [W[0] * u + sw * (x * W[0]), W[1] * u + sw * (x * W[1])]
            for j in range(nd):
                G.append(W[2 + j] * u + (p if j == d else 0) + sw * (rho * sK * x if j == d else x * (rho * v[j])))
            G.append((W[2 + nd] + p) * u + sw * (x * (W[2 + nd] + p) + (1 + x) * rho * ss * (ss - u)))
            G.append(W[3 + nd] * ss)
            out.append(torch.stack(G))
        return torch.where(ss > 0, out[0], torch.where(ss < 0, out[1], 0.5 * (out[0] + out[1]))), ss

    def rct(self, W):
        """rho c~^2 = rho e - pbar (Section 5.1)."""
        nd = self.nd
        m2 = sum(W[2 + j] * W[2 + j] for j in range(nd))
        return W[2 + nd] - 0.5 * m2 / (W[0] + W[1]) - W[3 + nd] * self.q1 / (self.gam(W[3 + nd]) + 1)

    def tested(self, W, which):
        A = 3 + self.nd
        return (W[0], W[1], W[A], 1 - W[A])[which] if which < 4 else self.rct(W)

    def theta(self, A, B, which):
        eps = (self.eps_ar, self.eps_ar, self.eps_a, self.eps_a, self.eps_rc)[which]
        fA, fB = self.tested(A, which), self.tested(B, which)
        one = torch.ones_like(fA)
        return torch.where(fA < eps, 0 * one, torch.where(fB < eps, (fA - eps) / (fA - fB), one))

    def hard(self, W):
        A = 3 + self.nd
        return (W[0] < self.hs_ar) | (W[1] < self.hs_ar) | (W[A] < self.hs_a) | (1 - W[A] < self.hs_a) | (self.rct(W) < self.hs_rc)

    def face(self, S, d, lam):
        """G^- and G^+ at the midpoint between nodes 2 and 3 of the six states S."""
        nd = self.nd
        E, A = 2 + nd, 3 + nd
        prim = [self.node(w) for w in S]
        V = [torch.stack([w[0], w[1], *v, p, w[A]]) for w, (v, p, _) in zip(S, prim)]
        Wi, Wj = S[2], S[3]
        (vi, p_i, ci), (vj, pj, cj) = prim[2], prim[3]
        r1, r2, cb = 0.5 * (Wi[0] + Wj[0]), 0.5 * (Wi[1] + Wj[1]), 0.5 * (ci + cj)
        rb = r1 + r2
        k1, k2 = r1 / (rb * cb * cb), r2 / (rb * cb * cb)
        U = []
        for v in V:
            v = v - V[2]
            U.append([v[2 + d] - v[E] / (rb * cb), v[0] - k1 * v[E], v[1] - k2 * v[E]] + [v[2 + j] for j in range(nd) if j != d]
                     + [v[A], v[2 + d] + v[E] / (rb * cb)])
        sides = []
        for idx in ((0, 1, 2, 3, 4), (5, 4, 3, 2, 1)):
            u = [self.wenois(*[U[k][f] for k in idx]) for f in range(nd + 4)]
            dac = u[-1] - u[0]
            X = [Wi[0] + u[1] + 0.5 * r1 / cb * dac, Wi[1] + u[2] + 0.5 * r2 / cb * dac]
            row = 3
            for j in range(nd):
                if j == d:
                    X.append(vi[j] + 0.5 * (u[0] + u[-1]))
                else:
                    X.append(vi[j] + u[row])
                    row += 1
            p, a = p_i + 0.5 * rb * cb * dac, Wi[A] + u[-2]
            rho = X[0] + X[1]
            W = torch.stack([X[0], X[1], *[rho * X[2 + j] for j in range(nd)],
                             p * self.gam(a) + a * self.q1 + 0.5 * rho * sum(X[2 + j] ** 2 for j in range(nd)), a])
            N = Wi if not sides else Wj
            for which in range(5):
                th = self.theta(N, W, which)
                W = torch.where(th < 1, (1 - th) * N + th * W, W)
            sides.append(torch.where(self.hard(W), N, W))
        (vL, pL, cL), (vR, pR, cR) = self.node(sides[0]), self.node(sides[1])
        Gt, ut = self.hllc(d, sides[0], vL, pL, cL, sides[1], vR, pR, cR)
        hcs = lambda t, g: 256.0 / 175.0 * t - 101.0 / 420.0 * (g[2] + g[3]) + (g[1] + g[4]) / 105.0 - (g[0] + g[5]) / 2100.0  # noqa: E731
        F = []
        for w, (v, p, _) in zip(S, prim):
            f = w * v[d]
            f[2 + d] = f[2 + d] + p
            f[E] = f[E] + p * v[d]
            F.append(f)
        G, uh = hcs(Gt, F), hcs(ut, [q[0][d] for q in prim])
        split = lambda g, u, w: torch.cat([g[:A], (g[A] - w[A] * u)[None]])  # noqa: E731
        Gm, Gp = split(G, uh, Wi), split(G, uh, Wj)
        H, uH = self.hllc(d, Wi, vi, p_i, ci, Wj, vj, pj, cj)
        Hm, Hp = split(H, uH, Wi), split(H, uH, Wj)
        Fi, Fj = torch.cat([F[2][:A], 0 * F[2][A:]]), torch.cat([F[3][:A], 0 * F[3][A:]])
        l2 = 2.0 * lam
        Ap, Am = Wi - l2 * (Hm - Fi), Wj + l2 * (Hp - Fj)
        for which in range(5):
            th = torch.minimum(self.theta(Ap, Wi - l2 * (Gm - Fi), which), self.theta(Am, Wj + l2 * (Gp - Fj), which))
            Gp, Gm = torch.where(th < 1, (1 - th) * Hp + th * Gp, Gp), torch.where(th < 1, (1 - th) * Hm + th * Gm, Gm)
        bad = self.hard(Wi - l2 * (Gm - Fi)) | self.hard(Wj + l2 * (Gp - Fj))
        return torch.where(bad, Hm, Gm), torch.where(bad, Hp, Gp)

    def speeds(self, W):
        """max(|u_d| + c) of every problem, by axis (nd, nprob)."""
        v, _, c = self.node(W)
        out = W.new_zeros(self.nd, self.nprob)
        for j in range(self.nd):
            s = v[j].abs() + c
            out[j] = s.max() if self.nprob == 1 else out[j].scatter_reduce(0, self.prob, s, "amax")
        return out

    def taus(self, W):
        return self.speeds(W) / self.dx

    def rhs(self, W, dt):
        N = W.shape[1]
        tau = self.taus(W)
        L = torch.zeros_like(W)
        for d in range(self.nd):
            lam = dt / self.dx[d] * (tau.sum(0) / tau[d])  # dt / (dx sigma)
            for c0 in range(0, N, self.chunk):
                sl = slice(c0, min(N, c0 + self.chunk))
                at = 0 if self.nprob == 1 else self.prob[sl]
                S = [self.stencil(W, d, o, sl) for o in range(-3, 4)]
                left, right = self.face(S[:6], d, lam[at])[1], self.face(S[1:], d, lam[at])[0]
                L[:, sl] += (left - right) / self.dx[d][at]
        return L

    def step(self, W, dt):
        c = 0 if self.nprob == 1 else self.prob
        W1 = W + dt[c] * self.rhs(W, dt)
        W2 = 0.75 * W + 0.25 * (W1 + dt[c] * self.rhs(W1, dt))
        return W / 3.0 + 2.0 / 3.0 * (W2 + dt[c] * self.rhs(W2, dt))


def exact(case, seed):
    if case["call"] == "batch":
        W, sizes = _batch_problem(case, seed)
        k, nd = sizes.shape
        cells = sizes.prod(axis=1)
        prob = torch.from_numpy(np.repeat(np.arange(k), cells)).cuda()
        dev = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()[prob]  # noqa: E731
        at = torch.arange(int(cells.sum()), device="cuda") - dev(np.cumsum(cells) - cells)
        nx = dev(sizes[:, 0])
        axes = [(at % nx, nx, 1), (torch.div(at, nx, rounding_mode="floor"), dev(sizes[:, 1]) if nd > 1 else 1, nx)][:nd]
        x = _Exact(WATER_AIR, axes, torch.from_numpy(np.ascontiguousarray((1.0 / sizes).T)).cuda(), ((TR, TR),) * nd, prob, k)
    else:
        W, n, lo, hi, bcs, eos = _grid_problem(case, seed)
        shape, N = W.shape, int(np.prod(n))
        i = torch.arange(N, device="cuda")
        axes, stride = [], 1
        for m in n:
            axes.append((torch.div(i, stride, rounding_mode="floor") % m, m, stride))
            stride *= m
        dx = torch.tensor([[(h - l) / m] for l, h, m in zip(lo, hi, n)], dtype=torch.float64, device="cuda")
        x = _Exact(eos, axes, dx, bcs, None, 1)
        W = W.reshape(W.shape[0], N)
    t = torch.zeros(x.nprob, dtype=torch.float64, device="cuda")
    dt = None if case["call"] not in ("rhs", "step") else torch.full_like(t, _dt_fixed(case, seed))
    if case["call"] == "rhs":
        return x.rhs(W, dt).reshape(shape)
    for _ in range(case["steps"]):
        h = dt if dt is not None else 0.5 / x.taus(W).sum(0)
        W = x.step(W, h)
        t = t + h
    if case["call"] == "batch":
        return {"W": W, "t": t}
    W = W.reshape(shape)
    return W if case["call"] == "step" else {"t": float(t[0]), "W": W.cpu() if case["call"] == "host" else W}
