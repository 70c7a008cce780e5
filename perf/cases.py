"""The work a user of this library has it do, as timed cases: each goes through the public entry points.

A case is a dict: "kind" says which entry point, the other keys its sizes and options.
  advance2d  a job on one 2D grid: load a state, advance `steps` CFL steps, read the state back
  step2d     the same with the caller's own loop: hw_cfl_dt, then hw_rk3_step with that dt
  rhs2d      one right-hand side of the semi-discrete scheme
  stage2d    one Runge-Kutta stage (right-hand side, limiter, combination)
  advance1d  a job on one 1D grid
  batch      many uneven 2D grids advancing together (continues from call to call)
  split      one 2D grid in px x py blocks on the GPU (continues from call to call)
  gradient   a gauge misfit and its gradient through torch's autograd
Inputs are smooth currents over Gaussian bumps with a hump of the surface and, for "strip", the small
discontinuous surface perturbation of the library's benchmark workload; all come from the seed.
"""
import math
import random

import numpy as np
import torch

import paper_2208_01260_gb300 as hw
from paper_2208_01260_gb300 import adjoint as hw_adj

G, CFL = 9.812, 0.6
PERIODIC, REFLECTIVE, OUTFLOW = 0, 1, 2


def listed():
    return [
        # the benchmark workload: a job of a few steps on the full-size grid
        dict(name="advance2d_2048", kind="advance2d", nx=2048, ny=2048, bc=REFLECTIVE, strip=True, steps=2, fp32=False),
        # an ordinary odd-sized grid in the caller's own time loop
        dict(name="step2d_701x389", kind="step2d", nx=701, ny=389, bc=PERIODIC, strip=False, steps=2),
        # a small grid, where launches and half-empty waves count (the batched workload's smallest sizes)
        dict(name="advance2d_64x66", kind="advance2d", nx=64, ny=66, bc=REFLECTIVE, strip=False, steps=10, fp32=False),
        # the spatial operator alone, for a caller's own integrator
        dict(name="rhs2d_512", kind="rhs2d", nx=512, ny=512, bc=REFLECTIVE, strip=True, char=True),
        # one stage, open boundaries, component-wise reconstruction, a long thin ragged grid
        dict(name="stage2d_1500x203", kind="stage2d", nx=1500, ny=203, bc=OUTFLOW, strip=True, char=False),
        # the single-precision variant at full size
        dict(name="fp32_2048", kind="advance2d", nx=2048, ny=2048, bc=REFLECTIVE, strip=True, steps=4, fp32=True),
        # the paper's 1D grids: N = 200 with a tiny pulse, and a large one
        dict(name="advance1d_200", kind="advance1d", nx=200, bc=REFLECTIVE, strip=True, eps=1e-10, steps=20),
        dict(name="advance1d_12801", kind="advance1d", nx=12801, bc=PERIODIC, strip=False, eps=1e-6, steps=10),
        # the batched workload: log-uniform uneven grids
        dict(name="batch_24", kind="batch", count=24, lo=64, hi=512, steps=2),
        # one grid in blocks
        dict(name="split_2x2_600x512", kind="split", nx=600, ny=512, px=2, py=2, bc=REFLECTIVE, strip=False, steps=2),
        # gradients: everything kept, and binomial checkpointing
        dict(name="gradient_256", kind="gradient", nx=256, ny=256, bc=REFLECTIVE, steps=4, gauges=32, snapshots=-1),
        dict(name="gradient_ckpt_150x97", kind="gradient", nx=150, ny=97, bc=PERIODIC, steps=8, gauges=8, snapshots=2),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["advance2d", "advance2d", "step2d", "rhs2d", "stage2d", "advance1d", "batch", "split", "gradient"])
    bc, strip = rng.choice([PERIODIC, REFLECTIVE, OUTFLOW]), rng.random() < 0.5
    nx, ny = _log(rng, 40, 1600), _log(rng, 40, 1600)
    if kind == "advance2d":
        return dict(kind=kind, nx=nx, ny=ny, bc=bc, strip=strip, steps=rng.choice([1, 2, 3]), fp32=rng.random() < 0.3)
    if kind == "step2d":
        return dict(kind=kind, nx=nx, ny=ny, bc=bc, strip=strip, steps=rng.choice([1, 2]))
    if kind in ("rhs2d", "stage2d"):
        return dict(kind=kind, nx=nx, ny=ny, bc=bc, strip=strip, char=rng.random() < 0.75)
    if kind == "advance1d":
        return dict(kind=kind, nx=_log(rng, 60, 40000), bc=bc, strip=strip, eps=rng.choice([1e-6, 1e-10]),
                    steps=rng.choice([4, 8, 16]))
    if kind == "batch":
        return dict(kind=kind, count=rng.randrange(4, 30), lo=64, hi=rng.choice([128, 256, 512]), steps=rng.choice([1, 2]))
    if kind == "split":
        return dict(kind=kind, nx=max(nx, 64), ny=max(ny, 64), px=rng.choice([1, 2, 3]), py=rng.choice([2, 3]), bc=bc,
                    strip=strip, steps=rng.choice([1, 2]))
    return dict(kind=kind, nx=_log(rng, 48, 300), ny=_log(rng, 48, 300), bc=bc, steps=rng.randrange(2, 6),
                gauges=rng.randrange(4, 40), snapshots=rng.choice([-1, -1, 2, 3]))


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------
def _axis(n, x1, bc):
    return (torch.arange(n, dtype=torch.float64, device="cuda") + (0.0 if bc == PERIODIC else 0.5)) * (x1 / n)


def _bumps(X, Y, r, count, lo, hi, s_lo, s_hi, x1, y1):
    f, fx, fy = torch.zeros_like(X), torch.zeros_like(X), torch.zeros_like(X)
    for _ in range(count):
        a, s = r.uniform(lo, hi), r.uniform(s_lo, s_hi)
        dx, dy = X - r.uniform(0.15, 0.85) * x1, Y - r.uniform(0.15, 0.85) * y1
        g = a * torch.exp(-(dx * dx + dy * dy) / s ** 2)
        f, fx, fy = f + g, fx - 2.0 * dx / s ** 2 * g, fy - 2.0 * dy / s ** 2 * g
    return f, fx, fy


def _fields2d(nx, ny, bc, strip, seed):
    """h, hu, hv, b and h_x, hu_x, hv_x, h_y, hu_y, hv_y, b_x, b_y on [0, 2] x [0, 1]."""
    r = random.Random(seed)
    x1, y1 = 2.0, 1.0
    X, Y = torch.meshgrid(_axis(nx, x1, bc), _axis(ny, y1, bc), indexing="xy")
    b, bx, by = _bumps(X, Y, r, 8, 0.02, 0.12, 0.03, 0.15, x1, y1)
    e, ex, ey = _bumps(X, Y, r, 2, 0.01, 0.05, 0.05, 0.2, x1, y1)
    eta = 1.0 + e
    if strip:
        eta = eta + torch.where((X >= 0.05) & (X <= 0.15), 0.01, 0.0)
    h, hx, hy = eta - b, ex - bx, ey - by
    kx, ky = math.pi * r.choice([2, 4]) / x1, math.pi * r.choice([2, 4]) / y1
    am, aw = r.uniform(0.05, 0.2), r.uniform(0.05, 0.2)
    sx, cx, sy, cy = torch.sin(kx * X), torch.cos(kx * X), torch.sin(ky * Y), torch.cos(ky * Y)
    hu, hux, huy = am * sx * cy, am * kx * cx * cy, -am * ky * sx * sy
    hv, hvx, hvy = aw * cx * sy, -aw * kx * sx * sy, aw * ky * cx * cy
    return [p.contiguous() for p in (h, hu, hv, b, hx, hux, hvx, hy, huy, hvy, bx, by)]


def _fields1d(nx, bc, strip, seed):
    """h, hu, b, h_x, hu_x, b_x on [0, 2]."""
    r = random.Random(seed)
    x = _axis(nx, 2.0, bc)
    b, bx = torch.zeros_like(x), torch.zeros_like(x)
    for _ in range(2):
        a, s, d = r.uniform(0.1, 0.4), r.uniform(0.05, 0.15), x - r.uniform(0.3, 1.7)
        g = a * torch.exp(-d * d / s ** 2)
        b, bx = b + g, bx - 2.0 * d / s ** 2 * g
    eta = torch.ones_like(x)
    etax = torch.zeros_like(x)
    if strip:
        s = r.uniform(0.2, 1.7)
        eta = eta + torch.where((x >= s) & (x <= s + 0.1), 1e-3, 0.0)
    k, a = math.pi * r.choice([1, 2]), r.uniform(0.05, 0.2)
    eta, etax = eta + 0.02 * torch.cos(k * x), etax - 0.02 * k * torch.sin(k * x)
    m, mx = a * torch.sin(k * x), a * k * torch.cos(k * x)
    return [p.contiguous() for p in (eta - b, m, b, etax - bx, mx, bx)]


def _batch_sizes(case, seed):
    r = random.Random(case["count"] * 1000 + case["hi"])  # the sizes belong to the case, the data to the seed
    return [(_log(r, case["lo"], case["hi"]), _log(r, case["lo"], case["hi"]), seed * 1000 + i) for i in range(case["count"])]


def _gradient_problem(case, seed):
    f = _fields2d(case["nx"], case["ny"], case["bc"], False, seed)
    state = torch.stack([f[0] + f[3], f[1], f[2], f[4] + f[10], f[5], f[6], f[7] + f[11], f[8], f[9]])
    static = torch.stack([f[3], f[10], f[11]])
    dx, dy = 2.0 / case["nx"], 1.0 / case["ny"]
    ax, ay = _alpha2d(state, static[0])
    dt = float(0.9 * CFL / (ax / dx + ay / dy))
    r = random.Random(seed + 7)
    idx = np.array(sorted(r.sample(range(case["nx"] * case["ny"]), case["gauges"])), dtype=np.int32)
    obs = np.array([[1.0 + r.uniform(-0.02, 0.05) for _ in range(case["gauges"])] for _ in range(case["steps"])])
    return state, static, [dt] * case["steps"], idx, obs


# ------------------------------------------------------------------------------------------------
# what a program holds, and one pass
# ------------------------------------------------------------------------------------------------
def _solver2d(case, f, **params):
    s = hw.Solver(hw.make_grid(case["nx"], case["ny"], 0.0, 2.0, 0.0, 1.0, case["bc"], case["bc"], dim=2),
                  hw.make_params(**params))
    hw.hw_init(s.h, f[0], f[1], f[2], f[3], f[4:])
    return s


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind in ("advance2d", "step2d", "rhs2d", "stage2d"):
        f = _fields2d(case["nx"], case["ny"], case["bc"], case["strip"], seed)
        st["solver"] = _solver2d(case, f, precision=hw.HW_FP32 if case.get("fp32") else hw.HW_FP64,
                                 char_decomp=int(case.get("char", True)))
        st["in"] = [f[0], f[1], f[2]] + f[4:10]
        if kind == "stage2d":
            st["dt"] = _dt2d(case, f)
    elif kind == "advance1d":
        f = _fields1d(case["nx"], case["bc"], case["strip"], seed)
        s = hw.Solver(hw.make_grid(case["nx"], 1, 0.0, 2.0, bc_x=case["bc"], dim=1), hw.make_params(eps_w=case["eps"]))
        hw.hw_init(s.h, f[0], f[1], None, f[2], f[3:])
        st["solver"], st["in"] = s, [f[0], f[1], f[3], f[4]]
    elif kind == "batch":
        sizes = _batch_sizes(case, seed)
        st["sizes"] = sizes
        st["batch"] = hw.hw_batch_create([hw.make_grid(nx, ny, 0.0, 2.0, 0.0, 1.0, REFLECTIVE, REFLECTIVE, dim=2)
                                          for nx, ny, _ in sizes], hw.make_params())
        for i, (nx, ny, sd) in enumerate(sizes):
            f = _fields2d(nx, ny, REFLECTIVE, False, sd)
            hw.hw_batch_init(st["batch"], i, f[0], f[1], f[2], f[3], f[4:])
    elif kind == "split":
        f = _fields2d(case["nx"], case["ny"], case["bc"], case["strip"], seed)
        g = hw.make_grid(case["nx"], case["ny"], 0.0, 2.0, 0.0, 1.0, case["bc"], case["bc"], dim=2)
        st["split"] = hw.hw_dd_create(g, hw.make_params(), case["px"], case["py"])
        hw.hw_dd_init(st["split"], f[0], f[1], f[2], f[3], f[4:])
    else:
        f = _fields2d(case["nx"], case["ny"], case["bc"], False, seed)
        st["solver"] = _solver2d(case, f)
        st["state"], st["static"], st["dts"], st["idx"], st["obs"] = _gradient_problem(case, seed)
    st["guard"] = _Guard(st)
    return st


class _Guard:
    """Frees the handles that have no object of their own when the state goes away."""

    def __init__(self, st):
        self.batch, self.split = st.get("batch"), st.get("split")

    def __del__(self):
        try:
            hw.hw_batch_destroy(self.batch)
            hw.hw_dd_destroy(self.split)
        except Exception:  # noqa: BLE001
            pass


def _empty(n, ny, nx):
    return torch.empty(n, ny, nx, dtype=torch.float64, device="cuda")


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        hw.hw_batch_run(state["batch"], case["steps"])
        outs = []
        for i, (nx, ny, _) in enumerate(state["sizes"]):
            outs.append(_empty(9, ny, nx))
            hw.hw_batch_get_state(state["batch"], i, list(outs[-1]))
        return outs
    if kind == "split":
        hw.hw_dd_advance(state["split"], case["steps"])
        out = _empty(9, case["ny"], case["nx"])
        hw.hw_dd_get_state(state["split"], list(out))
        return out
    s = state["solver"]
    if kind == "gradient":
        x, y = state["state"].detach().requires_grad_(True), state["static"].detach().requires_grad_(True)
        loss = hw_adj.GaugeMisfit.apply(x, y, s, state["dts"], state["idx"], state["obs"], case["snapshots"])
        loss.backward()
        return dict(loss=loss.detach(), state=x.grad, static=y.grad)
    hw.hw_set_state(s.h, state["in"], hw.HW_LAYOUT_PHYSICAL)
    if kind == "advance1d":
        out = torch.empty(4, case["nx"], dtype=torch.float64, device="cuda")
        s.advance(case["steps"])
        hw.hw_get_state(s.h, list(out), hw.HW_LAYOUT_EQUILIBRIUM)
        return dict(U=out[:2], V=out[2:])
    out = _empty(9, case["ny"], case["nx"])
    if kind == "rhs2d":
        hw.hw_rhs(s.h, list(out))
        return dict(U=out[:3], VQ=out[3:])
    if kind == "advance2d":
        s.advance(case["steps"])
    elif kind == "step2d":
        for _ in range(case["steps"]):
            s.rk3_step(s.cfl_dt())
    else:
        s.rk3_stage(1, state["dt"])
    hw.hw_get_state(s.h, list(out), hw.HW_LAYOUT_EQUILIBRIUM)
    if case.get("fp32"):
        out = out.float()  # the values are single-precision ones
    return dict(U=out[:3], VQ=out[3:])


# ------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------------
# Per node and stage: 9 state planes and 3 bottom planes read, 9 written, the step's base (read at two of
# three stages, written at one) on average 9; the scheme's operations (two interfaces, two node records,
# assembly, limiter, combination), an fma counted as 2. 1D: 4, 2, 4 and 4 planes.
FLOPS2D, FLOPS1D = 1911, 560


def work(case):
    kind = case["kind"]
    if kind == "advance1d":
        n = case["nx"]
        return dict(bytes=n * 8 * (8 + 14 * 3 * case["steps"]), flops=n * FLOPS1D * 3 * case["steps"])
    if kind == "batch":
        n, stages = sum(nx * ny for nx, ny, _ in _batch_sizes(case, 0)), 3 * case["steps"]
    else:
        n, stages = case["nx"] * case["ny"], 1 if kind in ("rhs2d", "stage2d") else 3 * case["steps"]
    if kind == "gradient":  # the forward run and its reverse (about twice the operations), the planes read and written twice
        return dict(bytes=n * 8 * (24 + 60 * stages), flops=n * FLOPS2D * 3 * stages)
    word = 4 if case.get("fp32") else 8
    return dict(bytes=n * (word * 30 * stages + 8 * 18), flops=n * FLOPS2D * stages)


# ------------------------------------------------------------------------------------------------
# the scheme in plain torch, 64 bits
# ------------------------------------------------------------------------------------------------
# Parities across a reflective wall normal to x of eta, m, w, their x-derivatives, their y-derivatives, b, b_x, b_y.
_PAR = [1, -1, 1, -1, 1, -1, 1, -1, 1, 1, -1, 1]


def _pad(p, par, bc, n):
    """n ghost nodes on either side of the last axis."""
    if bc == PERIODIC:
        return torch.cat([p[..., -n:], p, p[..., :n]], -1)
    if bc == REFLECTIVE:
        return torch.cat([par * p[..., :n].flip(-1), p, par * p[..., -n:].flip(-1)], -1)
    return torch.cat([p[..., :1]] * n + [p] + [p[..., -1:]] * n, -1)


def _alpha2d(S, b):
    h = S[0] - b
    c = torch.sqrt(G * h)
    return ((S[1] / h).abs() + c).max(), ((S[2] / h).abs() + c).max()


def _dt2d(case, f):
    c = torch.sqrt(G * f[0])
    ax, ay = ((f[1] / f[0]).abs() + c).max(), ((f[2] / f[0]).abs() + c).max()
    return float(CFL / (ax * case["nx"] / 2.0 + ay * case["ny"]))


def _weighted(f, p, eps):
    """Candidates' weights of one upwind side: f, p = values and dx * derivatives at three nodes."""
    d1, d2, p1 = f[0] - f[1], f[1] - f[2], p[1]
    B1, B2 = 2 * d1 + p[0] + p1, 2 * d2 + p1 + p[2]
    A1, A2, e, g = B1 + d1 + p1, B2 + d2 + p1, d1 - d2, f[0] - f[2] + 2 * p1
    w = [0.3 / (p1 * p1 + 13 / 3 * A1 * A1 + 781 / 20 * B1 * B1 + eps) ** 2,
         0.3 / (p1 * p1 + 13 / 3 * A2 * A2 + 781 / 20 * B2 * B2 + eps) ** 2,
         0.4 / (p1 * p1 + 13 / 12 * e * e + 781 / 80 * g * g + eps) ** 2]
    s = w[0] + w[1] + w[2]
    return [x / s for x in w]


def _cands(f, p):
    return [0.5 * (f[0] + f[1]) + (p[0] + 5 * p[1]) / 6, 0.5 * (f[1] + f[2]) + (p[1] - p[2]) / 6,
            (f[0] + 10 * f[1] + f[2]) / 12 + 0.5 * p[1]]


def _rows(u, v, c, char):
    """Left eigenvectors on (mass, normal, tangential), and the way back."""
    if not char:
        return (lambda a: list(a)), (lambda a: list(a))

    def left(a):
        return [((u + c) * a[0] - a[1]) / (2 * c), a[2] - v * a[0], (a[1] - (u - c) * a[0]) / (2 * c)]

    def right(a):
        return [a[0] + a[2], (u - c) * a[0] + (u + c) * a[2], v * (a[0] + a[2]) + a[1]]

    return left, right


def _sweep(S, b, bs, bm, par, bc, alpha, ds, eps, char, two=True):
    """Interfaces along the last axis. S: eta, n, t, and their derivatives along (s) and across (m) the
    sweep, n the normal and t the tangential momentum. Fluxes, source interface values, derivative
    fluxes and mixed terms, each on (mass, normal, tangential)."""
    P = [_pad(p, q, bc, 2) for p, q in zip(S, par)]
    eta, n, t = P[:3]
    B, Bs, Bm = (_pad(p, q, bc, 2) for p, q in zip((b, bs, bm), (1, -1, 1)))
    h = eta - B
    u, v = n / h, t / h
    F = [n, n * u + 0.5 * G * (eta * eta - 2 * eta * B), n * v]

    def chain(D, Db):
        return [D[1], 2 * u * D[1] + (G * h - u * u) * D[0] + (u * u - G * eta) * Db,
                u * v * (Db - D[0]) + v * D[1] + u * D[2]]

    Gs = chain(P[3:6], Bs)
    Gm = chain(P[6:9], Bm)
    k = h.shape[-1] - 3
    at = lambda a, o: a[..., o:o + k]
    hs = at(h, 1) + at(h, 2)
    ub, vb, c = (at(n, 1) + at(n, 2)) / hs, (at(t, 1) + at(t, 2)) / hs, torch.sqrt(0.5 * G * hs)
    left, right = _rows(ub, vb, c, char)
    zero = torch.zeros_like(ub)
    Fh, Bh, Gh = [0.0] * 3, [0.0] * 3, [0.0] * 3
    for side, order, sg in ((1.0, (0, 1, 2), 1.0), (-1.0, (3, 2, 1), -1.0)):
        f = [[at(0.5 * (F[q] + side * alpha * P[q]), o) for q in range(3)] for o in order]
        p = [[0.5 * ds * at(Gs[q] + side * alpha * P[3 + q], o) for q in range(3)] for o in order]
        lf, lp = [left(a) for a in f], [left([sg * x for x in a]) for a in p]
        lb = [left([zero, 0.5 * at(B, o), zero]) for o in order]
        ls = [left([zero, sg * 0.5 * ds * at(Bs, o), zero]) for o in order]
        vf, vb_ = [], []
        for q in range(3):
            fq, pq = [a[q] for a in lf], [a[q] for a in lp]
            w = _weighted(fq, pq, eps)
            vf.append(sum(x * y for x, y in zip(w, _cands(fq, pq))))
            vb_.append(sum(x * y for x, y in zip(w, _cands([a[q] for a in lb], [a[q] for a in ls]))))
        for q, (x, y) in enumerate(zip(right(vf), right(vb_))):
            Fh[q], Bh[q] = Fh[q] + x, Bh[q] + y
        for q in range(3):
            Gh[q] = Gh[q] + sg * _qprime([a[q] for a in f], [sg * a[q] / ds for a in p], ds)
    Mh = [(7 * (at(x, 1) + at(x, 2)) - at(x, 0) - at(x, 3)) / 12 for x in Gm]
    # the parts of the source that depend on the bottom only: along (quintic) and across (mixed)
    bq = sum(0.5 * sg * _qprime([at(B, o) for o in order], [sg * at(Bs, o) for o in order], ds)
             for order, sg in (((0, 1, 2), 1.0), ((3, 2, 1), -1.0)))
    bmx = (7 * (at(Bm, 1) + at(Bm, 2)) - at(Bm, 0) - at(Bm, 3)) / 12
    return Fh, Bh, Gh, Mh, bq, bmx


def _qprime(f, p, ds):
    """Derivative of the quintic at the interface from values and derivatives at three nodes."""
    return (f[0] - 8 * f[1] + 7 * f[2]) / (4 * ds) + (p[0] - 2 * p[1] - 5 * p[2]) / 12


def _limit(S, D, b, par, bc, ds, eps, char):
    """Limited derivatives along the last axis: S = eta, n, t; D their derivatives along it."""
    P = [_pad(p, q, bc, 1) for p, q in zip(S, par[:3])]
    Q = [ds * _pad(p, q, bc, 1) for p, q in zip(D, par[3:6])]
    n = S[0].shape[-1]
    at = lambda a, o: [x[..., o:o + n] for x in a]
    h = S[0] - b
    left, right = _rows(S[1] / h, S[2] / h, torch.sqrt(G * h), char)
    m0, m1, m2, nl, nr = left(at(P, 0)), left(at(P, 1)), left(at(P, 2)), left(at(Q, 0)), left(at(Q, 2))
    out = []
    for q in range(3):
        dl, dr = m1[q] - m0[q], m2[q] - m1[q]
        pl, pr, pc = 2 * dl - nl[q], 2 * dr - nr[q], 0.5 * (m2[q] - m0[q])
        w = [0.25 / (pl * pl + 13 / 3 * (dl - nl[q]) ** 2 + eps) ** 2,
             0.25 / (pr * pr + 13 / 3 * (dr - nr[q]) ** 2 + eps) ** 2,
             0.5 / (pc * pc + 13 / 12 * (dr - dl) ** 2 + eps) ** 2]
        out.append((w[0] * pl + w[1] * pr + w[2] * pc) / (w[0] + w[1] + w[2]))
    return [x / ds for x in right(out)]


_YX = [0, 2, 1, 6, 8, 7, 3, 5, 4]  # state planes seen by a y-sweep: eta, w, m, their y- then x-derivatives


def _rhs2d(S, st, bc, dx, dy, eps, char):
    ax, ay = _alpha2d(S, st[0])
    T = lambda a: a.transpose(-1, -2)
    X = _sweep(list(S), st[0], st[1], st[2], _PAR, bc, ax, dx, eps, char)
    Y = _sweep([T(S[q]) for q in _YX], T(st[0]), T(st[2]), T(st[1]), _PAR, bc, ay, dy, eps, char)
    d_x = lambda a: (a[..., 1:] - a[..., :-1]) / dx
    d_y = lambda a: T(a[..., 1:] - a[..., :-1]) / dy
    yo = [0, 2, 1]  # (mass, x-momentum, y-momentum) of a y-sweep's (mass, normal, tangential)
    out = [None] * 9
    sv = [0.0, d_x(X[4]), d_y(Y[5])]
    sq = [0.0, d_x(X[5]), d_y(Y[4])]
    for q in range(3):
        r = yo[q]
        db = d_x(X[1][q]) + d_y(Y[1][r])
        out[q] = -G * S[0] * db - d_x(X[0][q]) - d_y(Y[0][r])
        out[3 + q] = -G * S[3] * db - G * S[0] * sv[q] - d_x(X[2][q]) - d_y(Y[3][r])
        out[6 + q] = -G * S[6] * db - G * S[0] * sq[q] - d_x(X[3][q]) - d_y(Y[2][r])
    return out


def _limited2d(S, st, bc, dx, dy, eps, char):
    T = lambda a: a.transpose(-1, -2)
    V = _limit(list(S[:3]), list(S[3:6]), st[0], _PAR, bc, dx, eps, char)
    Q = _limit([T(S[0]), T(S[2]), T(S[1])], [T(S[6]), T(S[8]), T(S[7])], T(st[0]), _PAR, bc, dy, eps, char)
    return list(S[:3]) + V + [T(Q[0]), T(Q[2]), T(Q[1])]


def _stage2d(k, S, base, st, dt, bc, dx, dy, eps=1e-6, char=True):
    R, C = _rhs2d(S, st, bc, dx, dy, eps, char), _limited2d(S, st, bc, dx, dy, eps, char)
    new = [c + dt * r for c, r in zip(C, R)]
    if k > 1:
        a = 0.75 if k == 2 else 1.0 / 3.0
        new = [a * x + (1.0 - a) * y for x, y in zip(base, new)]
    return new, C if k == 1 else base


def _step2d(S, st, dt, bc, dx, dy):
    base = None
    for k in (1, 2, 3):
        S, base = _stage2d(k, S, base, st, dt, bc, dx, dy)
    return S


def _advance2d(f, bc, nx, ny, steps):
    S = [f[0] + f[3], f[1], f[2], f[4] + f[10], f[5], f[6], f[7] + f[11], f[8], f[9]]
    st, dx, dy = [f[3], f[10], f[11]], 2.0 / nx, 1.0 / ny
    for _ in range(steps):
        ax, ay = _alpha2d(S, st[0])
        S = _step2d(S, st, CFL / (ax / dx + ay / dy), bc, dx, dy)
    return torch.stack(S)


def _advance1d(f, bc, nx, steps, eps):
    """The 1D scheme is the 2D one without the tangential momentum and the second direction."""
    dx, b, bx = 2.0 / nx, f[2], f[5]
    z = torch.zeros_like(b)
    S = [f[0] + b, f[1], f[3] + bx, f[4]]
    d = lambda a: (a[1:] - a[:-1]) / dx
    for _ in range(steps):
        h = S[0] - b
        dt = CFL * dx / ((S[1] / h).abs() + torch.sqrt(G * h)).max()
        base = None
        for k in (1, 2, 3):
            h = S[0] - b
            alpha = ((S[1] / h).abs() + torch.sqrt(G * h)).max()
            X = _sweep([S[0], S[1], z, S[2], S[3], z, z, z, z], b, bx, z, _PAR, bc, alpha, dx, eps, True)
            V = _limit([S[0], S[1], z], [S[2], S[3], z], b, _PAR, bc, dx, eps, True)
            C = [S[0], S[1], V[0], V[1]]
            db = [d(X[1][q]) for q in range(2)]
            R = [-G * S[0] * db[q] - d(X[0][q]) for q in range(2)]
            R += [-G * S[2] * db[q] - (G * S[0] * d(X[4]) if q else 0.0) - d(X[2][q]) for q in range(2)]
            new = [c + dt * r for c, r in zip(C, R)]
            if k > 1:
                a = 0.75 if k == 2 else 1.0 / 3.0
                new = [a * x + (1.0 - a) * y for x, y in zip(base, new)]
            else:
                base = C
            S = new
    return torch.stack(S)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [_advance2d(_fields2d(nx, ny, REFLECTIVE, False, sd), REFLECTIVE, nx, ny, case["steps"])
                for nx, ny, sd in _batch_sizes(case, seed)]
    nx, bc = case["nx"], case["bc"]
    if kind == "advance1d":
        out = _advance1d(_fields1d(nx, bc, case["strip"], seed), bc, nx, case["steps"], case["eps"])
        return dict(U=out[:2], V=out[2:])
    ny = case["ny"]
    if kind == "gradient":
        state, static, dts, idx, obs = _gradient_problem(case, seed)
        state.requires_grad_(True)
        static.requires_grad_(True)
        S, loss = [state[q] for q in range(9)], 0.0
        at = torch.from_numpy(idx.astype(np.int64)).cuda()
        for dt, o in zip(dts, torch.from_numpy(obs).cuda()):
            S = _step2d(S, [static[q] for q in range(3)], dt, bc, 2.0 / nx, 1.0 / ny)
            loss = loss + ((S[0].reshape(-1)[at] - o) ** 2).sum()
        loss.backward()
        return dict(loss=loss.detach(), state=state.grad, static=static.grad)
    f = _fields2d(nx, ny, bc, case["strip"], seed)
    if kind == "split":
        return _advance2d(f, bc, nx, ny, case["steps"])
    if kind in ("advance2d", "step2d"):
        out = _advance2d(f, bc, nx, ny, case["steps"])
    else:
        S = [f[0] + f[3], f[1], f[2], f[4] + f[10], f[5], f[6], f[7] + f[11], f[8], f[9]]
        st, dx, dy = [f[3], f[10], f[11]], 2.0 / nx, 1.0 / ny
        if kind == "rhs2d":
            out = torch.stack(_rhs2d(S, st, bc, dx, dy, 1e-6, case["char"]))
        else:
            out = torch.stack(_stage2d(1, S, None, st, _dt2d(case, f), bc, dx, dy, 1e-6, case["char"])[0])
    return dict(U=out[:3], VQ=out[3:])
