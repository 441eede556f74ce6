"""Performance cases of the Dichotomy solver: what a user's program has it do, through its public classes.

A case is a dict of plain values.  ``kind`` says which entry points a pass calls:

  solve          Plan.solve: one system, one right-hand side
  series         Plan.solve_series: many right-hand sides, one matrix
  train          Plan.solve, then Plan.adjoint with the loss gradient: the two halves of a training step
  modes          Batch.solve: the mode systems of a 2-D Poisson problem, all of one length
  uneven         Batch.solve: systems of very different lengths, packed back to back
  batch_train    Batch.solve, then Batch.adjoint
  general        GenPlan.solve: a tridiagonal matrix with its own entries in every row
  poisson2d      Poisson2D.solve: transform, mode systems, transform back

Plans, batches and their device workspaces are made by ``prepare`` (a program plans once and solves
many times); right-hand sides are new for every seed.  Coefficients and sizes belong to the case.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1002_2469_gb300 as D
from paper_1002_2469_gb300.poisson import Poisson2D

_PREC = {"f64": D.PREC_F64, "mixed": D.PREC_MIXED, "auto": D.PREC_AUTO}

# strongly dominant symmetric, the headline system (unsymmetric), weakly dominant
_C1, _C2, _WEAK = (-1.0, 4.0, -1.0), (-1.2, 2.5, -0.8), (-1.0, 2.001, -1.0)


def _single(kind, t, N, precision, **more):
    return dict(kind=kind, tm1=t[0], t0=t[1], tp1=t[2], N=N, precision=precision, **more)


def listed():
    return [
        # the smallest call: a short system in the library's default precision (latency, launches, host path)
        dict(name="solve_short", **_single("solve", _C1, 3001, "f64")),
        # one mid-sized system inside a time loop: too short to fill the chip
        dict(name="solve_mid", **_single("solve", _C1, 65536, "auto")),
        # the headline system: one very long right-hand side
        dict(name="solve_long", **_single("solve", _C2, 1 << 26, "auto")),
        # the same matrix in the default precision, at an odd length
        dict(name="solve_long_f64", **_single("solve", _C2, 33554467, "f64")),
        # weak dominance (an implicit step of a stiff diffusion): the coupling outlasts a window
        dict(name="solve_weak", **_single("solve", _WEAK, 16777217, "auto")),
        # a constant matrix and a series of right-hand sides (one line of an alternating-direction step)
        dict(name="series", **_single("series", _C1, 20011, "f64", M=256)),
        # a training step through one solve: forward, then gradients of right-hand side and coefficients
        dict(name="train_single", **_single("train", _C2, 1000003, "f64")),
        # 2-D Poisson by separation of variables: one system per mode
        dict(name="modes", kind="modes", M=4096, My=4096, precision="auto"),
        # a series of unrelated systems from 256 to 2^20 rows
        dict(name="uneven", kind="uneven", nsys=1500, lo=256, hi=1 << 20, coef_seed=1, precision="auto"),
        # a training step through a batch of equal systems with their own coefficients
        dict(name="batch_train", kind="batch_train", nsys=512, N=65536, coef_seed=1, precision="auto"),
        # a matrix with its own entries in every row, default precision
        dict(name="general", kind="general", N=8388613, coef_seed=1, precision="f64"),
        # the whole Poisson solve: both sine transforms and the mode systems
        dict(name="poisson2d", kind="poisson2d", M=4095, My=4095, bc_y="dirichlet"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "series", "train", "modes", "uneven", "batch_train", "general", "poisson2d"])
    prec = rng.choice(["f64", "auto"])
    if kind in ("solve", "series", "train"):
        t = rng.choice([_C1, _C2, _C2, _WEAK, (rng.uniform(-1.0, -0.5), rng.uniform(2.05, 4.0), rng.uniform(-1.0, -0.5))])
        if kind == "solve":
            return _single(kind, t, _log_int(rng, 1000, 1 << 26), prec)
        if kind == "train":
            return _single(kind, t, _log_int(rng, 10000, 1 << 24), prec)
        N = _log_int(rng, 1000, 1 << 17)
        return _single(kind, t, N, prec, M=max(2, min(4096, _log_int(rng, 1 << 18, 1 << 25) // N)))
    if kind == "modes":
        return dict(kind=kind, M=_log_int(rng, 256, 4096), My=_log_int(rng, 256, 4096), precision=prec)
    if kind == "uneven":
        return dict(kind=kind, nsys=_log_int(rng, 50, 1500), lo=256, hi=_log_int(rng, 1 << 14, 1 << 18),
                    coef_seed=rng.randrange(1, 1000), precision=prec)
    if kind == "batch_train":
        return dict(kind=kind, nsys=_log_int(rng, 32, 512), N=_log_int(rng, 4096, 65536), coef_seed=rng.randrange(1, 1000),
                    precision=prec)
    if kind == "general":
        return dict(kind=kind, N=_log_int(rng, 1 << 16, 1 << 23), coef_seed=rng.randrange(1, 1000), precision=prec)
    return dict(kind=kind, M=_log_int(rng, 255, 4095), My=_log_int(rng, 255, 4095), bc_y=rng.choice(["dirichlet", "neumann"]))


# ------------------------------------------------------------------ sizes and coefficients of a case
def _systems(case):
    """Lengths and (t_-1, t_0, t_1) of a batch's systems."""
    kind = case["kind"]
    if kind == "modes":
        k = np.arange(1, case["M"] + 1, dtype=np.float64)
        one = np.ones(case["M"])
        t0 = 2.0 + 4.0 * np.sin(k * math.pi / (2.0 * (case["M"] + 1))) ** 2
        return np.full(case["M"], case["My"], dtype=np.int64), -one, t0, -one
    rng = np.random.default_rng(case["coef_seed"])
    n = case["nsys"]
    t0, tm1, tp1 = rng.uniform(2.05, 4.0, n), rng.uniform(-1.0, -0.5, n), rng.uniform(-1.0, -0.5, n)
    if kind == "uneven":
        N = np.rint(np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), n))).astype(np.int64)
    else:
        N = np.full(n, case["N"], dtype=np.int64)
    return N, tm1, t0, tp1


def _rows(case):
    """Sub-diagonal, diagonal and super-diagonal of the general matrix (dominant by 0.05 to 2)."""
    rng = np.random.default_rng(case["coef_seed"])
    N = case["N"]
    a, c = rng.uniform(-1.0, 1.0, N), rng.uniform(-1.0, 1.0, N)
    b = np.abs(a) + np.abs(c) + rng.uniform(0.05, 2.0, N)
    return a, b, c


def _unknowns(case):
    kind = case["kind"]
    if kind == "series":
        return case["M"] * case["N"]
    if kind in ("modes", "poisson2d"):
        return case["M"] * case["My"]
    if kind in ("uneven", "batch_train"):
        return int(_systems(case)[0].sum())
    return case["N"]


# ------------------------------------------------------------------ inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _normal(n, g):
    return torch.empty(n, dtype=torch.float64, device="cuda").normal_(0.0, 1.0, generator=g)


def _uniform(n, g):
    return torch.empty(n, dtype=torch.float64, device="cuda").uniform_(-1.0, 1.0, generator=g)


def _smooth(M, My, g):
    """A smooth source on the grid: eight Gaussian bumps that vanish on the boundary ([M, My])."""
    amp = torch.empty(8, dtype=torch.float64, device="cuda").normal_(0.0, 1.0, generator=g)
    at = torch.empty(8, 2, dtype=torch.float64, device="cuda").uniform_(0.2, 0.8, generator=g)
    x = torch.arange(1, M + 1, dtype=torch.float64, device="cuda") / (M + 1)
    y = torch.arange(1, My + 1, dtype=torch.float64, device="cuda") / (My + 1)
    gx = torch.exp(-((x[:, None] - at[:, 0]) ** 2) / 0.02) * (x * (1 - x))[:, None]
    gy = torch.exp(-((y[:, None] - at[:, 1]) ** 2) / 0.02) * (y * (1 - y))[:, None]
    return (gx * amp) @ gy.T


def _sine(M):
    """The orthonormal DST-I matrix of order M."""
    k = torch.arange(1, M + 1, dtype=torch.int64, device="cuda")
    turn = (k[:, None] * k[None, :]) % (2 * (M + 1))
    return torch.sin(turn.double() * (math.pi / (M + 1))) * math.sqrt(2.0 / (M + 1))


def _rhs(case, seed):
    """Right-hand side (and the loss gradient w of a training step), on the GPU."""
    g = _generator(seed)
    kind = case["kind"]
    if kind == "poisson2d":
        return _smooth(case["M"], case["My"], g), None
    if kind == "modes":   # spectrum of a smooth source: what the transform along x hands over
        h = 1.0 / (case["M"] + 1)
        return (-(h * h) * (_sine(case["M"]) @ _smooth(case["M"], case["My"], g))).reshape(-1), None
    if kind == "series":
        return _normal(case["M"] * case["N"], g).reshape(case["M"], case["N"]), None
    n = _unknowns(case)
    F = _uniform(n, g) if kind in ("uneven", "batch_train") else _normal(n, g)
    return F, (_uniform(n, g) if kind in ("train", "batch_train") else None)


class _State:
    def __init__(self, kind, solver, F, w):
        self.kind, self.solver, self.F, self.w = kind, solver, F, w


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("solve", "series", "train"):
        solver = D.Plan(case["tm1"], case["t0"], case["tp1"], case["N"], precision=_PREC[case["precision"]])
    elif kind in ("modes", "uneven", "batch_train"):
        solver = D.Batch(*_systems(case), precision=_PREC[case["precision"]])
    elif kind == "general":
        solver = D.GenPlan(*_rows(case), precision=_PREC[case["precision"]])
    else:
        solver = Poisson2D(case["M"], My=case["My"], bc_y=case["bc_y"])
    return _State(kind, solver, *_rhs(case, seed))


def run(state):
    s = state.solver
    if state.kind == "series":
        return s.solve_series(state.F)
    x = s.solve(state.F)
    if state.w is None:
        return x
    gF, gt = s.adjoint(state.w, x)
    return {"x": x, "gF": gF, "gt": gt}


def work(case):
    """Bytes: every right-hand side, matrix entry and forward solution read once, every result written
    once.  Operations: the five multiply-adds per unknown of two recurrences and a scaled correction
    (the general matrix: its elimination), three more for the gradient sums; the transforms' FFTs."""
    n = _unknowns(case)
    kind = case["kind"]
    if kind in ("train", "batch_train"):
        return {"bytes": 40 * n, "flops": 26 * n}   # F, x | w, x, gF
    if kind == "general":
        return {"bytes": 40 * n, "flops": 10 * n}   # three matrix entries, F, x
    if kind == "poisson2d":
        return {"bytes": 16 * n, "flops": n * (10 + 2 * 2.5 * math.log2(case["M"] + 1))}
    return {"bytes": 16 * n, "flops": 10 * n}


# ------------------------------------------------------------------ reference values, plain torch
def _two_sum(a, b):
    s = a + b
    t = s - a
    return s, (a - (s - t)) + (b - t)


def _two_prod(a, b):
    p = a * b
    ta, tb = a * 134217729.0, b * 134217729.0
    ah, bh = ta - (ta - a), tb - (tb - b)
    al, bl = a - ah, b - bh
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def _columns(a, b, c, f):
    """Independent tridiagonal systems, one per column of the [L, K] arrays: Gaussian elimination in
    64 bits, then one step of refinement with a residual in twice the precision."""
    L = f.shape[0]
    cp, inv = torch.empty_like(f), torch.empty_like(f)
    q = torch.zeros_like(f[0])
    for i in range(L):
        inv[i] = 1.0 / torch.addcmul(b[i], a[i], q, value=-1.0)
        q = torch.mul(c[i], inv[i], out=cp[i])

    def elim(r):
        d = torch.empty_like(r)
        y = torch.zeros_like(r[0])
        for i in range(L):
            y = torch.mul(torch.addcmul(r[i], a[i], y, value=-1.0), inv[i], out=d[i])
        for i in range(L - 2, -1, -1):
            d[i].addcmul_(cp[i], d[i + 1], value=-1.0)
        return d

    x = elim(f)
    zero = torch.zeros_like(f[:1])
    hi, lo = f, torch.zeros_like(f)
    for m, v in ((b, x), (a, torch.cat([zero, x[:-1]])), (c, torch.cat([x[1:], zero]))):
        p, e = _two_prod(m, v)
        hi, t = _two_sum(hi, -p)
        lo = lo + (t - e)
    return x + elim(hi + lo)


def _windows(N, t, F, gap):
    """x = T^-1 F for systems of lengths N (coefficients t = three arrays) packed in F: every system in
    pieces of 4096 rows, each solved with `gap` more rows on both sides (clipped at the system's ends;
    beyond them identity rows), past which nothing couples in 64 bits."""
    N = np.asarray(N, dtype=np.int64)
    off = np.concatenate([[0], np.cumsum(N)[:-1]])
    piece = 4096
    count = -(-N // piece)
    s = np.repeat(np.arange(N.size), count)
    k = np.arange(count.sum()) - np.repeat(np.concatenate([[0], np.cumsum(count)[:-1]]), count)
    own0, own1 = k * piece, np.minimum((k + 1) * piece, N[s])
    lo, hi = np.maximum(0, own0 - gap), np.minimum(N[s], own1 + gap)
    put = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
    lo_d, hi_d, o0, o1, base = put(lo), put(hi), put(own0), put(own1), put(off[s])
    row = lo_d[None, :] + torch.arange(int((hi - lo).max()), device="cuda")[:, None]
    live = row < hi_d[None, :]
    at = (base[None, :] + row).clamp_(max=F.numel() - 1)
    f = torch.where(live, F[at], 0.0)
    a, b, c = (put(np.asarray(v, dtype=np.float64)[s])[None, :].expand_as(f) for v in t)
    b = torch.where(live, b, 1.0)
    a = torch.where(live & (row > lo_d[None, :]), a, 0.0)
    c = torch.where(live & (row + 1 < hi_d[None, :]), c, 0.0)
    x = _columns(a, b, c, f)
    own = (row >= o0[None, :]) & (row < o1[None, :])
    out = torch.empty_like(F)
    out[at[own]] = x[own]
    return out


def _gap(tm1, t0, tp1):
    """Rows after which the slower of the two decaying solutions is below 2^-75 (at most 20000)."""
    tm1, t0, tp1 = (np.asarray(v, dtype=np.float64) for v in (tm1, t0, tp1))
    q = 0.5 * (np.abs(t0) + np.sqrt(np.maximum(0.0, t0 * t0 - 4.0 * tm1 * tp1)))
    r = float(np.max(np.maximum(np.abs(tm1), np.abs(tp1)) / q))
    return 20000 if r >= 0.9975 else int(math.ceil(75.0 * math.log(2.0) / -math.log(max(r, 1e-9)))) + 2


def _sums(lam, x, N):
    """-(sum lam_i x_{i-1}, sum lam_i x_i, sum lam_i x_{i+1}) of every system."""
    out, at = [], 0
    for n in N:
        v, u = lam[at:at + n], x[at:at + n]
        out.append(torch.stack([(v[1:] * u[:-1]).sum(), (v * u).sum(), (v[:-1] * u[1:]).sum()]))
        at += int(n)
    return -torch.stack(out)


def exact(case, seed):
    kind = case["kind"]
    F, w = _rhs(case, seed)
    if kind in ("solve", "series", "train"):
        t = (case["tm1"], case["t0"], case["tp1"])
        N = [case["N"]] * case.get("M", 1)
        full = lambda v: np.full(len(N), v)  # noqa: E731
        x = _windows(N, [full(v) for v in t], F.reshape(-1), _gap(*t))
        if w is None:
            return x.reshape(F.shape)
        lam = _windows(N, [full(v) for v in t[::-1]], w, _gap(*t))
        return {"x": x, "gF": lam, "gt": _sums(lam, x, N)[0]}
    if kind in ("uneven", "batch_train"):
        N, tm1, t0, tp1 = _systems(case)
        x = _windows(N, (tm1, t0, tp1), F, _gap(tm1, t0, tp1))
        if w is None:
            return x
        lam = _windows(N, (tp1, t0, tm1), w, _gap(tm1, t0, tp1))
        return {"x": x, "gF": lam, "gt": _sums(lam, x, N)}
    if kind == "modes":
        M, My = case["M"], case["My"]
        t0 = torch.from_numpy(_systems(case)[2]).cuda()
        one = torch.ones(My, M, dtype=torch.float64, device="cuda")
        return _columns(-one, one * t0, -one, F.reshape(M, My).T.contiguous()).T.reshape(-1)
    if kind == "general":
        N = case["N"]
        a, b, c = (torch.from_numpy(v).cuda() for v in _rows(case))
        a[0] = 0.0
        c[N - 1] = 0.0
        # pieces with 2000 rows more on both sides (the weakest rows decay by about 0.95 per row, most far faster)
        piece, gap = 4096, 2000
        K = -(-N // piece)
        row = torch.arange(K, device="cuda")[None, :] * piece - gap + torch.arange(piece + 2 * gap, device="cuda")[:, None]
        live = (row >= 0) & (row < N)
        at = row.clamp(0, N - 1)
        x = _columns(torch.where(live, a[at], 0.0), torch.where(live, b[at], 1.0), torch.where(live, c[at], 0.0),
                     torch.where(live, F[at], 0.0))
        return x[gap:gap + piece].T.reshape(-1)[:N].contiguous()
    M, My = case["M"], case["My"]
    neumann = case["bc_y"] == "neumann"
    hy = 1.0 / My if neumann else 1.0 / (My + 1)
    S = _sine(M)
    k = torch.arange(1, M + 1, dtype=torch.float64, device="cuda")
    t0 = 2.0 + (hy * (M + 1)) ** 2 * 4.0 * torch.sin(k * (math.pi / (2.0 * (M + 1)))) ** 2
    one = torch.ones(My, M, dtype=torch.float64, device="cuda")
    b = one * t0
    if neumann:
        b[0] -= 1.0
        b[-1] -= 1.0
    v = _columns(-one, b, -one, ((hy * hy) * (S @ F)).T.contiguous())
    return S @ v.T
