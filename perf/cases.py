"""The solves that users of this framework run, as measurable cases.

Every case goes through the package's public classes (``Solver``, ``Server``)
with the arguments a user's program passes.  ``listed()`` names twelve of them,
``draw(rng)`` gives one more of the same ranges, ``prepare`` makes the inputs
and the solver such a program keeps, ``run`` is one solve (or one served burst)
and ``exact`` the same solution from numpy and torch in 64 bits, evaluated from
the scheme's formulas without the package.

Kinds of case (``case["kind"]``):
  single  one trajectory, ``Solver.solve``: y0 and the solution in host memory
  batch   trajectories sharing the system, ``Solver.solve_batch`` into a CUDA tensor
  fresh   a new solver (its weights) for one solve, as a scan over orders does
  served  a burst of independent requests through one ``Server``
"""
from __future__ import annotations

import math
from decimal import Decimal, getcontext

import numpy as np
import torch

import paper_1710_01133_gb300 as fabm

DIM = {"linear": 1, "lorenz": 3, "duffing": 2, "lcr": 2}
LORENZ = (10.0, 28.0, 8.0 / 3.0)
DUFFING = (0.1, 1.2)                       # gamma, omega; the amplitude is swept
LCR = (1.015, 0.55, -1.02, -0.58)          # sigma, omega, a, b; the amplitude is swept
LCR_F_MAX = 0.1                            # limit cycles and equilibria; chaos begins above
SERVED = ("linear", "duffing", "lorenz")


def _case(name, kind, rhs, precision, alpha, h, N, B=1, uneven=False, alpha2=0.0):
    c = {"kind": kind, "rhs": rhs, "precision": precision, "alpha": alpha, "h": h, "N": N, "B": B,
         "uneven": uneven, "alpha2": alpha2}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a short scalar relaxation, as a parameter fit evaluates many times: launches and latency
        _case("scalar-500", "single", "linear", "fp64", 0.8, 1e-3, 500),
        # the scalar test equation over its whole run
        _case("scalar-10000", "single", "linear", "fp64", 0.8, 1e-3, 10_000),
        # one Lorenz-type trajectory over its full horizon
        _case("lorenz-262144", "single", "lorenz", "fp64", 0.98, 5e-4, 2 ** 18),
        # a parameter sweep of the LCR circuit in double, trajectories of uneven length
        _case("lcr-256-uneven", "batch", "lcr", "fp64", 0.9, 1e-2, 2 ** 13, 256, True),
        # an ensemble of Lorenz-type trajectories in double
        _case("lorenz-16", "batch", "lorenz", "fp64", 0.95, 1e-4, 2 ** 15, 16),
        # one trajectory with double-double weights and history (the extended-precision mode)
        _case("lorenz-16384-x2", "single", "lorenz", "fp64x2", 0.98, 5e-4, 2 ** 14),
        # one trajectory in split precision (compensated fp32 history)
        _case("lorenz-65536-split", "single", "lorenz", "split", 0.98, 5e-4, 2 ** 16),
        # the LCR sweep in split precision: tensor-core history, a narrow batch of short runs
        _case("lcr-1024-split", "batch", "lcr", "split", 0.9, 1e-2, 2 ** 14, 1024),
        # the bifurcation sweep of the forced oscillator, full size
        _case("duffing-4096-split", "batch", "duffing", "split", 0.95, 1e-3, 2 ** 16, 4096),
        # the long-horizon batch, a quarter of its horizon
        _case("lorenz-256-split", "batch", "lorenz", "split", 0.95, 1e-4, 2 ** 18, 256),
        # a scan over orders: a new solver with one order per component, one solve
        _case("lcr-orders-fresh", "fresh", "lcr", "fp64", 0.9, 1e-2, 2 ** 13, 1, False, 0.8),
        # a burst of mixed requests on the continuous-batching server
        _case("served-256", "served", "mixed", "split", 0.0, 1e-3, 2 ** 14, 256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    k = rng.choice(("single", "single", "single", "batch64", "batch64", "batch64", "split", "split",
                    "split", "narrow", "order", "x2", "fresh", "served"))
    if k == "single":
        rhs = rng.choice(("linear", "lorenz", "duffing"))
        N = _log_int(rng, 300, 150_000)
        alpha = round(rng.uniform(0.6, 0.99) if rhs == "linear" else rng.uniform(0.93, 0.99), 3)
        return _case("", "single", rhs, "fp64", alpha, 5e-4, N)
    if k == "batch64":
        rhs = rng.choice(("lcr", "lorenz", "duffing"))
        B = _log_int(rng, 2, 320)
        N = _log_int(rng, 1000, min(40_000, int(math.sqrt(2.4e10 / B))))
        h = {"lcr": 1e-2, "lorenz": 1e-4, "duffing": 1e-3}[rhs]
        return _case("", "batch", rhs, "fp64", round(rng.uniform(0.9, 0.98), 3), h, N, B,
                     rng.random() < 0.4)
    if k == "split":
        rhs = rng.choice(("lcr", "lorenz", "duffing"))
        B = _log_int(rng, 64, 4096)
        N = _log_int(rng, 1000, min(65_536, int(math.sqrt(1e12 / B))))
        h = {"lcr": 1e-2, "lorenz": 1e-4, "duffing": 1e-3}[rhs]
        if rhs == "lcr":
            N = min(N, 2 ** 14)
        return _case("", "batch", rhs, "split", round(rng.uniform(0.9, 0.98), 3), h, N, B,
                     rng.random() < 0.3)
    if k == "narrow":
        rhs = rng.choice(("linear", "lorenz"))
        return _case("", "single", rhs, "split", round(rng.uniform(0.93, 0.99), 3), 5e-4,
                     _log_int(rng, 1000, 80_000))
    if k == "order":  # 1 < alpha < 2 with y'(0)
        return _case("", "single", "linear", "fp64", round(rng.uniform(1.1, 1.8), 3), 1e-3,
                     _log_int(rng, 300, 30_000))
    if k == "x2":
        return _case("", "single", rng.choice(("linear", "lorenz")), "fp64x2",
                     round(rng.uniform(0.93, 0.99), 3), 5e-4, _log_int(rng, 500, 25_000))
    if k == "fresh":
        a = round(rng.uniform(0.85, 0.95), 3)
        return _case("", "fresh", "lcr", "fp64", a, 1e-2, _log_int(rng, 500, 12_000), 1, False,
                     round(a - rng.uniform(0.02, 0.1), 3))
    return _case("", "served", "mixed", "split", 0.0, 1e-3, 2 ** rng.choice((12, 13, 14)),
                 _log_int(rng, 20, 256))


# --------------------------------------------------------------- inputs ---

def _batch_inputs(case, seed):
    """(y0, shared params, per-trajectory params or None, N_each or None)."""
    r = np.random.default_rng(seed)
    B, N, rhs = case["B"], case["N"], case["rhs"]
    N_each = r.integers(N // 2, N + 1, B) if case["uneven"] else None
    if N_each is not None:
        N_each[r.integers(0, B)] = N
    if rhs == "linear":
        return r.uniform(0.8, 1.2, (B, 1)), (1.0,), None, N_each
    if rhs == "lorenz":
        return 1.0 + r.uniform(-0.05, 0.05, (B, 3)), LORENZ, None, N_each
    if rhs == "duffing":
        F = np.linspace(0.1, 2.0, B) if B > 1 else np.array([0.5])
        tp = np.stack([np.full(B, DUFFING[0]), np.full(B, DUFFING[1]), F], axis=1)
        return r.uniform(-0.01, 0.01, (B, 2)), DUFFING + (1.0,), tp, N_each
    f = np.linspace(0.0, LCR_F_MAX, B) if B > 1 else np.array([0.5 * LCR_F_MAX])
    tp = np.stack([np.full(B, v) for v in LCR] + [f], axis=1)
    return r.uniform(-0.1, 0.1, (B, 2)), LCR + (0.0,), tp, N_each


def _requests(case, seed):
    """The burst: systems uniform over three, orders U(0.7, 0.99), N = 2^12 up to case["N"]."""
    r = np.random.default_rng(seed)
    ks = list(range(12, int(round(math.log2(case["N"]))) + 1))
    out = []
    for j in range(case["B"]):
        rhs = SERVED[j % 3]
        alpha = float(r.uniform(0.7, 0.99))
        N = 2 ** ks[(j // 3) % len(ks)]
        if rhs == "linear":
            y0, p = r.uniform(0.5, 1.5, 1), (float(r.uniform(0.5, 1.5)),)
        elif rhs == "duffing":
            y0, p = r.uniform(-0.5, 0.5, 2), DUFFING + (float(r.uniform(0.1, 2.0)),)
        else:
            y0, p = 1.0 + r.uniform(-0.05, 0.05, 3), LORENZ
        out.append((rhs, DIM[rhs], alpha, case["h"], N, y0, p))
    return out


def _y1(case, seed):
    return np.random.default_rng(seed + 1).uniform(-0.5, 0.5, DIM[case["rhs"]])


def _alpha(case):
    return (case["alpha"], case["alpha2"]) if case["alpha2"] else case["alpha"]


def prepare(case, seed):
    st = {"case": case}
    if case["kind"] == "served":
        st["requests"] = _requests(case, seed)
        st["server"] = fabm.Server(16 << 30, precision=case["precision"], max_slots=1024)
        return st
    st["y0"], st["params"], st["traj"], st["N_each"] = _batch_inputs(case, seed)
    dim = DIM[case["rhs"]]
    if case["kind"] == "fresh":
        st["params"] = tuple(st["traj"][0])
        return st
    if case["kind"] == "single" and st["traj"] is not None:
        st["params"] = tuple(st["traj"][0])
    st["solver"] = fabm.Solver(case["rhs"], dim, _alpha(case), case["h"], case["N"], st["params"],
                               precision=case["precision"])
    if case["alpha"] > 1.0:
        st["y1"] = _y1(case, seed)
    if case["kind"] == "batch":
        st["out"] = torch.zeros((case["B"], case["N"] + 1, dim), dtype=torch.float64, device="cuda")
    return st


def run(st):
    case = st["case"]
    if case["kind"] == "single":
        return st["solver"].solve(st["y0"][0], y1=st.get("y1"))
    if case["kind"] == "batch":
        return st["solver"].solve_batch(st["y0"], traj_params=st["traj"], N_each=st["N_each"],
                                        out=st["out"])
    if case["kind"] == "fresh":
        with fabm.Solver(case["rhs"], DIM[case["rhs"]], _alpha(case), case["h"], case["N"],
                         st["params"], precision=case["precision"]) as s:
            return s.solve(st["y0"][0])
    srv = st["server"]
    tickets = [srv.submit(r[0], r[1], r[2], r[3], r[4], r[5], r[6]) for r in st["requests"]]
    while True:
        active, waiting = srv.step()
        if active == 0 and waiting == 0:
            break
    srv.finished()
    ys = [srv.result(t) for t in tickets]
    # one array per system: the requests' rows one after another
    return {q: np.concatenate([y for y, r in zip(ys, st["requests"]) if r[0] == q])
            for q in SERVED if any(r[0] == q for r in st["requests"])}


def work(case):
    """Inputs read and solutions written once; the two hereditary sums of every
    column by the cheapest known method (online Toeplitz convolution over
    doubling blocks: about 7.5 log2(2n) operations per step and level n, both
    sums) and about 40 operations per step for the scheme itself."""
    if case["kind"] == "served":
        sizes = [(r[4], r[1]) for r in _requests(case, 0)]
    elif case["uneven"]:
        sizes = [(int(n), DIM[case["rhs"]]) for n in _batch_inputs(case, 0)[3]]
    else:
        sizes = [(case["N"], DIM[case["rhs"]])] * case["B"]
    bytes_ = sum(8.0 * (n + 1) * d + 8.0 * (d + 5) for n, d in sizes)
    flops = 0.0
    for n, d in set(sizes):
        levels = sum(7.5 * (j + 1) for j in range(5, int(math.log2(n)) + 1))
        flops += sizes.count((n, d)) * n * d * (40.0 + levels)
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------- exact ---

def _weights(alpha, n):
    """B(d) = (d^a - (d-1)^a)/G(a+1), A(d) = ((d+1)^p - 2 d^p + (d-1)^p)/G(a+2),
    D(m) = C(m-1) - A(m), C(m-1) = ((m-1)^p - (m-p) m^a)/G(a+2), p = a+1, for
    d, m = 0..n (index 0: 0), without cancellation: 50 digits up to 64, series
    in 1/d beyond."""
    p = alpha + 1.0
    g1, g2 = math.gamma(alpha + 1.0), math.gamma(alpha + 2.0)
    d = np.arange(n + 1, dtype=np.float64)
    d[0] = 1.0
    x = 1.0 / np.maximum(d, 2.0)
    B = d ** alpha * -np.expm1(alpha * np.log1p(-x))
    even = np.zeros(n + 1)
    cs = np.zeros(n + 1)
    coef, xs = 1.0, np.ones(n + 1)
    for j in range(1, 14):
        coef *= (p - j + 1) / j
        xs = xs * x
        if j % 2 == 0:
            even += 2.0 * coef * xs
        if j >= 2:
            cs += coef * xs * (-1) ** j
    A, C = d ** p * even, d ** p * cs
    getcontext().prec = 50
    a_, p_ = Decimal(alpha), Decimal(alpha) + 1
    w = [Decimal(0)] + [(a_ * Decimal(i).ln()).exp() for i in range(1, 66)]
    v = [Decimal(0)] + [(p_ * Decimal(i).ln()).exp() for i in range(1, 66)]
    for i in range(1, min(n, 64) + 1):
        B[i] = float(w[i] - w[i - 1])
        A[i] = float(v[i + 1] - 2 * v[i] + v[i - 1])
        C[i] = float(v[i - 1] - (Decimal(i) - p_) * w[i])
    B, A, C = B / g1, A / g2, C / g2
    D = C - A
    B[0] = A[0] = D[0] = 0.0
    return B, A, D


def _rhs(rhs, t, y, p):
    """f(t, y): y (..., dim), p (..., n_params) or (n_params,)."""
    if rhs == "linear":
        return -p[..., 0:1] * y
    if rhs == "lorenz":
        a, b, c = y[..., 0], y[..., 1], y[..., 2]
        return np.stack([p[..., 0] * (b - a), a * (p[..., 1] - c) - b, a * b - p[..., 2] * c], -1)
    if rhs == "duffing":
        a, b = y[..., 0], y[..., 1]
        return np.stack([b, p[..., 2] * np.cos(p[..., 1] * t) - (p[..., 0] * b + a + a ** 3)], -1)
    a, b = y[..., 0], y[..., 1]
    ga, gb = p[..., 2], p[..., 3]
    g = np.where(a <= -1, gb * a - ga + gb, np.where(a >= 1, gb * a + ga - gb, ga * a))
    return np.stack([b - g, p[..., 4] * np.sin(p[..., 1] * t) - (p[..., 0] * b + a)], -1)


def _solve(rhs, alphas, h, N, y0, p, y1=None):
    """The scheme for groups of columns: alphas (R,) orders, y0 (R, C, dim),
    p broadcastable to (R, C, n_params); one order per group, or, with alphas
    (R, dim), one per component (R = 1); y1 = y'(0) where orders are above 1.  Returns (R, C, N+1, dim)."""
    R, Cn, dim = y0.shape
    L = 64
    per_comp = alphas.ndim == 2
    flat = alphas.reshape(-1)
    G = len(flat)                                   # weight sets
    cols = Cn if per_comp else Cn * dim             # columns of one weight set
    W = [_weights(float(a), N + L) for a in flat]
    WB, WA, WD = (np.stack([w[i] for w in W]) for i in range(3))
    ha = np.array([h ** float(a) for a in flat])
    ig = np.array([1.0 / math.gamma(float(a) + 2.0) for a in flat])
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    tW = torch.from_numpy(np.concatenate([WB, WA])).to(dev)          # (2G, N+L+1)
    tF = torch.zeros((G, N + 1, cols), dtype=torch.float64, device=dev)
    shape = (R, Cn, dim)
    # y (R, C, dim) <-> columns (G, cols)
    def to_g(v):
        return np.ascontiguousarray(v[0].T) if per_comp else v.reshape(G, cols)

    def from_g(v):
        return v.T.reshape(shape) if per_comp else v.reshape(shape)

    out = np.empty((N + 1,) + shape)
    out[0] = y0
    f = _rhs(rhs, 0.0, y0, p)
    f0 = to_g(f)
    Y0 = to_g(y0)
    Y1 = 0.0 if y1 is None else to_g(np.broadcast_to(y1, shape))
    blk = np.empty((G, L, cols))
    sc = (ha * ig)[:, None]
    for s0 in range(0, N, L):
        n = min(L, N - s0)
        # points k < s0 for the targets s0+1 .. s0+n
        if s0 > 0:
            idx = torch.arange(s0 + 1, s0 + n + 1, device=dev)[:, None] - torch.arange(s0, device=dev)[None, :]
            far = [torch.bmm(tW[i * G:(i + 1) * G][:, idx], tF[:, :s0]).cpu().numpy() for i in (0, 1)]
        else:
            far = [np.zeros((G, n, cols))] * 2
        blk[:, 0] = to_g(f)
        for s in range(n):
            m = s0 + s + 1
            pts = blk[:, :s + 1]
            wb, wa = WB[:, s + 1:0:-1][:, None, :], WA[:, s + 1:0:-1][:, None, :]
            P = far[0][:, s] + np.matmul(wb, pts)[:, 0]
            Cc = far[1][:, s] + np.matmul(wa, pts)[:, 0] + WD[:, m:m + 1] * f0
            T = Y0 + m * h * Y1
            yp = from_g(T + ha[:, None] * P)
            fp = to_g(_rhs(rhs, m * h, yp, p))
            y = from_g(T + ha[:, None] * Cc + sc * fp)
            out[m] = y
            f = _rhs(rhs, m * h, y, p)
            if s + 1 < L:
                blk[:, s + 1] = to_g(f)
        tF[:, s0:s0 + n] = torch.from_numpy(blk[:, :n]).to(dev)
    return np.moveaxis(out, 0, 2)


def exact(case, seed):
    N, B = case["N"], case["B"]
    if case["kind"] == "served":
        groups = {}
        reqs = _requests(case, seed)
        for j, r in enumerate(reqs):
            groups.setdefault((r[0], r[4]), []).append(j)
        ys = [None] * len(reqs)
        for (rhs, n), js in groups.items():
            got = _solve(rhs, np.array([reqs[j][2] for j in js]), case["h"], n,
                         np.stack([reqs[j][5] for j in js])[:, None, :],
                         np.array([reqs[j][6] for j in js])[:, None, :])
            for i, j in enumerate(js):
                ys[j] = got[i, 0]
        return {q: np.concatenate([y for y, r in zip(ys, reqs) if r[0] == q])
                for q in SERVED if any(r[0] == q for r in reqs)}
    cols = B * DIM[case["rhs"]]
    if N * 1.1e-4 * (1 + cols / 2000) + N * float(N) * cols / 5e11 > 18:  # seconds it would take
        return None
    y0, params, traj, N_each = _batch_inputs(case, seed)
    if traj is not None and case["kind"] != "batch":
        params, traj = tuple(traj[0]), None
    p = np.asarray(params if traj is None else traj)
    alphas = np.array([[case["alpha"], case["alpha2"]]]) if case["alpha2"] else np.array([case["alpha"]])
    y = _solve(case["rhs"], alphas, case["h"], N, y0[None], p,
               _y1(case, seed) if case["alpha"] > 1.0 else None)[0]
    if case["kind"] != "batch":
        return y[0]
    if N_each is not None:
        for b in range(B):
            y[b, N_each[b] + 1:] = 0.0
    return y
