"""The work that a program built on this library has it do, as measurable cases.

Kinds (a case's "kind"):
  step      one cycle of a model-predictive controller: new q, l, u for the plant's new state, then one
            FP32 solve warm-started from the last cycle's solution (what a control loop runs at its rate)
  random    a dense QP with equality and one-sided inequality rows, new q, l, u, cold solve to 1e-6 in
            FP64 or in the FP64-anchored form (the random-QP benchmark of the paper's Sec. V-A)
  batch     many QPs that share P and A, each with its own initial state (parametric update) or its own
            q, l, u rows, solved to 1e-3 with the BF16-split or the FP32 backend, cold or warm-started
            (sampling-based planning, scenario trees, fleets of the same robot)
  served    a burst of requests over two resident problem families, served by continuous batching until
            the last one is answered
  setup     the offline stage: a new plant's QP is set up (layer bank, batch buffers, tuning) and its
            first batch solved, as at a program's start or when the model changes
  condense  the condensing of a linear MPC problem into the dense QP (a new or re-linearised model)

Problems are condensed, LQR-preconditioned MPC problems (x+ = A x + B u, nx = 3 nu, |u| <= 1, horizon N,
n = m = N nu; with "extra" dense inequality rows: |u| <= 50 and block dynamics), with initial states
scaled so that the limits bind over part of the trajectory.
"""
import functools
import math

import numpy as np
import torch

import paper_2311_18056_gb300 as rq

SIGMA = 1e-6
BANK = (0.1, 1.0, 10.0)
CHECK = 25
MAX_ITER = 4000


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # control cycles of a small, a middle and the largest plant of the random-MPC sweep: launches,
        # copies and latency count in the small one, the bank's bytes in the large one
        {"name": "step_n20", "kind": "step", "nx": 6, "nu": 2, "N": 10},
        {"name": "step_n320", "kind": "step", "nx": 24, "nu": 8, "N": 40},
        {"name": "step_n1600", "kind": "step", "nx": 120, "nu": 40, "N": 40},
        # random dense QPs to 1e-6: a middle and a large size of the ten (one for each arithmetic)
        {"name": "random_fp64_n342", "kind": "random", "n": 342, "precision": "fp64"},
        {"name": "random_fp64r_n1110", "kind": "random", "n": 1110, "precision": "fp64r"},
        # batches of one plant: a small one, the library's headline size, a wide one with dense
        # inequality rows and warm starts, and the FP32 backend on ragged sizes with data by rows
        {"name": "batch_n800_b64", "kind": "batch", "nx": 60, "nu": 20, "N": 40, "extra": 0, "B": 64,
         "precision": "bf16x3", "data": "x0", "warm": False},
        {"name": "batch_n800_b1024", "kind": "batch", "nx": 60, "nu": 20, "N": 40, "extra": 0, "B": 1024,
         "precision": "bf16x3", "data": "x0", "warm": False},
        {"name": "batch_n600_m1000_b250_warm", "kind": "batch", "nx": 70, "nu": 30, "N": 20, "extra": 400, "B": 250,
         "precision": "bf16x3", "data": "x0", "warm": True},
        {"name": "batch_fp32_n210_b333", "kind": "batch", "nx": 21, "nu": 7, "N": 30, "extra": 0, "B": 333,
         "precision": "fp32", "data": "rows", "warm": False},
        # a burst of requests for a small plant and one with dense inequality rows
        {"name": "served_burst_240", "kind": "served", "requests": 240, "share": 0.67},
        # offline: a new plant's bank and first batch, and a new model's condensing
        {"name": "setup_n800", "kind": "setup", "nx": 60, "nu": 20, "N": 40, "B": 32},
        {"name": "condense_nx60_nu20_N40", "kind": "condense", "nx": 60, "nu": 20, "N": 40, "state": False},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "random", "batch", "batch", "batch", "served", "setup", "condense"])
    if kind == "step":
        nu = _log(rng, 2, 40)
        return {"kind": kind, "nx": 3 * nu, "nu": nu, "N": rng.randint(10, 40)}
    if kind == "random":
        return {"kind": kind, "n": _log(rng, 10, 1400), "precision": rng.choice(["fp64", "fp64r"])}
    if kind == "batch":
        nu = rng.randint(4, 20)
        extra = rng.choice([0, 0, rng.randint(1, 200)])
        return {"kind": kind, "nx": 3 * nu, "nu": nu, "N": rng.randint(10, 40), "extra": extra, "B": _log(rng, 10, 1000),
                "precision": rng.choice(["bf16x3", "bf16x3", "fp32"]), "data": rng.choice(["x0", "rows"]),
                "warm": rng.choice([False, True])}
    if kind == "served":
        return {"kind": kind, "requests": _log(rng, 20, 240), "share": round(rng.uniform(0.3, 0.9), 2)}
    nu = rng.randint(4, 20)
    if kind == "setup":
        return {"kind": kind, "nx": 3 * nu, "nu": nu, "N": rng.randint(10, 40), "B": rng.randint(9, 32)}
    return {"kind": kind, "nx": rng.randint(8, 60), "nu": rng.randint(2, 20), "N": rng.randint(8, 40),
            "state": rng.choice([False, True])}


# ---------------------------------------------------------------------------
# problems
# ---------------------------------------------------------------------------
def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _plant(rng, nx, nu, block):
    """A: I + 0.1 N(0,1), rescaled to spectral radius 1.05 (block-diagonal in 10 x 10 blocks: 1.0); B: N(0,1)."""
    A = np.zeros((nx, nx))
    step = 10 if block else nx
    for s in range(0, nx, step):
        k = min(step, nx - s)
        a = np.eye(k) + 0.1 * rng.standard_normal((k, k))
        A[s:s + k, s:s + k] = a * ((1.0 if block else 1.05) / np.max(np.abs(np.linalg.eigvals(a))))
    return A, rng.standard_normal((nx, nu))


def _lqr(A, B, Q, R):
    """Infinite-horizon gain by the Riccati recursion run to its fixed point."""
    X, K = Q.copy(), None
    for _ in range(100000):
        K = np.linalg.solve(R + B.T @ X @ B, B.T @ X @ A)
        Xn = Q + A.T @ X @ (A - B @ K)
        Xn = 0.5 * (Xn + Xn.T)
        done = np.max(np.abs(Xn - X)) <= 1e-14 * max(1.0, np.max(np.abs(Xn)))
        X = Xn
        if done:
            break
    return np.linalg.solve(R + B.T @ X @ B, B.T @ X @ A)


def _condensed(A, B, N):
    """P, A_con (control rows, then state rows), F, E, K for Q = Q_N = I, R = 0.1 I, in 64 bits on the GPU."""
    nx, nu = B.shape
    K = _lqr(A, B, np.eye(nx), 0.1 * np.eye(nu))
    Ad, Bd, Kd = _dev(A), _dev(B), _dev(K)
    Ab = Ad - Bd @ Kd
    n = N * nu
    Su, Sx = torch.zeros(N, nu, n, dtype=torch.float64, device="cuda"), torch.zeros(N, nx, n, dtype=torch.float64, device="cuda")
    Mu, Mx = torch.zeros(N, nu, nx, dtype=torch.float64, device="cuda"), torch.zeros(N, nx, nx, dtype=torch.float64, device="cuda")
    S = torch.zeros(nx, n, dtype=torch.float64, device="cuda")
    M = torch.eye(nx, dtype=torch.float64, device="cuda")
    one = torch.eye(nu, dtype=torch.float64, device="cuda")
    for k in range(N):
        Su[k] = -Kd @ S
        Su[k, :, k * nu:(k + 1) * nu] += one
        Mu[k] = -Kd @ M
        S = Ab @ S
        S[:, k * nu:(k + 1) * nu] += Bd
        M = Ab @ M
        Sx[k], Mx[k] = S, M
    su, sx, mu, mx = Su.reshape(-1, n), Sx.reshape(-1, n), Mu.reshape(-1, nx), Mx.reshape(-1, nx)
    P = 0.1 * (su.T @ su) + sx.T @ sx
    F = 0.1 * (su.T @ mu) + sx.T @ mx
    return 0.5 * (P + P.T), torch.cat([su, sx]), F, torch.cat([mu, mx]), K


class _Problem:
    """Parametric QP: q = F x0, l = l0 - E x0, u = u0 - E x0, and the states' scale."""

    def __init__(self, nx, nu, N, extra, seed):
        rng = np.random.default_rng(seed)
        A, B = _plant(rng, nx, nu, extra > 0)
        P, S, F, M, _ = _condensed(A, B, N)
        n, umax = N * nu, 50.0 if extra else 1.0
        self.P, self.F = P.cpu().numpy(), F.cpu().numpy()
        self.A, self.E = S[:n].cpu().numpy(), M[:n].cpu().numpy()
        self.l0, self.u0 = np.full(n, -umax), np.full(n, umax)
        # the median, over 64 draws, of the peak unconstrained control is 4 limits (1 with the wider limits)
        peak = np.max(np.abs(rng.standard_normal((64, nx)) @ self.E.T), axis=1) / umax
        self.std = (1.0 if extra else 4.0) / float(np.median(peak))
        if extra:
            self.A = np.vstack([self.A, rng.standard_normal((extra, n)) / math.sqrt(n)])
            self.E = np.vstack([self.E, np.zeros((extra, nx))])
            self.l0 = np.concatenate([self.l0, np.full(extra, -np.inf)])
            self.u0 = np.concatenate([self.u0, rng.uniform(1.0, 2.0, extra)])
        self.Ad, self.Bd, self.nx, self.nu, self.n, self.m = A, B, nx, nu, n, self.A.shape[0]

    def instance(self, X):
        return X @ self.F.T, self.l0 - X @ self.E.T, self.u0 - X @ self.E.T


@functools.lru_cache(maxsize=4)
def _problem(nx, nu, N, extra, sub=0):
    return _Problem(nx, nu, N, extra, [nx, nu, N, extra, sub])


def _random_qp(n, seed):
    """n/4 equality rows, then n/4 one-sided inequality rows, feasible by construction (rows >= 1)."""
    rng = np.random.default_rng([91, n, seed])
    k = max(1, n // 4)
    M = _dev(rng.standard_normal((n, n)))
    P = M @ M.T / n
    P = (0.5 * (P + P.T)).cpu().numpy() + 1e-2 * np.eye(n)
    A = rng.standard_normal((2 * k, n)) / math.sqrt(n)
    Ax = A @ rng.standard_normal(n)
    lo, up = Ax.copy(), Ax.copy()
    lo[k:] = -np.inf
    up[k:] += rng.uniform(0.0, 1.0, k)
    return P, rng.standard_normal(n), A, lo, up


# ---------------------------------------------------------------------------
# the method in 64 bits (plain torch): for warm starts and for exact()
# ---------------------------------------------------------------------------
def _admm(P, A, q, l, u, eps, x=None, lam=None, ri=None, most=MAX_ITER):
    """ADMM with a bank of penalties for a batch of QPs (rows of q, l, u) that share P and A: checks every
    25 steps, the penalty rule and the nearest bank entry.  Returns x, z, lam, status, rho index."""
    P, A, q, l, u = (_dev(v) for v in (P, A, q, l, u))
    B, n = q.shape
    eq = (l[0] == u[0]).double() * 999.0 + 1.0
    eye = torch.eye(n, dtype=torch.float64, device="cuda")
    D = [torch.cholesky_inverse(torch.linalg.cholesky(P + SIGMA * eye + A.T @ ((r * eq)[:, None] * A))) for r in BANK]
    x = torch.zeros_like(q) if x is None else _dev(x)
    z = x @ A.T
    lam = torch.zeros_like(l) if lam is None else _dev(lam)
    ri = torch.zeros(B, dtype=torch.long, device="cuda") if ri is None else torch.as_tensor(ri, device="cuda").long()
    bank = torch.tensor(BANK, dtype=torch.float64, device="cuda")
    out = [torch.empty_like(x), torch.empty_like(z), torch.empty_like(lam), torch.ones(B, dtype=torch.int64), ri.clone()]
    live = torch.arange(B, device="cuda")
    it = 0
    while live.numel():
        for r in range(len(BANK)):
            g = (ri == r).nonzero()[:, 0]
            if not g.numel():
                continue
            rho = bank[r] * eq
            xg, zg, yg, lg, ug = x[g], z[g], lam[g], l[g], u[g]
            qg, W = q[g], D[r]
            for _ in range(CHECK):
                xg = (SIGMA * xg - qg + (rho * zg - yg) @ A) @ W
                ax = xg @ A.T
                zg = torch.minimum(torch.maximum(ax + yg / rho, lg), ug)
                yg = yg + rho * (ax - zg)
            x[g], z[g], lam[g] = xg, zg, yg
        it += CHECK
        ax, px, aty = x @ A.T, x @ P, lam @ A
        top = lambda v: v.abs().amax(1)  # noqa: E731
        rp, rd = top(ax - z), top(px + q + aty)
        done = (rp <= eps) & (rd <= eps)
        stop = done | (it >= most)
        k = stop.nonzero()[:, 0]
        if k.numel():
            at = live[k]
            out[0][at], out[1][at], out[2][at], out[4][at] = x[k], z[k], lam[k], ri[k]
            out[3][at.cpu()] = (~done[k]).long().cpu()
        num = rp * torch.maximum(torch.maximum(top(px), top(aty)), top(q).clamp_min(1e-4))
        den = rd * torch.maximum(top(ax), top(z)).clamp_min(1e-4)
        est = bank[ri] * torch.sqrt(num / den)
        near = (est.log()[:, None] - bank.log()[None, :]).abs().argmin(1)
        ri = torch.where((num > 0) & (den > 0) & torch.isfinite(est), near, ri)
        keep = (~stop).nonzero()[:, 0]
        x, z, lam, q, l, u, ri, live = (v[keep] for v in (x, z, lam, q, l, u, ri, live))
    return [v.cpu().numpy() for v in out]


# ---------------------------------------------------------------------------
# inputs of a case
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=8)
def _inputs(key, seed):
    """Host data of a case (the same for prepare() and exact())."""
    c = dict(key)
    rng = np.random.default_rng([7, seed])
    if c["kind"] == "step":
        p = _problem(c["nx"], c["nu"], c["N"], 0)
        last = p.std * rng.standard_normal((1, p.nx))
        x, _, lam, _, ri = _admm(p.P, p.A, *p.instance(last), 1e-3)
        # the plant's next state: the first control applied, with a disturbance
        K = -p.E[:p.nu]
        new = last @ p.Ad.T + (x[:, :p.nu] - last @ K.T) @ p.Bd.T + 0.1 * rng.standard_normal((1, p.nx))
        return p, p.instance(new), x[0], lam[0], int(ri[0])
    if c["kind"] == "batch":
        p = _problem(c["nx"], c["nu"], c["N"], c["extra"])
        X = (p.std * rng.standard_normal((c["B"], p.nx))).astype(np.float32)
        warm = None
        if c["warm"]:
            # every QP's last solution, for a state a disturbance away
            last = X + 0.1 * rng.standard_normal(X.shape)
            w = _admm(p.P, p.A, *p.instance(last.astype(np.float64)), 1e-3)
            warm = (w[0].astype(np.float32), w[2].astype(np.float32), w[4].astype(np.int32))
        rows = tuple(v.astype(np.float32) for v in p.instance(X.astype(np.float64))) if c["data"] == "rows" else None
        return p, X, rows, warm
    if c["kind"] == "served":
        fam = (_problem(12, 4, 20, 0), _problem(70, 30, 20, 400))
        which = np.ones(c["requests"], int)
        which[:max(1, min(c["requests"] - 1, round(c["share"] * c["requests"])))] = 0
        rng.shuffle(which)
        X = [(fam[f].std * rng.standard_normal(fam[f].nx)).astype(np.float32) for f in which]
        return fam, which, X
    if c["kind"] == "setup":
        p = _problem(c["nx"], c["nu"], c["N"], 0, 1 + seed % 1000003)
        return p, (p.std * rng.standard_normal((c["B"], p.nx))).astype(np.float32)
    A, B = _plant(rng, c["nx"], c["nu"], False)
    return A, B


def _key(case):
    return tuple(sorted((k, v) for k, v in case.items() if k != "name"))


def _batch_handle(p, B, precision):
    h = rq.ReluQP(p.P, p.A, p.l0, p.u0, sigma=SIGMA, rho_bank=BANK, max_batch=B,
                  precision=rq.PREC_BF16X3 if precision == "bf16x3" else rq.PREC_FP32)
    h.set_parametric(p.F, p.E, p.l0, p.u0)
    return h


def _outputs(B, p):
    return tuple(torch.empty(B, k, dtype=torch.float32, device="cuda") for k in (p.n, p.m, p.m))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "random":
        P, q, A, l, u = _random_qp(case["n"], seed)
        h = rq.ReluQP(P, A, l, u, sigma=SIGMA, rho_bank=BANK,
                      single_precision=rq.PREC_FP64 if case["precision"] == "fp64" else rq.PREC_FP64R)
        return {"kind": kind, "h": h, "q": q, "l": l, "u": u}
    got = _inputs(_key(case), seed)
    if kind == "step":
        p, (q, l, u), x, lam, ri = got
        h = rq.ReluQP(p.P, p.A, l[0], u[0], sigma=SIGMA, rho_bank=BANK)
        return {"kind": kind, "h": h, "q": q[0], "l": l[0], "u": u[0], "x": x, "lam": lam, "ri": ri}
    if kind == "batch":
        p, X, rows, warm = got
        dev = lambda t: None if t is None else tuple(torch.from_numpy(v.copy()).cuda() for v in t)  # noqa: E731
        return {"kind": kind, "h": _batch_handle(p, case["B"], case["precision"]), "X": torch.from_numpy(X.copy()).cuda(),
                "rows": dev(rows), "warm": dev(warm) or (None, None, None), "out": _outputs(case["B"], p)}
    if kind == "served":
        fam, which, X = got
        server = rq.Server([_batch_handle(fam[0], 128, "bf16x3"), _batch_handle(fam[1], 64, "bf16x3")])
        return {"kind": kind, "server": server, "which": [int(f) for f in which], "X": X}
    if kind == "setup":
        p, X = got
        return {"kind": kind, "p": p, "X": torch.from_numpy(X.copy()).cuda(), "out": _outputs(case["B"], p), "B": case["B"]}
    A, B = got
    one, big = np.ones(case["nu"]), np.full(case["nx"], 1e3)
    return {"kind": kind, "A": A, "B": B, "Q": np.eye(case["nx"]), "R": 0.1 * np.eye(case["nu"]), "N": case["N"],
            "lim": dict(umin=-one, umax=one, **(dict(xmin=-big, xmax=big) if case["state"] else {}))}


def _batched(s, h):
    r = h.solve_batch(X_warm=s["warm"][0], Lam_warm=s["warm"][1], rho_warm=s["warm"][2], eps_abs=1e-3,
                      max_iter=MAX_ITER, out=s["out"])
    return {"x": r["x"], "z": r["z"], "lam": r["lam"], "status": r["status"], "rho_index": r["rho_index"]}


def run(state):
    s, kind = state, state["kind"]
    if kind in ("step", "random"):
        h = s["h"]
        h.update(s["q"], s["l"], s["u"])
        if kind == "step":
            r = h.solve(x_warm=s["x"], lam_warm=s["lam"], rho_index=s["ri"], eps_abs=1e-3, max_iter=MAX_ITER)
        else:
            r = h.solve(eps_abs=1e-6, max_iter=MAX_ITER)
        return {"x": r["x"], "z": r["z"], "lam": r["lam"], "status": r["status"], "rho_index": r["rho_index"]}
    if kind == "batch":
        h = s["h"]
        if s["rows"] is not None:
            h.update_batch(*s["rows"])
        else:
            h.update_batch_x0(s["X"])
        return _batched(s, h)
    if kind == "served":
        server = s["server"]
        for tag, (f, x0) in enumerate(zip(s["which"], s["X"])):
            server.submit(f, x0, tag=tag)
        got = []
        while len(got) < len(s["which"]):
            server.step()
            got += server.poll(max_results=len(s["which"]))
        got.sort(key=lambda r: r["tag"])
        return {"x%d" % f: np.stack([r["x"] for r in got if r["family"] == f]) for f in (0, 1)} | {
            "status": np.array([r["status"] for r in got])}
    if kind == "setup":
        h = _batch_handle(s["p"], s["B"], "bf16x3")
        h.update_batch_x0(s["X"])
        r = _batched(dict(s, warm=(None, None, None)), h)
        h.close()
        return r
    return rq.condense_mpc(s["A"], s["B"], s["Q"], s["R"], s["N"], **s["lim"])


def exact(case, seed):
    """A single solve: the same iterate in 64 bits.  A batch: the QPs' solutions, since among hundreds of QPs some
    residual lies within rounding of the tolerance, and no 64-bit run stops at the check where the measured one
    does (the iterates' own rounding is far below the stop test's)."""
    kind = case["kind"]
    if kind == "random":
        P, q, A, l, u = _random_qp(case["n"], seed)
        r = _admm(P, A, q[None], l[None], u[None], 1e-6)
        return {"x": r[0][0], "z": r[1][0], "lam": r[2][0], "status": int(r[3][0]), "rho_index": int(r[4][0])}
    got = _inputs(_key(case), seed)
    if kind == "step":
        p, (q, l, u), x, lam, ri = got
        r = _admm(p.P, p.A, q, l, u, 1e-3, x[None], lam[None], [ri])
        return {"x": r[0][0], "z": r[1][0], "lam": r[2][0], "status": int(r[3][0]), "rho_index": int(r[4][0])}
    if kind in ("batch", "setup"):
        p, X = got[:2]
        rows = got[2] if kind == "batch" and got[2] is not None else p.instance(X.astype(np.float64))
        x, lam, ri = got[3] if kind == "batch" and got[3] is not None else (None, None, None)
        r = _admm(p.P, p.A, *rows, 1e-7, x, lam, ri, 40000)
        return {"x": r[0], "z": r[1], "lam": r[2], "status": None, "rho_index": None}
    if kind == "served":
        fam, which, X = got
        out = {"status": None}
        for f in (0, 1):
            p, at = fam[f], np.nonzero(which == f)[0]
            r = _admm(p.P, p.A, *p.instance(np.stack([X[i] for i in at]).astype(np.float64)), 1e-7, most=40000)
            out["x%d" % f] = r[0]
        return out
    A, B = got
    P, S, F, M, K = _condensed(A, B, case["N"])
    n, rows = case["N"] * case["nu"], None if case["state"] else case["N"] * case["nu"]
    lim = np.concatenate([np.ones(n)] + ([np.full(case["N"] * case["nx"], 1e3)] if case["state"] else []))
    return {"P": P.cpu().numpy(), "A": S[:rows].cpu().numpy(), "F": F.cpu().numpy(), "E": M[:rows].cpu().numpy(),
            "l0": -lim, "u0": lim, "K": K}


# ---------------------------------------------------------------------------
# work and tolerances
# ---------------------------------------------------------------------------
def work(case):
    """Layers as these problems take on average: about 50 for a warm-started step, 100 for a random QP,
    200 for a cold solve (75 with the wide limits).  One product of the (n + m)^2 layer each, in the width
    of the solve; the layer bank, or for a setup P and A, and the data and results once."""
    kind = case["kind"]
    if kind == "random":
        n = case["n"]
        R = n + 2 * max(1, n // 4)
        return {"bytes": 8.0 * (R * R + n * R + 4 * R), "flops": 100 * 2.0 * R * R}
    if kind == "served":
        a, b = 160, 1600
        ka, kb = case["requests"] * case["share"], case["requests"] * (1 - case["share"])
        return {"bytes": 4.0 * (a * a + b * b + ka * 100 + kb * 700), "flops": 2.0 * (150 * ka * a * a + 75 * kb * b * b)}
    nx, nu, N = case["nx"], case["nu"], case["N"]
    n = N * nu
    if kind == "condense":
        rows = N * (nu + (nx if case["state"] else 0))
        # the powers' blocks, and the upper triangle of S'HS with S block lower triangular
        return {"bytes": 8.0 * (nx * nx * 2 + nx * nu + n * n + rows * (n + nx) + n * nx),
                "flops": N * 2.0 * nx * nx * (nx + nu) + n * n * N * (nx + nu) / 3.0}
    m = n + case.get("extra", 0)
    R = n + m
    if kind == "step":
        return {"bytes": 4.0 * (R * R + n * (R + m) + 8 * R), "flops": 50 * 2.0 * R * R}
    if kind == "batch":
        B = case["B"]
        layers = 50 if case["warm"] else (75 if case["extra"] else 200)
        return {"bytes": 4.0 * (R * R + B * (2 * nx + n + 2 * m)), "flops": layers * 2.0 * R * R * B}
    # setup: per bank entry A'rho A, the factor, the inverse and A D A' (symmetric halves), D A'
    flops = len(BANK) * (m * n * n + n ** 3 + 3.0 * n * n * m)
    return {"bytes": 8.0 * (n * n + m * n) + 4.0 * len(BANK) * R * (R + n), "flops": flops + 200 * 2.0 * R * R * case["B"]}


def tolerance(case):
    """Solves: the stop tests' own resolution.  The same iterate differs by 3e-7 (plain limits) to 4e-5 (dense rows)
    in FP32 and by 1e-8 in the FP64 forms, but a QP whose residual lies within rounding of the tolerance may
    stop one check earlier or later.  Condensing: F, the gradient's matrix, cancels to 5e-10 of its terms."""
    if case["kind"] == "condense":
        return {"rel": 2e-9}
    if case["kind"] == "random":
        return {"rel": 1e-6}
    return {"rel": 1e-3, "max": 0.05, "differ": 0.01}
