"""Performance cases of the tensor-train solver: what a user's program has it do.

A case is one of
  points    hopf_eval_points on a state (probing Phi between steps);
  moments   hopf_eval_moments on a state (mean and covariance);
  rate      hopf_apply_op and the moments of G Phi (the initial rate of the
            moments, no rounding);
  step      one step of a scheme from a kept state, then what the user reads
            from the new state (moments of Phi, or values of the CDF);
  ensemble  hopf_step_ensemble: independent states advanced together, each on
            its own stream and share of the SMs;
  round     tt_sum of several states and tt_round (a stage sum made by hand);
  train     hopf_mlp_train: Adam steps of the surrogate network;
  predict   hopf_mlp_predict: a batch of surrogate queries.

States.  A solver state in use is smooth in every variable, vanishes at the
edge of the box and has bond spectra that decay towards the rounding
tolerance.  The cores made here are random combinations of Gaussian
characteristic functions exp(i mu a - s a^2 / 2) (Gaussian CDFs for the CDF
equation), with weights on the bonds that fall over `decay` decades: to near
the tolerance where the rank cap resolves the state, over one or two where
the cap binds long before (the largest configuration).  Every interior rank
is the given one, so a state sits at its rank cap as those of long solves do.

A TT's cores are determined only up to unitary factors on the bonds, so a
state is read through its values: moments, and values at grid points.
"""
import math

import numpy as np
import torch

from paper_2403_04946_gb300 import binding as B

BOX = 1.3  # half-width of the CDF equation's box
SCHEMES = {"rk4": B.HOPF_RK4, "euler": B.HOPF_EULER, "midpoint": B.HOPF_MIDPOINT}


# ---- the cases ---------------------------------------------------------------

def _step(name, d, n, r, tol, precision, scheme="rk4", dt=1.2e-5, nu=0.01, L=12.4, equation="phi", points=2048,
          decay=2.0):
    return {"name": name, "kind": "step", "d": d, "n": n, "r": r, "tol": tol, "decay": decay, "precision": precision,
            "scheme": scheme, "dt": dt, "nu": nu, "L": L, "equation": equation, "points": points}


def listed():
    return [
        # Probing Phi at a few points of a mid-size state between steps: the
        # smallest call, all latency.
        {"name": "points_c2", "kind": "points", "d": 16, "n": 64, "r": 32, "tol": 1e-9, "decay": 7.0, "nu": 0.02,
         "L": 12.4, "points": 64},
        # Mean and covariance of the largest configured state (d = 32,
        # n = 128, rank 64): read after every output interval.
        {"name": "moments_c3", "kind": "moments", "d": 32, "n": 128, "r": 64, "tol": 1e-7, "decay": 2.0,
         "nu": 0.01, "L": 12.4},
        # Initial rate of the moments (one operator apply), as every
        # surrogate query starts, at the mid-size configuration.
        {"name": "rate_c2", "kind": "rate", "d": 16, "n": 64, "r": 32, "tol": 1e-9, "decay": 7.0, "nu": 0.02,
         "L": 12.4},
        # One RK4 step of the small configuration in FP64 (d = 4, n = 24,
        # rank 16): the solves behind the surrogate's data set, step by step.
        _step("rk4_c1_fp64", 4, 24, 16, 1e-10, "fp64", dt=1e-3, nu=0.05, L=15.0, points=512, decay=9.0),
        # Eight such solves advanced together on shares of the SMs.
        {"name": "ensemble_c1", "kind": "ensemble", "members": 8, "d": 4, "n": 24, "r": 16, "tol": 1e-10,
         "decay": 9.0, "dt": 1e-2, "nu": 0.05, "L": 15.0, "points": 256},
        # One FP64 RK4 step of the mid-size configuration (n = 64, rank 32,
        # tol 1e-9), on eight of its sixteen modes.
        _step("rk4_c2_fp64", 8, 64, 32, 1e-9, "fp64", dt=5e-4, nu=0.02, decay=7.0),
        # The headline step (n = 128, rank 64, tol 1e-7) in FP64, on a slice
        # of its 32 modes.
        _step("rk4_c3_fp64", 4, 128, 64, 1e-7, "fp64"),
        # The headline step in mixed precision, on a longer slice.
        _step("rk4_c3_mixed", 6, 128, 64, 1e-7, "mixed"),
        # The paper's own workload: the CDF equation by the explicit midpoint
        # scheme at rank 128 (n = 64), mixed precision, on a slice of its 20
        # modes: factors of 6 r = 768 columns and more.
        _step("cdf_midpoint_mixed", 4, 64, 128, 1e-7, "mixed", scheme="midpoint", dt=1e-4, equation="cdf", L=BOX,
              decay=5.0),
        # A stage sum made by hand and rounded: three states of uneven, odd
        # ranks on an odd-sized problem, FP64.
        {"name": "sum_round_odd", "kind": "round", "d": 7, "n": 90, "r": 37, "terms": 3, "cap": 41, "tol": 1e-8,
         "decay": 6.0, "precision": "fp64", "nu": 0.02, "L": 12.4, "points": 512},
        # Training steps of the surrogate networks (26 -> 256 x 4 -> 14, four
        # members, batch 128).
        {"name": "surrogate_train", "kind": "train", "n_in": 26, "width": 256, "depth": 4, "n_out": 14, "members": 4,
         "batch": 128, "iters": 10, "samples": 1280},
        # A large batch of surrogate queries through the same networks.
        {"name": "surrogate_predict", "kind": "predict", "n_in": 26, "width": 256, "depth": 4, "n_out": 14,
         "members": 4, "queries": 4096},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw(rng):
    kind = rng.choice(["points", "moments", "rate", "step", "step", "step", "step", "ensemble", "round", "round",
                       "train", "predict"])
    if kind == "train":
        return {"kind": kind, "n_in": _log(rng, 12, 60), "width": _log(rng, 32, 256), "depth": rng.randint(2, 4),
                "n_out": _log(rng, 5, 44), "members": rng.randint(1, 4), "batch": _log(rng, 16, 512),
                "iters": rng.randint(4, 20), "samples": _log(rng, 512, 4096)}
    if kind == "predict":
        return {"kind": kind, "n_in": _log(rng, 12, 60), "width": _log(rng, 32, 256), "depth": rng.randint(2, 4),
                "n_out": _log(rng, 5, 44), "members": rng.randint(1, 4), "queries": _log(rng, 16, 8192)}
    n = 2 * _log(rng, 12, 64)
    c = {"kind": kind, "d": rng.randint(4, 16), "n": n, "r": _log(rng, 8, 64),
         "tol": 10.0 ** -rng.randint(7, 10), "decay": round(rng.uniform(1.0, 6.0), 2),
         "nu": round(rng.uniform(0.01, 0.1), 4), "L": 12.4}
    if kind in ("points", "moments", "rate"):
        if kind == "points":
            c["points"] = _log(rng, 16, 2048)
        return c
    c["points"] = _log(rng, 64, 1024)
    if kind == "ensemble":
        c.update(members=rng.randint(2, 16), d=rng.randint(3, 5), n=2 * _log(rng, 8, 16), r=_log(rng, 6, 20),
                 tol=1e-10, decay=9.0, dt=1e-3, L=15.0)
        return c
    if kind == "round":
        c.update(d=rng.randint(3, 9), terms=rng.randint(2, 5), cap=_log(rng, 8, 64),
                 precision=rng.choice(["fp64", "mixed"]))
        return c
    c.update(d=rng.randint(3, 8), precision=rng.choice(["fp64", "mixed"]), equation="phi",
             scheme=rng.choice(["rk4", "rk4", "euler", "midpoint"]), dt=1.2e-5)
    if rng.random() < 0.25:
        c.update(equation="cdf", scheme=rng.choice(["euler", "midpoint"]), dt=1e-4, L=BOX, n=min(c["n"], 64))
    if c["precision"] == "mixed":
        c["tol"] = max(c["tol"], 1e-7)
    return c


def draw(rng):
    # the costliest listed case of each precision bounds the drawn ones
    most = {p: max(work(c)["flops"] for c in listed() if c.get("precision", "fp64") == p and c["kind"] == "step")
            for p in ("fp64", "mixed")}
    while True:
        c = _draw(rng)
        if c["kind"] in ("train", "predict") or work(c)["flops"] <= most[c.get("precision", "fp64")]:
            return c


# ---- inputs --------------------------------------------------------------------

def _ranks(d, n, r):
    return [min(r, n ** min(k, d - k, 4)) for k in range(d + 1)]


def _grid(c):
    """Grid of one variable and its spacing."""
    n = c["n"]
    if c.get("equation") == "cdf":
        du = 2.0 * BOX / (n - 1)
        return -BOX + np.arange(n) * du, du
    da = 2.0 * c["L"] / n
    return (np.arange(n) - n // 2) * da, da


def _cores(c, r, seed):
    """Cores (r_{k-1}, n, r_k) of one state (module docstring)."""
    rng = np.random.default_rng(seed)
    d, n = c["d"], c["n"]
    x, _ = _grid(c)
    ranks = _ranks(d, n, r)
    cores = []
    for k in range(d):
        a, b = ranks[k], ranks[k + 1]
        g = (rng.standard_normal((a, b)) + 1j * rng.standard_normal((a, b))) / math.sqrt(2.0)
        mu, s = rng.normal(0.0, 0.5, (a, b)), rng.uniform(0.15, 0.35, (a, b))
        if c.get("equation") == "cdf":
            z = (x[None, :, None] - mu[:, None, :]) / (np.sqrt(2.0 * s)[:, None, :])
            f = 0.5 * torch.special.erfc(torch.from_numpy(-z)).numpy() + 0j
        else:
            f = np.exp(1j * mu[:, None, :] * x[None, :, None] - 0.5 * s[:, None, :] * (x * x)[None, :, None])
            f[:, 0, :] = 0.0  # the box boundary
        w = np.ones(b)
        if b > 1:
            w = 10.0 ** (-c["decay"] * np.arange(b) / (b - 1.0))
            w /= np.linalg.norm(w)
        cores.append(np.asfortranarray(g[:, None, :] * f * w[None, None, :]))
    return cores


def _points(c, seed):
    rng = np.random.default_rng(seed + 77)
    n = c["n"]
    lo, hi = (0, n) if c.get("equation") == "cdf" else (n // 2 - n // 4, n // 2 + n // 4)
    return rng.integers(lo, hi, size=(c["points"], c["d"])).astype(np.int32)


def _term_ranks(c):
    """Uneven ranks of the terms of a sum, the largest c['r']."""
    return [max(1, c["r"] - 6 * t) for t in range(c["terms"])]


def _mlp(c, seed):
    rng = np.random.default_rng(seed)
    dims = [c["n_in"]] + [c["width"]] * c["depth"] + [c["n_out"]]
    init = np.stack([np.concatenate([np.concatenate([rng.normal(0.0, math.sqrt(2.0 / fi), fi * fo), np.zeros(fo)])
                                     for fi, fo in zip(dims[:-1], dims[1:])]) for _ in range(c["members"])])
    ns = c.get("samples", 1024)
    x = rng.normal(size=(ns, c["n_in"])) * rng.uniform(0.1, 3.0, c["n_in"]) + rng.normal(size=c["n_in"])
    y = np.tanh(x @ rng.normal(0.0, 0.3, (c["n_in"], c["n_out"]))) + 0.1 * rng.normal(size=(ns, c["n_out"]))
    return dims, init.astype(np.float32), x, y, rng


class _State:
    """Contexts, tensors and networks of a case, released with it."""

    def __init__(self, case):
        self.case, self.ctxs, self.tts, self.nets = case, [], [], []

    def context(self, rank_cap, stream=None):
        c = self.case
        ctx = B.Context(d=c["d"], n=c["n"], nu=c["nu"], tol=c["tol"], rank_cap=rank_cap, L=c["L"], stream=stream,
                        precision=B.HOPF_MIXED if c.get("precision") == "mixed" else B.HOPF_FP64)
        if c.get("equation") == "cdf":
            ctx.hopf_set_equation(B.HOPF_EQ_CDF, BOX)
        self.ctxs.append(ctx)
        return ctx

    def tensor(self, ctx, cores=None, cap=None):
        t = ctx.tt_create(cap) if cores is None else ctx.tt_from_host(cores, max_rank=cap)
        self.tts.append((ctx, t))
        return t

    def __del__(self):
        for net in self.nets:
            net.close()
        for ctx, t in self.tts:
            ctx.tt_free(t)
        for ctx in self.ctxs:
            ctx.close()


def prepare(case, seed):
    c, s = case, _State(case)
    kind = c["kind"]
    if kind in ("train", "predict"):
        ctx = B.Context(d=4, n=8, nu=0.05, tol=1e-10, rank_cap=4, L=3.0)
        s.ctxs.append(ctx)
        dims, init, x, y, rng = _mlp(c, seed)
        net = B.Mlp(ctx, dims[0], c["width"], c["depth"], dims[-1], c["members"],
                    c["batch"] if kind == "train" else 4096, init)
        s.nets.append(net)
        net.set_data(x, y)
        if kind == "train":
            s.idx = rng.integers(0, len(x), size=(c["iters"], c["members"], c["batch"])).astype(np.int32)
            s.lr = np.full(c["iters"], 1e-3, dtype=np.float32)
        else:
            s.x = x[rng.integers(0, len(x), c["queries"])] + 0.01 * rng.normal(size=(c["queries"], c["n_in"]))
        return s
    if kind == "ensemble":
        m = c["members"]
        share = torch.cuda.get_device_properties(torch.cuda.current_device()).multi_processor_count // m
        s.streams = [torch.cuda.Stream() for _ in range(m)]
        s.members, s.kept = [], []
        for k, st in enumerate(s.streams):
            ctx = s.context(c["r"], stream=st.cuda_stream)
            ctx.hopf_set_max_ctas(share)
            s.kept.append(s.tensor(ctx, _cores(c, c["r"], 1000 * seed + k), c["r"]))
            s.members.append((ctx, s.tensor(ctx, cap=c["r"])))
        s.idx = _points(c, seed)
        return s
    if kind == "round":
        ranks = _term_ranks(c)
        ctx = s.context(c["cap"])
        s.terms = [s.tensor(ctx, _cores(c, r, 1000 * seed + k), r) for k, r in enumerate(ranks)]
        s.out = s.tensor(ctx, cap=sum(ranks))
        s.coefs = np.exp(1j * np.arange(len(ranks)))
        s.idx = _points(c, seed)
        return s
    ctx = s.context(c["r"])
    s.t = s.tensor(ctx, _cores(c, c["r"], seed), c["r"])
    if kind == "rate":
        s.g = s.tensor(ctx, cap=6 * c["r"])
    if kind == "step":
        s.next = s.tensor(ctx, cap=c["r"])
    if "points" in c:
        s.idx = _points(c, seed)
    return s


def run(s):
    c, kind = s.case, s.case["kind"]
    if kind == "train":
        loss = s.nets[0].train(s.idx, s.lr)
        return {"loss": loss, "params": s.nets[0].get_params()}
    if kind == "predict":
        y, bound, members = s.nets[0].predict(s.x, 1.0, members=True)
        return {"y": y, "bound": bound, "members": members}
    if kind == "ensemble":
        for (ctx, t), kept in zip(s.members, s.kept):
            ctx.tt_copy(kept, t)
        B.hopf_step_ensemble(s.members, c["dt"], 1)
        out = []
        for ctx, t in s.members:
            mean, cov, _ = ctx.hopf_eval_moments(t)
            out.append({"mean": mean, "cov": cov, "phi": ctx.hopf_eval_points(t, s.idx)})
        return out
    ctx = s.ctxs[0]
    if kind == "points":
        return {"phi": ctx.hopf_eval_points(s.t, s.idx)}
    if kind == "moments":
        mean, cov, _ = ctx.hopf_eval_moments(s.t)
        return {"mean": mean, "cov": cov}
    if kind == "rate":
        ctx.hopf_apply_op(s.t, s.g)
        mean, cov, _ = ctx.hopf_eval_moments(s.g)
        return {"mean": mean, "cov": cov}
    if kind == "round":
        ctx.tt_sum(s.terms, s.coefs, s.out)
        ctx.tt_round(s.out, c["tol"], c["cap"])
        return {"phi": ctx.hopf_eval_points(s.out, s.idx)}
    ctx.tt_copy(s.t, s.next)  # the kept state stays for the next pass
    ctx.hopf_step_scheme(s.next, SCHEMES[c["scheme"]], c["dt"], 1)
    out = {"phi": ctx.hopf_eval_points(s.next, s.idx)}
    if c["equation"] == "phi":
        out["mean"], out["cov"], _ = ctx.hopf_eval_moments(s.next)
    return out


# ---- the work of a pass -----------------------------------------------------------

def _tt_bytes(d, n, r):
    q = _ranks(d, n, r)
    return 16.0 * sum(q[k] * n * q[k + 1] for k in range(d))


def _round_flops(d, n, rin, cap):
    """Householder sweeps of one rounding from interior rank rin to cap:
    QR of every flattening, its Q applied, QR of the projected flattening,
    bidiagonalisation of the factor, the projection (complex arithmetic, 8
    real operations per multiply-add)."""
    qr = lambda m, k: 8.0 * m * k * k - 8.0 * k ** 3 / 3.0 if m >= k else 8.0 * k * m * m - 8.0 * m ** 3 / 3.0
    rin_k = [1] + [rin] * (d - 1) + [1]
    p, total = [1] * (d + 1), 0.0
    for k in range(d - 1, 0, -1):
        m = n * p[k + 1]
        p[k] = min(m, rin_k[k])
        total += qr(m, rin_k[k]) + 8.0 * rin_k[k - 1] * n * rin_k[k] * p[k]
    rho = 1
    for k in range(d - 1):
        m = rho * n
        pp = min(m, p[k + 1])
        new = min(cap, pp)
        total += qr(m, p[k + 1]) + 32.0 * pp ** 3 / 3.0 + 16.0 * m * new * pp - 8.0 * new * pp * pp
        total += 8.0 * new * pp * p[k + 1]
        mq = n * p[k + 2] if k + 2 <= d else n
        total += 16.0 * mq * new * p[k + 1] - 8.0 * new * p[k + 1] ** 2
        rho = new
    return total


def work(case):
    c, kind = case, case["kind"]
    if kind in ("train", "predict"):
        dims = [c["n_in"]] + [c["width"]] * c["depth"] + [c["n_out"]]
        params = sum((a + 1) * b for a, b in zip(dims[:-1], dims[1:]))
        mac = sum(a * b for a, b in zip(dims[:-1], dims[1:]))
        if kind == "train":
            rows = c["batch"] * c["iters"]
            return {"bytes": c["members"] * (4.0 * 7 * params * c["iters"] + 4.0 * rows * (dims[0] + dims[-1])),
                    "flops": 6.0 * c["members"] * rows * mac}
        return {"bytes": 4.0 * c["members"] * params + 8.0 * c["queries"] * (dims[0] + dims[-1] * (1 + c["members"])),
                "flops": 2.0 * c["members"] * c["queries"] * mac}
    d, n, r = c["d"], c["n"], c["r"]
    state = _tt_bytes(d, n, r)
    if kind in ("points", "moments"):
        npts = c["points"] if kind == "points" else 1 + 2 * d * d
        return {"bytes": min(state, npts * state / n), "flops": 8.0 * npts * d * r * r}
    if kind == "rate":
        return {"bytes": state + 36.0 * state, "flops": 36.0 * 8.0 * state / 16.0}
    if kind == "round":
        ranks = _term_ranks(c)
        return {"bytes": sum(_tt_bytes(d, n, q) for q in ranks) + _tt_bytes(d, n, c["cap"]),
                "flops": _round_flops(d, n, sum(ranks), c["cap"])}
    if kind == "ensemble":
        one = 4.0 * _round_flops(d, n, 6 * r, r) + 3.0 * _round_flops(d, n, 2 * r, r) + _round_flops(d, n, 5 * r, r)
        return {"bytes": c["members"] * 2.0 * state, "flops": c["members"] * one}
    flops = {"rk4": [6, 6, 6, 6, 2, 2, 2, 5], "euler": [6, 2], "midpoint": [6, 12, 2]}[c["scheme"]]
    return {"bytes": 2.0 * state, "flops": sum(_round_flops(d, n, m * r, r) for m in flops)}


# ---- the same in 64 bits, by torch and numpy alone ------------------------------------

_DEV = "cuda" if torch.cuda.is_available() else "cpu"


def _up(cores):
    return [torch.from_numpy(np.ascontiguousarray(x)).to(_DEV) for x in cores]


def _operator(c):
    """Matrix-product form of the generator: {(alpha, beta): n x n} per site."""
    d, n, nu = c["d"], c["n"], c["nu"]
    x, dx = _grid(c)
    h = 2.0 * math.pi / d
    e = nu / h ** 2
    eye = np.eye(n)
    A, D, S, J = np.diag(x), np.zeros((n, n)), np.zeros((n, n)), np.zeros((n, n))
    for i in range(n):
        S[i, i] = -2.0 / dx ** 2
        for j, sign in ((i - 1, -1.0), (i + 1, 1.0)):
            if 0 <= j < n:
                D[i, j], S[i, j] = sign / (2.0 * dx), 1.0 / dx ** 2
    if c.get("equation") == "cdf":
        D[0, :] = D[-1, :] = 0.0
        for k in range(1, n):
            J[k, 0] = J[k, k] = dx / 2.0
            J[k, 1:k] = dx
        K, AD = A - J, A @ D
        P, Q, Z = AD / (2.0 * h) - e * D, -AD / (2.0 * h) - e * D, 2.0 * e * AD
        first = [eye, P, K, Z, K, Q]
        last = [Z, K, Q, eye, P, K]
    else:
        for M in (A, D, S):
            M[0, :] = 0.0
            M[:, 0] = 0.0
        P, Q, Z = 1j / (4.0 * h) * S + e * D, -1j / (4.0 * h) * S + e * D, -2.0 * e * (A @ D)
        first = [eye, A, Q, Z, P, A]
        last = [Z, P, A, eye, A, Q]
    mid = {(0, b): first[b] for b in range(4)}
    mid.update({(1, 3): last[1], (2, 3): last[2], (3, 3): eye, (4, 4): eye, (5, 5): eye})
    sites = [{(0, b): first[b] for b in range(6)}] + [mid] * (d - 2) + [{(a, 0): last[a] for a in range(6)}]
    return [{k: torch.from_numpy(np.asarray(v, dtype=complex)).to(_DEV) for k, v in w.items()} for w in sites]


def _apply(cores, W):
    out = []
    for k, (X, w) in enumerate(zip(cores, W)):
        a, n, b = X.shape
        na, nb = (1 if k == 0 else 6), (1 if k == len(cores) - 1 else 6)
        Y = torch.zeros((na, a, n, nb, b), dtype=X.dtype, device=X.device)
        for (al, be), M in w.items():
            Y[al, :, :, be, :] = torch.einsum("mp,ipj->imj", M, X)
        out.append(Y.reshape(na * a, n, nb * b))
    return out


def _sum(terms):
    out, d = [], len(terms[0][1])
    for k in range(d):
        a = 1 if k == 0 else sum(t[k].shape[0] for _, t in terms)
        b = 1 if k == d - 1 else sum(t[k].shape[2] for _, t in terms)
        Y = torch.zeros((a, terms[0][1][k].shape[1], b), dtype=torch.complex128, device=_DEV)
        i = j = 0
        for co, t in terms:
            x = t[k] * co if k == 0 else t[k]
            Y[i:i + x.shape[0], :, j:j + x.shape[2]] = x
            i += x.shape[0] if k > 0 else 0
            j += x.shape[2] if k < d - 1 else 0
        out.append(Y)
    return out


def _round(cores, tol, cap):
    Y, d = list(cores), len(cores)
    for k in range(d - 1, 0, -1):
        a, n, b = Y[k].shape
        q, r = torch.linalg.qr(Y[k].reshape(a, n * b).mH)
        Y[k] = q.mH.reshape(-1, n, b)
        Y[k - 1] = torch.einsum("inj,jk->ink", Y[k - 1], r.mH)
    eps = tol * float(torch.linalg.norm(Y[0])) / math.sqrt(d - 1)
    for k in range(d - 1):
        a, n, b = Y[k].shape
        q, r = torch.linalg.qr(Y[k].reshape(a * n, b))
        u, s, vh = np.linalg.svd(r.cpu().numpy(), full_matrices=False)
        tail = np.sqrt(np.concatenate([np.cumsum((s ** 2)[::-1])[::-1], [0.0]]))
        rho = min(max(1, int(np.argmax(tail <= eps))), cap)
        Y[k] = (q @ torch.from_numpy(np.ascontiguousarray(u[:, :rho])).to(_DEV)).reshape(a, n, rho)
        sv = torch.from_numpy(s[:rho, None] * vh[:rho]).to(_DEV)
        Y[k + 1] = torch.einsum("ij,jnk->ink", sv, Y[k + 1])
    return Y


def _values(cores, idx):
    v = torch.ones((len(idx), 1, 1), dtype=torch.complex128, device=_DEV)
    at = torch.from_numpy(np.asarray(idx, dtype=np.int64)).to(_DEV)
    for k, X in enumerate(cores):
        v = v @ X[:, at[:, k], :].permute(1, 0, 2)
    return v[:, 0, 0].cpu().numpy()


def _moments(c, cores):
    d, mid = c["d"], c["n"] // 2
    da = 2.0 * c["L"] / c["n"]
    pts, where = [], {}

    def at(*offsets):
        p = [mid] * d
        for k, o in offsets:
            p[k] += o
        return where.setdefault(tuple(p), len(where))

    plan = [[at()]] + [[at((k, 1)), at((k, -1))] for k in range(d)]
    pairs = {(j, k): [at((j, p), (k, q)) for p in (1, -1) for q in (1, -1)] for j in range(d) for k in range(j + 1, d)}
    pts = np.array(list(where), dtype=np.int64)
    v = np.concatenate([_values(cores, pts[i:i + 256]) for i in range(0, len(pts), 256)])
    mean = np.array([(-1j * (v[p] - v[q]) / (2.0 * da)).real for p, q in plan[1:]])
    second = np.zeros((d, d))
    for k in range(d):
        p, q = plan[1 + k]
        second[k, k] = -((v[p] - 2.0 * v[0] + v[q]) / da ** 2).real
    for (j, k), (pp, pm, mp, mm) in pairs.items():
        second[j, k] = second[k, j] = -((v[pp] - v[pm] - v[mp] + v[mm]) / (4.0 * da ** 2)).real
    return mean, second - np.outer(mean, mean)


def _advance(c, f):
    W, dt, T = _operator(c), c["dt"], lambda x: _round(x, c["tol"], c["r"])
    G = lambda x: _apply(x, W)
    k1 = T(G(f))
    scheme = c.get("scheme", "rk4")
    if scheme == "euler":
        return T(_sum([(1.0, f), (dt, k1)]))
    if scheme == "midpoint":
        return T(_sum([(1.0, f), (dt, T(G(_sum([(1.0, f), (dt / 2, k1)]))))]))
    k2 = T(G(T(_sum([(1.0, f), (dt / 2, k1)]))))
    k3 = T(G(T(_sum([(1.0, f), (dt / 2, k2)]))))
    k4 = T(G(T(_sum([(1.0, f), (dt, k3)]))))
    return T(_sum([(1.0, f), (dt / 6, k1), (dt / 3, k2), (dt / 3, k3), (dt / 6, k4)]))


def _bf16(w):
    return w.to(torch.float32).to(torch.bfloat16).to(torch.float64)


def _net(p, x, dims):
    """Output of one network whose weights are used as BF16 values."""
    off, h = 0, x
    for l, (fi, fo) in enumerate(zip(dims[:-1], dims[1:])):
        w, b = p[off:off + fi * fo].reshape(fo, fi), p[off + fi * fo:off + fi * fo + fo]
        off += fi * fo + fo
        # straight through the rounding: the gradient is taken at the rounded weights
        h = h @ (w + (_bf16(w.detach()) - w.detach())).T + b
        if l < len(dims) - 2:
            h = torch.nn.functional.gelu(h)
    return h


def _exact_mlp(c, seed):
    dims, init, x, y, rng = _mlp(c, seed)
    stats = lambda a: (a.mean(0), np.where(a.std(0) > 0, a.std(0), 1.0))
    (mx, sx), (my, sy) = stats(x), stats(y)
    up = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).to(_DEV)
    if c["kind"] == "predict":
        q = x[rng.integers(0, len(x), c["queries"])] + 0.01 * rng.normal(size=(c["queries"], c["n_in"]))
        m = np.stack([my + sy * _net(up(p), up((q - mx) / sx), dims).cpu().numpy() for p in init])
        ybar = m.mean(0)
        spread = np.sqrt(((m - ybar) ** 2).mean(0))
        return {"y": ybar, "bound": np.linalg.norm(spread, axis=1) / np.linalg.norm(ybar, axis=1), "members": m}
    idx = rng.integers(0, len(x), size=(c["iters"], c["members"], c["batch"])).astype(np.int64)
    lr = float(np.float32(1e-3))
    X, Y = up((x - mx) / sx), up((y - my) / sy)
    losses, params = np.zeros((c["iters"], c["members"])), []
    for e in range(c["members"]):
        p = up(init[e]).requires_grad_(True)
        m, v = torch.zeros_like(p), torch.zeros_like(p)
        for t in range(c["iters"]):
            at = torch.from_numpy(idx[t, e]).to(_DEV)
            loss = ((_net(p, X[at], dims) - Y[at]) ** 2).mean()
            g, = torch.autograd.grad(loss, p)
            losses[t, e] = float(loss.detach())
            with torch.no_grad():
                m = 0.9 * m + 0.1 * g
                v = 0.999 * v + 0.001 * g * g
                p -= lr * (m / (1 - 0.9 ** (t + 1))) / (torch.sqrt(v / (1 - 0.999 ** (t + 1))) + 1e-8)
        params.append(p.detach().cpu().numpy())
    return {"loss": losses, "params": np.stack(params)}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("train", "predict"):
        return _exact_mlp(c, seed)
    if kind == "ensemble":
        out = []
        for k in range(c["members"]):
            f = _advance(c, _up(_cores(c, c["r"], 1000 * seed + k)))
            mean, cov = _moments(c, f)
            out.append({"mean": mean, "cov": cov, "phi": _values(f, _points(c, seed))})
        return out
    if kind == "round":
        ranks = _term_ranks(c)
        co = np.exp(1j * np.arange(len(ranks)))
        f = _sum([(complex(z), _up(_cores(c, r, 1000 * seed + k))) for k, (z, r) in enumerate(zip(co, ranks))])
        return {"phi": _values(_round(f, c["tol"], c["cap"]), _points(c, seed))}
    f = _up(_cores(c, c["r"], seed))
    if kind == "points":
        return {"phi": _values(f, _points(c, seed))}
    if kind in ("moments", "rate"):
        mean, cov = _moments(c, _apply(f, _operator(c)) if kind == "rate" else f)
        return {"mean": mean, "cov": cov}
    if c.get("equation") == "cdf" and c["r"] > 64:
        return None  # factors of rank 12 r: more than a reference in 64 bits does in the time
    f = _advance(c, f)
    out = {"phi": _values(f, _points(c, seed))}
    if c["equation"] == "phi":
        out["mean"], out["cov"] = _moments(c, f)
    return out
