"""Timed cases: the calls that a user of the library makes, over the sizes it is used at.

Each case is one of five kinds of call:

* ``pf``       particle-filter log-likelihoods of N parameter vectors on a context
               (``SMC2.pf_loglik``), for the three models, both precisions, the
               default filter and the paper's (multinomial below ESS M/2);
* ``noalloc``  the same through the allocation-free entry point;
* ``run``      a whole SMC^2 run on a context (reset, K iterations, statistics,
               final population, recycled estimate), with the random-walk or the
               learned proposal, one dataset or several;
* ``train``    the surrogate network's training call;
* ``resample`` the systematic resampling primitive.

Observations, parameters and weights are simulated from the seed.  ``exact``
evaluates the same calls in 64 bits with torch alone, on the same random
numbers; a run or a binomial filter in mixed precision has no such value,
because a rounding moves a resampling decision or a binomial draw and the run
then follows other random numbers.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2311_12973_gb300 import inputs as I
from paper_2311_12973_gb300 import smc2 as S

BASE = {"lg": "lg_t50_n64", "seir": "seir_t100_n1024", "sir": "sir_t30_n1024"}
# algorithmic lane operations per particle-step: each model with the default filter
# (systematic resampling every step) and with the paper's
OPS = {"lg": (67.0, 87.0), "seir": (108.0, 128.0), "sir": (242.0, 276.0)}
# rough cost of a particle-step against the mixed-precision default filter's, for the sizes of drawn cases
COST = {("lg", "mixed"): 1, ("lg", "fp64"): 25, ("seir", "mixed"): 1, ("seir", "fp64"): 40,
        ("sir", "mixed"): 15, ("sir", "fp64"): 500}
MAX_COST = 2.1e9


def listed():
    return [
        # A whole run of the smallest benchmark configuration: 64 filters, FP64, launch and latency bound.
        {"name": "lg_fp64_run", "kind": "run", "model": "lg", "precision": "fp64", "paper": False,
         "learned": False, "datasets": 1, "N": 64, "M": 128, "T": 50, "K": 10},
        # The smallest call in use: a few filters from a program that owns all device memory itself.
        {"name": "lg_fp64_noalloc_small", "kind": "noalloc", "model": "lg", "precision": "fp64", "paper": False,
         "N": 8, "M": 100, "T": 20},
        # The resampling primitive at an odd size, as a program with its own weights calls it.
        {"name": "resample_odd", "kind": "resample", "n": 10007},
        # Scoring a ragged set of parameters with ragged filters, mixed precision.
        {"name": "seir_mixed_pf_ragged", "kind": "pf", "model": "seir", "precision": "mixed", "paper": False,
         "N": 1001, "M": 300, "T": 73},
        # The main benchmark configuration as a user runs it: SEIR-type, mixed precision, 20 iterations.
        {"name": "seir_mixed_run", "kind": "run", "model": "seir", "precision": "mixed", "paper": False,
         "learned": False, "datasets": 1, "N": 1024, "M": 512, "T": 100, "K": 20},
        # One iteration's filters of the largest configuration (the benchmark headline).
        {"name": "seir_mixed_pf_large", "kind": "pf", "model": "seir", "precision": "mixed", "paper": False,
         "N": 8192, "M": 1024, "T": 200},
        # The plain FP64 form of the main configuration.
        {"name": "seir_fp64_pf", "kind": "pf", "model": "seir", "precision": "fp64", "paper": False,
         "N": 1024, "M": 512, "T": 100},
        # Several datasets of uneven length and size in one context.
        {"name": "seir_batched_run", "kind": "run", "model": "seir", "precision": "mixed", "paper": False,
         "learned": False, "datasets": 12, "N": 0, "M": 0, "T": 0, "K": 3},
        # The paper's own experiment, its filter (multinomial below ESS M/2), both precisions.
        {"name": "sir_mixed_pf", "kind": "pf", "model": "sir", "precision": "mixed", "paper": True,
         "N": 1024, "M": 500, "T": 30},
        {"name": "sir_fp64_pf", "kind": "pf", "model": "sir", "precision": "fp64", "paper": True,
         "N": 256, "M": 500, "T": 30},
        # The learned proposal: the network trains beside the sampler.
        {"name": "seir_learned_run", "kind": "run", "model": "seir", "precision": "mixed", "paper": False,
         "learned": True, "datasets": 1, "N": 1024, "M": 512, "T": 100, "K": 20},
        # The training call alone, on the rows of four iterations of 1024 samples.
        {"name": "train_ring", "kind": "train", "D": 4, "R": 4096, "steps": 16},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _whole_groups(M):
    """Whether a filter of M particles fills a power of two of threads at 1, 2 or 4 particles each:
    the shapes that a context takes for the paper's filter and the SIR model."""
    groups = [-(-M // (32 * ppt)) for ppt in (1, 2, 4)]
    return any(g & (g - 1) == 0 for g in groups)


def draw(rng):
    kind = rng.choices(["pf", "noalloc", "run", "train", "resample"], [12, 2, 3, 1, 2])[0]
    if kind == "resample":
        return {"kind": kind, "n": _log_int(rng, 32, 16384)}
    if kind == "train":
        return {"kind": kind, "D": rng.choice([2, 3, 4]), "R": _log_int(rng, 256, 8192),
                "steps": rng.choice([1, 4, 16, 32])}
    while True:
        model = rng.choice(["lg", "seir", "seir", "sir"])
        c = {"kind": kind, "model": model, "precision": rng.choice(["mixed", "mixed", "fp64"]),
             "paper": rng.random() < 0.8 if model == "sir" else rng.random() < 0.15,
             "N": _log_int(rng, 1, 8192), "M": _log_int(rng, 16, 1024), "T": _log_int(rng, 5, 400)}
        if model == "sir":
            c["T"] = min(c["T"], 100)
        if kind != "noalloc" and (model == "sir" or c["paper"]) and not _whole_groups(c["M"]):
            continue
        if kind == "noalloc":
            c["N"] = min(c["N"], 1024)
        if kind == "run":
            c.update(learned=model == "seir" and c["precision"] == "mixed" and rng.random() < 0.3, datasets=1,
                     N=_log_int(rng, 64, 4096), K=rng.randint(2, 12))
            if c["learned"]:
                c["N"], c["paper"] = min(c["N"], 2048), False
        if COST[model, c["precision"]] * c["N"] * c["M"] * c["T"] * c.get("K", 1) <= MAX_COST:
            return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _workload(case, seed):
    # the LG and SEIR workloads run the default filter unless the case asks for the paper's
    over = {"pf_scheme": I.PF_MULTINOMIAL, "pf_ess_frac": 0.5} if case["paper"] else \
        {"pf_scheme": I.PF_SYSTEMATIC, "pf_ess_frac": 0.0}
    if case.get("learned"):
        over["proposal"] = I.PROP_MLP
    if case["precision"] == "mixed" and case["model"] != "sir" and not case["paper"]:
        # the FP32 filter, as a program asks for that wants the same numbers on every machine
        # (the other kernel rounds differently, and the tuner picks by time)
        over["pf_family"] = S.PF_FP32
    return I.workload(BASE[case["model"]], N=case["N"], M=case["M"], T=case["T"], K=case.get("K", 1),
                      precision=I.PREC_FP64 if case["precision"] == "fp64" else I.PREC_MIXED,
                      seed=1 + seed % 1000003, data_seed=seed, **over)


def _datasets(case, seed):
    # the sizes are the workload's own; the data and the sampler's random numbers are the seed's
    return [w.with_(pf_family=S.PF_FP32, data_seed=seed + w.dataset, seed=1 + seed % 1000003)
            for w in I.batched_workloads(case["datasets"], K=case["K"])]


def _theta(w, seed):
    """Draws about the prior's centre, as narrow as a population after a few iterations; the
    uniform prior's whole support for the SIR model."""
    return I.theta_near_prior(w, w.N, seed + 1, 1.0 if w.model == I.SIR else 0.3)


def _weights(n, seed):
    rng = np.random.default_rng(seed)
    lw = 2.0 * rng.standard_normal(n)
    bits = min(52, 63 - (0 if n <= 1 else (n - 1).bit_length()))
    q = np.floor(np.exp(lw - lw.max()) * 2.0 ** bits).astype(np.int64)
    return q, int(rng.integers(0, 2 ** 32))


def _ring(case, seed):
    """Rows (theta, log pi^) as the sampler stores them, and a network's initial state."""
    rng = np.random.default_rng(seed)
    D, R, H = case["D"], case["R"], 64
    th = 0.5 * rng.standard_normal((R, D)) - 1.0
    lp = -400.0 - 30.0 * ((th + 1.0) ** 2).sum(1) + 2.0 * rng.standard_normal(R)
    parts = [rng.uniform(-1, 1, (D, H)) * math.sqrt(6.0 / (D + H)), np.zeros(H),
             rng.uniform(-1, 1, (H, H)) * math.sqrt(3.0 / H), np.zeros(H),
             rng.uniform(-1, 1, H) * math.sqrt(6.0 / (H + 1)), np.zeros(1)]
    f32 = lambda a: np.ascontiguousarray(a, dtype=np.float32)  # noqa: E731
    return f32(th), f32(lp), f32(np.concatenate([a.reshape(-1) for a in parts]))


def prepare(case, seed):
    kind = case["kind"]
    dev = torch.device("cuda")
    if kind == "resample":
        q, U = _weights(case["n"], seed)
        return {"kind": kind, "q": torch.from_numpy(q).to(dev), "U": U,
                "anc": torch.empty(case["n"], dtype=torch.int32, device=dev)}
    if kind == "train":
        th, lp, p = (torch.from_numpy(a).to(dev) for a in _ring(case, seed))
        return {"kind": kind, "th": th, "lp": lp, "p": p, "m": torch.zeros_like(p), "v": torch.zeros_like(p),
                "step": torch.zeros(1, dtype=torch.int32, device=dev), "steps": case["steps"]}
    if kind == "run" and case["datasets"] > 1:
        ws = _datasets(case, seed)
        ctx = S.SMC2(S.make_config(ws[0]), np.concatenate([w.y for w in ws]),
                     datasets=[(w.N, w.M, w.T) for w in ws])
        return {"kind": kind, "ctx": ctx, "K": case["K"], "seed": ws[0].seed}
    w = _workload(case, seed)
    cfg = S.make_config(w)
    if kind == "run":
        return {"kind": kind, "ctx": S.SMC2(cfg, w.y), "K": w.K, "seed": w.seed}
    theta = torch.from_numpy(np.ascontiguousarray(_theta(w, seed).T)).to(dev)
    if kind == "noalloc":
        return {"kind": kind, "cfg": cfg, "y": torch.from_numpy(w.y).to(dev), "theta": theta}
    return {"kind": kind, "ctx": S.SMC2(cfg, w.y), "theta": theta}


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    kind = state["kind"]
    if kind == "pf":
        return {"loglik": state["ctx"].pf_loglik(state["theta"], iteration=1)}
    if kind == "noalloc":
        return {"loglik": S.pf_loglik_noalloc(state["cfg"], state["y"], state["theta"], iteration=1)}
    if kind == "resample":
        return {"ancestors": S.resample_systematic(state["q"], state["U"], state["anc"])}
    if kind == "train":
        x, y, stdz = S.mlp_train_ring(state["p"], state["m"], state["v"], state["step"], state["th"], state["lp"],
                                      state["steps"], 5e-3)
        return {"params": state["p"], "m": state["m"], "v": state["v"], "x": x, "y": y, "stdz": stdz}
    ctx = state["ctx"]
    ctx.reset(state["seed"])
    stats = ctx.run(state["K"])
    out = {name: np.array([[d[name] for d in row] for row in stats]) for name in ("ess", "lse", "logz", "est", "cov")}
    if ctx.n_ds == 1:
        k, theta, logprior, loglik, logw = ctx.get_state()
        mean, logz, ess_sum = ctx.estimate()
        out.update(theta=theta, logprior=logprior, loglik=loglik, logw=logw, mean=mean, ess_sum=ess_sum)
    else:
        out["mean"] = np.array([ctx.estimate(d)[0] for d in range(ctx.n_ds)])
    return out


def _sizes(case):
    """(N, M, T) of each dataset of a filter or run case."""
    if case.get("datasets", 1) > 1:
        return [(w.N, w.M, w.T) for w in I.batched_workloads(case["datasets"], K=case["K"])]
    return [(case["N"], case["M"], case["T"])]


def work(case):
    if case["kind"] == "resample":
        return {"bytes": 12.0 * case["n"], "flops": 20.0 * case["n"]}
    if case["kind"] == "train":
        D, R, P = case["D"], case["R"], 64 * case["D"] + 4289
        return {"bytes": 4.0 * R * (2 * D + 2) + 24.0 * P, "flops": 6.0 * P * R * case["steps"]}
    D = {"lg": 3, "seir": 4, "sir": 2}[case["model"]]
    K = case.get("K", 1)
    steps = sum(n * m * t for n, m, t in _sizes(case)) * K
    size = sum(n * (8 * D + 8) + 8 * t for n, m, t in _sizes(case))
    return {"bytes": float(size), "flops": steps * OPS[case["model"]][case["paper"]]}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 words (int64 tensors holding 32-bit words) of broadcast counters."""
    c = torch.broadcast_tensors(*(torch.as_tensor(v, dtype=torch.int64, device="cuda") for v in (c0, c1, c2, c3)))
    x, y, z, w = c
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        p0, p1 = x * 0xD2511F53, z * 0xCD9E8D57
        x, y, z, w = ((p1 >> 32) & M32) ^ y ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ w ^ k1, p0 & M32
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return x, y, z, w


def _box_muller(wa, wb):
    ua = ((wa >> 9).double() + 0.5) * 2.0 ** -23
    ub = ((wb >> 9).double() + 0.5) * 2.0 ** -23
    r = torch.sqrt(-2.0 * torch.log(ua))
    quarter = torch.round(4.0 * ub)
    f = 2.0 * math.pi * (ub - 0.25 * quarter)
    s, c = torch.sin(f), torch.cos(f)
    turn = quarter.to(torch.int64) & 3
    cos = torch.where(turn == 0, c, torch.where(turn == 1, -s, torch.where(turn == 2, -c, s)))
    sin = torch.where(turn == 0, s, torch.where(turn == 1, c, torch.where(turn == 2, -s, -c)))
    return r * cos, r * sin


def _normals(c0, c1, c2, c3, seed):
    a, b, c, d = _philox(c0, c1, c2, c3, seed)
    return _box_muller(a, b) + _box_muller(c, d)


def _bits(n):
    return min(52, 63 - (0 if n <= 1 else (n - 1).bit_length()))


def _log_fact(v):
    """log v! for an integer v >= 0 less v log v - v: no cancellation at large v."""
    if v < 30:
        return math.lgamma(v + 1.0) - (v * math.log(v) - v if v > 0 else 0.0)
    i = 1.0 / v
    return 0.5 * math.log(2 * math.pi * v) + i * (1 / 12 - i * i * (1 / 360 - i * i * (1 / 1260 - i * i / 1680)))


def _log_poisson(lam, y):
    """log Poisson(y; lam), lam > 0."""
    if y <= 0:
        return -lam
    d = (lam - y) / y
    return y * (torch.log1p(d) - d) - _log_fact(y)


def _binomial(n, p, ctr, pos, seed):
    """Bin(n, p) from each element's word stream (counter ctr, words from pos on): inversion where
    n min(p, 1-p) < 10, else Hormann's BTRS.  Returns the draws and the words' new positions."""
    out = torch.where(p >= 1.0, n, torch.zeros_like(n))
    pos = pos.clone()
    todo = torch.nonzero((p > 0) & (p < 1) & (n > 0)).squeeze(1)
    N, flip = n[todo], p[todo] > 0.5
    P = torch.where(flip, 1.0 - p[todo], p[todo])
    res = torch.zeros_like(N)

    def uniform(idx):
        c0, c1, c2, c3 = (c[todo[idx]] for c in ctr)
        at = pos[todo[idx]]
        words = torch.stack(_philox(c0 + 4096 * (at >> 2), c1, c2, c3, seed))
        pos[todo[idx]] = at + 1
        return (words.gather(0, (at & 3)[None])[0].double() * 2.0 + 1.0) * 2.0 ** -33

    live = torch.nonzero(N * P < 10.0).squeeze(1)
    while live.numel():
        nn, pp = N[live], P[live]
        s = pp / (1.0 - pp)
        a = (nn + 1.0) * s
        u, r, k = uniform(live), torch.exp(nn * torch.log1p(-pp)), torch.zeros_like(nn)
        while True:
            on = (u > r) & (k <= nn)
            if not bool(on.any()):
                break
            u = torch.where(on, u - r, u)
            k = torch.where(on, k + 1.0, k)
            r = torch.where(on, r * (a / torch.clamp(k, min=1.0) - s), r)
        res[live] = k
        live = live[k > nn]
    live = torch.nonzero(N * P >= 10.0).squeeze(1)
    while live.numel():
        nn, pp = N[live], P[live]
        q = 1.0 - pp
        spq = torch.sqrt(nn * pp * q)
        b = 1.15 + 2.53 * spq
        a = -0.0873 + 0.0248 * b + 0.01 * pp
        u = uniform(live) - 0.5
        v = uniform(live)
        us = 0.5 - u.abs()
        k = torch.floor((2.0 * a / us + b) * u + nn * pp + 0.5)
        inside = (k >= 0) & (k <= nn)
        m = torch.floor((nn + 1.0) * pp)
        lf = lambda t: torch.lgamma(torch.clamp(t, min=0.0) + 1.0)  # noqa: E731
        rhs = lf(m) + lf(nn - m) - lf(k) - lf(nn - k) + (k - m) * torch.log(pp / q)
        lhs = torch.log(v * (2.83 + 5.1 / b) * spq / (a / (us * us) + b))
        ok = inside & (((us >= 0.07) & (v <= 0.92 - 4.2 / b)) | (lhs <= rhs))
        res[live[ok]] = k[ok]
        live = live[~ok]
    out[todo] = torch.where(flip, N - res, res)
    return out, pos


def _filter64(w, theta, iteration, dataset=0):
    """log p^(y | theta_i) of each row of theta by the bootstrap filter, in 64 bits."""
    dev = torch.device("cuda")
    th = torch.as_tensor(theta, dtype=torch.float64, device=dev)
    n, M, seed = th.shape[0], w.M, w.seed
    i = torch.arange(n, device=dev)[:, None] | (dataset << 20)
    j = torch.arange(M, device=dev)[None, :]
    tag = lambda t: t | (iteration << 4)  # noqa: E731
    col = lambda d: th[:, d:d + 1]  # noqa: E731
    full = lambda v: torch.zeros((n, M), dtype=torch.float64, device=dev) + v  # noqa: E731
    if w.model == I.LG:
        x = [_normals(j, 0, i, tag(4), seed)[0]]
        phi, sx, sy = col(0), torch.exp(col(1)), torch.exp(col(2))
    elif w.model == I.SEIR:
        x = [full(w.npop - w.e0 - w.i0), full(w.e0), full(w.i0), full(col(0))]
        srw, kappa, gamma, dt = torch.exp(col(1)), torch.exp(col(2)), torch.exp(col(3)), 1.0 / w.n_sub
    else:
        x = [full(w.npop - w.i0), full(w.i0)]
        p_ir = full(-torch.expm1(-col(1)))
    B = _bits(M)
    loglik, common = torch.zeros(n, dtype=torch.float64, device=dev), torch.zeros(n, dtype=torch.float64, device=dev)
    carried = full(0.0)
    dead = torch.zeros(n, dtype=torch.bool, device=dev)
    for t in range(1, w.T + 1):
        y = float(w.y[t - 1])
        if w.model != I.SIR:
            if (t - 1) % 4 == 0:
                z4 = _normals(j, (t - 1) >> 2, i, tag(5), seed)
            z = z4[(t - 1) % 4]
        if w.model == I.LG:
            x = [phi * x[0] + sx * z]
            r = (y - x[0]) / sy
            ell = -0.5 * math.log(2 * math.pi) - col(2) - 0.5 * r * r
        elif w.model == I.SEIR:
            s, e, f, lb = x
            lb = lb + srw * z
            beta, lam = torch.exp(lb), 0.0
            for _ in range(w.n_sub):
                inf, onset, rec = beta * s * f / w.npop, kappa * e, gamma * f
                lam = lam + dt * onset
                s = torch.clamp(s - dt * inf, min=0.0)
                e = torch.clamp(e + dt * (inf - onset), min=0.0)
                f = torch.clamp(f + dt * (onset - rec), min=0.0)
            x = [s, e, f, lb]
            ell = _log_poisson(torch.clamp(lam, min=w.lambda_floor), y)
        else:
            s, f = (v.reshape(-1) for v in x)
            ctr = [c.reshape(-1) for c in torch.broadcast_tensors(j, torch.full((1, 1), t, device=dev), i,
                                                                  torch.full((1, 1), tag(9), device=dev))]
            pos = torch.zeros_like(ctr[0])
            p_si = -torch.expm1(-(full(col(0)).reshape(-1) * f / w.npop))
            n_si, pos = _binomial(s, p_si, ctr, pos, seed)
            n_ir, pos = _binomial(f, p_ir.reshape(-1), ctr, pos, seed)
            x = [(s - n_si).reshape(n, M), (f + n_si - n_ir).reshape(n, M)]
            f = x[1]
            ell = torch.where(f > 0, _log_poisson(torch.clamp(f, min=1.0), y), full(-math.inf if y > 0 else 0.0))
        ell = torch.where(torch.isnan(ell), -math.inf, carried + ell)
        top = ell.max(1).values
        dead |= ~(top > -math.inf)
        top = torch.where(dead, 0.0, top)
        q = torch.floor(torch.exp(ell - top[:, None]) * 2.0 ** B).to(torch.int64)
        C = torch.cumsum(q, 1)
        total = C[:, -1].double()
        loglik = common + top + torch.log(total * 2.0 ** -B) - math.log(M)
        if t == w.T:
            break
        again = torch.ones(n, dtype=torch.bool, device=dev)
        if w.pf_ess_frac > 0:
            qd = q.double()
            again = total * total / (qd * qd).sum(1) < w.pf_ess_frac * M
        share = C.double() / total[:, None]
        if w.pf_scheme == I.PF_MULTINOMIAL:
            words = torch.stack(_philox(j >> 2, t, i, tag(8), seed))
            u = (words.gather(0, (j & 3).expand(n, M)[None])[0].double() * 2.0 + 1.0) * 2.0 ** -33
        else:
            U = _philox(0, t, i, tag(6), seed)[0].double()
            share = share * M
            u = j + (2.0 * U + 1.0) * 2.0 ** -33
        anc = torch.clamp(torch.searchsorted(share, u.contiguous(), right=True), max=M - 1)
        anc = torch.where(again[:, None], anc, j)
        x = [v.gather(1, anc) for v in x]
        carried = torch.where(again[:, None], 0.0, ell)
        common = torch.where(again, loglik, common)
    return torch.where(dead, -math.inf, loglik)


def _log_gauss(x, mean, cov):
    """log N(x; mean, cov) of each row."""
    L = np.linalg.cholesky(cov)
    v = np.linalg.solve(L, (x - mean).T)
    return -0.5 * len(cov) * math.log(2 * math.pi) - np.log(np.diag(L)).sum() - 0.5 * (v * v).sum(0)


def _run64(w):
    """The statistics and final population of a random-walk run with the Gaussian L-kernel, in 64 bits."""
    N, D, seed = w.N, w.D, w.seed
    i = torch.arange(N, device="cuda")
    got = {name: [] for name in ("ess", "lse", "logz", "est", "cov")}
    A = logw = old = None
    for k in range(1, w.K + 1):
        t = (1 if k == 1 else 2) | (k << 4)
        if k == 1 and w.prior_kind == I.PRIOR_UNIFORM:
            u = torch.stack(_philox(0, 0, i, t, seed)[:D], 1).double().cpu().numpy()
            lo, hi = np.array(w.prior_lo), np.array(w.prior_hi)
            th = lo + (hi - lo) * ((u * 2.0 + 1.0) * 2.0 ** -33)
        else:
            z = torch.stack(_normals(0, 0, i, t, seed)[:D], 1).cpu().numpy()
            th = np.array(w.prior_mean) + np.array(w.prior_sd) * z if k == 1 else A + w.rw_scale * z
        if w.prior_kind == I.PRIOR_UNIFORM:
            inside = ((th >= np.array(w.prior_lo)) & (th <= np.array(w.prior_hi))).all(1)
            lp = np.where(inside, -np.log(np.array(w.prior_hi) - np.array(w.prior_lo)).sum(), -math.inf)
        else:
            lp = _log_gauss(th, np.array(w.prior_mean), np.diag(np.array(w.prior_sd) ** 2))
        ll = _filter64(w, th, k).cpu().numpy()
        with np.errstate(invalid="ignore"):
            if k == 1:
                lw = ll + lp - lp
            else:
                step = np.eye(D) * w.rw_scale ** 2
                pw = np.exp(logw - logw.max())
                pw /= pw.sum()
                pair = np.concatenate([A, th], 1)
                mu = pw @ pair
                c = (pair - mu).T @ ((pair - mu) * pw[:, None])
                gain = c[:D, D:] @ np.linalg.inv(c[D:, D:])
                back = _log_gauss(A - (th - mu[D:]) @ gain.T, mu[:D], c[:D, :D] - gain @ c[D:, :D])
                lw = logw + (lp + ll) - old + back - _log_gauss(th, A, step)
        lw = np.where(np.isnan(lw), -math.inf, lw)
        top = lw.max()
        e = np.exp(lw - top)
        lse = top + math.log(e.sum())
        p = e / e.sum()
        est = p @ th
        ess = 1.0 / (p @ p)
        for name, v in (("ess", ess), ("lse", lse), ("logz", lse - math.log(N)), ("est", est),
                        ("cov", (th - est).T @ ((th - est) * p[:, None]))):
            got[name].append([v])
        anc = np.arange(N)
        if ess < w.ess_frac * N:
            q = np.floor(e * 2.0 ** _bits(N)).astype(np.int64)
            U = int(_philox(0, 0, 0, 3 | (k << 4), seed)[0])
            total = int(q.sum())
            C = np.cumsum(q)
            tau = [((j << 33) + 2 * U + 1) * total // (N << 33) for j in range(N)]
            anc = np.searchsorted(C, np.array(tau, dtype=np.int64), side="right")
            lw = np.full(N, lse - math.log(N))
        A, logw, old = th[anc], lw, (lp + ll)[anc]
        lp, ll = lp[anc], ll[anc]
    got = {name: np.array(v) for name, v in got.items()}
    mean = (got["ess"] * got["est"][:, 0]).sum(0) / got["ess"].sum()
    return dict(got, theta=A, logprior=lp, loglik=ll, logw=logw, mean=mean, ess_sum=float(got["ess"].sum()))


def _train64(case, seed):
    th, lp, p = (torch.from_numpy(a).double().cuda() for a in _ring(case, seed))
    D, H = case["D"], 64
    top, tau = lp.max(), max(2.0, float(D))
    z = torch.clamp((lp - top) / tau, min=-8.0)
    zm, zs = z.mean(), z.var(unbiased=False).sqrt()
    keep = z > -8.0
    if int(keep.sum()) < 2 * D + 2:
        keep = torch.ones_like(keep)
    mu, sd = th[keep].mean(0), th[keep].var(0, unbiased=False).sqrt()
    x, y = (th - mu) / sd, (z - zm) / zs
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    loss = torch.zeros(())
    for step in range(1, case["steps"] + 1):
        q = p.clone().requires_grad_(True)
        W1, b1, W2, b2, w3, b3 = torch.split(q, [D * H, H, H * H, H, H, 1])
        h = torch.tanh(torch.tanh(x @ W1.view(D, H) + b1) @ W2.view(H, H) + b2)
        loss = ((h @ w3 + b3 - y) ** 2).mean()
        g, = torch.autograd.grad(loss, q)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        p = p - 5e-3 * (m / (1 - 0.9 ** step)) / (torch.sqrt(v / (1 - 0.999 ** step)) + 1e-8)
    stdz = {"mu": mu, "sd": sd, "tau": tau, "zmean": zm, "zsd": zs, "var_y": 1.0, "loss": loss.detach(), "ymax": top}
    return {"params": p, "m": m, "v": v, "x": x, "y": y, "stdz": stdz}


def exact(case, seed):
    kind = case["kind"]
    if kind == "resample":
        return None  # whole numbers
    if kind == "train":
        return _train64(case, seed)
    if case.get("datasets", 1) > 1 or (case["precision"] == "mixed" and (kind == "run" or case["model"] == "sir")):
        return None
    w = _workload(case, seed)
    if kind == "run":
        return _run64(w)
    return {"loglik": _filter64(w, _theta(w, seed), 1)}
