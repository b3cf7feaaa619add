"""The calls a user of this framework makes, as measurable cases.

Every case is one call (or one round of calls) through the public entry
points of ``paper_1408_1664_gb300.binding``: a whole job from host data, a
whole job on device data, a batch of small jobs with new data, a round of
served jobs, a job with an order prior and family weights.  Sizes are those
of the package's named workloads and of the n and d sweep of the benchmark
(8 to 29 variables, in-degree bounds 2 to 8, 100 to 2000 samples).

Outputs are the edge posteriors and log P(D).  The single-precision form
computes in FP32 and promises 1e-4, so its results are kept as float32; the
FP64 form's are kept as float64.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1408_1664_gb300 import binding, datagen


def listed():
    return [
        # the smallest everyday job: host arrays in, host posteriors out; its
        # time is the launches and the host path
        {"name": "host_n12", "kind": "host", "n": 12, "d": 3, "m": 200, "arity": 2,
         "precision": "fp32"},
        # an ordinary small job in the accuracy reference precision
        {"name": "host_n16_fp64", "kind": "host", "n": 16, "d": 3, "m": 500, "arity": 3,
         "precision": "fp64"},
        # an order prior q_i(|S|) and per-family weights on mixed arities
        {"name": "priors_n21", "kind": "host", "n": 21, "d": 3, "m": 700, "arity": 0,
         "precision": "fp32", "priors": True},
        # the mid-size workload (ternary data), both precisions, device data
        {"name": "mid_n20", "kind": "device", "n": 20, "d": 4, "m": 1000, "arity": 3,
         "precision": "fp32"},
        {"name": "mid_n20_fp64", "kind": "device", "n": 20, "d": 4, "m": 1000, "arity": 3,
         "precision": "fp64"},
        # a size of the paper's n sweep in FP64
        {"name": "sweep_n23_fp64", "kind": "device", "n": 23, "d": 4, "m": 500, "arity": 2,
         "precision": "fp64"},
        # the benchmark's flagship: the full 2^26 lattice
        {"name": "large_n26", "kind": "device", "n": 26, "d": 4, "m": 2000, "arity": 2,
         "precision": "fp32"},
        # the paper's d sweep at n = 25: many parents, so many families
        {"name": "sweep_n25_d6", "kind": "device", "n": 25, "d": 6, "m": 500, "arity": 2,
         "precision": "fp32"},
        {"name": "sweep_n25_d8", "kind": "device", "n": 25, "d": 8, "m": 500, "arity": 2,
         "precision": "fp32"},
        # the large end of the n sweep: 36 GB of arrays
        {"name": "sweep_n29", "kind": "device", "n": 29, "d": 4, "m": 500, "arity": 2,
         "precision": "fp32"},
        # the batched workload: 256 small jobs, new data in, all results out
        {"name": "batch_256", "kind": "batch", "jobs": 256, "n": 10, "n_hi": 18, "d": 3,
         "m": 1000, "precision": "fp32"},
        # the served workload: a round of 64 jobs in flight together
        {"name": "serve_64", "kind": "serve", "jobs": 64, "n": 8, "n_hi": 22, "d": 3,
         "m": 500, "precision": "fp32"},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["host", "host", "device", "device", "device", "batch", "serve"])
    if kind == "batch":
        lo = rng.randint(8, 12)
        return {"kind": kind, "jobs": _log_uniform(rng, 16, 256), "n": lo,
                "n_hi": rng.randint(lo + 2, 18), "d": rng.randint(2, 4),
                "m": _log_uniform(rng, 150, 1000), "precision": "fp32"}
    if kind == "serve":
        lo = rng.randint(6, 14)
        return {"kind": kind, "jobs": _log_uniform(rng, 8, 96), "n": lo,
                "n_hi": rng.randint(lo + 2, 22), "d": rng.randint(2, 4),
                "m": _log_uniform(rng, 100, 1000), "precision": "fp32"}
    precision = rng.choice(["fp32", "fp32", "fp64"])
    arity = rng.choice([2, 2, 3, 0])
    # the cost doubles with n: uniform in n is uniform in its logarithm
    top = 22 if kind == "host" else (24 if precision == "fp64" else 28)
    n = rng.randint(9 if kind == "host" else 14, top)
    if arity == 2:
        d = rng.randint(2, 8) if n <= 25 else rng.randint(2, 4)
    else:
        d = rng.randint(2, 4)
    c = {"kind": kind, "n": n, "d": d, "m": _log_uniform(rng, 100, 2000), "arity": arity,
         "precision": precision}
    if kind == "host" and rng.random() < 0.35:
        c["priors"] = True
        c["d"] = min(d, 4)
    return c


# ---- inputs ----------------------------------------------------------------

def _arities(n, arity):
    """Every variable's arity; 0 stands for mixed arities 2, 3 and 4."""
    return [2 + (5 * i + i // 3) % 3 for i in range(n)] if arity == 0 else [arity] * n


def _dataset(n, m, arity, d, seed):
    return datagen.random_dag_data(n, m, _arities(n, arity), min(d, 4), 1.0, seed=seed)


def _families(n, d):
    return sum(math.comb(n - 1, k) for k in range(min(d, n - 1) + 1))


def _priors(case, seed):
    """An order prior by |S| and family weights around 1 (natural logs)."""
    if not case.get("priors"):
        return None, None
    n = case["n"]
    rng = np.random.default_rng([seed, 17])
    log_q = -0.3 * rng.random((n, n))
    log_w = 0.5 * rng.standard_normal((n, _families(n, case["d"])))
    return log_q, log_w


def _many(case, seed):
    """The jobs of a batch or a served round: sizes from the case alone, data
    from the seed."""
    sizes = np.random.default_rng(case["jobs"] * 1000 + case["n_hi"])
    out = []
    for j in range(case["jobs"]):
        n = int(sizes.integers(case["n"], case["n_hi"] + 1))
        if case["kind"] == "batch":
            arity, m = int(sizes.integers(2, 4)), int(sizes.integers(100, case["m"] + 1))
        else:
            arity, m = 2, case["m"]
        out.append(_dataset(n, m, arity, case["d"], [seed, j]))
    return out


@functools.lru_cache(maxsize=None)
def _context():
    """A program keeps one context for all its jobs."""
    return binding.Context(0, slots=8)


class _Batch(binding.Batch):
    """A batch whose device memory goes with its state."""

    def __del__(self):
        self.close()


@functools.lru_cache(maxsize=None)
def _stream():
    return torch.cuda.Stream()


def prepare(case, seed):
    ctx, kind, prec = _context(), case["kind"], case["precision"]
    state = {"kind": kind, "ctx": ctx, "precision": prec, "d": case["d"]}
    if kind in ("batch", "serve"):
        state["jobs"] = [binding.Job(ds.data, ds.arity, case["d"], precision=prec)
                         for ds in _many(case, seed)]
        if kind == "batch":
            state["batch"] = _Batch(ctx.h, state["jobs"])
        return state
    ds = _dataset(case["n"], case["m"], case["arity"], case["d"], seed)
    if kind == "host":
        state["data"], state["arity"] = ds.data, ds.arity
        state["log_q"], state["log_w"] = _priors(case, seed)
        return state
    n = case["n"]
    state["stream"] = _stream()
    state["data"] = torch.from_numpy(ds.data).cuda()
    state["job"] = binding.Job(state["data"], ds.arity, case["d"], precision=prec)
    # posteriors and log P(D) in one buffer: post = out[:-1], log P(D) = out[-1]
    state["out"] = torch.empty(n * n + 1, dtype=torch.float64, device="cuda")
    state["result"] = (state["out"] if prec == "fp64"
                       else torch.empty(n * n + 1, dtype=torch.float32, device="cuda"))
    torch.cuda.current_stream().synchronize()
    return state


def _kept(post, log_PD, precision):
    t = np.float64 if precision == "fp64" else np.float32
    return {"post": np.asarray(post, t), "log_PD": np.asarray(log_PD, t)}


def run(state):
    kind, ctx = state["kind"], state["ctx"]
    if kind == "host":
        job = binding.Job(state["data"], state["arity"], state["d"], precision=state["precision"],
                          log_q=state["log_q"], log_w=state["log_w"])
        post, log_PD = binding.bn_edge_posteriors(ctx.h, job)
        return _kept(post, log_PD, state["precision"])
    if kind == "device":
        out = state["out"]
        binding.bn_edge_posteriors_async(ctx.h, state["job"], out, out.data_ptr() + 8 * (out.numel() - 1),
                                         state["stream"])
        if state["result"] is not out:
            with torch.cuda.stream(state["stream"]):
                state["result"].copy_(out)
        return {"post": state["result"][:-1], "log_PD": state["result"][-1:]}
    if kind == "batch":
        batch = state["batch"]
        batch.upload(state["jobs"])
        batch.run()
        posts, log_PD = batch.download()
        return _kept(np.concatenate([p.reshape(-1) for p in posts]), log_PD, state["precision"])
    ids = [binding.bn_submit(ctx.h, j) for j in state["jobs"]]
    posts, log_PD = [], []
    for i, j in zip(ids, state["jobs"]):
        rc, p, l = binding.bn_wait(ctx.h, i, j.n)
        if rc != binding.BN_OK:
            raise binding.BnError(rc, "bn_wait")
        posts.append(p.reshape(-1))
        log_PD.append(l)
    return _kept(np.concatenate(posts), log_PD, state["precision"])


# ---- what a pass cannot do without -----------------------------------------

def _job_work(n, d, m, word):
    """Bytes: the data and the posteriors, A (n 2^(n-1) values) written once
    and read by F and by R', F and R' written and read once, their halves
    read for every endpoint.  Operations: the two zeta transforms' additions
    (half the values of each dimension), a multiplication and an addition per
    term of F, of R' and of the down-zeta's input, and one count per sample
    of every variable set of at most d + 1 members."""
    cells, A = float(2 ** n), n * float(2 ** (n - 1))
    sets = sum(math.comb(n, k) for k in range(min(d, n - 1) + 2))
    return {"bytes": m * n + 8.0 * n * n + word * (3.0 * A + 4.0 * cells + n * cells),
            "flops": A * (n - 1) + 6.0 * A + float(m) * sets}


def work(case):
    word = 8.0 if case["precision"] == "fp64" else 4.0
    if case["kind"] in ("host", "device"):
        return _job_work(case["n"], case["d"], case["m"], word)
    total = {"bytes": 0.0, "flops": 0.0}
    sizes = np.random.default_rng(case["jobs"] * 1000 + case["n_hi"])
    for _ in range(case["jobs"]):
        n, m = int(sizes.integers(case["n"], case["n_hi"] + 1)), case["m"]
        if case["kind"] == "batch":
            sizes.integers(2, 4)
            m = int(sizes.integers(100, case["m"] + 1))
        w = _job_work(n, case["d"], m, word)
        total = {k: total[k] + w[k] for k in total}
    return total


# ---- the same results in plain torch, 64 bits ------------------------------

def _subsets(n, k, device):
    """All k-element subsets of n variables as rows of increasing members."""
    c = torch.arange(n, device=device).reshape(-1, 1) if k else torch.zeros(1, 0, dtype=torch.long, device=device)
    for _ in range(1, k):
        more = (n - 1 - c[:, -1]).clamp_min(0)
        at = torch.repeat_interleave(torch.arange(len(c), device=device), more)
        start = torch.cumsum(more, 0) - more
        step = torch.arange(len(at), device=device) - start[at]
        c = torch.cat([c[at], (c[at, -1] + 1 + step).reshape(-1, 1)], 1)
    return c


def _set_scores(data, arity, d, masks, device, ess=1.0):
    """H(X) = sum over the joint states of X of lgamma(a + N) - lgamma(a),
    a = ess / states, for every X of at most d + 1 variables; the BDeu score
    of (i, G) is H(G + i) - H(G)."""
    m, n = data.shape
    x = torch.as_tensor(np.ascontiguousarray(data), device=device).long().T.contiguous()
    r = torch.as_tensor(np.asarray(arity, np.int64), device=device)
    H = torch.zeros(2 ** n, dtype=torch.float64, device=device)
    for k in range(min(d, n - 1) + 2):
        sets = masks[k]
        for c in torch.split(sets, max(1, 2 ** 27 // max(m, 1) // 8)):
            states = torch.ones(len(c), dtype=torch.long, device=device)
            key = torch.zeros(len(c), m, dtype=torch.long, device=device)
            for t in range(k):
                key += x[c[:, t]] * states.reshape(-1, 1)
                states = states * r[c[:, t]]
            N = torch.zeros(len(c), int(states.max()), dtype=torch.float64, device=device)
            N.scatter_add_(1, key, torch.ones(1, 1, dtype=torch.float64, device=device).expand(len(c), m))
            a = (ess / states.double()).reshape(-1, 1)
            at = (1 << c).sum(1) if k else torch.zeros(1, dtype=torch.long, device=device)
            H[at] = (torch.lgamma(a + N) - torch.lgamma(a)).sum(1)
    return H


def _squeeze(mask, i):
    low = mask & ((1 << i) - 1)
    return low | ((mask >> 1) & ~((1 << i) - 1))


def _spread(c, i):
    low = c & ((1 << i) - 1)
    return low | ((c & ~((1 << i) - 1)) << 1)


def _exact_job(data, arity, d, log_q=None, log_w=None):
    """Edge posteriors (n, n) and log P(D): the forward-backward sums over
    the subset lattice in natural logs, one torch call per dimension."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    n = int(data.shape[1])
    d = min(d, n - 1)
    half, ninf = 2 ** (n - 1), -math.inf
    sets = [_subsets(n, k, dev) for k in range(d + 2)]
    H = _set_scores(data, arity, d, sets, dev)
    masks = torch.cat([(1 << s).sum(1) if k else torch.zeros(1, dtype=torch.long, device=dev)
                       for k, s in enumerate(sets[:d + 1])])
    size = torch.cat([torch.full((len(s),), k, device=dev) for k, s in enumerate(sets[:d + 1])])
    c = torch.arange(half, device=dev)
    pop = torch.zeros(half, dtype=torch.long, device=dev)
    for b in range(n - 1):
        pop += (c >> b) & 1
    B, A, shift = [], [], 0.0
    for i in range(n):
        ok = (masks >> i) & 1 == 0
        G = masks[ok]
        b = H[G | (1 << i)] - H[G]
        if log_w is not None:
            # canonical family order: size, then mask
            order = torch.argsort(size[ok] * 2 ** n + G)
            w = torch.empty_like(b)
            w[order] = torch.as_tensor(log_w[i], dtype=torch.float64, device=dev)
            b = b + w
        top = b.max()
        shift += float(top)
        B.append((G, b - top))
        a = torch.full((half,), ninf, dtype=torch.float64, device=dev)
        a[_squeeze(G, i)] = b - top
        for t in range(n - 1):
            v = a.view(-1, 2, 2 ** t)
            v[:, 1] = torch.logaddexp(v[:, 1], v[:, 0])
        if log_q is not None:
            a += torch.as_tensor(log_q[i], dtype=torch.float64, device=dev)[pop]
        A.append(a)
    full = torch.arange(2 ** n, device=dev)
    pop2 = torch.zeros(2 ** n, dtype=torch.uint8, device=dev)
    for b in range(n):
        pop2 += ((full >> b) & 1).to(torch.uint8)
    levels = [torch.nonzero(pop2 == k).reshape(-1) for k in range(n + 1)]
    del full, pop2
    F = torch.zeros(2 ** n, dtype=torch.float64, device=dev)
    R = torch.zeros(2 ** n, dtype=torch.float64, device=dev)   # R[P]: the orders after prefix P
    for k in range(1, n + 1):
        S, T = levels[k], levels[n - k]
        f = torch.full((len(S),), ninf, dtype=torch.float64, device=dev)
        r = torch.full((len(T),), ninf, dtype=torch.float64, device=dev)
        for i in range(n):
            P = S & ~(1 << i)
            f = torch.where(P != S, torch.logaddexp(f, F[P] + A[i][_squeeze(P, i)]), f)
            Q = T | (1 << i)
            r = torch.where(Q != T, torch.logaddexp(r, R[Q] + A[i][_squeeze(T & ~(1 << i), i)]), r)
        F[S], R[T] = f, r
    Z = float(F[-1])
    post = torch.zeros(n, n, dtype=torch.float64, device=dev)
    for v in range(n):
        A[v] = None
        S = _spread(c, v)
        g = F[S] + R[S | (1 << v)]
        if log_q is not None:
            g += torch.as_tensor(log_q[v], dtype=torch.float64, device=dev)[pop]
        for t in range(n - 1):
            x = g.view(-1, 2, 2 ** t)
            x[:, 0] = torch.logaddexp(x[:, 0], x[:, 1])
        G, b = B[v]
        w = torch.exp(b + g[_squeeze(G, v)] - Z)
        for u in range(n):
            post[u, v] = (w * ((G >> u) & 1)).sum()
    return post.cpu().numpy(), Z + shift


def exact(case, seed):
    if case["kind"] in ("batch", "serve"):
        got = [_exact_job(ds.data, ds.arity, case["d"]) for ds in _many(case, seed)]
        return {"post": np.concatenate([p.reshape(-1) for p, _ in got]),
                "log_PD": np.array([l for _, l in got])}
    if case["n"] > 26:
        return None                       # tens of seconds and over 100 GB
    ds = _dataset(case["n"], case["m"], case["arity"], case["d"], seed)
    post, log_PD = _exact_job(ds.data, ds.arity, case["d"], *_priors(case, seed))
    if case["kind"] == "device":
        return {"post": post.reshape(-1), "log_PD": np.array([log_PD])}
    return {"post": post, "log_PD": np.float64(log_PD)}
