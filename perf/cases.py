"""The calls of this framework that are timed, with inputs, exact results and work.

Every case goes through the public Python entry points as a program that
compares GPU-kernel control-flow graphs makes them.  The graphs are drawn here:
nested sequence / if-then-else / while-loop regions with early returns, loop
breaks and (for the large ones) unrolled loop bodies, branch probabilities on
the edges, instruction-category counts and a register count or block frequency
as attributes.  Block counts follow from the case alone (the quantiles of a
log-uniform or uniform range), so that a case's work does not depend on the
seed; structure, weights and attributes follow from the seed.

    corpus of kernels  similarity() of all pairs, scores only: the default call
    small_set          the same on a handful of small kernels, with the matrices
                       and matchings: the smallest calls, launches and latency
    query              new kernels against a corpus under a chosen configuration
                       with kept buffers, then the best of each row
    mid_pairs          pairs of 150-400 blocks (too large for one SM's shared memory)
    large_set          all pairs of kernels of 500-2000 blocks (unrolled loops)
    large_pair         one pair of such kernels: latency of a single comparison
    train              one training step: scores, then gradients of all edge
                       weights and of the feature weights
    match / optimal    matchings of matrices in hand, greedy or maximum weight
    distances          the element-wise distances of all pairs, scaled to [0, 1]
    topk               the best k of every row of a score matrix
    ward               the clustering of similarity profiles
"""
from __future__ import annotations

import math
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_1707_02423_gb300 import api

DEV = "cuda"


# ----------------------------------------------------------------------------- sizes
def block_counts(lo, hi, count, log=True, salt=0):
    """`count` block counts spread evenly (over the logarithm) in [lo, hi], in a
    fixed shuffled order."""
    out = []
    for k in range(count):
        q = (k + 0.5) / count
        v = lo * (hi / lo) ** q if log else lo + (hi - lo) * q
        out.append(max(lo, min(hi, int(round(v)))))
    random.Random(1000 * count + salt).shuffle(out)
    return out


def sizes(case):
    """(blocks of side A, blocks of side B or None when both sides are one set,
    pair list) of a case on graphs."""
    kind = case["kind"]
    if kind in ("small_set", "corpus", "large_set", "distances", "match", "optimal"):
        na = block_counts(case["lo"], case["hi"], case["cfgs"], case.get("log", True))
        i, j = np.triu_indices(len(na), k=1)
        return na, None, np.stack([i, j], 1).astype(np.int32)
    if kind == "query":
        na = block_counts(case["lo"], case["hi"], case["queries"])
        nb = block_counts(case["lo"], case["hi"], case["corpus"], salt=1)
        i, j = np.meshgrid(np.arange(len(na)), np.arange(len(nb)), indexing="ij")
        return na, nb, np.stack([i.ravel(), j.ravel()], 1).astype(np.int32)
    if kind in ("mid_pairs", "train"):
        na = block_counts(case["lo"], case["hi"], 2 * case["pairs"])
        k = 2 * np.arange(case["pairs"])
        return na, None, np.stack([k, k + 1], 1).astype(np.int32)
    if kind == "large_pair":
        return [case["na"], case["nb"]], None, np.array([[0, 1]], dtype=np.int32)
    raise ValueError(kind)


# ----------------------------------------------------------------------------- graphs
def structure(rnd, n, depth, unroll):
    """Edges of a structured control-flow graph of exactly n blocks: START 0,
    STOP n - 1, and the open blocks that may get an early return or a break."""
    edges, plain = [], []
    top = [0]

    def new(k):
        v = top[0]
        top[0] += k
        return v

    def chain(k, brk):
        v = new(k)
        edges.extend((u, u + 1) for u in range(v, v + k - 1))
        plain.extend((u, brk) for u in range(v, v + k))
        return v, v + k - 1

    def region(budget, depth, brk):
        if depth <= 0 or budget < 3:
            return chain(budget, brk)
        kind = rnd.random()
        if kind < 0.40:  # a sequence of 2 to 4 regions
            k = rnd.randint(2, min(4, budget))
            cuts = [0] + sorted(rnd.sample(range(1, budget), k - 1)) + [budget]
            first = last = None
            for a, b in zip(cuts, cuts[1:]):
                e0, e1 = region(b - a, depth - 1, brk)
                if first is None:
                    first = e0
                else:
                    edges.append((last, e0))
                last = e1
            return first, last
        inner = budget - 2
        head = new(1)
        if kind < 0.75:  # if-then or if-then-else
            two = inner >= 2 and rnd.random() < 0.6
            b1 = rnd.randint(1, inner - 1) if two else inner
            arms = [region(b1, depth - 1, brk)]
            if two:
                arms.append(region(inner - b1, depth - 1, brk))
            join = new(1)
            for e0, e1 in arms:
                edges.extend([(head, e0), (e1, join)])
            if not two:
                edges.append((head, join))
            return head, join
        # a while loop: header, body (its template repeated when unrolled), exit
        exit_ = [None]
        u = rnd.randint(4, 16) if unroll and inner >= 8 else 1
        body = max(1, inner // u)
        u = min(u, inner // body)
        if u == 1:
            b0, b1 = region(inner, depth - 1, exit_)
        else:
            at, ne, np_ = top[0], len(edges), len(plain)
            b0, b1 = region(body, depth - 1, exit_)
            tmpl, opened = edges[ne:], plain[np_:]
            for k in range(1, u):
                off = new(body) - at
                edges.extend((a + off, b + off) for a, b in tmpl)
                plain.extend((v + off, e) for v, e in opened)
                edges.append((b1, b0 + off))
                b1 += body
            rest = inner - u * body
            if rest:
                c0, c1 = chain(rest, exit_)
                edges.append((b1, c0))
                b1 = c1
        edges.extend([(head, b0), (b1, head)])
        exit_[0] = new(1)
        edges.append((head, exit_[0]))
        return head, exit_[0]

    if n >= 3:
        start = new(1)
        r0, r1 = region(n - 2, depth, None)
        stop = new(1)
        edges.extend([(start, r0), (r1, stop)])
        for v, brk in plain:
            x = rnd.random()
            if x < 0.03:
                edges.append((v, stop))
            elif brk is not None and x < 0.08:
                edges.append((v, brk[0]))
    elif n == 2:
        edges.append((0, 1))
    return sorted(set(edges))


def graphs(counts, F, seed, depth, unroll, salt=0, shape=None):
    """`shape`: the seed of the structure, where it is not the inputs' seed."""
    rnd = random.Random((seed if shape is None else shape) * 7919 + salt)
    rng = np.random.default_rng([seed, salt])
    out = []
    for n in counts:
        e = np.array(structure(rnd, n, depth, unroll), dtype=np.int32).reshape(-1, 2)
        src, dst = np.ascontiguousarray(e[:, 0]), np.ascontiguousarray(e[:, 1])
        w = rng.exponential(size=len(src))  # Dirichlet(1, ..., 1) over the out-edges of each block
        w = w / np.bincount(src, weights=w, minlength=n)[src]
        attr = np.empty((n, F), dtype=np.float32)
        attr[:, :-1] = rng.poisson(rng.uniform(0.0, 20.0, size=(n, F - 1)))
        attr[:, -1] = rng.lognormal(0.0, 2.0, size=n) if unroll else rng.integers(8, 65, size=n)
        out.append(SimpleNamespace(n=n, src=src, dst=dst, w=w.astype(np.float32), attr=attr))
    return out


def workload(case, seed):
    na, nb, pairs = sizes(case)
    large = case["kind"] in ("large_set", "large_pair")
    depth = 8 if large else 5
    # a training program fits the weights of fixed graphs: the edges stay, their weights follow from the seed
    A = graphs(na, case["F"], seed, depth, large, shape=case["pairs"] if case["kind"] == "train" else None)
    Bs = A if nb is None else graphs(nb, case["F"], seed, depth, large, salt=1)
    return A, Bs, pairs


def feature_weights(case, seed):
    return np.random.default_rng([seed, 77]).uniform(0.5, 1.5, case["F"]).astype(np.float32)


def given_matrices(case, seed):
    """Matrices as a program holds them after similarity(want_x=True): positive,
    norm 1, dominated by one singular direction with structure under it."""
    na, _, pairs = sizes(case)
    n = np.array(na, dtype=np.int64)
    g = torch.Generator(device=DEV).manual_seed(seed)
    P = len(pairs)
    off = np.concatenate([[0], np.cumsum(n)])
    base = np.concatenate([[0], np.cumsum(n[pairs[:, 0]] * n[pairs[:, 1]])])
    u = torch.rand(int(off[-1]), generator=g, device=DEV) * 0.9 + 0.1
    h = torch.rand(int(off[-1]), 2, generator=g, device=DEV) - 0.5
    X = torch.empty(int(base[-1]), device=DEV)
    noise = torch.rand(int(base[-1]), generator=g, device=DEV)
    pid = torch.repeat_interleave(torch.arange(P, device=DEV), torch.from_numpy(np.diff(base)).to(DEV))
    local = torch.arange(int(base[-1]), device=DEV) - torch.from_numpy(base).to(DEV)[pid]
    nb = torch.from_numpy(n[pairs[:, 1]]).to(DEV)[pid]
    i = torch.from_numpy(off[pairs[:, 0]]).to(DEV)[pid] + local // nb
    j = torch.from_numpy(off[pairs[:, 1]]).to(DEV)[pid] + local % nb
    X = u[i] * u[j] * (1.0 + 0.6 * (h[i] * h[j]).sum(1)) * (0.9 + 0.2 * noise)
    nrm = torch.zeros(P, dtype=torch.float64, device=DEV).index_add_(0, pid, X.double() ** 2).sqrt()
    return (X.double() / nrm[pid]).float()


def score_rows(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    return torch.rand(case["rows"], case["cols"], generator=g, device=DEV) * 2.0 + 1.0


def profiles(case, seed):
    """Similarity profiles of kernels from a few families, with spread."""
    rng = np.random.default_rng([seed, 5])
    n, dim = case["points"], case["points"]
    centre = rng.uniform(1.0, 3.0, (max(2, n // 20), dim))
    return (centre[rng.integers(0, len(centre), n)] + rng.normal(0, 0.15, (n, dim))).astype(np.float32)


# ----------------------------------------------------------------------------- cases
def listed():
    return [
        # eight small kernels compared in full: the first thing a user runs
        dict(name="small_set", kind="small_set", cfgs=8, lo=5, hi=20, F=13, alpha=0.8, K=40),
        # every pair of a benchmark suite's kernels (the 19,900-pair workload), the default call
        dict(name="corpus", kind="corpus", cfgs=200, lo=8, hi=120, F=13, alpha=0.8, K=40, tune=0),
        # new kernels looked up in a corpus, step after step with kept buffers under a tuned configuration
        dict(name="query", kind="query", queries=8, corpus=613, lo=5, hi=400, F=25, alpha=0.8, K=40, top=16, tune=182),
        # pairs of mid-size kernels whose matrices are wanted
        dict(name="mid_pairs", kind="mid_pairs", pairs=48, lo=150, hi=400, F=13, alpha=0.8, K=40),
        # kernels with unrolled loops, all pairs
        dict(name="large_set", kind="large_set", cfgs=24, lo=500, hi=2000, log=False, F=13, alpha=0.8, K=40),
        # two such kernels: an analyst's single comparison
        dict(name="large_pair", kind="large_pair", na=1371, nb=1998, F=13, alpha=0.8, K=40),
        # fitting edge and feature weights: one step over 256 pairs
        dict(name="train", kind="train", pairs=256, lo=10, hi=300, F=13, alpha=0.8, K=40),
        # matchings of matrices already computed
        dict(name="match", kind="match", cfgs=100, lo=8, hi=120, F=13),
        dict(name="optimal", kind="optimal", cfgs=100, lo=8, hi=120, F=13),
        # the element-wise measures over the same suite
        dict(name="distances", kind="distances", cfgs=200, lo=8, hi=120, F=13, p=3.0),
        # the best 16 of 10,000 for 32 queries
        dict(name="topk", kind="topk", rows=32, cols=10000, top=16),
        # the dendrogram of a suite
        dict(name="ward", kind="ward", points=200),
    ]


def log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["small_set", "corpus", "query", "mid_pairs", "large_set", "large_pair", "train", "match",
                       "optimal", "distances", "topk", "ward"])
    c = dict(kind=kind)
    if kind == "topk":
        cols = log_int(rng, 100, 10000)
        return dict(c, rows=rng.randint(1, 32), cols=cols, top=log_int(rng, 1, min(64, cols)))
    if kind == "ward":
        return dict(c, points=log_int(rng, 12, 400))
    c.update(F=rng.choice([7, 13, 16, 25]))
    if kind == "small_set":
        c.update(cfgs=rng.randint(2, 8), lo=rng.randint(2, 6), hi=rng.randint(9, 20))
    elif kind in ("corpus", "distances"):
        c.update(cfgs=log_int(rng, 24, 200), lo=rng.randint(5, 12), hi=rng.randint(40, 120))
    elif kind in ("match", "optimal"):
        c.update(cfgs=log_int(rng, 16, 100), lo=rng.randint(5, 12), hi=rng.randint(40, 120))
    elif kind == "query":
        c.update(queries=rng.randint(1, 8), corpus=log_int(rng, 100, 613), lo=rng.randint(5, 12),
                 hi=rng.randint(150, 400), top=rng.choice([5, 10, 16]))
    elif kind == "mid_pairs":
        c.update(pairs=log_int(rng, 3, 48), lo=rng.randint(130, 180), hi=rng.randint(250, 400))
    elif kind == "large_set":
        c.update(cfgs=rng.randint(3, 24), lo=rng.randint(450, 600), hi=rng.randint(900, 2000), log=False)
    elif kind == "large_pair":
        c.update(na=log_int(rng, 450, 2000), nb=log_int(rng, 450, 2000))
    elif kind == "train":
        c.update(pairs=log_int(rng, 8, 256), lo=rng.randint(8, 16), hi=rng.randint(100, 300))
    if kind == "distances":
        c.update(p=rng.choice([1.5, 2.0, 3.0, 4.0]))
    if kind not in ("match", "optimal", "distances"):
        c.update(alpha=rng.choice([0.5, 0.8, 0.9]), K=rng.choice([10, 25, 40]))
    if kind in ("corpus", "query"):
        c.update(tune=rng.choice([0, 2, 182]))
    return c


# ----------------------------------------------------------------------------- the calls
def prepare(case, seed):
    kind = case["kind"]
    if kind == "topk":
        return dict(case=case, scores=score_rows(case, seed))
    if kind == "ward":
        return dict(case=case, points=torch.from_numpy(profiles(case, seed)).to(DEV))
    A, Bs, pairs = workload(case, seed)
    pa = api.Pack(A, case["F"], device=DEV)
    pb = pa if Bs is A else api.Pack(Bs, case["F"], device=DEV)
    st = dict(case=case, pa=pa, pb=pb, pairs=pairs)
    if kind in ("match", "optimal"):
        st["X"] = given_matrices(case, seed)
    elif kind != "distances":
        st["omega"] = torch.from_numpy(feature_weights(case, seed)).to(DEV)
    if kind == "train":
        st["w"] = torch.from_numpy(np.concatenate([g.w for g in A])).to(DEV).requires_grad_(True)
        st["omega"].requires_grad_(True)
    if kind == "query":  # a serving program keeps its buffers
        st["d_pairs"] = torch.from_numpy(pairs).to(DEV)
        st["out"] = {"scores": torch.empty(len(pairs), device=DEV)}
        st["ws"] = api.Workspace(DEV)
        Q, k = case["queries"], case["top"]
        st["top"] = (torch.empty(Q, k, device=DEV), torch.empty(Q, k, dtype=torch.int32, device=DEV))
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "topk":
        top, idx = api.topk(state["scores"], case["top"])
        return {"top": top, "idx": idx}
    if kind == "ward":
        merge, height, size = api.ward(state["points"])
        return {"merge": merge, "height": height, "size": size}
    pa, pb, pairs = state["pa"], state["pb"], state["pairs"]
    if kind == "distances":
        return {"d": api.distances(pa, pb, pairs, case["p"], scale01=True)}
    if kind in ("match", "optimal"):
        r = api.match(pa, pb, pairs, state["X"], optimal=kind == "optimal")
        return {"scores": r.scores, "match": r.match}
    omega, alpha, K = state["omega"], case["alpha"], case["K"]
    if kind == "small_set":
        r = api.similarity(pa, pb, pairs, omega, alpha, K, want_x=True, want_match=True)
        return {"scores": r.scores, "X": r.X, "match": r.match}
    if kind in ("mid_pairs", "large_pair"):
        r = api.similarity(pa, pb, pairs, omega, alpha, K, want_x=True)
        return {"scores": r.scores, "X": r.X}
    if kind == "query":
        r = api.similarity(pa, pb, pairs, omega, alpha, K, d_pairs=state["d_pairs"], out=state["out"],
                           ws=state["ws"], check_status=False, tune=case["tune"])
        top, idx = api.topk(r.scores.view(case["queries"], case["corpus"]), case["top"], out=state["top"])
        return {"scores": r.scores, "top": top, "idx": idx}
    if kind == "train":
        scores = api.CFSimilarity.apply(state["w"], None, omega, pa, pb, pairs, alpha, K)
        gw, go = torch.autograd.grad(scores.sum(), [state["w"], omega])
        return {"scores": scores.detach(), "grad_w": gw, "grad_omega": go}
    return {"scores": api.similarity(pa, pb, pairs, omega, alpha, K, tune=case.get("tune", 0)).scores}


# ----------------------------------------------------------------------------- work
EDGES = 1.15  # edges per block of these graphs, on average


def work(case):
    kind = case["kind"]
    if kind == "topk":
        R, Cn, k = case["rows"], case["cols"], case["top"]
        return {"bytes": 4 * R * Cn + 8 * R * k, "flops": R * Cn}
    if kind == "ward":
        n = case["points"]
        return {"bytes": 4 * n * n + 16 * n, "flops": 3 * n * n * n // 2 + 8 * n * n}
    na, nb, pairs = sizes(case)
    blocks = sum(na) + (0 if nb is None else sum(nb))
    a = np.array(na, dtype=np.float64)[pairs[:, 0]]
    b = np.array(na if nb is None else nb, dtype=np.float64)[pairs[:, 1]]
    P, cells, F = len(pairs), float((a * b).sum()), case["F"]
    graph = blocks * (4.0 * F + 12 * EDGES)  # attributes; source, target and weight of each edge
    if kind in ("match", "optimal"):
        return {"bytes": int(4 * cells + 8 * P + 4 * P + 4 * a.sum()), "flops": int(cells)}
    if kind == "distances":
        N = np.maximum(a, b)
        return {"bytes": int(12 * EDGES * blocks + 8 * P + 20 * P), "flops": int((20 * N * N).sum())}
    # per step and entry: a multiply-add for each pair of out-edges and of in-edges, blend, norm
    step = cells * (4 * EDGES * EDGES + 4)
    out = {"bytes": int(graph + 8 * P + 4 * P), "flops": int(case["K"] * step + 2 * F * cells)}
    if kind in ("small_set", "mid_pairs", "large_pair"):
        out["bytes"] += int(4 * cells)
    if kind == "small_set":
        out["bytes"] += int(4 * a.sum())
    if kind == "train":  # the reverse pass: the transposed step and two terms for each pair of edges
        out["flops"] += int(case["K"] * (step + cells * 8 * EDGES * EDGES))
        out["bytes"] += int(8 * EDGES * blocks + 8 * F)
    return out


# ----------------------------------------------------------------------------- 64-bit results
def dense(cfgs, n, ws=None):
    """Zero-padded adjacency matrices [len(cfgs), n, n] in 64 bits."""
    k = np.concatenate([np.full(len(c.src), q) for q, c in enumerate(cfgs)]) if cfgs else np.zeros(0)
    idx = tuple(torch.from_numpy(np.concatenate(x).astype(np.int64)).to(DEV)
                for x in ([k], [c.src for c in cfgs], [c.dst for c in cfgs]))
    w = torch.cat(ws) if ws is not None else torch.from_numpy(np.concatenate([c.w for c in cfgs])).to(DEV).double()
    return torch.zeros(len(cfgs), n, n, dtype=torch.float64, device=DEV).index_put(idx, w, accumulate=True)


def padded(cfgs, n, F):
    out = np.zeros((len(cfgs), n, F))
    for q, c in enumerate(cfgs):
        out[q, :c.n] = c.attr
    return torch.from_numpy(out).to(DEV)


def similarity64(A, Bs, omega, alpha, K, wa=None, wb=None):
    """X_K of the pairs (A[q], Bs[q]), zero-padded to one size."""
    na, nb, F = max(c.n for c in A), max(c.n for c in Bs), A[0].attr.shape[1]
    a, b = padded(A, na, F), padded(Bs, nb, F)
    WA, WB = dense(A, na, wa), dense(Bs, nb, wb)
    r = ((a * a) @ omega).clamp_min(0)
    c = ((b * b) @ omega).clamp_min(0)
    live = (r > 0).double()[:, :, None] * (c > 0).double()[:, None, :]
    den = torch.where(r > 0, r, torch.ones_like(r)).sqrt()[:, :, None] * \
        torch.where(c > 0, c, torch.ones_like(c)).sqrt()[:, None, :]
    E = ((a * omega) @ b.transpose(1, 2)) / den * live
    eh = E / E.square().sum((1, 2), keepdim=True).sqrt()
    X = eh
    for _ in range(K):
        Y = 0.5 * alpha * (WA @ X @ WB.transpose(1, 2) + WA.transpose(1, 2) @ X @ WB) + (1 - alpha) * eh
        X = Y / Y.square().sum((1, 2), keepdim=True).sqrt()
    return X


def greedy64(X, A, Bs):
    """Greedy matchings [len(A), rows] (-1: unmatched) of padded matrices: largest
    live entry first, the first in row-major order among equals."""
    P, n, m = X.shape
    M = X.detach().clone()
    rows = torch.tensor([c.n for c in A], device=DEV)
    cols = torch.tensor([c.n for c in Bs], device=DEV)
    M.masked_fill_(torch.arange(n, device=DEV)[None, :, None] >= rows[:, None, None], -1.0)
    M.masked_fill_(torch.arange(m, device=DEV)[None, None, :] >= cols[:, None, None], -1.0)
    match = torch.full((P, n), -1, dtype=torch.int64, device=DEV)
    q = torch.arange(P, device=DEV)
    for _ in range(min(n, m)):
        best = M.view(P, -1).max(1)
        flat = (M.view(P, -1) == best.values[:, None]).to(torch.int8).argmax(1)
        ok = best.values >= 0
        i, j = flat // m, flat % m
        match[q[ok], i[ok]] = j[ok]
        M[q, i, :] = -1.0
        M[q, :, j] = -1.0
    return match


def chunks(pairs, na, nb, most):
    """Pair indices sorted by size, in runs whose padded matrices hold at most
    `most` entries."""
    order = sorted(range(len(pairs)), key=lambda p: (max(na[pairs[p][0]], nb[pairs[p][1]]), na[pairs[p][0]]))
    run_, hi = [], 0
    for p in order:
        h = max(hi, na[pairs[p][0]], nb[pairs[p][1]])
        if run_ and (len(run_) + 1) * h * h > most:
            yield run_
            run_, h = [], max(na[pairs[p][0]], nb[pairs[p][1]])
        run_, hi = run_ + [p], h
    if run_:
        yield run_


def exact(case, seed):
    kind = case["kind"]
    if kind == "topk":
        s = score_rows(case, seed).double()
        top, idx = torch.sort(s, dim=1, descending=True, stable=True)
        return {"top": top[:, :case["top"]], "idx": idx[:, :case["top"]].int()}
    if kind == "ward":
        return exact_ward(profiles(case, seed).astype(np.float64))
    if kind == "optimal":
        return None
    na, nb, pairs = sizes(case)
    nb = na if nb is None else nb
    if kind == "large_set" or (kind == "large_pair" and case["na"] * case["nb"] > 3e6):
        return None
    A, Bs, _ = workload(case, seed)
    P = len(pairs)
    if kind == "match":
        X = given_matrices(case, seed).double()
        off = np.concatenate([[0], np.cumsum([na[i] * nb[j] for i, j in pairs])])
    if kind == "distances":
        return {"d": exact_distances(A, pairs, case["p"])}
    scores = torch.zeros(P, dtype=torch.float64, device=DEV)
    Xs, Ms, gw = [None] * P, [None] * P, None
    if kind != "match":
        omega = torch.from_numpy(feature_weights(case, seed)).to(DEV).double()
    if kind == "train":
        omega.requires_grad_(True)
        ws = [torch.from_numpy(c.w).to(DEV).double().requires_grad_(True) for c in A]
    for run_ in chunks(pairs, na, nb, 4_000_000 if kind == "train" else 40_000_000):
        a = [A[pairs[p][0]] for p in run_]
        b = [Bs[pairs[p][1]] for p in run_]
        if kind == "match":
            Y = torch.zeros(len(run_), max(c.n for c in a), max(c.n for c in b), dtype=torch.float64, device=DEV)
            for q, p in enumerate(run_):
                Y[q, :a[q].n, :b[q].n] = X[off[p]:off[p + 1]].view(a[q].n, b[q].n)
        elif kind == "train":
            Y = similarity64(a, b, omega, case["alpha"], case["K"], [ws[pairs[p][0]] for p in run_],
                             [ws[pairs[p][1]] for p in run_])
        else:
            Y = similarity64(a, b, omega, case["alpha"], case["K"])
        m = greedy64(Y, a, b)
        s = (Y.gather(2, m.clamp_min(0)[:, :, None])[:, :, 0] * (m >= 0)).sum(1)
        if kind == "train":
            s.sum().backward()
        scores[torch.tensor(run_, device=DEV)] = s.detach()
        if kind in ("small_set", "mid_pairs", "large_pair", "match"):
            for q, p in enumerate(run_):
                Ms[p] = m[q, :a[q].n].int()
                Xs[p] = Y[q, :a[q].n, :b[q].n].reshape(-1) if kind != "match" else None
    if kind == "match":
        return {"scores": scores, "match": torch.cat(Ms)}
    if kind == "small_set":
        return {"scores": scores, "X": torch.cat(Xs), "match": torch.cat(Ms)}
    if kind in ("mid_pairs", "large_pair"):
        return {"scores": scores, "X": torch.cat(Xs)}
    if kind == "train":
        return {"scores": scores, "grad_w": torch.cat([w.grad for w in ws]), "grad_omega": omega.grad}
    if kind == "query":
        top, idx = torch.sort(scores.view(case["queries"], case["corpus"]), dim=1, descending=True, stable=True)
        return {"scores": scores, "top": top[:, :case["top"]], "idx": idx[:, :case["top"]].int()}
    return {"scores": scores}


def exact_distances(cfgs, pairs, p):
    """The five distances of the resized transition matrices, min-max scaled."""
    n = [c.n for c in cfgs]
    out = torch.zeros(len(pairs), 5, dtype=torch.float64, device=DEV)
    for run_ in chunks(pairs, n, n, 40_000_000):
        a = [cfgs[pairs[q][0]] for q in run_]
        b = [cfgs[pairs[q][1]] for q in run_]
        N = max(max(c.n for c in a), max(c.n for c in b))

        def spread(side, other):
            R = np.zeros((len(run_), N, N))  # row t: the weights of the two source rows it samples
            for q, (c, o) in enumerate(zip(side, other)):
                k = max(c.n, o.n)
                x = np.arange(k) * ((c.n - 1) / (k - 1) if k > 1 else 0.0)
                i = np.minimum(x.astype(np.int64), max(c.n - 2, 0))
                R[q, np.arange(k), i] += 1 - (x - i)
                R[q, np.arange(k), np.minimum(i + 1, c.n - 1)] += x - i
            R = torch.from_numpy(R).to(DEV)
            return R @ dense(side, N) @ R.transpose(1, 2)

        x, y = spread(a, b), spread(b, a)
        d = (x - y).abs()
        xx, yy, xy = x.square().sum((1, 2)), y.square().sum((1, 2)), (x * y).sum((1, 2))
        den = xx + yy - xy
        jac = torch.where(den != 0, d.square().sum((1, 2)) / den, torch.zeros_like(den))
        nn = (xx * yy).sqrt()
        cos = torch.where(nn > 0, 1 - xy / nn, ((xx > 0) != (yy > 0)).double())
        out[torch.tensor(run_, device=DEV)] = torch.stack(
            [d.square().sum((1, 2)).sqrt(), d.sum((1, 2)), d.pow(p).sum((1, 2)).pow(1 / p), jac, cos], 1)
    lo, hi = out.min(0).values, out.max(0).values
    return torch.where(hi > lo, (out - lo) / torch.where(hi > lo, hi - lo, torch.ones_like(hi)), torch.zeros_like(out))


def exact_ward(X):
    n = len(X)
    D = ((X[:, None, :] - X[None, :, :]) ** 2).sum(2) if n <= 250 else None
    if D is None:
        D = np.empty((n, n))
        for i in range(n):
            D[i] = ((X - X[i]) ** 2).sum(1)
    np.fill_diagonal(D, np.inf)
    size, ident = np.ones(n), list(range(n))
    merge, height, count = [], [], []
    for k in range(n - 1):
        i, j = divmod(int(D.argmin()), n)
        i, j = min(i, j), max(i, j)
        merge.append(sorted((ident[i], ident[j])))
        height.append(math.sqrt(D[i, j]))
        t = size[i] + size[j] + size
        row = ((size[i] + size) * D[i] + (size[j] + size) * D[j] - size * D[i, j]) / t
        dead = np.isinf(D[i]) | np.isinf(D[j])
        row[dead] = np.inf
        size[i] += size[j]
        count.append(int(size[i]))
        D[i], D[:, i] = row, row
        D[i, i] = np.inf
        D[j], D[:, j] = np.inf, np.inf
        ident[i] = n + k
    return {"merge": np.array(merge, dtype=np.int32), "height": np.array(height),
            "size": np.array(count, dtype=np.int32)}
