"""The calls a user of the library makes, at the sizes they make them, for timing and comparison.

A case is either a batched search on a resident forest (``gf_query``) or the construction of one
(``gf_build`` + ``gf_forest_add_screen`` + ``gf_forest_export``).  Points and queries are drawn on
the GPU from the mixture laws of the repository's workloads (``synth``): "A" 20 isotropic
components, "B" 100 components with decaying per-dimension deviations (GIST-like), "C" the same
with 50 components for very high dimensions, "K" a noisy Klein bottle (low intrinsic dimension).
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1603_09596_gb300 as gf

DEV = "cuda"
PREC = {"fp32": gf.GF_FP32, "bf16": gf.GF_BF16_RERANK, "fp8": gf.GF_FP8_RERANK}
SPLIT_T = 5  # gf_build's default: split dimension drawn from the 5 of largest variance


def _query(name, law, n, d, T, p, m, k, precision, R=0, checks=0):
    return {"name": name, "op": "query", "law": law, "n": n, "d": d, "T": T, "p": p, "m": m, "k": k,
            "precision": precision, "R": R, "checks": checks}


def _build(name, law, n, d, T, p, precision):
    return {"name": name, "op": "build", "law": law, "n": n, "d": d, "T": T, "p": p, "precision": precision}


def listed():
    return [
        # the smallest workload: a small forest asked a hundred nearest-neighbour questions; latency
        _query("tiny_fp32", "A", 10_000, 128, 8, 32, 100, 1, "fp32"),
        # one interactive query against the large index (the operating point with recall@1 >= 0.9)
        _query("single_bf16", "B", 1_000_000, 960, 32, 1024, 1, 10, "bf16", 32),
        # an ordinary serving batch (27 requests, the mean at 200k q/s) on a mid-sized forest
        _query("serve_small_fp32", "B", 50_000, 512, 16, 256, 27, 10, "fp32"),
        # a busy serving batch on one of the large resident forests
        _query("serve_bf16", "B", 500_000, 960, 32, 512, 199, 10, "bf16", 32),
        # offline batch, plain float32, the 10^5-point index with small leaves
        _query("batch_fp32", "B", 100_000, 960, 16, 64, 10_000, 10, "fp32"),
        # the 10^6-point index with the small leaves of its specification, one leaf per tree
        _query("one_leaf_bf16", "B", 1_000_000, 960, 32, 64, 10_000, 10, "bf16", 32),
        # the headline: recall@1 >= 0.9 on 10^6 x 960, bf16 screen and float32 rerank
        _query("wide_bf16", "B", 1_000_000, 960, 32, 1024, 10_000, 10, "bf16", 32),
        # the same search in plain float32
        _query("wide_fp32", "B", 1_000_000, 960, 32, 1024, 10_000, 10, "fp32"),
        # the priority search over small leaves (512 leaf checks a query), the other way to that recall
        _query("priority_bf16", "B", 1_000_000, 960, 32, 64, 10_000, 10, "bf16", 16, 512),
        # very high dimension, E4M3 screen
        _query("highd_fp8", "C", 200_000, 10_000, 24, 32, 2_000, 10, "fp8", 32),
        # low intrinsic dimension, odd sizes throughout (rows that end inside a 16-byte piece)
        _query("manifold_fp32", "K", 700_001, 101, 32, 64, 5_003, 5, "fp32"),
        # making an index: the forest, its bf16 copy, and the structure brought to the host
        _build("build_bf16", "B", 500_000, 960, 32, 512, "bf16"),
    ]


def _log_int(rng: random.Random, lo: int, hi: int) -> int:
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng: random.Random):
    kind = rng.choice(["small", "serve", "serve", "batch", "batch", "batch", "priority", "highd", "manifold", "build"])
    precision = rng.choice(["fp32", "bf16", "fp8"])
    k = rng.choice([1, 5, 7, 10, 10, 16])
    if kind == "small":
        c = _query("", "A", _log_int(rng, 2_000, 50_000), _log_int(rng, 48, 512), rng.randint(4, 16),
                   _log_int(rng, 16, 256), _log_int(rng, 1, 1_000), k, precision, 32)
    elif kind == "serve":
        c = _query("", "B", _log_int(rng, 30_000, 1_000_000), _log_int(rng, 100, 960), rng.randint(16, 32),
                   _log_int(rng, 128, 1024), _log_int(rng, 1, 1_024), k, precision, 32)
    elif kind == "batch":
        c = _query("", "B", _log_int(rng, 30_000, 1_000_000), _log_int(rng, 100, 960), rng.randint(8, 32),
                   _log_int(rng, 32, 1024), _log_int(rng, 1_500, 10_000), k, precision, rng.choice([16, 24, 32, 64]))
    elif kind == "priority":
        T, checks = rng.randint(8, 32), _log_int(rng, 48, 512)
        c = _query("", "B", _log_int(rng, 30_000, 1_000_000), _log_int(rng, 100, 960), T, _log_int(rng, 32, 128),
                   _log_int(rng, 1, 10_000), min(k, 10), precision, 16, checks)
    elif kind == "highd":
        c = _query("", "C", _log_int(rng, 10_000, 200_000), _log_int(rng, 2_000, 10_000), rng.randint(8, 24),
                   _log_int(rng, 32, 256), _log_int(rng, 20, 2_000), k, precision, 32)
    elif kind == "manifold":
        c = _query("", "K", _log_int(rng, 10_000, 1_000_000), _log_int(rng, 60, 200), rng.randint(8, 32),
                   _log_int(rng, 32, 256), _log_int(rng, 100, 10_000), k, precision, 32)
    else:
        c = _build("", "B", _log_int(rng, 20_000, 500_000), _log_int(rng, 100, 960), rng.randint(8, 32),
                   _log_int(rng, 64, 512), precision)
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs

LAWS = {"A": (20, 0.0, False), "B": (100, 32.0, True), "C": (50, 256.0, True)}  # components, decay, shift
ROWS = 1 << 17  # rows drawn at a time


def _mixture(law, n, d, m, g):
    comps, decay, shift = LAWS[law]
    centers = torch.randn(comps, d, generator=g, device=DEV) * 2.0
    j = torch.arange(d, device=DEV, dtype=torch.float32)
    sigma = torch.rsqrt(1.0 + j / decay) if decay else torch.ones(d, device=DEV)

    def points(rows):
        out = torch.empty(rows, d, device=DEV)
        for lo in range(0, rows, ROWS):
            o = out[lo:lo + ROWS]
            o.normal_(generator=g).mul_(sigma)
            o += centers[torch.randint(0, comps, (o.shape[0],), generator=g, device=DEV)]
        return out

    X, Q = points(n), points(m)
    if shift:
        low = X.amin(0)
        X -= low
        Q -= low
    return X, Q


def _klein(n, d, m, g):
    frame = torch.randn(4, d, generator=g, device=DEV)
    for c in range(4):  # orthonormal rows (Gram-Schmidt)
        for b in range(c):
            frame[c] -= (frame[c] @ frame[b]) * frame[b]
        frame[c] /= frame[c].norm()

    def points(rows):
        u, v = (2 * math.pi * torch.rand(2, rows, generator=g, device=DEV))
        P = torch.stack([(2 + v.cos()) * u.cos(), (2 + v.cos()) * u.sin(), v.sin() * (u / 2).cos(),
                         v.sin() * (u / 2).sin()], 1)
        out = torch.empty(rows, d, device=DEV).normal_(generator=g).mul_(0.05)
        for c in range(4):
            out.addcmul_(P[:, c:c + 1], frame[c])
        return out

    return points(n), points(m)


def _inputs(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * (seed + 1))
    m = case.get("m", 0)
    if case["law"] == "K":
        return _klein(case["n"], case["d"], m, g)
    return _mixture(case["law"], case["n"], case["d"], m, g)


def prepare(case, seed):
    X, Q = _inputs(case, seed)
    if case["op"] == "build":
        return {"case": case, "X": X, "seed": seed}
    F = gf.gf_build(X, case["T"], case["p"], t=SPLIT_T, seed=seed)
    if case["precision"] != "fp32":
        gf.gf_forest_add_screen(F, PREC[case["precision"]])
    return {"case": case, "F": F, "Q": Q}


def run(state):
    c = state["case"]
    if c["op"] == "build":
        F = gf.gf_build(state["X"], c["T"], c["p"], t=SPLIT_T, seed=state["seed"])
        if c["precision"] != "fp32":
            gf.gf_forest_add_screen(F, PREC[c["precision"]])
        dims, vals, perm = gf.gf_forest_export(F)
        F.free()
        return {"split_dim": dims, "split_val": vals, "perm": perm}
    ids, dists = gf.gf_query(state["F"], state["Q"], c["k"], precision=PREC[c["precision"]],
                             rerank_R=0 if c["precision"] == "fp32" else c["R"], checks=c["checks"])
    return {"ids": ids, "dists": dists}


# ---------------------------------------------------------------- the work of a pass

def _depth(n, p):
    L = 0
    while -(-n // (1 << L)) > p:
        L += 1
    return L


def work(case):
    n, d, T = case["n"], case["d"], case["T"]
    L = _depth(n, case["p"])
    tree = T * ((1 << L) - 1) * 8 + T * n * 4
    if case["op"] == "build":
        # the points in, the nodes and leaf orders out (twice: on the device and to the host), the
        # copy out; one subtract, multiply and two adds per point, dimension, tree and level
        copy = {"fp32": 0, "bf16": 2, "fp8": 1}[case["precision"]]
        return {"bytes": 4 * n * d + 2 * tree + copy * n * d, "flops": 4 * n * d * T * L}
    m, k = case["m"], case["k"]
    leaves = max(T, case["checks"])
    leaf = -(-n // (1 << L))
    # of the ids gathered from a query's leaves a third at the least are distinct (0.3 to 0.6 on
    # these laws); every row some query needs is read once
    cand = max(leaf, min(n, leaves * leaf // 3))
    rows = min(n, m * cand)
    size = {"fp32": 4, "bf16": 2, "fp8": 1}[case["precision"]]
    rerank = 0 if case["precision"] == "fp32" else min(case["R"], cand)
    return {"bytes": rows * d * size + min(n, m * rerank) * d * 4 + m * d * 4 + min(T * n, m * leaves * leaf) * 4 + m * k * 12,
            "flops": 3 * m * d * (cand + rerank)}


# ---------------------------------------------------------------- the same in float64, plain torch

def _mix64(s0, i):
    with np.errstate(over="ignore"):
        z = np.uint64(s0) + (np.asarray(i, dtype=np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _fmix32(h):
    for shift, mul in ((16, 0x85EBCA6B), (13, 0xC2B2AE35)):
        h = ((h ^ (h >> shift)) * mul) & 0xFFFFFFFF
    return h ^ (h >> 16)


def _tree(X, L, seed, t):
    """Tree t of the forest: (split dims, split values, leaf order), by sorting (Alg. 1)."""
    n, d = X.shape
    key = _mix64(seed, t)
    seq = torch.arange(n, device=X.device)
    rank = _fmix32(seq ^ int(_mix64(key, 0) & np.uint64(0xFFFFFFFF)))
    dims = torch.zeros((1 << L) - 1, dtype=torch.int32)
    vals = torch.zeros((1 << L) - 1, dtype=torch.float32)
    for level in range(L):
        nodes = np.arange(1 << level, dtype=np.int64)
        lo, hi, mid = nodes * n >> level, (nodes + 1) * n >> level, (2 * nodes + 1) * n >> (level + 1)
        draws = (_mix64(key, (1 << level) + nodes) % np.uint64(SPLIT_T)).astype(np.int64)
        out = torch.empty_like(seq)
        for size, left in sorted(set(zip((hi - lo).tolist(), (mid - lo).tolist()))):
            sel = nodes[(hi - lo == size) & (mid - lo == left)]
            per = max(1, (1 << 28) // (size * d))
            for b in range(0, len(sel), per):
                part = sel[b:b + per]
                pos = torch.from_numpy(lo[part]).to(X.device)[:, None] + torch.arange(size, device=X.device)
                rows = seq[pos]
                var = torch.zeros(len(part), d, dtype=torch.float64, device=X.device)
                if size > 1:
                    step = max(1, (1 << 27) // (len(part) * size))
                    for c in range(0, d, step):
                        V = X[:, c:c + step][rows].double()
                        var[:, c:c + step] = V.sub_(V[:, :1].clone()).var(1, correction=1)
                        del V
                top = var.topk(SPLIT_T, 1).indices
                s = top.gather(1, torch.from_numpy(draws[part]).to(X.device)[:, None])
                x = X[rows, s] + 0.0
                bits = x.view(torch.int32).long() & 0xFFFFFFFF
                bits = torch.where(bits >= 1 << 31, 0xFFFFFFFF - bits, bits + (1 << 31))
                keys = ((bits - (1 << 31)) << 32) | rank[rows]
                order = keys.argsort(1)
                goes_left = torch.zeros_like(keys, dtype=torch.bool)
                goes_left.scatter_(1, order[:, :left], True)
                out[pos] = rows.gather(1, torch.sort((~goes_left).to(torch.int8), dim=1, stable=True).indices)
                at = (1 << level) - 1 + torch.from_numpy(part)
                dims[at] = s[:, 0].int().cpu()
                vals[at] = x.gather(1, order[:, left:left + 1])[:, 0].cpu() if left < size else math.inf
        seq = out
    return dims, vals, seq.int()


def _rounded(X, precision):
    if precision == "bf16":
        return lambda ids: X[ids].bfloat16().double()

    def codes(ids):
        V = X[ids]
        a = V.abs().amax(1, keepdim=True)
        scale = torch.where(a > 0, a / 448.0, torch.ones_like(a))
        inv = torch.where(a > 0, 448.0 / a, torch.zeros_like(a))
        return (V * inv).to(torch.float8_e4m3fn).double() * scale.double()

    return codes


def exact(case, seed):
    if case.get("checks", 0) > case["T"]:
        return None  # one shared priority queue per query, popped hundreds of times: minutes
    X, Q = _inputs(case, seed)
    n, T, L = case["n"], case["T"], _depth(case["n"], case["p"])
    trees = [_tree(X, L, seed, t) for t in range(T)]
    if case["op"] == "build":
        return {"split_dim": None, "split_val": torch.stack([v for _, v, _ in trees]), "perm": None}
    leaf = []
    for dims, vals, _ in trees:
        dims, vals = dims.to(DEV).long(), vals.to(DEV)
        j = torch.zeros(len(Q), dtype=torch.long, device=DEV)
        for _level in range(L):
            j = 2 * j + 2 - (Q.gather(1, dims[j][:, None])[:, 0] < vals[j]).long()
        leaf.append(j - ((1 << L) - 1))
    lo = torch.stack([b * n >> L for b in leaf], 1)
    size = torch.stack([(b + 1) * n >> L for b in leaf], 1) - lo
    perm = torch.cat([s for _, _, s in trees])
    base = lo + torch.arange(T, device=DEV) * n
    span = torch.arange(-(-n // (1 << L)), device=DEV)
    screen = None if case["precision"] == "fp32" else _rounded(X, case["precision"])
    dists = torch.full((len(Q), case["k"]), math.inf, dtype=torch.float64, device=DEV)
    for i, q in enumerate(Q.double()):
        at = base[i][:, None] + span
        ids = perm[at[span < size[i][:, None]]].unique().long()  # ascending
        if screen is not None and len(ids) > case["R"]:
            ids = ids[(screen(ids) - q).square_().sum(1).sort(stable=True).indices[:case["R"]]]
        near = (X[ids].double() - q).square_().sum(1).sort().values[:case["k"]]
        dists[i, :len(near)] = near
    return {"ids": None, "dists": dists}
