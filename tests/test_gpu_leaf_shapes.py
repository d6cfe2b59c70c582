"""The leaf-major path at the edges of its row tiles, chunk groups and query counts: the float32
kernel's one, two and four warps a chunk (leaves of 64 / 65 and 128 / 129 rows), every number of
queries a chunk can hold, and rows that end inside a slab; the tensor-core kernel's row groups of four
and its tiles of one and two chunks."""
import numpy as np
import pytest
import torch

import oracle
import synth
from parity import assert_screened_close, assert_topk_close
from oracle import screen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gf():
    import paper_1603_09596_gb300 as g
    g.lib()
    return g


# (rows of the largest leaf, leaves a tree, d, queries)
SHAPES = [(1, 64, 3, 40), (31, 16, 130, 24), (63, 8, 33, 60), (64, 8, 96, 130), (65, 4, 64, 44), (128, 4, 100, 66),
          (129, 4, 31, 66), (257, 2, 960, 50), (600, 2, 47, 7)]


def forest(gf, leaf, leaves, d, m):
    n = leaf * leaves - (leaves // 2 if leaf > 1 else 0)  # leaves of `leaf` and of `leaf` - 1 rows
    X, Q = synth.mixture(n, d, m, "B", seed=leaf + d, qseed=m)
    F = oracle.build_forest(X, 5, leaf, t=min(5, d), seed=2)
    assert 1 << F.L == leaves and -(-n // leaves) == leaf
    G = gf.gf_forest_import(torch.from_numpy(X).cuda(), F.T, F.leaf_size, F.split_dim, F.split_val, F.perm)
    return X, Q, F, G


@pytest.mark.parametrize("leaf,leaves,d,m", SHAPES)
@pytest.mark.parametrize("k", [1, 9, 32])
def test_leaf_float32_shapes(gf, leaf, leaves, d, m, k):
    X, Q, F, G = forest(gf, leaf, leaves, d, m)
    gi, gd = gf.gf_query(G, torch.from_numpy(Q).cuda(), k, algo=gf.GF_ALGO_LEAF)
    oi, od = oracle.search(F, X, Q, k)
    assert_topk_close(X, Q, gi.cpu().numpy(), gd.cpu().numpy(), oi, od)


@pytest.mark.parametrize("leaf,leaves,d,m", SHAPES)
@pytest.mark.parametrize("prec", ["bf16", "fp8"])
@pytest.mark.parametrize("ctas", [0, 1])
def test_leaf_screen_shapes(gf, leaf, leaves, d, m, prec, ctas):
    X, Q, F, G = forest(gf, leaf, leaves, d, m)
    p = gf.PRECISIONS[prec]
    gf.gf_forest_add_screen(G, p)
    gi, gd = gf.gf_query(G, torch.from_numpy(Q).cuda(), 8, precision=p, rerank_R=24, algo=gf.GF_ALGO_LEAF, ctas_per_sm=ctas)
    assert gf.gf_kernel_status() == 0
    offs, ids = oracle.candidates(F, oracle.descend(F, Q))
    oi, od, _ = screen.screened_search(F, X, Q, 8, 24, prec, offs, ids)
    assert_screened_close(X, Q, gi.cpu().numpy(), gd.cpu().numpy(), oi, od, offs, ids, prec, 24, "norm")


@pytest.mark.parametrize("d", [8177, 8208, 50_001, 56_000])
@pytest.mark.parametrize("precision", ["bf16", "fp8"])
def test_leaf_merge_rescores_long_rows(gf, d, precision):
    """Rows on both sides of the merge's own set in length, up to what a CTA's shared memory holds.
    One leaf of well separated points: the k nearest of all, which any screen keeps."""
    rng = np.random.default_rng(d)
    X = rng.standard_normal((60, d)).astype(np.float32)
    Q = X[:12] + rng.standard_normal((12, d)).astype(np.float32) * np.float32(0.01)
    G = gf.gf_build(torch.from_numpy(X).cuda(), 1, 64, t=1)
    prec = {"bf16": gf.GF_BF16_RERANK, "fp8": gf.GF_FP8_RERANK}[precision]
    gf.gf_forest_add_screen(G, prec)
    ids, dists = gf.gf_query(G, torch.from_numpy(Q).cuda(), 1, precision=prec, rerank_R=32, algo=gf.GF_ALGO_LEAF)
    want = np.square(X[:12].astype(np.float64) - Q).sum(1)
    assert ids.cpu().numpy()[:, 0].tolist() == list(range(12))
    # float32 sums of d squares by 32 lanes: at most d / 32 + 10 roundings of 2^-24 each
    assert np.all(np.abs(dists.cpu().numpy()[:, 0] - want) <= want * (d / 32 + 10) * 2.0 ** -24)


@pytest.mark.parametrize("scale", [1e-17, 1.0, 4e17])
@pytest.mark.parametrize("d", [7, 300, 1025])
def test_bf16_norms_of_small_and_large_values(gf, scale, d):
    """The screen ranks by |x|^2 - 2 x q: norms whose squares leave float32's comfortable range."""
    rng = np.random.default_rng(d)
    s = np.float32(scale * (300 / d) ** 0.5)
    X = rng.standard_normal((60, d)).astype(np.float32) * s
    Q = X[:12] + rng.standard_normal((12, d)).astype(np.float32) * (s * np.float32(0.03))
    G = gf.gf_build(torch.from_numpy(X).cuda(), 1, 64, t=1)
    gf.gf_forest_add_screen(G, gf.GF_BF16_RERANK)
    ids, dists = gf.gf_query(G, torch.from_numpy(Q).cuda(), 1, precision=gf.GF_BF16_RERANK, rerank_R=32, algo=gf.GF_ALGO_LEAF)
    want = np.square(X[:12].astype(np.float64) - Q).sum(1)
    assert ids.cpu().numpy()[:, 0].tolist() == list(range(12))
    # float32 sums of d squares by 32 lanes, plus a float32 subnormal step a square
    assert np.all(np.abs(dists.cpu().numpy()[:, 0] - want) <= want * (d / 32 + 10) * 2.0 ** -24 + d * 2.0 ** -148)
