"""The staged per-query path (what GF_ALGO_AUTO takes when the caller fixes no kernel and no
workspace) answers bit for bit as the streaming kernel, whose answers the oracle checks: at the edges
of its hash set, bitmaps, row blocks, selection and waves."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gf():
    import paper_1603_09596_gb300 as g
    g.lib()
    return g


# (asking for candidate counts keeps every batch off the leaf-major path, which does not report them)
def same_as_stream(gf, F, Q, k, prec="fp32", R=32, checks=0):
    p = gf.PRECISIONS[prec]
    if p:
        gf.gf_forest_add_screen(F, p)
    nc = torch.zeros(Q.shape[0], dtype=torch.int32, device="cuda")
    nr = torch.zeros_like(nc)
    a = gf.gf_query(F, Q, k, precision=p, rerank_R=R if p else 0, checks=checks, ncand_out=nc)
    b = gf.gf_query(F, Q, k, precision=p, rerank_R=R if p else 0, checks=checks, algo=gf.GF_ALGO_STREAM, ncand_out=nr)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and torch.equal(nc, nr)
    c = gf.gf_query(F, Q, k, precision=p, rerank_R=R if p else 0, checks=checks, ncand_out=nc, order=gf.GF_ORDER_GIVEN)
    assert torch.equal(c[0], b[0]) and torch.equal(c[1], b[1])


# (n, d, T, p, m, k): hash set of few ids and at its limit (2 T ceil(n / 2^L) <= 16384) and past it
# (bitmaps), leaf_size 1, one tree of one leaf, rows of 1 to over 256 sixteen-byte pieces, a lone query
SHAPES = [
    (3, 1, 1, 1, 1, 1), (500, 7, 3, 1, 9, 4), (1000, 33, 2, 1000, 5, 128), (4096, 128, 8, 1024, 3, 10),
    (4097, 130, 8, 1025, 2, 10), (8200, 96, 2, 4200, 1, 100), (20_000, 65, 16, 700, 40, 10),
    (3000, 1030, 6, 50, 600, 7), (6000, 257, 12, 30, 1, 1), (30_000, 24, 40, 500, 130, 17),
    (2_000_000, 4, 10, 100, 1100, 5), (2_000_000, 4, 20, 1000, 30, 5),  # bitmaps past shared memory, L = 15
]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp8"])
def test_list_path_equals_streaming(gf, shape, prec):
    n, d, T, p, m, k = shape
    X, Q = synth.mixture(n, d, m, "B", seed=61, qseed=62)
    F = gf.gf_build(torch.from_numpy(X).cuda(), T, p, t=min(5, d), seed=3)
    same_as_stream(gf, F, torch.from_numpy(Q).cuda(), k, prec, R=max(32, k))


@pytest.mark.parametrize("n,T,p,checks,m", [(20_000, 8, 32, 9, 3), (20_000, 4, 16, 700, 50), (9000, 5, 40, 300, 600)])
def test_list_path_priority_search(gf, n, T, p, checks, m):
    X, Q = synth.mixture(n, 48, m, "B", seed=63, qseed=64)
    F = gf.gf_build(torch.from_numpy(X).cuda(), T, p, seed=5)
    same_as_stream(gf, F, torch.from_numpy(Q).cuda(), 10, checks=checks)


def test_list_path_in_waves(gf):
    """60,000 candidates a query and a bitmap of 7.5 KB: about 550 queries fit a wave of the scratch."""
    X, Q = synth.mixture(60_000, 16, 1200, "A", seed=65, qseed=66)
    F = gf.gf_build(torch.from_numpy(X).cuda(), 64, 1000, seed=7)
    same_as_stream(gf, F, torch.from_numpy(Q).cuda(), 40)


def test_selection_with_the_near_points_in_few_groups(gf):
    """One leaf lists its ids in order; the near points fall into 100 of the 256 groups whose minima
    bound the 128th key, so 3100 keys lie below the bound, more than the selection's buffer."""
    n, d = 8000, 8
    rng = np.random.default_rng(67)
    X = rng.standard_normal((n, d)).astype(np.float32)
    X[np.arange(n) % 256 >= 100] += 50.0
    F = gf.gf_build(torch.from_numpy(X).cuda(), 1, n, seed=1)
    Q = torch.from_numpy(rng.standard_normal((3, d)).astype(np.float32)).cuda()
    same_as_stream(gf, F, Q, 128)


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 3e38])
def test_list_path_queries_that_are_not_finite(gf, value):
    X, Q = synth.mixture(5000, 40, 20, "A", seed=68, qseed=69)
    Q[3, 5] = value
    Q[7, :] = value
    F = gf.gf_build(torch.from_numpy(X).cuda(), 6, 64, seed=9)
    Qg = torch.from_numpy(Q).cuda()
    a = gf.gf_query(F, Qg, 5)
    b = gf.gf_query(F, Qg, 5, algo=gf.GF_ALGO_STREAM)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1].view(torch.int32), b[1].view(torch.int32))


def test_list_path_under_capture_and_on_two_streams(gf):
    X, Q = synth.mixture(30_000, 64, 400, "B", seed=70, qseed=71)
    F = gf.gf_build(torch.from_numpy(X).cuda(), 8, 128, seed=11)
    Qg = torch.from_numpy(Q).cuda()
    want = gf.gf_query(F, Qg, 10, algo=gf.GF_ALGO_STREAM)
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    outs = []
    for i in range(6):
        with torch.cuda.stream(streams[i % 2]):
            outs.append(gf.gf_query(F, Qg, 10))
    torch.cuda.synchronize()
    assert all(torch.equal(o[0], want[0]) and torch.equal(o[1], want[1]) for o in outs)
    out = (torch.empty_like(want[0]), torch.empty_like(want[1]))
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        gf.gf_query(F, Qg, 10, out=out)
    for _ in range(2):
        out[0].zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out[0], want[0]) and torch.equal(out[1], want[1])
