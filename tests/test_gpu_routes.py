"""Which kernels GF_ALGO_AUTO takes, by what that means for the caller."""
import ctypes as C

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gf():
    import paper_1603_09596_gb300 as g
    g.lib()
    return g


def cudart():
    for name in ("libcudart.so.13", "libcudart.so"):
        try:
            return C.CDLL(name)
        except OSError:
            pass
    pytest.skip("the CUDA runtime cannot be opened by name")


# calls within the sort kernel's reach: the staged steps', and the single launch's
@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp8"])
@pytest.mark.parametrize("n,d,T,p,m", [(10_000, 960, 16, 64, 100), (50_000, 512, 16, 256, 27), (10_000, 128, 8, 32, 100)])
def test_small_calls_are_captured_without_memory_nodes(gf, prec, n, d, T, p, m):
    """Two instances of the captured graph live side by side and give the uncaptured call's answers: a
    graph that allocates can have only one."""
    rt = cudart()
    X, Q = synth.mixture(n, d, m, "B", seed=81, qseed=82)
    F = gf.gf_build(torch.from_numpy(X).cuda(), T, p, seed=1)
    P, R = gf.PRECISIONS[prec], 0 if prec == "fp32" else 32
    if P:
        gf.gf_forest_add_screen(F, P)
    Qg = torch.from_numpy(Q).cuda()
    want = gf.gf_query(F, Qg, 10, precision=P, rerank_R=R, algo=gf.GF_ALGO_SORT)
    out = (torch.empty_like(want[0]), torch.empty_like(want[1]))
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = C.c_void_p()
    st = C.c_void_p(s.cuda_stream)
    assert rt.cudaStreamBeginCapture(st, 2) == 0  # relaxed
    try:
        gf.gf_query(F, Qg, 10, precision=P, rerank_R=R, out=out, stream=s)
    finally:
        assert rt.cudaStreamEndCapture(st, C.byref(graph)) == 0
    instances = []
    try:
        for _ in range(2):
            h = C.c_void_p()
            assert rt.cudaGraphInstantiate(C.byref(h), graph, C.c_ulonglong(0)) == 0
            instances.append(h)
        for h in instances:
            out[0].zero_()
            torch.cuda.synchronize()
            assert rt.cudaGraphLaunch(h, st) == 0
            torch.cuda.synchronize()
            assert torch.equal(out[0], want[0]) and torch.equal(out[1], want[1])
    finally:
        rt.cudaGetLastError()
        for h in instances:
            rt.cudaGraphExecDestroy(h)
        rt.cudaGraphDestroy(graph)


# (n, d, T, p, m, k): on both sides of the lines between the sort kernel and the staged path or the single
# launch: leaves of 2 to 9 points, 8 and 9 candidates, 96 and 97, fewer than k and more, short rows and long
@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp8"])
@pytest.mark.parametrize("n,d,T,p,m,k", [
    (4217, 26, 40, 3, 300, 5), (4217, 26, 12, 9, 400, 5), (512, 300, 12, 8, 400, 5), (4000, 128, 4, 2, 1100, 3),
    (900, 128, 9, 1, 1100, 3), (3072, 1100, 8, 12, 40, 10), (3104, 1100, 1, 97, 50, 10), (5000, 2200, 6, 20, 30, 128),
    (3000, 5, 20, 3, 9000, 2), (30_000, 60, 4, 32, 6000, 33), (2000, 1500, 4, 1, 3, 1),
])
def test_routes_of_few_candidates_answer_alike(gf, prec, n, d, T, p, m, k):
    X, Q = synth.mixture(n, d, m, "B", seed=83, qseed=84)
    F = gf.gf_build(torch.from_numpy(X).cuda(), T, p, t=min(5, d), seed=1)
    P, R = gf.PRECISIONS[prec], 0 if prec == "fp32" else max(k, 40)  # (no leaf-major batch at 40)
    if P:
        gf.gf_forest_add_screen(F, P)
    Qg = torch.from_numpy(Q).cuda()
    for order in (gf.GF_ORDER_AUTO, gf.GF_ORDER_GIVEN):
        a = gf.gf_query(F, Qg, k, precision=P, rerank_R=R, order=order)
        if prec == "fp32" and k <= 32 and m >> F.info.L >= 4:  # leaf-major: another order of additions
            continue
        for algo in (gf.GF_ALGO_SORT, gf.GF_ALGO_STREAM):
            b = gf.gf_query(F, Qg, k, precision=P, rerank_R=R, algo=algo)
            assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


def test_tuning_leaves_autos_path_alone(gf):
    """One query on a forest tuned to any shape takes the path, and the time, of an untuned one: the staged
    steps are some ten times as fast here as the streaming kernel with any shape."""
    from paper_1603_09596_gb300 import autotune
    g = torch.Generator(device="cuda").manual_seed(85)
    X, Q = torch.randn(200_000, 512, generator=g, device="cuda"), torch.randn(1, 512, generator=g, device="cuda")

    def ms(F, **kw):
        return autotune._time(lambda: gf.gf_query(F, Q, 10, **kw), reps=15)

    F = gf.gf_build(X, 32, 1024, seed=1)
    plain, stream = ms(F), ms(F, algo=gf.GF_ALGO_STREAM)
    assert stream > 4 * plain
    for shape in ((16, 0, 0, 0), (4, 2, 0, 2), (8, 1, 0, 0)):
        gf.gf_forest_set_tuning(F, gf.GF_FP32, *shape)
        assert ms(F) < 2 * plain
    res = autotune.tune(F, Q, 10, gf.GF_FP32)
    assert res["ms"] < 2 * plain < res["shape_ms"]
    assert ms(F) < 2 * plain


# Device bitmaps in three waves of reordered queries (n above 1.8 million, T ceil(n / 2^L) above 8192), and the
# single launch with rows of 513 to 1024 dimensions.
@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp8"])
@pytest.mark.parametrize("n,d,T,p,m,k", [(2_000_000, 4, 20, 1000, 1500, 33), (3000, 600, 8, 50, 200, 10), (3000, 1024, 8, 50, 200, 10)])
def test_staged_path_in_its_less_usual_forms(gf, prec, n, d, T, p, m, k):
    X, Q = synth.mixture(n, d, m, "A", seed=87, qseed=88)
    F = gf.gf_build(torch.from_numpy(X).cuda(), T, p, t=min(5, d), seed=1)
    P, R = gf.PRECISIONS[prec], 0 if prec == "fp32" else 40
    if P:
        gf.gf_forest_add_screen(F, P)
    Qg = torch.from_numpy(Q).cuda()
    counts = [torch.zeros(m, dtype=torch.int32, device="cuda") for _ in range(2)]
    # (asking for the candidates' number keeps a batch off the leaf-major path)
    a = gf.gf_query(F, Qg, k, precision=P, rerank_R=R, ncand_out=counts[0])
    b = gf.gf_query(F, Qg, k, precision=P, rerank_R=R, algo=gf.GF_ALGO_STREAM, ncand_out=counts[1])
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and torch.equal(counts[0], counts[1])
