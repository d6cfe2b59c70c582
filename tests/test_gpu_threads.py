"""Host threads that query forests of different shapes at once: a kernel's limits are the process's, and
no thread's launch may depend on what another's needs."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gf():
    import paper_1603_09596_gb300 as g
    g.lib()
    return g


# (n, d, T, p) of two forests whose queries run the same kernels with different shared memory, above the
# default limit: bitmaps over the points (staged path), rows of the shortlist's query (one CTA a query)
@pytest.mark.parametrize("algo,shapes", [
    ("auto", [(450_000, 8, 8, 2048), (1_300_000, 8, 8, 2048)]),
    ("stream", [(3000, 13_000, 2, 100), (3000, 30_000, 2, 100)]),
    ("sort", [(3000, 13_000, 2, 100), (3000, 30_000, 2, 100)]),
])
def test_two_threads_with_different_shared_memory(gf, algo, shapes):
    algo = {"auto": gf.GF_ALGO_AUTO, "stream": gf.GF_ALGO_STREAM, "sort": gf.GF_ALGO_SORT}[algo]
    calls, errors = 3000, []
    work = []
    for n, d, T, p in shapes:
        g = torch.Generator(device="cuda").manual_seed(n + d)
        F = gf.gf_build(torch.randn(n, d, generator=g, device="cuda"), T, p, seed=1)
        Q = torch.randn(2, d, generator=g, device="cuda")
        work.append((F, Q, gf.gf_query(F, Q, 5, algo=algo)))
    torch.cuda.synchronize()
    go = threading.Barrier(len(work))

    def run(F, Q, want):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            out = (torch.empty_like(want[0]), torch.empty_like(want[1]))
        go.wait()
        try:
            for _ in range(calls):
                gf.gf_query(F, Q, 5, algo=algo, out=out, stream=stream)
            stream.synchronize()
            assert torch.equal(out[0], want[0]) and torch.equal(out[1], want[1])
        except Exception as e:  # reported by the test's own thread
            errors.append(e)

    threads = [threading.Thread(target=run, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
