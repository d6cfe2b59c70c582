"""The screening copies and their norms at the ends of float32's range."""
import numpy as np
import pytest
import torch

from oracle import screen
from parity import U32

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gf():
    import paper_1603_09596_gb300 as g
    g.lib()
    return g


@pytest.mark.parametrize("d", [5, 10, 16, 33])
def test_fp8_rows_too_small_for_the_inverse_scale(gf, d):
    """448 / a overflows for a row whose largest value a lies below 1.3e-36: its codes are +-448 and the
    padding's stay zero, so the row's screened distances are those of the oracle's codes."""
    rng = np.random.default_rng(d)
    n, m = 200, 3
    X = rng.uniform(0.5, 1.0, (n, d)).astype(np.float32) * rng.choice([-1.0, 1.0], (n, d)).astype(np.float32)
    X[::2] *= np.float32(1e-37)
    Q = rng.standard_normal((m, d)).astype(np.float32)
    F = gf.gf_build(torch.from_numpy(X).cuda(), 1, n, t=1, seed=1)
    gf.gf_forest_add_screen(F, gf.GF_FP8_RERANK)
    cand = torch.arange(n, dtype=torch.int32, device="cuda").repeat(m, 1)
    nc = torch.full((m,), n, dtype=torch.int32, device="cuda")
    got = gf.gf_score_screened(F, torch.from_numpy(Q).cuda(), cand, nc, gf.GF_FP8_RERANK).cpu().numpy()
    # the tiny rows' values, and the others as the oracle rounds them
    deq = np.sign(X) * 448.0 * (np.abs(X).max(1, keepdims=True) / np.float32(448.0)).astype(np.float64)
    deq[1::2] = screen.dequantized_rows(X, np.arange(1, n, 2), "fp8")
    for i in range(m):
        want = ((deq - Q[i].astype(np.float64)) ** 2).sum(1)
        assert np.all(np.abs(got[i] - want) <= (np.ceil(d / 32) + 16) * U32 * want)  # parity.screen_bounds, "direct"
