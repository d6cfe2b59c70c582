"""The screening copies and their norms at the ends of float32's range."""
import ctypes as C
import math
import os
import subprocess

import numpy as np
import pytest
import torch

from conftest import ROOT
from oracle import screen
from paper_1603_09596_gb300 import _build
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


@pytest.mark.parametrize("d", [1, 33, 960, 3000])
def test_sums_of_squares_round_like_float64_ones(tmp_path, d):
    """bfloat16 values over twenty binary orders: a lane rounds three times every 32 squares (2^-53 of a sum
    that is at most the total), and the warp five times more."""
    lib = str(tmp_path / "squares.so")
    subprocess.run([_build.nvcc(), "-gencode", _build.GENCODE, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                    "-cudart", "shared", "-I", _build.CSRC, "-o", lib,
                    os.path.join(ROOT, "tests", "native", "square_sums.cu")], check=True)
    rng = np.random.default_rng(d)
    n = 300
    X = screen.bf16_round((rng.standard_normal((n, d)) * 2.0 ** rng.uniform(-10, 10, (n, d))).astype(np.float32))
    X = np.ascontiguousarray(X)
    out = np.zeros(n)
    f = C.CDLL(lib).square_sums
    f.argtypes = [C.c_void_p, C.c_longlong, C.c_int, C.c_void_p]
    assert f(X.ctypes.data, n, d, out.ctypes.data) == 0
    want = np.array([math.fsum(r * r) for r in X.astype(np.float64)])
    assert np.all(np.abs(out - want) <= (3 * -(-d // 1024) + 6) * 2.0 ** -53 * want)
