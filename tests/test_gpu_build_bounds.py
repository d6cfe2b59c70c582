"""The build's fixed-point variance bounds (which dimensions can be among the t of largest variance)
on data that stretch them: the forest must still be the oracle's, node for node."""
import numpy as np
import pytest
import torch

import oracle
import synth
from test_gpu_build import assert_same_forest, gpu_build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gf():
    import paper_1603_09596_gb300 as g
    g.lib()
    return g


def offset(X):      # all values far from zero: few float32 digits left for the spread
    return X + np.float32(4096.0)


def outliers(X):    # a few far values set a coarse step for some dimensions
    X[5, ::7] = 3e4
    X[-3, 3::5] = -2e4
    return X


def twins(X):       # 80 equal columns of the largest variance: more than a node's list holds
    X[:, :80] = 10 * X[:, :1]
    return X


def flat(X):        # constant dimensions, and some whose range is too small for the fixed point
    X[:, 1::3] = 2.5
    X[:, 2::9] *= np.float32(1e-33)
    return X


def bytes_(X):      # small integers: exact variance ties between dimensions are rare, equal values common
    return synth.quantize_u8(X, 20.0)


# (n, d, T, p): chunked levels and small ones, odd widths, one row group and many, deep trees
@pytest.mark.parametrize("change", [offset, outliers, twins, flat, bytes_])
@pytest.mark.parametrize("n,d,T,p", [(20_011, 101, 3, 40), (9000, 1100, 2, 300), (70_000, 90, 2, 4000)])
def test_build_with_stretched_bounds_matches_oracle(gf, change, n, d, T, p):
    X, _ = synth.mixture(n, d, 1, "B", seed=n + d)
    X = np.ascontiguousarray(change(X))
    G, Fg = gpu_build(gf, X, T, p, seed=5)
    Fo = oracle.build_forest(X, T, p, seed=5)
    assert_same_forest(X, Fg, Fo, 5)


def test_build_derived_sums_agree_with_direct_ones(gf):
    """Widths past 65,536 nodes' sums of 16 bytes a dimension: the last levels sum every node."""
    X, _ = synth.mixture(70_000, 600, 1, "B", seed=12)
    G, Fg = gpu_build(gf, X, 4, 2, seed=6)
    Fo = oracle.build_forest(X, 4, 2, seed=6)
    assert_same_forest(X, Fg, Fo, 5)


@pytest.mark.parametrize("most", [1, 3, 90])  # float32 steps a dimension spans
@pytest.mark.parametrize("n,d,T,p", [(20_011, 101, 3, 40), (9000, 1100, 2, 300)])
def test_build_on_few_float32_steps_equals_the_shifted_build(gf, most, n, d, T, p):
    """Small even integers on 2^24, where float32 steps by 2: all differences between points, and so
    the sums, the choices and the order, are those of the integers themselves."""
    rng = np.random.default_rng(n + most)
    span = rng.integers(1, most + 1, d)
    X = 2.0 * rng.binomial(span, rng.uniform(0.05, 0.95, d), (n, d))
    _, A = gpu_build(gf, np.ascontiguousarray(X, dtype=np.float32), T, p, seed=5)
    _, B = gpu_build(gf, np.ascontiguousarray(X + 2.0 ** 24, dtype=np.float32), T, p, seed=5)
    assert np.array_equal(A.split_dim, B.split_dim)
    assert np.array_equal(A.perm, B.perm)
    assert np.array_equal(A.split_val + np.float32(2.0 ** 24), B.split_val)
