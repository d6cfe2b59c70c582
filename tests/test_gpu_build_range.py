"""Builds of points at the ends of float32's range, where the variances leave it."""
import numpy as np
import pytest
import torch

import oracle
import synth
from parity import check_forest
from test_gpu_build import gpu_build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gf():
    import paper_1603_09596_gb300 as g
    g.lib()
    return g


@pytest.mark.parametrize("form", ["node", "global", "reflected"])
@pytest.mark.parametrize("n,d,T,p", [(9001, 90, 2, 300), (2000, 101, 3, 40), (600, 5, 2, 10)])
def test_variances_beyond_float32_count_as_equal_largest(gf, form, n, d, T, p):
    """Points of about 1e24: every variance overflows, so the ranking is that of the dimensions and the
    drawn one is the draw itself; the rest of the forest is a forest of those dimensions."""
    X, _ = synth.mixture(n, d, 1, "A", seed=n)
    X = X * np.float32(2.0 ** 80)
    scope = gf.GF_VAR_GLOBAL if form == "global" else gf.GF_VAR_NODE
    U = np.zeros((T, d), np.float32) if form == "reflected" else None  # (x - 0 u: the points themselves)
    G, F = gpu_build(gf, X, T, p, t=5, var_scope=scope, seed=3, U=U)
    for tree in range(T):
        assert F.split_dim[tree].tolist() == [oracle.node_draw(3, tree, j) % 5 for j in range(F.split_dim.shape[1])]
    check_forest(F, X, 5, 3, 1, 0, check_dims=False)


def ramp(X):    # dimensions of every size at which squares of float32 vanish, pair by pair of columns
    return X * (10.0 ** np.linspace(-26, -9, X.shape[1])).astype(np.float32)


def steep(X):   # from vanishing squares to overflowing ones
    return X * (10.0 ** np.linspace(-30, 30, X.shape[1])).astype(np.float32)


def speck(X):   # ordinary points, one dimension in three far below them, one dimension far above
    X[:, ::3] *= np.float32(1e-22)
    X[:, 7] *= np.float32(1e13)
    return X


def faint(X):   # equal spreads, at which float32 keeps a few bits of the squares
    return (np.random.default_rng(X.shape[0]).standard_normal(X.shape) * 1e-22).astype(np.float32)


SCALES = [1e-12, 1e-15, 1e-16, 1e-17, 1e-18, 1e-20, 1e-22, 1e-26, 1e-37, 1e15, 1e19]


@pytest.mark.parametrize("change", SCALES + [ramp, steep, speck, faint])
@pytest.mark.parametrize("n,d,T,p", [(9001, 90, 2, 300), (2500, 101, 3, 20), (3000, 40, 2, 30)])
def test_fixed_point_bounds_hold_where_squares_leave_float32(gf, change, n, d, T, p):
    """Reflections by the zero vector leave the points as they are and the build without the bounds: it
    sums every dimension, and the forest has to be that one, node for node."""
    X, _ = synth.mixture(n, d, 1, "B", seed=n + d)
    X = np.ascontiguousarray(change(X) if callable(change) else X * np.float32(change))
    _, A = gpu_build(gf, X, T, p, t=5, seed=4)
    _, B = gpu_build(gf, X, T, p, t=5, seed=4, U=np.zeros((T, d), np.float32))
    assert np.array_equal(A.split_dim, B.split_dim)
    assert np.array_equal(A.split_val, B.split_val)
    assert np.array_equal(A.perm, B.perm)


@pytest.mark.parametrize("n", [2, 2047, 2048, 2049])
def test_builds_around_the_fixed_point_pass_smallest_size(gf, n):
    X, _ = synth.mixture(n, 70, 1, "B", seed=n)
    _, A = gpu_build(gf, X, 3, 8, t=5, seed=4)
    _, B = gpu_build(gf, X, 3, 8, t=5, seed=4, U=np.zeros((3, 70), np.float32))
    assert np.array_equal(A.split_dim, B.split_dim)
    assert np.array_equal(A.split_val, B.split_val)
    assert np.array_equal(A.perm, B.perm)


def two_far(X):     # two far points set every dimension's step: the upper nodes stay undecided, small ones not
    X = np.random.default_rng(1).standard_normal(X.shape).astype(np.float32)
    X[0], X[1] = 1000.0, -1000.0
    return X


def one_far(X):     # no node without it tells its dimensions apart
    X[0] = 1e6
    return X


def tied(X):        # three columns over and over
    return np.tile(X[:, :3], (1, X.shape[1]))[:, :X.shape[1]]


@pytest.mark.parametrize("change", [two_far, one_far, tied])
@pytest.mark.parametrize("n,d,T,p", [(20_000, 300, 3, 20), (40_000, 90, 1, 9), (5000, 260, 40, 700), (3000, 600, 600, 5)])
def test_levels_the_bounds_leave_undecided(gf, change, n, d, T, p):
    """The pass stops where it decides too few nodes and may come back (by derived sums or direct ones; the
    last shape has more nodes than a sums buffer)."""
    X, _ = synth.mixture(n, d, 1, "A", seed=n)
    X = np.ascontiguousarray(change(X))
    _, A = gpu_build(gf, X, T, p, t=3, seed=4)
    _, B = gpu_build(gf, X, T, p, t=3, seed=4, U=np.zeros((T, d), np.float32))
    assert np.array_equal(A.split_dim, B.split_dim)
    assert np.array_equal(A.split_val, B.split_val)
    assert np.array_equal(A.perm, B.perm)
