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
