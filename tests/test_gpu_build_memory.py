"""The build's memory that it can do without (the fixed-point copy of the points and its sums)."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gf():
    import paper_1603_09596_gb300 as g
    g.lib()
    yield g
    g.gf_debug_fail_alloc(-1)


@pytest.mark.parametrize("n,d,T,p", [(20_000, 48, 8, 40), (3000, 300, 2, 16)])
def test_build_without_its_spare_memory_gives_the_same_forest(gf, n, d, T, p):
    """Every allocation of a build is made to fail in turn: all but one fail the build, and without that
    one (the refusal is used up: the screen added next gets its memory) the forest is the same."""
    X, _ = synth.mixture(n, d, 1, "B", seed=91)
    Xg = torch.from_numpy(X).cuda()
    ref = gf.gf_build(Xg, T, p, seed=3)
    want = gf.gf_forest_export(ref)
    ref.free()
    for after in range(32):
        gf.gf_debug_fail_alloc(after)
        try:
            F = gf.gf_build(Xg, T, p, seed=3)
        except gf.GFError as e:
            assert e.code == gf.GF_ENOMEM
            continue
        gf.gf_forest_add_screen(F, gf.GF_BF16_RERANK)
        gf.gf_debug_fail_alloc(-1)
        assert all(np.array_equal(a, b) for a, b in zip(gf.gf_forest_export(F), want))
        F.free()
        break
    else:
        pytest.fail("every refused allocation failed the build")
    assert after >= 3
