"""The shapes of the direct sums' parity tests are summed directly, those of the tile tests
run over tiles: a change of the rule between them must not move a test to other kernels
unseen."""
import itertools

import pytest

import test_gpu_direct as direct
import test_gpu_tiles as tiles
from gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gft():
    from paper_2010_10199_gb300 import build, gft as g
    build.build()
    g.load()
    return g


@pytest.mark.parametrize("basis,shape", direct.SHAPES)
def test_direct_shapes(gft, basis, shape):
    for M in (1, 31, 65, 1999, 2001, 4133):
        P = direct._case(gft, basis, shape[0], shape[1], M)[0]
        assert gft.anova_debug_plan_form(P.handle) == gft.FORM_DIRECT, M


@pytest.mark.parametrize("basis,shape,M", [(0, (4, (26, 6, 4)), 40001), (0, (6, (16, 10)), 22222), (1, (5, (40, 9)), 20481),
                                           (0, (20, (8,)), 5), (0, (40, (16, 8)), 700), (0, (5, (16, 6, 4)), 3000)])
def test_larger_direct_shapes(gft, basis, shape, M):
    P = direct._case(gft, basis, shape[0], shape[1], M)[0]
    assert gft.anova_debug_plan_form(P.handle) == gft.FORM_DIRECT


@pytest.mark.parametrize("bw", [(64,), (30, 32), (16, 8), (16, 8, 4), (20, 12, 10)])
def test_tile_shapes(gft, bw):
    import torch
    for counts in (tiles.COUNTS, [1] * 9, [16], [8], [700]):
        x = tiles._nodes(counts, 3)
        terms = [u for s in range(len(bw) + 1) for u in itertools.combinations(range(3), s)]
        P = gft.Plan(to_dev(x, torch.float32), terms, [bw[len(u) - 1] if u else 0 for u in terms], n_ctas=5)
        assert gft.anova_debug_plan_form(P.handle) == gft.FORM_TILES, len(counts)
