"""Third-order terms with few nodes per cell: the forward runs over records beside the tiles
(default options), right on both sides of the rule, and no slower than over records alone.
"""
import pytest

from oracle import anova
from paper_2010_10199_gb300 import inputs

from gpu_util import cplx_dev, to_dev
from test_gpu_trafo import _pair_check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gft():
    import torch
    from paper_2010_10199_gb300 import build, gft as g
    assert torch.cuda.is_available()
    build.build()
    g.load()
    return g


# n = 12, 20: five nodes per cell at 8640 and 40000
@pytest.mark.parametrize("N3,M", [(6, 1), (6, 33), (6, 1999), (6, 8639), (6, 8640), (10, 3001), (10, 39999), (10, 40000)])
def test_both_sides_of_the_rule(gft, N3, M):
    terms = anova.term_set(4, 3)
    _pair_check(gft, inputs.uniform_points(7, 4, M), terms, [(0, 32, 16, N3)[len(u)] for u in terms])


@pytest.mark.parametrize("basis", [0, 1])
def test_mixed_grids(gft, basis):
    """Terms of every order and of several grids; the records' slots are of two sizes."""
    import torch
    from oracle import ndct, ndft
    from gpu_util import f32_nodes, host, rel_l2
    M = 2001
    terms = [(), (2,), (0, 1, 2), (0, 3), (1, 2, 3), (3,), (0, 1, 3)]
    bw = [0, 40, 10, 20, 6, 12, 8] if not basis else [0, 20, 5, 12, 3, 15, 4]
    x = inputs.uniform(3, 8, 4 * M).reshape(4, M) - (0.0 if basis else 0.5)
    P = gft.Plan(to_dev(x, torch.float32), terms, bw, basis=basis)
    fhat, y = inputs.complex_normal(5, 2, P.n_coeffs), inputs.complex_normal(5, 4, M)
    ref = ndct if basis else ndft
    assert rel_l2(host(P.trafo(cplx_dev(fhat))), ref.trafo(f32_nodes(x), terms, bw, fhat)) <= 1e-5
    assert rel_l2(host(P.adjoint(cplx_dev(y))), ref.adjoint(f32_nodes(x), terms, bw, y)) <= 1e-5


def _ms(P):
    import torch
    fhat = cplx_dev(inputs.complex_normal(1, 2, P.n_coeffs))
    times = []
    for _ in range(4):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(20):
            P.trafo(fhat)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b) / 20)
    return min(times)


@pytest.mark.parametrize("d,by,M", [(10, (64, 24, 10), 3000), (6, (64, 16, 8), 2000)])
def test_forward_is_as_fast_as_over_records(gft, d, by, M):
    """Over tiles it took three to four times as long at these sizes."""
    import torch
    terms = anova.term_set(d, 3)
    bw = [by[len(u) - 1] if u else 0 for u in terms]
    x = to_dev(inputs.uniform_points(7, d, M), torch.float32)
    P, Q = gft.Plan(x, terms, bw), gft.Plan(x, terms, bw, cell_kernel=1)
    assert gft.anova_debug_plan_form(P.handle) == gft.FORM_TILES
    assert _ms(P) <= 1.5 * _ms(Q)
