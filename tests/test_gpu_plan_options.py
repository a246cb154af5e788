"""Options that name a part of the NFFT are obeyed at bandwidths that a default plan sums
directly: a window or oversampling study measures the grids that it asked for."""
import numpy as np
import pytest

from oracle import anova, ndft
from paper_2010_10199_gb300 import inputs

from gpu_util import cplx_dev, f32_nodes, host, rel_l2, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gft():
    from paper_2010_10199_gb300 import build, gft as g
    build.build()
    g.load()
    return g


@pytest.mark.parametrize("kw,nfft", [({}, False), (dict(eps=1e-4), False), (dict(eps=1e-7), False), (dict(sigma=2.0), True),
                                     (dict(sigma=1.75), True), (dict(window_m_row=3), True), (dict(window_m_row=4), True),
                                     (dict(n_ctas=1), True), (dict(node_sort=-1), True), (dict(cell_kernel=1), True)])
def test_which_options_keep_the_nfft(gft, kw, nfft):
    import torch
    terms = anova.term_set(5, 2)
    bw = [0] + [16] * 5 + [8] * 10
    P = gft.Plan(to_dev(inputs.uniform_points(3, 5, 2000), torch.float32), terms, bw, **kw)
    assert (gft.anova_debug_plan_form(P.handle) != gft.FORM_DIRECT) == nfft


def test_a_narrow_window_shows_its_error(gft):
    """6 row taps hold 3e-5 but not the 1e-6 that FP32 sums reach at this size."""
    import torch
    x = inputs.uniform_points(3, 5, 2000)
    terms = anova.term_set(5, 2)
    bw = [0] + [16] * 5 + [8] * 10
    y = inputs.complex_normal(1, 4, 2000)
    ref = ndft.adjoint(f32_nodes(x), terms, bw, y)
    err = [rel_l2(host(gft.Plan(to_dev(x, torch.float32), terms, bw, **kw).adjoint(cplx_dev(y))), ref)
           for kw in ({}, dict(window_m_row=3))]
    assert err[0] <= 1e-6 < err[1] <= 3e-5
