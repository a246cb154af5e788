"""The kernels over node tiles at bandwidths that a default plan sums directly: an explicit
chunk count keeps the plan on the NFFT.  Long runs of one cell, axes shorter than the
window, third-order cosine terms, scales far from 1, non-finite data, failing
allocations of the sorted copy; every test asserts which kernels its plan runs.

Bar of the other parity tests: 1e-5 relative l2 for the whole vectors, every adjoint
block and every order alone.
"""
import numpy as np
import pytest

from oracle import anova, ndct, ndft
from paper_2010_10199_gb300 import inputs

from gpu_util import cplx_dev, f32_nodes, host, rel_l2, to_dev
from test_gpu_trafo import _pair_check

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def gft():
    import torch
    from paper_2010_10199_gb300 import build, gft as g
    assert torch.cuda.is_available()
    build.build()
    g.load()
    return g


class _Forms:
    """The binding, with every plan's form checked."""

    def __init__(self, gft, form):
        self.gft, self.form = gft, form

    def Plan(self, *a, **kw):
        P = self.gft.Plan(*a, **kw)
        assert self.gft.anova_debug_plan_form(P.handle) == self.form
        return P


def _tiles(gft):
    return _Forms(gft, gft.FORM_TILES)


def _bw(terms, *by_order):
    return [by_order[len(u) - 1] if u else 0 for u in terms]


def test_forms(gft):
    import torch
    x = to_dev(inputs.uniform_points(3, 5, 2000), torch.float32)
    terms = anova.term_set(5, 2)
    for want, bw, kw in ((gft.FORM_DIRECT, (16, 8), {}), (gft.FORM_TILES, (64, 32), {}),
                         (gft.FORM_TILES, (16, 8), dict(n_ctas=4)), (gft.FORM_RECORDS, (16, 8), dict(cell_kernel=1)),
                         (gft.FORM_OWN_ORDER, (16, 8), dict(node_sort=-1)),
                         (gft.FORM_TILES, (16, 8), dict(precision=gft.PREC_F16)),
                         (gft.FORM_RECORDS, (16, 8), dict(precision=gft.PREC_F64))):
        P = gft.Plan(x, terms, _bw(terms, *bw), **kw)
        assert gft.anova_debug_plan_form(P.handle) == want, (bw, kw)
    assert gft.anova_debug_plan_form(None) == -1


@pytest.mark.parametrize("M", [1, 255, 256, 257, 1000, 4099])
def test_ragged_sizes(gft, M):
    terms = anova.term_set(5, 3)
    _pair_check(_tiles(gft), inputs.uniform_points(7, 5, M), terms, _bw(terms, 16, 8, 4), n_ctas=4)


@pytest.mark.parametrize("chunks", [1, 64])
@pytest.mark.parametrize("M", [300000, 300001])
def test_long_cell_runs(gft, M, chunks):
    """Thousands of nodes per cell in every order: sums must not drift with the run."""
    terms = [(), (0,), (1,), (0, 1), (0, 1, 2)]
    _pair_check(_tiles(gft), inputs.uniform_points(20, 3, M), terms, [0, 8, 4, 4, 4], n_ctas=chunks)


@pytest.mark.parametrize("N", [2, 4, 6])
def test_axes_shorter_than_the_window(gft, N):
    """n = 4, 8 and 12 against windows of 8 columns and 8 rows."""
    terms = [(0,), (1, 2), (0, 1, 2)]
    _pair_check(_tiles(gft), inputs.uniform_points(11, 3, 1500), terms, [N] * 3, n_ctas=4)


@pytest.mark.parametrize("N", [2, 4, 6])
def test_axes_shorter_than_the_window_of_6_rows(gft, N):
    """The 6-row window's own error on a sum of 1500 values that cancels to 2 % of their
    magnitudes is 4.2e-5 at N = 2 (FP64 evaluation of the same window), so the tiles are
    compared with the record kernels on the same window; 5e-6 is the bar for rounding."""
    import torch
    terms = [(0,), (1, 2), (0, 1, 2)]
    x = to_dev(inputs.uniform_points(11, 3, 1500), torch.float32)
    P = _tiles(gft).Plan(x, terms, [N] * 3, n_ctas=4, window_m_row=3)
    Q = _Forms(gft, gft.FORM_RECORDS).Plan(x, terms, [N] * 3, n_ctas=4, window_m_row=3, cell_kernel=1)
    fhat, y = cplx_dev(inputs.complex_normal(5, 2, P.n_coeffs)), cplx_dev(inputs.complex_normal(1, 4, 1500))
    assert rel_l2(host(P.trafo(fhat)), host(Q.trafo(fhat))) <= 5e-6
    assert rel_l2(host(P.adjoint(y)), host(Q.adjoint(y))) <= 5e-6


def test_wrap_boundary_nodes(gft):
    x = inputs.uniform_points(13, 3, 600)
    x[:, :50] = -0.5
    x[:, 50:100] = 0.5 - 1e-9
    x[:, 100:150] = x[:, 150:200]
    x[0, 200:260] = 0.49999997
    terms = anova.term_set(3, 3)
    _pair_check(_tiles(gft), x, terms, _bw(terms, 16, 8, 4), n_ctas=4)


@pytest.mark.parametrize("scale", [1e-25, 1.0, 1e25])
def test_scales_of_third_order_terms(gft, scale):
    terms = anova.term_set(4, 3)
    bw = _bw(terms, 32, 16, 10)
    x = inputs.uniform_points(29, 4, 3001)
    _pair_check(_tiles(gft), x, terms, bw, fhat=scale * inputs.decaying_coefficients(3, terms, bw),
                y=scale * inputs.complex_normal(3, 4, x.shape[1]), n_ctas=4)


@pytest.mark.parametrize("M", [500, 20001])
def test_third_order_cosine_terms(gft, M):
    import torch
    x = inputs.uniform(5, 9, 4 * M).reshape(4, M)
    terms = anova.term_set(4, 3)
    bw = _bw(terms, 9, 5, 5)
    P = _tiles(gft).Plan(to_dev(x, torch.float32), terms, bw, basis=gft.BASIS_COS, n_ctas=4)
    fhat, y = inputs.complex_normal(5, 2, P.n_coeffs), inputs.complex_normal(5, 4, M)
    xo = f32_nodes(x)
    assert rel_l2(host(P.trafo(cplx_dev(fhat))), ndct.trafo(xo, terms, bw, fhat)) <= TOL
    assert rel_l2(host(P.adjoint(cplx_dev(y))), ndct.adjoint(xo, terms, bw, y)) <= TOL


@pytest.mark.parametrize("order", [2, 3])
def test_forward_over_tiles_is_deterministic(gft, order):
    import torch
    terms = anova.term_set(6, order)
    bw = _bw(terms, 16, 8, 8)
    x = to_dev(inputs.uniform_points(3, 6, 4001), torch.float32)
    fh = cplx_dev(inputs.decaying_coefficients(3, terms, bw))
    P = _tiles(gft).Plan(x, terms, bw, n_ctas=8)
    f = host(P.trafo(fh))
    assert np.array_equal(f, host(P.trafo(fh)))
    Q = gft.Plan(x, terms, bw, node_sort=-1)
    assert rel_l2(f, host(Q.trafo(fh))) <= 1e-6


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_solvers_report_non_finite_data(gft, bad):
    import torch
    w = inputs.c1_small()
    P = _tiles(gft).Plan(to_dev(w["x"], torch.float32), w["terms"], w["bandwidths"], n_ctas=4)
    yb = w["y"].copy()
    yb[17] = bad
    for solve in (lambda y: P.lsqr(cplx_dev(y), 1e-3, max_it=20), lambda y: P.fista(cplx_dev(y), [1.0], max_it=20)):
        with pytest.raises(gft.AnovaError) as e:
            solve(yb)
        assert e.value.status == -7   # ANOVA_ERR_NOT_FINITE
        assert np.all(np.isfinite(host(solve(w["y"])[0])))   # the plan stays usable


def test_failing_allocations_of_the_sorted_copy(gft):
    import torch
    w = inputs.c1_small()
    x, terms, bw, y = w["x"], w["terms"], w["bandwidths"], w["y"]
    xd, xo = to_dev(x, torch.float32), f32_nodes(x)
    fhat = inputs.decaying_coefficients(5, terms, bw)
    f_ref, g_ref = ndft.trafo(xo, terms, bw, fhat), ndft.adjoint(xo, terms, bw, y)
    fh_d, y_d = cplx_dev(fhat), cplx_dev(y)
    P = _tiles(gft).Plan(xd, terms, bw, n_ctas=4)   # loads every kernel module
    P.trafo(fh_d), P.adjoint(y_d)
    P.close()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    forms = []
    try:
        for k in range(1, 48):
            gft.anova_debug_fail_allocation(k)
            try:
                P = gft.Plan(xd, terms, bw, n_ctas=4)
            except gft.AnovaError as e:
                assert e.status == -3, f"k={k}"
                continue
            finally:
                gft.anova_debug_fail_allocation(0)
            forms.append(gft.anova_debug_plan_form(P.handle))
            assert rel_l2(host(P.trafo(fh_d)), f_ref) <= TOL and rel_l2(host(P.adjoint(y_d)), g_ref) <= TOL, f"k={k}"
            P.close()
    finally:
        gft.anova_debug_fail_allocation(0)
    # without each of the sorted copy's parts (tiles, cells, counts), then with tiles but
    # without each part of the accumulators, then past the last allocation
    assert gft.FORM_TILES not in forms[:3] and forms[3:] == [gft.FORM_TILES] * len(forms[3:]) and len(forms) >= 6
    torch.cuda.synchronize()
    assert free0 - torch.cuda.mem_get_info()[0] <= (4 << 20)
