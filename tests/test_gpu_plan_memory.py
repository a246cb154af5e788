"""Plans where memory for a form of the nodes is lacking take one that needs less: the NFFT
in place of direct sums, records in place of tiles."""
import numpy as np
import pytest

from oracle import ndft
from paper_2010_10199_gb300 import inputs

from gpu_util import cplx_dev, f32_nodes, host, rel_l2, to_dev

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def gft():
    from paper_2010_10199_gb300 import build, gft as g
    build.build()
    g.load()
    return g


def _forms_under_failures(gft, **kw):
    """Per k, the form of the plan whose k-th allocation failed (None: no memory); every
    plan that is built is right, and all memory comes back."""
    import torch
    w = inputs.c1_small()
    x, terms, bw, y = w["x"], w["terms"], w["bandwidths"], w["y"]
    xd, xo = to_dev(x, torch.float32), f32_nodes(x)
    fhat = inputs.decaying_coefficients(5, terms, bw)
    f_ref, g_ref = ndft.trafo(xo, terms, bw, fhat), ndft.adjoint(xo, terms, bw, y)
    fh_d, y_d = cplx_dev(fhat), cplx_dev(y)
    for more in ({}, dict(n_ctas=4), dict(cell_kernel=1), dict(node_sort=-1)):   # loads every kernel module
        P = gft.Plan(xd, terms, bw, **more)
        P.trafo(fh_d), P.adjoint(y_d)
        P.close()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    forms = []
    try:
        for k in range(1, 48):
            gft.anova_debug_fail_allocation(k)
            try:
                P = gft.Plan(xd, terms, bw, **kw)
            except gft.AnovaError as e:
                assert e.status == -3, f"k={k}"
                forms.append(None)
                continue
            finally:
                gft.anova_debug_fail_allocation(0)
            forms.append(gft.anova_debug_plan_form(P.handle))
            assert rel_l2(host(P.trafo(fh_d)), f_ref) <= TOL and rel_l2(host(P.adjoint(y_d)), g_ref) <= TOL, f"k={k}"
            P.close()
    finally:
        gft.anova_debug_fail_allocation(0)
    torch.cuda.synchronize()
    assert free0 - torch.cuda.mem_get_info()[0] <= (4 << 20)
    return forms


def test_direct_sums_without_memory_become_the_nfft(gft):
    forms = _forms_under_failures(gft)
    # units, items, two counters, exp(2 pi i x), the adjoint's and the forward's partial
    # sums, two host lists
    assert forms.count(gft.FORM_TILES) == 9
    assert forms.count(None) >= 20 and forms[-1] == gft.FORM_DIRECT


def test_tiles_without_memory_become_records(gft):
    forms = _forms_under_failures(gft, n_ctas=4)
    # the tiles, their cells and their counts; without accumulators the tiles stay
    assert forms.count(gft.FORM_RECORDS) == 3 and gft.FORM_OWN_ORDER not in forms
    assert forms.count(None) >= 20 and forms[-1] == gft.FORM_TILES


@pytest.mark.parametrize("M,kw", [(40000, dict(n_ctas=1)), (39000, {})], ids=["tiles", "records_beside"])
def test_sorting_without_memory(gft, M, kw):
    """Many order-1 terms beside a third-order one: the sorts' histograms (8000 cells per term,
    two slices into tiles) do not fit in the partial grids.  Where they cannot be allocated one
    slice's have to do, and the forward runs over the tiles instead of records beside them."""
    import torch
    terms = [(t,) for t in range(100)] + [(0, 1, 2)]
    bw = [16] * 100 + [10]
    x = inputs.uniform_points(5, 100, M)
    xd, xo = to_dev(x, torch.float32), f32_nodes(x)
    fhat, y = inputs.complex_normal(5, 2, 100 * 15 + 9 ** 3), inputs.complex_normal(5, 4, M)
    f_ref, g_ref = ndft.trafo(xo, terms, bw, fhat), ndft.adjoint(xo, terms, bw, y)
    built = []
    try:
        for k in range(1, 48):
            gft.anova_debug_fail_allocation(k)
            try:
                P = gft.Plan(xd, terms, bw, **kw)
            except gft.AnovaError as e:
                assert e.status == -3, f"k={k}"
                built.append(False)
                continue
            finally:
                gft.anova_debug_fail_allocation(0)
            built.append(True)
            assert rel_l2(host(P.trafo(cplx_dev(fhat))), f_ref) <= TOL and rel_l2(host(P.adjoint(cplx_dev(y))), g_ref) <= TOL
            P.close()
    finally:
        gft.anova_debug_fail_allocation(0)
    # every allocation after those that a plan cannot do without has something in its place
    assert built.count(False) >= 15 and all(built[built.index(True):])
