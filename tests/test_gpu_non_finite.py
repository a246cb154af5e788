"""Coefficients and nodes that are not finite show in the forward transform, whichever
kernels run it: a coefficient reaches every node, a node coordinate its own node."""
import numpy as np
import pytest

from oracle import anova, ndft
from paper_2010_10199_gb300 import inputs

from gpu_util import cplx_dev, f32_nodes, host, rel_l2, to_dev

pytestmark = pytest.mark.gpu
TOL = 1e-5
M = 3001


@pytest.fixture(scope="module")
def gft():
    from paper_2010_10199_gb300 import build, gft as g
    build.build()
    g.load()
    return g


PATHS = {"tiles": (dict(n_ctas=4), 2), "records": (dict(cell_kernel=1), 1), "own order": (dict(node_sort=-1), 0),
         "sums": ({}, 3)}


def _problem(order, path):
    terms = anova.term_set(5, order)
    by = (16, 6, 4) if path == "sums" else (32, 16, 10)
    bw = [by[len(u) - 1] if u else 0 for u in terms]
    x = inputs.uniform_points(23, 5, M)
    return x, terms, bw, inputs.decaying_coefficients(3, terms, bw)


def _plan(gft, x, terms, bw, path):
    import torch
    kw, form = PATHS[path]
    P = gft.Plan(to_dev(x, torch.float32), terms, bw, **kw)
    assert gft.anova_debug_plan_form(P.handle) == form
    return P


@pytest.mark.parametrize("path", list(PATHS))
@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_a_coefficient(gft, path, order, bad):
    x, terms, bw, fhat = _problem(order, path)
    P = _plan(gft, x, terms, bw, path)
    ref = ndft.trafo(f32_nodes(x), terms, bw, fhat)
    for k in (1, len(fhat) // 2, len(fhat) - 1):
        h = fhat.copy()
        h[k] = bad
        f = host(P.trafo(cplx_dev(h)))
        assert not np.any(np.isfinite(f)), k
        assert rel_l2(host(P.trafo(cplx_dev(fhat))), ref) <= TOL   # nothing is left behind


@pytest.mark.parametrize("path", list(PATHS))
@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_node(gft, path, order, bad):
    x, terms, bw, fhat = _problem(order, path)
    ref = ndft.trafo(f32_nodes(x), terms, bw, fhat)
    x[1, 17] = bad
    f = host(_plan(gft, x, terms, bw, path).trafo(cplx_dev(fhat)))
    ok = np.arange(M) != 17
    assert not np.isfinite(f[17]) and rel_l2(f[ok], ref[ok]) <= TOL


@pytest.mark.parametrize("what", ["coefficient", "node"])
def test_one_problem_of_a_batch(gft, what):
    import torch
    x, terms, bw, fhat = _problem(2, "tiles")
    ref = ndft.trafo(f32_nodes(x), terms, bw, fhat)
    xb, h = x.copy(), fhat.copy()
    if what == "node":
        xb[1, 17] = np.nan
    else:
        h[7] = np.inf
    B = gft.Batch([to_dev(x, torch.float32), to_dev(xb, torch.float32)], [terms, terms], [bw, bw])
    f = host(B.trafo(cplx_dev(np.concatenate([fhat, h]))))
    assert rel_l2(f[:M], ref) <= TOL
    bad = ~np.isfinite(f[M:])
    assert np.array_equal(bad, np.arange(M) == 17) if what == "node" else bad.all()
