"""Direct sums over many nodes and over many terms: the FP32 chains are broken.

An FP32 chain of n additions of like size leaves a relative error of about
u sqrt(n / 6) in its sum, u = 2^-24 (each rounding is below u of a partial sum that
grows with the root of its length); the products add about 2 u.  A thread of the adjoint
adds at most 128 nodes (4.6 u) before the sums go on in FP64: together 5 u, and the
bound is 8 u.  One chain over the 2344 nodes of these plans' threads would leave 20 u.
"""
import itertools

import numpy as np
import pytest

from oracle import ndct, ndft
from paper_2010_10199_gb300 import inputs

from gpu_util import cplx_dev, f32_nodes, host, rel_l2, to_dev

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


@pytest.fixture(scope="module")
def gft():
    from paper_2010_10199_gb300 import build, gft as g
    build.build()
    g.load()
    return g


def _plan(gft, basis, d, bws, M):
    import torch
    terms = [u for s in range(len(bws) + 1) for u in itertools.combinations(range(d), s)]
    bw = [bws[len(u) - 1] if u else 0 for u in terms]
    x = inputs.uniform(7, M + d, d * M).reshape(d, M)
    x = x if basis else x - 0.5
    P = gft.Plan(to_dev(x, torch.float32), terms, bw, basis=basis)
    assert gft.anova_debug_plan_form(P.handle) == gft.FORM_DIRECT
    return P, terms, bw, f32_nodes(x)


# 4526 groups of 30 coordinates: one node chunk each, 128 threads' chains over all nodes
@pytest.mark.parametrize("basis,bws", [(0, (16, 4, 2)), (0, (16, 8, 2)), (1, (9, 3, 2))])
@pytest.mark.parametrize("M", [16383, 16384, 16385, 32769, 300000])
def test_adjoint_over_many_nodes(gft, basis, bws, M):
    P, terms, bw, x = _plan(gft, basis, 30, bws, M)
    y = inputs.complex_normal(3, 4, M)
    g = host(P.adjoint(cplx_dev(y)))
    pick = [0, 1, 7, 30, 31, 200, 465, 466, 467, 1500, 3000, len(terms) - 1]
    ref = (ndct if basis else ndft).adjoint(x, [terms[u] for u in pick], [bw[u] for u in pick], y)
    off = np.concatenate([[0], np.cumsum([(b - 1) ** len(u) for u, b in zip(terms, bw)])])
    got = np.concatenate([g[off[u]:off[u + 1]] for u in pick])
    assert rel_l2(got, ref) <= 8 * U


@pytest.mark.parametrize("basis,bws", [(0, (16, 4, 2)), (0, (16, 8)), (1, (9, 3, 2)), (1, (20, 8))])
@pytest.mark.parametrize("M", [60, 2500, 30001])
def test_forward_over_many_terms(gft, basis, bws, M):
    """A warp's chain is at most 8 units of 9 rows of two additions (144: 4.9 u), its
    total at most one addition per 8 of 566 units (3.4 u), the products 2 u: 6.3 u as
    independent errors, bound 8 u."""
    P, terms, bw, x = _plan(gft, basis, 30, bws, M)
    fhat = inputs.complex_normal(3, 2, P.n_coeffs)
    f = host(P.trafo(cplx_dev(fhat)))
    pick = np.linspace(0, M - 1, min(M, 500)).astype(int)
    ref = (ndct if basis else ndft).trafo(x[:, pick], terms, bw, fhat)
    assert rel_l2(f[pick], ref) <= 8 * U


def test_forward_over_many_terms_and_nodes(gft):
    """Enough nodes that a block's eight warps share all 4526 terms: rows of about 700 in
    one chain would leave 15 u."""
    import torch
    d, M, bws = 30, 4000000, (16, 4, 2)
    terms = [u for s in range(4) for u in itertools.combinations(range(d), s)]
    bw = [bws[len(u) - 1] if u else 0 for u in terms]
    x = torch.rand(d, M, generator=torch.Generator("cuda").manual_seed(5), device="cuda") - 0.5
    P = gft.Plan(x, terms, bw)
    assert gft.anova_debug_plan_form(P.handle) == gft.FORM_DIRECT
    fhat = inputs.complex_normal(3, 2, P.n_coeffs)
    f = P.trafo(cplx_dev(fhat))
    pick = torch.linspace(0, M - 1, 500, dtype=torch.float64, device="cuda").long()
    ref = ndft.trafo(f32_nodes(x[:, pick].cpu().numpy()), terms, bw, fhat)
    assert rel_l2(host(f[pick]), ref) <= 8 * U
