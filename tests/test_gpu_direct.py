"""Plans whose terms all have small bandwidths are summed directly: parity with the
FP64 oracles over every kernel instance and node-count edge, and with the same plan on
the NFFT path.

Bounds, from u = 2^-24: a node's value is a sum of products of at most three powers
(each at most 12 roundings of a unit number) with a coefficient, added over at most 9
positions of two axes, the terms and the warps in chains of at most 30, so its error is
below 128 u sum |fhat|; a coefficient's is below the same with sum |y|, its chain being
the nodes of a thread (at most 4133 / 128) and the chunks.
"""
import itertools

import numpy as np
import pytest

from oracle import anova, ndct, ndft
from paper_2010_10199_gb300 import inputs

from gpu_util import cplx_dev, f32_nodes, host, rel_l2, to_dev

pytestmark = pytest.mark.gpu
U = 2.0 ** -24
EXP = [(3, (2, 2, 2)), (4, (26, 4, 4)), (4, (6, 6, 6)), (5, (18, 8)), (4, (16, 10, 4)), (6, (64,)), (3, (254, 2, 6))]
COS = [(3, (2, 2, 2)), (4, (82, 10)), (4, (9, 3, 3)), (4, (8, 4, 4)), (3, (17, 5, 5)), (5, (30, 6)), (5, (7, 7, 2)),
       (4, (5, 8)), (4, (128, 9))]


@pytest.fixture(scope="module")
def gft():
    from paper_2010_10199_gb300 import build, gft as g
    build.build()
    g.load()
    return g


def _case(gft, basis, d, bws, M, empty=True, **kw):
    import torch
    terms = [u for s in range(0 if empty else 1, len(bws) + 1) for u in itertools.combinations(range(d), s)]
    bw = [bws[len(u) - 1] if u else 0 for u in terms]
    x = inputs.uniform(7, M + d, d * M).reshape(d, M)
    x = x if basis else x - 0.5
    if M > 3:   # coordinates at the ends and the middle of the period
        x[:, 0], x[:, 1], x[:, 2] = (0.0, 1.0, 0.5) if basis else (-0.5, 0.0, 0.49999997)
    P = gft.Plan(to_dev(x, torch.float32), terms, bw, basis=basis, **kw)
    return P, terms, bw, f32_nodes(x), ndct if basis else ndft


SHAPES = [(0, c) for c in EXP] + [(1, c) for c in COS]


@pytest.mark.parametrize("M", [1, 31, 65, 1999, 2001, 4133])
@pytest.mark.parametrize("basis,shape", SHAPES)
def test_direct_against_the_sums(gft, basis, shape, M):
    P, terms, bw, x, ref = _case(gft, basis, shape[0], shape[1], M, empty=M != 65)
    n = P.n_coeffs
    fhat, y = inputs.complex_normal(3, 2, n), inputs.complex_normal(3, 4, M)
    amp = 2.0 ** 1.5 if basis else 1.0
    f, g = host(P.trafo(cplx_dev(fhat))), host(P.adjoint(cplx_dev(y)))
    assert np.abs(f - ref.trafo(x, terms, bw, fhat)).max() <= 128 * U * amp * np.abs(fhat).sum()
    assert np.abs(g - ref.adjoint(x, terms, bw, y)).max() <= 128 * U * amp * np.abs(y).sum()
    # a second pass finds the counters at zero and gives the same bits
    assert np.array_equal(f, host(P.trafo(cplx_dev(fhat)))) and np.array_equal(g, host(P.adjoint(cplx_dev(y))))


@pytest.mark.parametrize("basis,shape,M", [(0, (4, (26, 6, 4)), 40001), (0, (6, (16, 10)), 22222), (1, (5, (40, 9)), 20481),
                                           (0, (20, (8,)), 5), (0, (40, (16, 8)), 700)])
def test_direct_against_the_nfft(gft, basis, shape, M):
    """Four nodes per lane, several node chunks and term sets, many coordinates (a table
    too large for several nodes per lane); both paths hold 1e-5 of the exact sums."""
    P, terms, bw, _, _ = _case(gft, basis, shape[0], shape[1], M)
    fhat, y = cplx_dev(inputs.complex_normal(5, 2, P.n_coeffs)), cplx_dev(inputs.complex_normal(5, 4, M))
    f, g = host(P.trafo(fhat)), host(P.adjoint(y))
    for kw in ({"n_ctas": 8}, {"node_sort": -1}, {"cell_kernel": 1}):
        Q = _case(gft, basis, shape[0], shape[1], M, **kw)[0]
        assert rel_l2(host(Q.trafo(fhat)), f) <= 2e-5, kw
        assert rel_l2(host(Q.adjoint(y)), g) <= 2e-5, kw


def test_direct_with_a_group_mask(gft):
    """One proximal step from zero at step 1 / L: masked groups stay zero, the others
    are within the adjoints' 2e-5 (the prox does not expand)."""
    M, L = 3000, 5e4
    paths = []
    for kw in ({}, {"n_ctas": 8}):
        P, terms, bw, _, _ = _case(gft, 0, 5, (16, 6, 4), M, **kw)
        y = cplx_dev(inputs.complex_normal(9, 4, M))
        mask = [i % 3 != 1 for i in range(len(terms))]
        path, _, _ = P.fista(y, [1.0], max_it=1, tol=0.0, L0=L, group_mask=mask)
        paths.append(host(path[0]))
        whole = host(P.adjoint(y))
    offs, _ = anova.layout(terms, bw)
    for u, (o, N) in enumerate(zip(offs, bw)):
        if not mask[u]:
            assert not paths[0][o:o + (N - 1) ** len(terms[u])].any()
    assert np.linalg.norm(paths[0]) > 0
    assert np.linalg.norm(paths[0] - paths[1]) <= 2e-5 * np.linalg.norm(whole) / L
