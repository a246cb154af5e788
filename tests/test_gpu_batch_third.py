"""Batches with third-order terms: the forward runs over records beside the tiles where the
whole batch has fewer than five nodes per third-order cell, and over tiles from there on.
Every problem within 1e-5 of its result's expected norm on both sides of the rule, uneven problems and
one without third-order terms among them.
"""
import numpy as np
import pytest

from oracle import anova, ndft
from paper_2010_10199_gb300 import inputs

from gpu_util import cplx_dev, f32_nodes, host, to_dev

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def gft():
    from paper_2010_10199_gb300 import build, gft as g
    build.build()
    g.load()
    return g


def _batch(gft, problems, seed=5):
    """problems: (d, bandwidths by order, M)."""
    import torch
    P = []
    for i, (d, by, M) in enumerate(problems):
        terms = anova.term_set(d, len(by))
        bw = [by[len(u) - 1] if u else 0 for u in terms]
        P.append((inputs.uniform_points(seed + i, d, M), terms, bw))
    B = gft.Batch([to_dev(x, torch.float32) for x, _, _ in P], [t for _, t, _ in P], [b for _, _, b in P])
    return B, P


# n = 8, 12, 16: 512, 1728 and 4096 cells per term
@pytest.mark.parametrize("problems", [
    [(4, (16, 8, 4), M) for M in (1, 100, 2560, 7579)],                    # 10240 nodes: 5 per cell
    [(4, (16, 8, 4), M) for M in (1, 100, 2560, 7578)],                    # one node fewer
    [(3, (32, 16, 8), 900), (4, (26, 6, 4), 33), (5, (64, 32), 4001)],     # records; one of order 2 only
    [(3, (32, 16, 8), 900), (4, (26, 6, 4), 60001), (5, (64, 32), 4001)],  # tiles
    [(3, (2, 2, 2), 5), (3, (8, 6, 6), 1729)],
], ids=["five", "below_five", "sparse", "dense", "short_axes"])
def test_batch_against_the_sums(gft, problems):
    B, P = _batch(gft, problems)
    co, no = B.coef_off, B.node_off
    fhat, y = inputs.complex_normal(3, 2, co[-1]), inputs.complex_normal(3, 4, no[-1])
    for _ in range(2):   # the second pass finds accumulators and counters as the first left them
        f, g = host(B.trafo(cplx_dev(fhat))), host(B.adjoint(cplx_dev(y)))
        for i, (x, terms, bw) in enumerate(P):
            xo = f32_nodes(x)
            ff, yy = fhat[co[i]:co[i + 1]], y[no[i]:no[i + 1]]
            # both results' expected norm: one node's or a few coefficients' sum may cancel
            size = np.sqrt(len(yy) * len(ff))
            assert np.linalg.norm(f[no[i]:no[i + 1]] - ndft.trafo(xo, terms, bw, ff)) <= TOL * size, i
            assert np.linalg.norm(g[co[i]:co[i + 1]] - ndft.adjoint(xo, terms, bw, yy)) <= TOL * size, i


def test_forward_is_as_fast_as_over_records(gft):
    """Four problems of an eighth of a node per cell: over tiles the forward took 1.4 times as
    long as CUDA-core plans one after the other."""
    import torch
    problems = [(6, (64, 24, 10), 1000)] * 4
    B, P = _batch(gft, problems)
    Q = [gft.Plan(to_dev(x, torch.float32), t, b, cell_kernel=1) for x, t, b in P]
    fhat = [cplx_dev(inputs.complex_normal(i, 2, q.n_coeffs)) for i, q in enumerate(Q)]
    whole = torch.cat(fhat)

    def ms(fn):
        times = []
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                fn()
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) / 20)
        return min(times)
    one_by_one = ms(lambda: [q.trafo(v) for q, v in zip(Q, fhat)])
    assert ms(lambda: B.trafo(whole)) <= 0.8 * one_by_one
