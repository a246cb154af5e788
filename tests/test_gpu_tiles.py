"""The tensor-core kernels over cell-aligned node tiles at the counts where a tile's
layout can go wrong: cells of 1 .. 49 nodes (half tiles, full tiles, one node more),
runs of one or two tiles per warp, every order, both row windows, axes as short as the
window.

Bounds: the window's error is at most 1e-5 of the sum of the coefficients' (adjoint:
the values') magnitudes with 8 row taps and 3e-5 with 6, FP32 rounding well below; a
node lost, doubled or put in the wrong cell is an error of about one of the 500 to 1000
values, 1e-3 of their sum.
"""
import itertools

import numpy as np
import pytest

from oracle import ndft
from paper_2010_10199_gb300 import inputs

from gpu_util import cplx_dev, f32_nodes, host, to_dev

pytestmark = pytest.mark.gpu
COUNTS = [1, 2, 7, 8, 9, 15, 16, 17, 23, 24, 25, 31, 32, 33, 40, 41, 47, 48, 49]


@pytest.fixture(scope="module")
def gft():
    from paper_2010_10199_gb300 import build, gft as g
    build.build()
    g.load()
    return g


def _nodes(counts, d):
    """Clusters of the given sizes, each 1e-3 wide around a node of its own."""
    c = inputs.uniform(11, len(counts), d * len(counts)).reshape(d, -1) - 0.5
    x = np.repeat(c, counts, axis=1)
    x += 1e-3 * (inputs.uniform(12, x.shape[1], x.size).reshape(d, -1) - 0.5)
    x = np.mod(x + 0.5, 1.0) - 0.5
    return x[:, np.argsort(inputs.uniform(13, 1, x.shape[1]))]   # in no order of cells


@pytest.mark.parametrize("m_row", [3, 4])
@pytest.mark.parametrize("chunks", [1, 5])
@pytest.mark.parametrize("bw", [(64,), (30, 32), (16, 8), (16, 8, 4), (20, 12, 10)])
@pytest.mark.parametrize("counts", [COUNTS, [1] * 9, [16], [8], [700]], ids=["edges", "singles", "tile", "half", "run"])
def test_tiles_against_the_sums(gft, counts, bw, chunks, m_row):
    import torch
    d = 3
    x = _nodes(counts, d)
    terms = [u for s in range(len(bw) + 1) for u in itertools.combinations(range(d), s)]
    bws = [bw[len(u) - 1] if u else 0 for u in terms]
    # a chunk count keeps the plan on the NFFT
    P = gft.Plan(to_dev(x, torch.float32), terms, bws, n_ctas=chunks, window_m_row=m_row)
    fhat, y = inputs.complex_normal(5, 2, P.n_coeffs), inputs.complex_normal(5, 4, x.shape[1])
    f, g = host(P.trafo(cplx_dev(fhat))), host(P.adjoint(cplx_dev(y)))
    tol = 1e-5 if m_row == 4 else 3e-5
    xo = f32_nodes(x)
    assert np.abs(f - ndft.trafo(xo, terms, bws, fhat)).max() <= tol * np.abs(fhat).sum()
    assert np.abs(g - ndft.adjoint(xo, terms, bws, y)).max() <= tol * np.abs(y).sum()


@pytest.mark.parametrize("M", [16383, 16385, 32769, 1048576, 1048577, 1300001])
def test_sort_slices_and_parts(gft, M):
    """One to sixteen slices, of one part and of two (more than 65536 nodes): the same
    plan over records, which are sorted node by node; both hold 1e-5 of the sums."""
    import torch
    x = to_dev(inputs.uniform(31, M, 2 * M).reshape(2, M) - 0.5, torch.float32)
    terms, bws = [(), (0,), (1,), (0, 1)], [0, 100, 64, 32]
    out = []
    for kernel in (0, 1):
        P = gft.Plan(x, terms, bws, n_ctas=16, cell_kernel=kernel)
        fhat, y = cplx_dev(inputs.complex_normal(5, 2, P.n_coeffs)), cplx_dev(inputs.complex_normal(5, 4, M))
        out.append((host(P.trafo(fhat)), host(P.adjoint(y))))
    for a, b in zip(*out):
        assert np.linalg.norm(a - b) <= 2e-5 * np.linalg.norm(b)
