"""The adjoint of third-order terms over node tiles is not short of its value.

Its three stages of tensor-core products (a tile's moments, the two window products) cut
their sums off at 24 bits: half a unit of 2^-23 each, 0.72 u of a value with an evenly
spread mantissa on average, u = 2^-24; together 2.2 u.  Operands that were cut off into
high and low parts, rather than rounded, would leave out a product of the low parts that
has the result's sign, (2^-11 x 0.72)^2 = 2 u on average.  The bound is 3 u.
"""
import numpy as np
import pytest

from oracle import ndft
from paper_2010_10199_gb300 import inputs

from gpu_util import cplx_dev, f32_nodes, host, to_dev

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


@pytest.fixture(scope="module")
def gft():
    from paper_2010_10199_gb300 import build, gft as g
    build.build()
    g.load()
    return g


@pytest.mark.parametrize("N", [8, 10])
@pytest.mark.parametrize("M", [3000, 20000, 100003])
def test_third_order_adjoint(gft, N, M):
    import torch
    x = inputs.uniform_points(5, 3, M)
    P = gft.Plan(to_dev(x, torch.float32), [(0, 1, 2)], [N], n_ctas=16)
    assert gft.anova_debug_plan_form(P.handle) == gft.FORM_TILES
    y = inputs.complex_normal(5, 4, M).astype(np.complex64).astype(np.complex128)
    g, ref = host(P.adjoint(cplx_dev(y))), ndft.adjoint(f32_nodes(x), [(0, 1, 2)], [N], y)
    assert abs(np.vdot(ref, g - ref).real) <= 3 * U * np.vdot(ref, ref).real
