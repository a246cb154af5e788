"""The forward over node tiles is not short of its value.

u = 2^-24.  The tensor core cuts its sums off: half a unit of the last place is 0.72 u of a
value with an evenly spread mantissa, and with what the smaller addends lose a stage of
products leaves its value short by about 1 u, three stages (order 1: two) by 3 u.  That is
taken back on average.  The CUDA cores' gather evaluates the same window with rounding to
nearest; the bound on the difference along the result is 1.2 u.
"""
import numpy as np
import pytest

from paper_2010_10199_gb300 import inputs

from gpu_util import cplx_dev, host, to_dev

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


@pytest.fixture(scope="module")
def gft():
    from paper_2010_10199_gb300 import build, gft as g
    build.build()
    g.load()
    return g


@pytest.mark.parametrize("terms,N", [([(0,)], 64), ([(0, 1)], 32), ([(0, 1)], 16), ([(0, 1, 2)], 4), ([(0, 1, 2)], 10)])
@pytest.mark.parametrize("M", [20000, 100003])
def test_bias(gft, terms, N, M):
    import torch
    x = to_dev(inputs.uniform_points(5, len(terms[0]), M), torch.float32)
    P, Q = gft.Plan(x, terms, [N], n_ctas=16), gft.Plan(x, terms, [N], n_ctas=16, cell_kernel=1)
    assert gft.anova_debug_plan_form(P.handle) == gft.FORM_TILES
    fhat = cplx_dev(inputs.complex_normal(5, 2, P.n_coeffs))
    f, ref = host(P.trafo(fhat)), host(Q.trafo(fhat))
    assert abs(np.vdot(ref, f - ref).real) <= 1.2 * U * np.vdot(ref, ref).real
