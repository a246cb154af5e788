"""The autotuner at bandwidths that a default plan sums directly: that plan is a candidate,
what is timed is what the returned options build, and tuning does not slow a plan down."""
import pytest

from oracle import anova
from paper_2010_10199_gb300 import inputs

from gpu_util import cplx_dev, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gft():
    from paper_2010_10199_gb300 import build, gft as g
    build.build()
    g.load()
    return g


def _pair_ms(P, reps=50):
    import torch
    fhat, y = cplx_dev(inputs.complex_normal(1, 2, P.n_coeffs)), cplx_dev(inputs.complex_normal(1, 4, P.M))
    times = []
    for _ in range(4):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(reps):
            P.trafo(fhat)
            P.adjoint(y)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b) / reps)
    return min(times)


@pytest.mark.parametrize("d,by,M", [(6, (16, 8), 2000), (9, (26, 6, 4), 10000)])
def test_tuning_does_not_slow_a_plan_down(gft, d, by, M):
    import torch
    terms = anova.term_set(d, len(by))
    bw = [by[len(u) - 1] if u else 0 for u in terms]
    x = to_dev(inputs.uniform_points(31, d, M), torch.float32)
    D = gft.Plan(x, terms, bw)
    assert gft.anova_debug_plan_form(D.handle) == gft.FORM_DIRECT
    chosen, trials = gft.autotune(x, terms, bw, eps=1e-5, reps=10)
    assert trials[0]["sigma"] == 0.0 and trials[0]["window_m_row"] == 0 and trials[0]["est_error"] <= 1e-5
    assert all(t["sigma"] >= 1.75 for t in trials[1:])
    P = gft.Plan(x, terms, bw, **chosen)
    # the sums take less than half of the NFFT's time at these sizes
    assert gft.anova_debug_plan_form(P.handle) == gft.FORM_DIRECT
    assert _pair_ms(P) <= 1.3 * _pair_ms(D)


def test_no_such_candidate_where_a_default_plan_runs_the_nfft(gft):
    import torch
    terms = anova.term_set(4, 2)
    bw = [0] + [64] * 4 + [32] * 6
    _, trials = gft.autotune(to_dev(inputs.uniform_points(31, 4, 20000), torch.float32), terms, bw, eps=1e-5, reps=2)
    assert all(t["sigma"] >= 1.75 for t in trials)
