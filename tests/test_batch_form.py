"""The problems of a batch may keep their nodes in different forms (a problem whose padded
tiles would pass 2^31 places keeps records beside others' tiles).  A kernel reads one
form, so the choice has to be one that every problem holds."""
import ctypes
import itertools

import pytest

OWN_ORDER, RECORDS, TILES = 0, 1, 2


@pytest.fixture(scope="module")
def lib():
    from paper_2010_10199_gb300 import build, gft
    build.build()
    return gft.load()


@pytest.mark.parametrize("n", [1, 2, 3, 4])
def test_a_batch_reads_a_form_that_every_problem_holds(lib, n):
    for forms in itertools.product((OWN_ORDER, RECORDS, TILES), repeat=n):
        got = lib.anova_debug_batch_form((ctypes.c_int32 * n)(*forms), n)
        assert got == (forms[0] if len(set(forms)) == 1 else OWN_ORDER), forms


def test_no_problems_is_invalid(lib):
    assert lib.anova_debug_batch_form(None, 2) == -1
    assert lib.anova_debug_batch_form((ctypes.c_int32 * 1)(1), 0) == -1
