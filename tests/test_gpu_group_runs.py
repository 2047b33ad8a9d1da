"""Group mapping: runs of consecutive minors that keep the elimination of their unchanged columns.
Every run length around the group width, both widths, ragged last runs, and minors with failing
pivots, against the oracle; the error bound must not depend on how the ranks are cut into runs
beyond the rounding of its sums."""
from fractions import Fraction

import numpy as np
import pytest

import oracle.radic_oracle as orc
from paper_1508_01326_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def R():
    import paper_1508_01326_gb300 as mod

    return mod


@pytest.mark.parametrize("run", [1, 2, 15, 16, 17, 33, 1000])
@pytest.mark.parametrize("m,n,width", [(1, 40, 16), (3, 11, 16), (11, 14, 16), (16, 18, 16), (5, 12, 32), (17, 19, 32)])
def test_runs_match_oracle(m, n, width, run):
    a = W.uniform_matrix(800 + m, m, n)
    val, abs_sum = orc.radic_det_exact(a)
    opts = dict(mapping="group", group_width=width, ranks_per_task=run)
    for mode, tol in (("fp64", 1e-12), ("mixed", 8 * m * 2.0 ** -24)):
        r = R().det(a, mode=mode, options=opts)
        assert abs(float(Fraction(r["value"]) - val)) <= tol * float(abs_sum)
        assert abs(float(Fraction(r["abs_sum"]) - abs_sum)) <= tol * float(abs_sum)
        assert abs(Fraction(r["value"]) - val) <= Fraction(r["err_bound"])
    one = R().det(a, mode="fp64", options=dict(opts, ranks_per_task=1))
    many = R().det(a, mode="fp64", options=opts)
    # bounds are summed in binary32 over at most 256 minors of a run
    assert abs(many["err_bound"] - one["err_bound"]) <= 256 * 2.0 ** -24 * one["err_bound"]


@pytest.mark.parametrize("run", [1, 16, 200])
def test_failed_pivots_inside_runs(run):
    a = W.uniform_matrix(820, 11, 14)
    a[:, 4] = a[:, 2]                      # singular minors
    a[:, 9] = a[:, 7] * (1 + 2.0 ** -52)   # pivots whose enclosure reaches zero
    val, abs_sum = orc.radic_det_exact(a)
    r = R().det(a, mode="fp64", options=dict(mapping="group", ranks_per_task=run))
    assert abs(Fraction(r["value"]) - val) <= Fraction(1e-12) * abs_sum
    assert abs(Fraction(r["value"]) - val) <= Fraction(r["err_bound"])
