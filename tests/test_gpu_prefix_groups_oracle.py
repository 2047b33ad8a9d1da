"""Binary64 prefixes factored a lane each (depth 3, runs of prefixes): the plans that take that kernel, against
the oracle's exact value and the sum of the minors' magnitudes by an independent LU."""
import itertools
from fractions import Fraction

import numpy as np
import pytest

import oracle.radic_oracle as orc
from paper_1508_01326_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def R():
    import paper_1508_01326_gb300 as mod

    return mod


def _abs_sum(a):
    m, n = a.shape
    cols = np.array(list(itertools.combinations(range(n), m)))
    return float(np.abs(np.linalg.det(np.moveaxis(a[:, cols], 1, 0))).sum())


@pytest.mark.parametrize("degenerate", [False, True])
@pytest.mark.parametrize("m,n,lanes", [(7, 23, 0), (7, 24, 32), (8, 20, 0), (8, 22, 16), (9, 19, 0), (9, 20, 16),
                                       (10, 19, 0), (10, 20, 0)])
def test_shared_runs_match_oracle(m, n, lanes, degenerate):
    # groups of lanes share runs only where that halves the tasks at least;
    # without sharing these shapes have one prefix per run
    options = dict(lanes_per_prefix=lanes)
    tasks = [R().radic_plan_info(m, n, "fp64", o)["run_or_tasks"] for o in (options, dict(options, ranks_per_task=1))]
    assert 2 * tasks[0] <= tasks[1]
    a = np.array(W.uniform_matrix(870 + m + n, m, n), dtype=np.float64)
    if degenerate:
        a[:, 5] = a[:, 2]
        a[:, 9] = 0.0
        a[1, :7] = a[0, :7]
    got = R().det(a, mode="fp64", options=options)
    want = orc.radic_det_pfaffian([[Fraction(x) for x in row] for row in a.tolist()])
    total = _abs_sum(a)
    # binary64 elimination: 1e-12 of the sum of magnitudes, as for every binary64 result
    assert abs(float(Fraction(got["value"]) - want)) <= 1e-12 * total
    assert abs(got["abs_sum"] - total) <= 1e-12 * total
    assert abs(Fraction(got["value"]) - want) <= Fraction(got["err_bound"])
