"""Group mapping on grids that hold fewer groups than there are runs: a group then takes consecutive runs and
goes on with its elimination, and every run's sums are closed as before."""
from fractions import Fraction

import numpy as np
import pytest

import oracle.radic_oracle as orc
from paper_1508_01326_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def R():
    import paper_1508_01326_gb300 as mod

    return mod


@pytest.mark.parametrize("blocks", [1, 2, 7])
@pytest.mark.parametrize("m,n,width,run", [(1, 40, 16, 3), (5, 12, 16, 7), (11, 14, 16, 1), (16, 19, 16, 5),
                                           (5, 12, 32, 9), (18, 21, 32, 1), (21, 24, 32, 4), (32, 34, 32, 2)])
def test_consecutive_runs_match_separate_runs(m, n, width, run, blocks):
    a = W.uniform_matrix(840 + m + n, m, n)
    want = orc.radic_det_pfaffian([[Fraction(x) for x in row] for row in a.tolist()])
    opts = dict(mapping="group", group_width=width, ranks_per_task=run, flag_capacity=1400)
    for mode in ("fp64", "mixed"):
        one = R().det(a, mode=mode, options=dict(opts, blocks=600))  # every group at most one run
        few = R().det(a, mode=mode, options=dict(opts, blocks=blocks))
        assert abs(Fraction(few["value"]) - want) <= Fraction(few["err_bound"])
        # the same sums per run, added in another order in binary64
        for key in ("abs_sum", "err_bound"):
            assert abs(few[key] - one[key]) <= 1e-13 * one[key]
        assert few["minors"] == one["minors"] and few["flagged"] == one["flagged"]


@pytest.mark.parametrize("m,n", [(18, 21), (20, 23), (21, 24), (22, 25)])
def test_single_minors_fill_one_wave(m, n):
    # 1330 to 2300 minors, one per run: the grid is what a kernel of groups of 32
    # leaves resident, three blocks per SM
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    info = R().radic_plan_info(m, n, "fp64", dict(mapping="group"))
    assert info["run_or_tasks"] == 1 and info["blocks"] <= 3 * sms
    a = W.uniform_matrix(860 + m, m, n)
    want = orc.radic_det_pfaffian([[Fraction(x) for x in row] for row in a.tolist()])
    got = R().det(a, mode="fp64", options=dict(mapping="group"))
    assert abs(Fraction(got["value"]) - want) <= Fraction(got["err_bound"])
