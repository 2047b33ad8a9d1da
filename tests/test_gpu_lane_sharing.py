"""Lanes that share a prefix in binary64 (small batches and small single matrices): values, sums of
|terms| and error bounds against the oracle and against the same matrices in a plan whose tasks are
large enough not to share, for both prefix depths, heads, degenerate pivots and every lane count the
shapes lead to."""
from fractions import Fraction

import numpy as np
import pytest
import torch

import oracle.radic_oracle as orc
from paper_1508_01326_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def R():
    import paper_1508_01326_gb300 as mod

    return mod


def _check(res, mat):
    val, abs_sum = orc.radic_det_exact(mat)
    assert res["status"] == 0
    assert abs(Fraction(res["value"]) - val) <= Fraction(1e-12) * abs_sum
    assert abs(Fraction(res["abs_sum"]) - abs_sum) <= Fraction(1e-12) * abs_sum
    assert abs(Fraction(res["value"]) - val) <= Fraction(res["err_bound"])
    # the bound of binary64 elimination stays near its rounding
    assert res["err_bound"] <= 1e-11 * float(abs_sum)


SHAPES = [(3, 4), (3, 9), (4, 5), (4, 12), (5, 7), (5, 13), (6, 8), (6, 13), (7, 12), (8, 11), (8, 13), (9, 13), (10, 13)]


def _batch(shapes, tuning=None):
    mats = [W.uniform_matrix(500 + i, m, n) for i, (m, n) in enumerate(shapes)]
    data, ms, ns, offs = W.pack_batch(mats, np.float64)
    plan = R().BatchPlan(list(zip(ms, ns)), offs, mode="fp64", tuning=tuning)
    out = plan.radic_det_batched(torch.from_numpy(data).cuda())
    res = R().parse_results(out)
    plan.close()
    return mats, res


@pytest.mark.parametrize("depth", [0, 2, 3])
def test_small_batches_match_oracle(depth):
    tun = R().make_tuning(prefix_depth={m: depth for m in range(4, 11)}) if depth else None
    mats, res = _batch(SHAPES, tun)
    for mat, r in zip(mats, res):
        _check(r, mat)


def test_bounds_do_not_depend_on_task_size():
    # tasks of one prefix per lane and of long runs: the same prefixes, split
    # over other lanes; binary32 bound sums per prefix stay the same bits, so
    # the totals differ by their binary64 sums only
    tuned = [R().make_tuning(task_cost={m: c for m in range(1, 11)}) for c in (100.0, 1e9)]
    (_, a), (_, b) = (_batch(SHAPES, t) for t in tuned)
    for x, y in zip(a, b):
        assert abs(x["err_bound"] - y["err_bound"]) <= 1e-13 * y["err_bound"]
        assert abs(x["value"] - y["value"]) <= 1e-13 * y["abs_sum"]


@pytest.mark.parametrize("m,n", [(4, 6), (4, 13), (5, 11), (6, 12)])
def test_small_single_matrices_match_one_lane(m, n):
    a = W.uniform_matrix(600 + m, m, n)
    auto = R().det(a, mode="fp64")
    _check(auto, a)
    one = R().det(a, mode="fp64", options=dict(mapping="prefix", lanes_per_prefix=1))
    assert abs(auto["err_bound"] - one["err_bound"]) <= 1e-13 * one["err_bound"]
    for lanes in (2, 8, 32):
        r = R().det(a, mode="fp64", options=dict(mapping="prefix", prefix_depth=2, lanes_per_prefix=lanes))
        _check(r, a)


@pytest.mark.parametrize("m,n", [(5, 10), (6, 12), (9, 12)])
def test_failed_enclosures_in_shared_prefixes(m, n):
    # nearly repeated columns: prefixes whose pivots cannot be bounded take
    # the per-minor path, split over the lanes that share them
    a = W.uniform_matrix(700 + m, m, n)
    a[:, 1] = a[:, 0] * (1 + 2.0 ** -52)
    a[:, 3] = a[:, 0]
    data, ms, ns, offs = W.pack_batch([a, W.uniform_matrix(710 + m, m, n)], np.float64)
    plan = R().BatchPlan(list(zip(ms, ns)), offs, mode="fp64")
    res = R().parse_results(plan.radic_det_batched(torch.from_numpy(data).cuda()))
    plan.close()
    val, abs_sum = orc.radic_det_exact(a)
    assert abs(Fraction(res[0]["value"]) - val) <= Fraction(1e-12) * abs_sum
    assert abs(Fraction(res[0]["value"]) - val) <= Fraction(res[0]["err_bound"])
