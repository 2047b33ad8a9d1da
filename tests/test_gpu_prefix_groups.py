"""Binary64 prefixes factored a lane each and shared by the lane group (depth 3, runs of prefixes): value,
sum of |terms| and error bound against the same lanes with one prefix per task, where every lane factors
the prefix it shares.  The operations on each prefix are the same, so the bounds agree to the rounding of
their binary64 sums."""
import numpy as np
import pytest

from paper_1508_01326_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def R():
    import paper_1508_01326_gb300 as mod

    return mod


def _compare(a, **options):
    got = R().det(a, mode="fp64", options=dict(options))
    ref = R().det(a, mode="fp64", options=dict(options, ranks_per_task=1))
    assert got["status"] == ref["status"] == 0
    # sums of at most C(20, 10) terms of one sign, in another order: 2^-53 * log2 of their number, per lane
    # and block, is below 1e-13
    assert abs(got["value"] - ref["value"]) <= 1e-13 * ref["abs_sum"]
    assert abs(got["abs_sum"] - ref["abs_sum"]) <= 1e-13 * ref["abs_sum"]
    assert abs(got["err_bound"] - ref["err_bound"]) <= 1e-13 * ref["err_bound"]


@pytest.mark.parametrize("m,n", [(7, 18), (7, 20), (8, 17), (8, 20), (9, 16), (9, 20), (10, 15), (10, 20)])
@pytest.mark.parametrize("deterministic", [False, True])
def test_runs_match_single_prefixes(m, n, deterministic):
    _compare(W.uniform_matrix(700 + 31 * m + n, m, n), deterministic=deterministic)


@pytest.mark.parametrize("lanes", [2, 4, 8, 16, 32])
@pytest.mark.parametrize("m,n", [(7, 19), (8, 19), (9, 19), (10, 18)])
def test_runs_of_every_lane_count(m, n, lanes):
    _compare(W.uniform_matrix(800 + m, m, n), lanes_per_prefix=lanes)


@pytest.mark.parametrize("m", [7, 8, 9, 10])
def test_degenerate_prefixes(m):
    # equal and zero columns, and a row that repeats another on the first columns: prefixes whose
    # enclosures fail take the per-minor path from the lane that works their leaves
    a = np.array(W.uniform_matrix(900 + m, m, 19), dtype=np.float64)
    a[:, 5] = a[:, 2]
    a[:, 9] = 0.0
    a[1, :8] = a[0, :8]
    _compare(a)
