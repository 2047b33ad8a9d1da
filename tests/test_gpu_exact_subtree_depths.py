"""Exact mode, deep subtrees: shapes whose plan sums subtrees of four to six columns, with small integers and
with matrices whose leading pivots vanish modulo the first prime (the row-exchange path of every depth)."""
import numpy as np
import pytest

from oracle import radic_oracle as orc
from paper_1508_01326_gb300 import workloads as W
from tests.test_gpu_exact_subtree import P0, _solve_unit_triangular, _unimodular

pytestmark = pytest.mark.gpu

# the depth is the plan's for both entry points (few and many primes), on 152 SMs
SHAPES = [(7, 36, 4), (9, 21, 4), (8, 40, 5), (9, 41, 6), (10, 30, 6), (11, 27, 6), (12, 24, 6)]


def R():
    import paper_1508_01326_gb300 as mod

    return mod


@pytest.fixture(autouse=True)
def sms():
    import torch

    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the depths are those of the plan for 152 SMs")


@pytest.mark.parametrize("m,n,depth", SHAPES)
def test_small_integers(m, n, depth):
    assert R().radic_plan_info(m, n, "exact")["subtree_depth"] == depth
    a = W.integer_matrix(980 + m, m, n, 3, np.int8)
    want = orc.radic_det_pfaffian(a.astype(np.int64))
    res = R().det(a, mode="exact")
    assert res["exact"] == want and res["status"] == 0
    assert R().det_exact_wide(a)["integer"] == want


@pytest.mark.parametrize("ones", [2, 3, 5])
@pytest.mark.parametrize("m,n,depth", SHAPES)
def test_vanishing_leading_pivots(m, n, depth, ones):
    # T A is congruent to a sparse matrix modulo the first prime only; the
    # other primes see random residues, so a wrong residue cannot cancel
    assert R().radic_plan_info(m, n, "exact")["subtree_depth"] == depth
    L, U = _unimodular(m)
    rng = np.random.default_rng(990 + m + ones)
    a = np.zeros((m, n), dtype=np.int64)
    for j in range(n):
        b = [0] * m
        for i in rng.choice(m, ones, replace=False):
            b[i] = int(rng.integers(1, 3))
        x = _solve_unit_triangular(U, _solve_unit_triangular(L, b, True), False)
        a[:, j] = [v if v <= P0 // 2 else v - P0 for v in x]
    a = a.astype(np.int32)
    res = R().det_exact_wide(a, options=dict(mapping="prefix"))
    assert res["status"] == 0 and res["integer"] == orc.radic_det_pfaffian(a.astype(np.int64))
