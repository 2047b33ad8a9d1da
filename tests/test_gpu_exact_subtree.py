"""Exact mode, prefix mapping: subtree sums of the eliminated heads (Definition 3, Eq. (1)) against
the oracle's closed form: every row count and subtree depth, square to long matrices, and matrices
whose leading pivots vanish modulo the first prime (the row-exchange path)."""
import numpy as np
import pytest

from oracle import radic_oracle as orc
from paper_1508_01326_gb300 import workloads as W

pytestmark = pytest.mark.gpu

P0 = 2147483647  # first prime of the exact mode


def R():
    import paper_1508_01326_gb300 as mod

    return mod


@pytest.mark.parametrize("m", range(3, 13))
@pytest.mark.parametrize("extra", [0, 1, 4, 9])
def test_default_depth_matches_oracle(m, extra):
    a = W.integer_matrix(900 + 16 * m + extra, m, m + extra, 4, np.int8)
    want = orc.radic_det_pfaffian(a.astype(np.int64))
    res = R().det(a, mode="exact")
    assert res["exact"] == want and res["status"] == 0
    wide = R().det_exact_wide(a)
    assert wide["integer"] == want and wide["n_primes"] == res["n_primes"]


@pytest.mark.parametrize("m,n", [(3, 64), (4, 64), (5, 40), (6, 30), (12, 26)])
def test_long_rows_match_oracle(m, n):
    a = W.integer_matrix(950 + m, m, n, 9, np.int32)
    want = orc.radic_det_pfaffian(a.astype(np.int64))
    assert R().det(a, mode="exact")["exact"] == want


@pytest.mark.parametrize("opts", [dict(prefix_depth=2), dict(prefix_depth=3), dict(prefix_depth=2, ranks_per_task=3),
                                  dict(blocks=1, threads_per_block=32), dict(blocks=7, ranks_per_task=5)])
@pytest.mark.parametrize("m,n", [(4, 9), (7, 15), (10, 16)])
def test_plan_options_match_oracle(m, n, opts):
    a = W.integer_matrix(960 + m, m, n, 5, np.int32)
    want = orc.radic_det_pfaffian(a.astype(np.int64))
    assert R().det(a, mode="exact", options=dict(mapping="prefix", **opts))["exact"] == want


def _mix64(z):
    mask = (1 << 64) - 1
    z = ((z ^ (z >> 30)) * 0xbf58476d1ce4e5b9) & mask
    z = ((z ^ (z >> 27)) * 0x94d049bb133111eb) & mask
    return z ^ (z >> 31)


def _unimodular(m):
    """L and U of the staging's row transform modulo the first prime (slot 0)."""
    rinv = pow(1 << 32, -1, P0)
    L, U = np.eye(m, dtype=object), np.eye(m, dtype=object)
    for i in range(m):
        for j in range(m):
            if j > i:
                h = _mix64((0x9e3779b97f4a7c15 * (i * 64 + j) + 1) % 2 ** 64)
                U[i, j] = (h >> 33) % P0 * rinv % P0
            elif j < i:
                h = _mix64((0xd1b54a32d192ed03 * (i * 64 + j) + 7) % 2 ** 64)
                L[i, j] = (h >> 33) % P0 * rinv % P0
    return L, U


def _solve_unit_triangular(T, b, lower):
    m = len(b)
    x = [0] * m
    for i in (range(m) if lower else reversed(range(m))):
        s = b[i]
        for j in (range(i) if lower else range(i + 1, m)):
            s -= T[i, j] * x[j]
        x[i] = s % P0
    return x


@pytest.mark.parametrize("depth", [0, 2, 3])
@pytest.mark.parametrize("m,n,ones", [(4, 9, 2), (5, 10, 3), (7, 11, 4), (8, 12, 3)])
def test_vanishing_leading_pivots(m, n, ones, depth):
    # A with T A congruent to a sparse 0/1 matrix modulo the first prime: zero
    # pivots at every step, singular heads among them; the other primes see
    # random residues, so that a wrong residue cannot cancel
    if depth >= m - 1:
        pytest.skip("subtree depth below m - 1")
    L, U = _unimodular(m)
    rng = np.random.default_rng(970 + m)
    a = np.zeros((m, n), dtype=np.int64)
    for j in range(n):
        b = [0] * m
        for i in rng.choice(m, ones, replace=False):
            b[i] = int(rng.integers(1, 3))
        x = _solve_unit_triangular(U, _solve_unit_triangular(L, b, True), False)
        a[:, j] = [v if v <= P0 // 2 else v - P0 for v in x]
    a = a.astype(np.int32)
    want = orc.radic_det_pfaffian(a.astype(np.int64))
    res = R().det_exact_wide(a, options=dict(mapping="prefix", prefix_depth=depth))
    assert res["integer"] == want
