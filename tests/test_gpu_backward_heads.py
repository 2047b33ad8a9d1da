"""Head kernel of the backward (subtrees of 2 to 4 columns): every row count from square to long
matrices and small to large batches (depth, blocks per matrix and partly filled warps follow from
them), and heads with exactly zero pivots, against the oracle's exact gradient."""
import numpy as np
import pytest
import torch

import oracle.radic_oracle as orc
from paper_1508_01326_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def R():
    import paper_1508_01326_gb300 as mod

    return mod


def _check(mats, mode, tol, which=None):
    g_out = torch.linspace(0.5, 2.0, len(mats), dtype=torch.float64, device="cuda")
    grad = R().radic_det_backward(torch.from_numpy(mats).cuda(), g_out, mode=mode).cpu().numpy()
    for b in which if which is not None else range(len(mats)):
        want = np.array([[float(x) for x in row] for row in orc.radic_grad_exact(mats[b], use_pfaffian=True)])
        assert np.abs(grad[b] - float(g_out[b]) * want).max() <= tol * max(np.abs(want).max(), 1e-300), b


# binary64 and pair rounding of the elimination and of sums over at most 14 columns
TOL = {"fp64": 1e-11, "pair": 1e-11}


@pytest.mark.parametrize("mode", ["fp64", "pair"])
@pytest.mark.parametrize("m,n,batch", [(3, 3, 1), (3, 4, 2), (3, 13, 1), (4, 4, 1), (4, 6, 3), (4, 13, 70), (5, 6, 1),
                                       (5, 14, 40), (6, 7, 2), (6, 14, 300), (7, 8, 1), (7, 13, 9), (8, 8, 2),
                                       (8, 9, 1), (8, 14, 5)])
def test_gradient_matches_oracle(m, n, batch, mode):
    mats = np.random.default_rng(3000 + 20 * m + n).uniform(-1, 1, (batch, m, n))
    _check(mats, mode, TOL[mode], sorted({0, batch // 2, batch - 1}))


@pytest.mark.parametrize("mode", ["fp64", "pair"])
@pytest.mark.parametrize("m,n", [(3, 8), (4, 9), (5, 9), (6, 11), (7, 11), (8, 11)])
def test_singular_heads_match_oracle(m, n, mode):
    # zero, repeated and dependent columns at the start, in the middle and at
    # the end: integer entries make the pivots exactly zero
    a = W.integer_matrix(3100 + m, m, n, 4, np.int32).astype(np.float64)
    b = a.copy()
    a[:, 0] = 0.0
    a[:, n - 2] = a[:, 1]
    b[:, 1] = b[:, 0]
    b[:, n // 2] = 2.0 * b[:, 0]
    c = W.integer_matrix(3200 + m, m, n, 4, np.int32).astype(np.float64)
    c[1] = c[0]  # two equal rows: every minor is zero, its cofactors are not
    _check(np.stack([a, b, c]), mode, 1e-11)
