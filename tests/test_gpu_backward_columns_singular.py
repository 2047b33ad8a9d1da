"""Backward of heads with an exactly zero pivot when later columns differ in size: integer entries, a zero
and a repeated column, and large columns by powers of two (the pivots stay exactly zero), against the
oracle's exact gradient, column by column."""
import numpy as np
import pytest
import torch

import oracle.radic_oracle as orc
from paper_1508_01326_gb300 import workloads as W
from tests.test_gpu_backward_columns import _bound

pytestmark = pytest.mark.gpu


def R():
    import paper_1508_01326_gb300 as mod

    return mod


@pytest.mark.parametrize("mode,unit", [("fp64", 2.0 ** -53), ("pair", 2.0 ** -44)])
@pytest.mark.parametrize("m,n,copies", [(3, 12, 1), (4, 12, 1), (4, 24, 50), (5, 12, 1), (5, 30, 30), (6, 12, 1),
                                        (6, 22, 30), (7, 12, 1), (7, 16, 50), (8, 12, 1), (8, 16, 50), (8, 24, 1)])
@pytest.mark.parametrize("bits", [7, 14, 20])
def test_singular_heads_with_large_columns(m, n, copies, bits, mode, unit):
    mats = []
    for where in ([n - 1], [n // 2], [n // 2, n - 2], list(range(2, n, 2))):
        a = W.integer_matrix(3400 + m + n, m, n, 4, np.int32).astype(np.float64)
        a[:, 0] = 0.0
        a[:, 2] = a[:, 1]
        a[:, where] *= 2.0 ** (min(bits, 100 // (m - 1)) if len(where) > 2 else bits)
        mats.append(a)
    A = torch.from_numpy(np.tile(np.stack(mats), (copies, 1, 1))).cuda()
    grad = R().radic_det_backward(A, torch.ones(len(A), dtype=torch.float64, device="cuda"), mode=mode).cpu().numpy()
    for b, a in enumerate(mats):
        want = np.array([[float(x) for x in row] for row in orc.radic_grad_exact(a, use_pfaffian=True)])
        err = np.abs(grad[b] - want).max(axis=0)
        assert np.all(err <= _bound(a, unit)), (b, err)
