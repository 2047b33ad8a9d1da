"""Backward of matrices whose columns differ in size, against the oracle's exact gradient, column by
column: one column times a large factor (first, middle, last), two, every other one, and sizes that grow
geometrically.  A column's own gradient does not contain its entries, so the gradient of a large column is
small next to the others' and shows any rounding that came from them."""
import numpy as np
import pytest
import torch

import oracle.radic_oracle as orc

pytestmark = pytest.mark.gpu


def R():
    import paper_1508_01326_gb300 as mod

    return mod


def _factors(n, s):
    f = np.ones((6, n))
    f[0, 0] = f[1, n // 2] = f[2, n - 1] = f[3, n // 3] = f[3, 2 * n // 3] = s
    f[4, ::2] = s
    f[5] = s ** (np.arange(n) / (n - 1))
    return f


def _bound(a, unit):
    """Per column j: every cofactor in it is at most the product of m-1 other columns' norms, and an
    elimination's error m^2 units of that times its growth (8, as for the terms); summed over all choices
    of m-1 other columns."""
    m, n = a.shape
    norms = np.sqrt((a * a).sum(axis=0))
    out = np.zeros(n)
    for j in range(n):
        e = np.zeros(m)  # elementary symmetric sums
        e[0] = 1.0
        for c in range(n):
            if c != j:
                e[1:] += norms[c] * e[:-1].copy()
        out[j] = 8 * m * m * unit * e[m - 1]
    return out


# batches that take subtrees of 2 to 4 columns: m = 3 and 4 of 2; 64 matrices of 4 x 24 of 3; single small
# matrices of m >= 5 of 3; larger batches of long rows of 4
@pytest.mark.parametrize("mode,unit", [("fp64", 2.0 ** -53), ("pair", 2.0 ** -44)])
@pytest.mark.parametrize("scale", [1e2, 1e4, 1e6, 1e9])
@pytest.mark.parametrize("m,n,copies", [(3, 13, 1), (4, 12, 1), (4, 24, 50), (5, 13, 1), (5, 30, 50), (6, 13, 1),
                                        (6, 22, 50), (7, 13, 1), (7, 16, 50), (8, 12, 1), (8, 16, 50)])
def test_columns_of_unequal_size(m, n, copies, scale, mode, unit):
    if mode == "pair":
        scale = min(scale, 10.0 ** (30 / (m - 1)))  # gradients within the binary32 range
    a = np.random.default_rng(3300 + 20 * m + n).uniform(-1, 1, (m, n)) * _factors(n, scale)[:, None, :]
    A = torch.from_numpy(np.tile(a, (copies, 1, 1))).cuda()
    grad = R().radic_det_backward(A, torch.ones(len(A), dtype=torch.float64, device="cuda"), mode=mode).cpu().numpy()
    for b in range(len(a)):
        want = np.array([[float(x) for x in row] for row in orc.radic_grad_exact(a[b], use_pfaffian=True)])
        err = np.abs(grad[b] - want).max(axis=0)
        assert np.all(err <= _bound(a[b], unit)), (b, err / np.abs(want).max(axis=0))
