"""Prefix kernels with blocks of one to four warps: the column buffers behind the reduction scratch are read
as 16-byte vectors, whatever the number of warps."""
from fractions import Fraction

import pytest

import oracle.radic_oracle as orc
from paper_1508_01326_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def R():
    import paper_1508_01326_gb300 as mod

    return mod


@pytest.mark.parametrize("threads", [32, 64, 96, 128])
@pytest.mark.parametrize("mode", ["fp64", "mixed", "pair"])
@pytest.mark.parametrize("m,n,depth", [(3, 8, 2), (4, 9, 2), (4, 9, 3), (5, 11, 2), (7, 12, 2), (7, 12, 3), (10, 14, 2),
                                       (10, 14, 3)])
def test_every_block_size(m, n, depth, mode, threads):
    a = W.uniform_matrix(1200 + m + depth, m, n)
    val, abs_sum = orc.radic_det_exact(a)
    r = R().det(a, mode=mode, options=dict(mapping="prefix", prefix_depth=depth, threads_per_block=threads))
    tol = 8 * m * 2.0 ** -24 if mode == "mixed" else 1e-11
    assert abs(Fraction(r["value"]) - val) <= Fraction(tol) * abs_sum
    if mode != "pair":  # pairs sum the magnitudes of a prefix in binary32
        assert abs(Fraction(r["abs_sum"]) - abs_sum) <= Fraction(tol) * abs_sum
    assert abs(Fraction(r["value"]) - val) <= Fraction(r["err_bound"])
