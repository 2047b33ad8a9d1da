"""Host-only plans of binary64 prefixes of depth 2 that several lanes share (no GPU)."""
import pytest

import paper_1508_01326_gb300 as R


@pytest.mark.parametrize("m", [4, 5, 6])
@pytest.mark.parametrize("per_sm", [2, 3, 4])
def test_shared_prefixes_do_not_repeat_eliminations_for_nothing(m, per_sm):
    # every lane that shares a prefix repeats its elimination, m (m-2)^2
    # operations: once the tasks fill the chip, that stays below twice the
    # work of the launch with one lane per prefix
    sms = 152
    for n in range(m + 1, 65):
        plan = R.prefix_plan_host(m, n, "fp64", sms=sms, blocks_per_sm=per_sm)
        if plan["tasks"] <= sms * per_sm * 4:
            continue
        red = m * (m - 2) ** 2
        total = repeated = 0
        for v, g in plan["groups"].items():
            k = n - 1 - v
            total += g["count"] * (red + k * (m + 4 * (m - 2)) + 3 * k * (k - 1))
            repeated += g["count"] * g["lanes"] * red
        assert repeated <= 2 * total, (n, plan["tasks"], repeated / total)
