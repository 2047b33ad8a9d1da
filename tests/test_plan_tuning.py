"""Host-only task lists of tuned batch plans (no GPU)."""
import pytest

import paper_1508_01326_gb300 as R

SHAPES = [(8, 30), (9, 29), (10, 24), (10, 30)]


@pytest.mark.parametrize("cost", [1000.0, 4000.0, 12000.0, 80000.0])
def test_low_tier_segments_do_not_follow_the_task_cost(cost):
    # the pair and binary32 tiers round their bounds per lane total, so the
    # segments of a head's last columns stay as they are whatever the tuning
    tuning = dict(prefix_depth={8: 2})
    plain = R.batch_tasks_host(SHAPES, mode="mixed", tuning=R.make_tuning(**tuning))
    tuned = R.batch_tasks_host(SHAPES, mode="mixed",
                               tuning=R.make_tuning(task_cost={m: cost for m, _ in SHAPES}, **tuning))
    cuts = lambda ts: {(t["b"], t["group"], t["vlo"], t["vhi"]) for t in ts}
    assert all(t["shared"] and t["tier"] != 0 for t in plain)
    assert cuts(tuned) == cuts(plain)
