"""Binary64 batches: a named task cost pins the split, so a matrix has the same bits in every batch; without
one the split follows the batch and values differ by rounding only."""
import numpy as np
import pytest
import torch

from paper_1508_01326_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def R():
    import paper_1508_01326_gb300 as mod

    return mod


SHAPES = [(2, 20), (3, 14), (4, 16), (5, 15), (6, 14), (7, 13), (8, 14), (9, 14), (10, 14)]


def _solve(mats, tuning):
    data, ms, ns, offs = W.pack_batch(mats, np.float64)
    plan = R().BatchPlan(list(zip(ms, ns)), offs, mode="fp64", tuning=tuning)
    out = plan.radic_det_batched(torch.from_numpy(data).cuda())
    return out.view(torch.float64)[:, :3].cpu().numpy(), plan.info()


@pytest.mark.parametrize("cost", [0.0, 1500.0, 6000.0, 30000.0])
def test_results_in_batches_of_different_size(cost):
    mats = [W.uniform_matrix(560 + i, m, n) for i, (m, n) in enumerate(SHAPES)]
    others = [W.uniform_matrix(600 + i, 2 + i % 9, 14 + i % 9) for i in range(300)]
    tuning = R().make_tuning(task_cost={m: cost for m in range(2, 11)}) if cost else None
    small, _ = _solve(mats, tuning)
    large, _ = _solve(mats + others, tuning)
    if cost:
        assert np.array_equal(small, large[:len(mats)])
    else:
        assert np.all(np.abs(small - large[:len(mats)])[:, 0] <= 1e-13 * small[:, 1])
        assert np.all(np.abs(small - large[:len(mats)])[:, 1] <= 1e-13 * small[:, 1])


def test_host_task_list_matches_the_device_plan():
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the host list is planned for 152 SMs")
    shapes = SHAPES * 20
    _, info = _solve([W.uniform_matrix(700 + i, m, n) for i, (m, n) in enumerate(shapes)], None)
    assert info["tasks_fp64"] == len(R().batch_tasks_host(shapes, mode="fp64"))
