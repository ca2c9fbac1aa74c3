"""Re-validation with and without a block's box grid: a short trajectory alone
is checked against every box, its steps' boxes dealt out over the warp; among
others of its block it is checked through the grid.  Both end at the same state
with the same verdict."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_02846_gb300 import refine, scenes  # noqa: E402


@pytest.mark.parametrize("steps", [1, 2, 3, 8, 9, 16, 17, 24])
@pytest.mark.parametrize("n_boxes,large", [(1, 0), (31, 0), (130, 0), (1000, 0), (60, 1), (500, 500)])
def test_alone_equals_among_others(steps, n_boxes, large):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    count, check = 32 * sms, 24  # 32 trajectories a block: more than 24 steps together
    prob = scenes.quad_scene(0, clutter=-1).replace(goal_c=[0.3, 0.5, 0.5], goal_r=0.2)
    rng = np.random.default_rng([steps, n_boxes, large])
    u = np.zeros((count, 2, 4), np.float32)
    u[:, :, 0] = prob.param[0] * prob.param[1] + rng.uniform(-0.8, 0.8, (count, 2))
    u[:, :, 1:] = rng.uniform(-0.004, 0.004, (count, 2, 3))
    k = np.stack([np.full(count, steps // 2), np.full(count, steps - steps // 2)], 1).astype(np.int32)
    x0 = np.tile(np.asarray(prob.start, np.float32), (count, 1))
    x0[:, :3] = rng.uniform(0.1, 0.9, (count, 3))
    x0[:, 6:9] = rng.uniform(-0.9, 0.9, (count, 3))
    c, e = rng.uniform(0, 1, (n_boxes, 3)), rng.uniform(0.004, 0.04, (n_boxes, 3))
    e[:large] = rng.uniform(0.2, 0.3, (large, 3))  # boxes of many cells; 500 of them: lists that do not fit
    obs = np.concatenate([c - e, c + e], 1).astype(np.float32)
    n = np.full(count, 2, np.int32)
    valid, cost, xe = refine.validate(refine.Batch(prob, x0, u, k, n, obstacles=obs))
    # one call for each trajectory alone
    for i in range(check):
        vi, ci, xi = refine.validate(refine.Batch(prob, x0[i:i + 1], u[i:i + 1], k[i:i + 1], n[i:i + 1],
                                                  obstacles=obs))
        assert torch.equal(valid[i:i + 1], vi) and torch.equal(cost[i:i + 1], ci) and torch.equal(xe[i:i + 1], xi), i
    # and the verdicts against the boxes: no end state lies in one unless that ended the trajectory
    p = xe[:, None, :3].cpu().numpy()
    inside = ((p >= obs[None, :, :3]) & (p <= obs[None, :, 3:])).all(-1).any(-1)
    assert not (inside & valid.cpu().numpy()).any() and (large == 500 or not inside.all())
