"""The refinement passes at the edges of their layout: a block's 32
trajectories, one wave of blocks, checkpoint intervals of 32 steps, segments
without steps, the box counts that change where boxes are kept and how fine
their grid is, and an inertia that is not isotropic.

A trajectory's objective and gradient do not depend on the batch it is in, so
a large batch is compared with the same trajectories in small ones, exactly.
Against the FP64 oracle the tolerances are those of test_gpu_refine.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_2602_02846_gb300 import refine, scenes  # noqa: E402

SPEC = dict(w_obs=1.0, beta=200.0, margin=0.01, w_goal=10.0, goal=[0.95, 0.5, 0.5], w_effort=1.0)


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _inputs(B, S, steps, n_boxes, seed, aniso=False):
    prob = scenes.quad_scene(0, clutter=-1)
    if aniso:
        par = list(prob.param)
        par[3], par[4] = scenes.f32(1.25 * par[2]), scenes.f32(1.75 * par[2])
        prob = prob.replace(param=par)
    rng = np.random.default_rng([0xADF, seed])
    n_seg = rng.integers(0, S + 1, B).astype(np.int32)
    n_seg[0] = S
    k = rng.integers(steps[0], steps[1] + 1, (B, S)).astype(np.int32)
    u = np.zeros((B, S, 4), np.float32)
    u[:, :, 0] = prob.param[0] * prob.param[1] + rng.uniform(-0.8, 0.8, (B, S))
    u[:, :, 1:] = rng.uniform(-0.004, 0.004, (B, S, 3))
    live = np.arange(S)[None, :] < n_seg[:, None]
    u *= live[:, :, None]
    k *= live
    x0 = np.tile(np.asarray(prob.start, np.float32), (B, 1))
    x0[:, 6] = 0.8
    c = np.column_stack([rng.uniform(0.0, 0.6, n_boxes), 0.5 + rng.uniform(-0.3, 0.3, (n_boxes, 2))])
    e = rng.uniform(0.004, 0.015, (n_boxes, 3))
    obs = np.concatenate([c - e, c + e], 1).astype(np.float32).reshape(-1, 6)
    return prob, x0, u, k, n_seg, obs


@pytest.mark.parametrize("count,steps,n_boxes,aniso", [
    (1, (1, 3), 0, False), (2, (31, 33), 1, False), (33, (0, 40), 40, True), (153, (5, 9), 300, False),
    (305, (0, 2), 1500, False), (64, (10, 20), 4096, True), (152 * 32 + 5, (3, 12), 60, False),
])
def test_batch_equals_its_trajectories_alone(count, steps, n_boxes, aniso):
    prob, x0, u, k, n_seg, obs = _inputs(count, 9, steps, n_boxes, count, aniso)
    J, g = refine.evaluate(refine.Batch(prob, x0, u, k, n_seg, obstacles=obs), SPEC, grad=True)
    assert torch.equal(J, refine.evaluate(refine.Batch(prob, x0, u, k, n_seg, obstacles=obs), SPEC))
    for i in sorted({0, 1 % count, 31 % count, 32 % count, count // 2, count - 1}):
        part = slice(i, i + 1)
        Ji, gi = refine.evaluate(refine.Batch(prob, x0[part], u[part], k[part], n_seg[part], obstacles=obs), SPEC,
                                 grad=True)
        assert torch.equal(J[part], Ji) and torch.equal(g[part], gi), i
        assert not g[i, n_seg[i]:].any()
        if n_seg[i] > 0 and n_boxes <= 300:
            n = int(n_seg[i])
            J64, g64 = oracle.refine_grad(prob, SPEC, x0[i].astype(np.float64), u[i, :n].astype(np.float64), k[i, :n],
                                          obstacles=obs.astype(np.float64))
            assert abs(float(J[i]) - J64) <= 1e-4 * abs(J64), i
            assert np.abs(g[i, :n].cpu().numpy() - g64).max() <= 2e-3 * np.abs(g64).max(), i


@pytest.mark.parametrize("eps", [-1e-3, -1e-20, 0.0, 1e-40, 1e-30, 1e-20, 8e-16, 9e-16, 1e-15, 1e-7, 1e-3])
@pytest.mark.parametrize("far_box", [False, True])
def test_distance_near_a_face(eps, far_box):
    """A hovering point at x = eps beside a box's face at x = 0 (the hover
    keeps x exactly), around the distance where the root changes its form, on
    the face and inside; far_box: with boxes at infinite squared distance in
    the same list (they begin in the cell of the point, which is that large).
    Against the FP64 oracle."""
    prob = scenes.quad_scene(0, clutter=-1)
    x0 = np.zeros((1, 12), np.float32)
    x0[0, :3] = [eps, 0.5, 0.5]
    u = np.zeros((1, 3, 4), np.float32)
    u[:, :, 0] = prob.param[0] * prob.param[1]
    k = np.full((1, 3), 7, np.int32)
    obs = np.float32([[-0.2, 0.2, 0.2, 0.0, 0.8, 0.8], [-0.1, 0.4, 0.4, 0.0, 0.6, 0.6]])
    if far_box:
        far = np.float32([[1e23, 0, 0, 1e25, 1, 1]])
        obs = np.concatenate([far, obs[:1], far, far, obs[1:], far])
    J, g = refine.evaluate(refine.Batch(prob, x0, u, k, np.int32([3]), obstacles=obs), SPEC, grad=True)
    J64, g64 = oracle.refine_grad(prob, SPEC, x0[0].astype(np.float64), u[0].astype(np.float64), k[0],
                                  obstacles=obs.astype(np.float64))
    assert abs(float(J[0]) - J64) <= 1e-4 * abs(J64)
    assert np.abs(g[0].cpu().numpy() - g64).max() <= 2e-3 * np.abs(g64).max()


def test_segments_without_steps_drop_out():
    """A sequence with empty segments in between (more than a window of 32 of
    them) is the sequence without them."""
    prob, x0, u, k, n_seg, obs = _inputs(3, 60, (20, 40), 40, 5)
    n_seg[:] = 60
    k[:, 3:58] = 0
    keep = [0, 1, 2, 58, 59]
    J, g = refine.evaluate(refine.Batch(prob, x0, u, k, n_seg, obstacles=obs), SPEC, grad=True)
    Jk, gk = refine.evaluate(refine.Batch(prob, x0, u[:, keep], k[:, keep], np.full(3, 5, np.int32), obstacles=obs),
                             SPEC, grad=True)
    assert torch.equal(J, Jk) and torch.equal(g[:, keep], gk) and not g[:, 3:58].any()


def test_trajectory_over_the_step_limit():
    """A trajectory of more than max_total_steps steps gets J = NaN and a zero
    gradient; its neighbours are unaffected."""
    prob, x0, u, k, n_seg, obs = _inputs(5, 6, (4, 8), 20, 7)
    ref = refine.Batch(prob, x0, u, k, n_seg, obstacles=obs)
    J0, g0 = refine.evaluate(ref, SPEC, grad=True)
    b = refine.Batch(prob, x0, u, k, n_seg, obstacles=obs)
    totals = k.sum(1)
    b.max_total_steps = int(totals.max()) - 1
    J, g = refine.evaluate(b, SPEC, grad=True)
    for i in range(5):
        if totals[i] > b.max_total_steps:
            assert torch.isnan(J[i]) and not g[i].any()
        else:
            assert J[i] == J0[i] and torch.equal(g[i], g0[i])


@pytest.mark.parametrize("count,steps,n_boxes,repeat,aniso", [
    (1, (1, 3), 0, 1, False), (2, (31, 33), 1, 1, False), (33, (0, 40), 40, 1, True), (153, (5, 9), 300, 1, False),
    (64, (10, 20), 40, 90, False), (152 * 32 + 5, (3, 12), 60, 1, False),
])
def test_validation_batch_equals_its_trajectories_alone(count, steps, n_boxes, repeat, aniso):
    """Re-validation: a batch against its trajectories alone (exactly) and the
    FP64 oracle away from boundaries; repeat: the boxes listed many times over
    and five that fill the workspace's far half, so that the block's grid does
    not hold them."""
    prob, x0, u, k, n_seg, obs = _inputs(count, 9, steps, n_boxes, count, aniso)
    if repeat > 1:
        obs = np.concatenate([obs, np.tile(np.float32([0.7, 0, 0, 1, 1, 1]), (5, 1))])
    prob = prob.replace(goal_c=[0.25, 0.5, 0.5], goal_r=0.2)
    valid, cost, xe = refine.validate(refine.Batch(prob, x0, u, k, n_seg, obstacles=np.tile(obs, (repeat, 1))))
    agree = 0
    for i in sorted({0, 1 % count, 31 % count, 32 % count, count // 2, count - 1}):
        part = slice(i, i + 1)
        vi, ci, xi = refine.validate(refine.Batch(prob, x0[part], u[part], k[part], n_seg[part], obstacles=obs))
        assert torch.equal(valid[part], vi) and torch.equal(cost[part], ci) and torch.equal(xe[part], xi), i
        n = int(n_seg[i])
        r = oracle.validate_controls(prob.replace(obstacles=obs), x0[i].astype(np.float64), u[i, :n], k[i, :n])
        assert abs(float(cost[i]) - r["cost"]) <= 1e-12 * max(r["cost"], 1.0)
        if abs(r["min_clearance"]) >= 1e-4 and abs(r["goal_dist"] - prob.goal_r) >= 1e-4:
            assert bool(valid[i]) == r["valid"], i
            agree += 1
    assert agree >= 1
