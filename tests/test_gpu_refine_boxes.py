"""Where the refinement kernels keep their boxes: blocks of 32 trajectories that
leave no room for them in shared memory (gradient and re-validation read the
caller's array), and boxes that reach so many cells that no lists fit (every box
is tested).  Batches against the same trajectories alone, exactly, and against
the FP64 oracle with the tolerances of test_gpu_refine.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_2602_02846_gb300 import refine, scenes  # noqa: E402

LIMIT = 226 * 1024  # dynamic shared memory of a block


def _batch(count, n_boxes, aniso, beta):
    prob = scenes.quad_scene(0, clutter=-1)
    if aniso:
        par = list(prob.param)
        par[3], par[4] = scenes.f32(1.25 * par[2]), scenes.f32(1.75 * par[2])
        prob = prob.replace(param=par)
    rng = np.random.default_rng([count, n_boxes, aniso])
    S = 3
    n_seg = rng.integers(1, S + 1, count).astype(np.int32)
    k = rng.integers(2, 16, (count, S)).astype(np.int32)
    u = np.zeros((count, S, 4), np.float32)
    u[:, :, 0] = prob.param[0] * prob.param[1] + rng.uniform(-0.8, 0.8, (count, S))
    u[:, :, 1:] = rng.uniform(-0.004, 0.004, (count, S, 3))
    live = np.arange(S)[None, :] < n_seg[:, None]
    u *= live[:, :, None]
    k *= live
    x0 = np.tile(np.asarray(prob.start, np.float32), (count, 1))
    x0[:, 6] = rng.uniform(-0.8, 0.8, count)
    c, e = rng.uniform(0, 1, (n_boxes, 3)), rng.uniform(0.004, 0.015, (n_boxes, 3))
    obs = np.concatenate([c - e, c + e], 1).astype(np.float32)
    spec = dict(w_obs=1.0, beta=beta, margin=0.01, w_goal=10.0, goal=[0.95, 0.5, 0.5], w_effort=1.0)
    return prob, spec, x0, u, k, n_seg, obs


@pytest.mark.parametrize("whole_blocks,aniso", [(False, False), (True, False), (True, True)])
@pytest.mark.parametrize("n_boxes,beta", [(1300, 200.0), (1300, 15.0)])
def test_gradient_and_validation(whole_blocks, aniso, n_boxes, beta):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    count = 32 * sms if whole_blocks else 3
    # one trajectory's part of a backward block (floats; kpx_adjoint.cu: states,
    # segments, two chunks of 8 records) and of a validating block (bytes)
    part = 2 * 32 * 9 + 3 * 32 + 16 * (4 * (20 if aniso else 16) + 4 + 1)
    assert (33 * part * 4 + 32 * n_boxes > LIMIT) and (part * 4 + 32 * n_boxes <= LIMIT)
    assert 33 * 4352 + 49152 + 32 * n_boxes > LIMIT
    prob, spec, x0, u, k, n_seg, obs = _batch(count, n_boxes, aniso, beta)
    batch = refine.Batch(prob, x0, u, k, n_seg, obstacles=obs)
    J, g = refine.evaluate(batch, spec, grad=True)
    tests = refine.box_tests(batch)
    # with beta = 15 a term reaches 2 units: 16^3 cells of 1,300 boxes each
    assert (tests[0] == tests[2] == int(k.sum()) * n_boxes) == (beta == 15.0)
    valid, cost, xe = refine.validate(batch)
    for i in sorted({0, 1, 2, count // 2, count - 1}):
        part_i = slice(i, i + 1)
        alone = refine.Batch(prob, x0[part_i], u[part_i], k[part_i], n_seg[part_i], obstacles=obs)
        Ji, gi = refine.evaluate(alone, spec, grad=True)
        assert torch.equal(J[part_i], Ji) and torch.equal(g[part_i], gi), i
        for a, b in zip((valid, cost, xe), refine.validate(alone)):
            assert torch.equal(a[part_i], b), i
        n = int(n_seg[i])
        if i < 2:
            J64, g64 = oracle.refine_grad(prob, spec, x0[i].astype(np.float64), u[i, :n].astype(np.float64), k[i, :n],
                                          obstacles=obs.astype(np.float64))
            assert abs(float(J[i]) - J64) <= 1e-4 * abs(J64), i
            assert np.abs(g[i, :n].cpu().numpy() - g64).max() <= 2e-3 * np.abs(g64).max(), i
