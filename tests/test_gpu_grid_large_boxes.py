"""The obstacle grid's build over few cells with long lists (large boxes: 32
threads a cell), in one block and several, against the oracle, which tests
every box."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2602_02846_gb300 as kpx  # noqa: E402
from paper_2602_02846_gb300 import scenes  # noqa: E402
from tests import gpu_helpers as gh  # noqa: E402


@pytest.mark.parametrize("n_boxes,edge", [(1, 0.9), (33, 0.5), (300, 0.45), (1100, 0.3), (1100, 0.08), (3000, 0.15)])
def test_obstacle_grid_verdicts(n_boxes, edge):
    prob = scenes.di_scene(n_boxes, n_obstacles=0, grid_pos=16, tree_cap=16384, lam=64)
    rng = np.random.default_rng([n_boxes, 5])
    c, e = rng.uniform(0, 1, (n_boxes, 3)), 0.5 * edge * rng.uniform(0.4, 1, (n_boxes, 3))
    boxes = np.clip(np.concatenate([c - e, c + e], 1), 0, 1).astype(np.float32)
    start = np.asarray(prob.start[:3])
    near = ((boxes[:, :3] <= start + 0.1) & (boxes[:, 3:] >= start - 0.1)).all(1)
    boxes[near] = [0.8, 0.1, 0.1, 0.9, 0.9, 0.9]  # away from the start, the same box many times over
    pl = kpx.Planner(prob.replace(obstacles=boxes))
    hits = 0
    for _ in range(3):
        rep = gh.step_phases(pl, prob.replace(obstacles=boxes))
        hits += rep["slots"] - rep["valid"]
    assert hits > 0
    pl.close()
