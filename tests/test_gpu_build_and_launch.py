"""The obstacle grid's one-launch build at the edges of its lists (a block's
256 threads, 1,024 listed boxes, the 6,000 boxes a problem may have), and the
ways an iteration is launched: the allocation-free call's hand-over from the
one-cluster kernel to the phase kernels, at iteration counts around its look
at the planner's state, against kpx_iterate with and without that kernel."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2602_02846_gb300 as kpx  # noqa: E402
from paper_2602_02846_gb300 import scenes  # noqa: E402
from tests import gpu_helpers as gh  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("n_boxes,edge,walls", [(1, 0.2, 0), (255, 0.02, 3), (257, 0.02, 0), (1100, 0.01, 40),
                                                (6000, 0.006, 2)])
def test_obstacle_grid_verdicts(n_boxes, edge, walls):
    """Every phase against the oracle, which tests every box: a box missing
    from a cell's list, or listed in another's, changes a verdict.  walls: thin
    boxes across the whole workspace, listed in many cells."""
    rng = np.random.default_rng([0x6B1D, n_boxes])
    boxes = scenes.di_obstacles(n_boxes, n_boxes - walls, edge=(0.5 * edge, edge))
    thin = rng.uniform(0.2, 0.8, walls)
    thin = np.stack([thin, 0 * thin, 0 * thin, thin + 1e-3, 0 * thin + 0.4, 0 * thin + 1], 1).astype(np.float32)
    boxes = np.concatenate([boxes, thin.reshape(-1, 6)])[rng.permutation(n_boxes)]
    prob = scenes.di_scene(n_boxes, n_obstacles=0, grid_pos=16, tree_cap=16384, lam=64).replace(
        obstacles=np.ascontiguousarray(boxes))
    pl = kpx.Planner(prob)
    hits = 0
    for _ in range(3):
        rep = gh.step_phases(pl, prob)
        hits += rep["slots"] - rep["valid"]
    assert hits > 0
    pl.close()


@pytest.mark.parametrize("iters", [0, 1, 4, 8, 9, 13, 40])
@pytest.mark.parametrize("cap", [700, 16384])
def test_static_call_equals_workspace_call(iters, cap):
    prob = scenes.di_scene(7, grid_pos=12, tree_cap=cap)
    ref = []
    for flags in (0, kpx.KPX_FLAG_NO_FUSED):
        pl = kpx.Planner(prob, flags=flags)
        pl.iterate(iters)
        ref.append(pl.best_trajectory())
        pl.close()
        st, tr = kpx.kpx_plan_static(prob, iters, stream=torch.cuda.current_stream(), flags=flags)
        assert st == (kpx.KPX_NO_SOLUTION if ref[-1] is None else kpx.KPX_OK)
        ref.append(tr)
    for tr in ref[1:]:
        assert (tr is None) == (ref[0] is None)
        if tr is not None:
            assert tr["cost"] == ref[0]["cost"]
            for k in ("states", "controls", "steps"):
                assert np.array_equal(tr[k], ref[0][k])
    if iters == 40 and cap == 16384:
        assert ref[0] is not None
