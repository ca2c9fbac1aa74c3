"""The one-cluster kernel's two forms and the wide one's split of a rollout
over several warps: at slot counts around the line between them and each number
of parts' limit (and one slot, one warp, and the largest iteration taken), with the obstacle grid absent, copied into
shared memory and too large for that, against the phase kernels, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2602_02846_gb300 as kpx  # noqa: E402
from paper_2602_02846_gb300 import scenes  # noqa: E402
from tests.test_gpu_fused import _same, _state  # noqa: E402

SLOTS = [1, 31, 33, 511, 512, 513, 1023, 1024, 1025, 2048, 2049, 4096, 4097, 8191, 8192, 8193]


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("lam", SLOTS)
@pytest.mark.parametrize("make,boxes,early", [(scenes.di_scene, 60, 0), (scenes.di_scene, 0, 0),
                                              (scenes.dubins_scene, 200, 0), (scenes.dubins_scene, 6000, 0),
                                              (scenes.dubins_scene, 200, 1)])
def test_split_equals_phase_kernels(make, boxes, early, lam):
    """The first iteration has lam slots (the tree is its root); the next ones
    have lam per active node: other part counts, until the phase kernels take
    over."""
    prob = make(lam, n_obstacles=boxes, tree_cap=1 << 16, lam=lam)
    flags = kpx.KPX_FLAG_EARLY_REJECT if early else 0
    fused, plain = kpx.Planner(prob, flags=flags), kpx.Planner(prob, flags=flags | kpx.KPX_FLAG_NO_FUSED)
    for n in (1, 3):
        fused.iterate(n)
        plain.iterate(n)
        _same(_state(plain, not early), _state(fused, not early), "%d iterations of %d slots a node" % (n, lam))
    assert (fused.header().fused_iterations > 0) == (lam <= 8192)
    fused.close()
    plain.close()
