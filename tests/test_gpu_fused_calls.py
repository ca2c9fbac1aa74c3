"""The one-cluster kernel's forms by call and problem: calls of one or two
iterations (one form alone), of more (both), problems whose slots cannot need
one of the forms; grown past every hand-over, against the phase kernels, bit
for bit."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2602_02846_gb300 as kpx  # noqa: E402
from paper_2602_02846_gb300 import scenes  # noqa: E402
from tests.test_gpu_fused import _same, _state  # noqa: E402


@pytest.mark.parametrize("make,lam,cap", [
    (scenes.di_scene, 16, 1 << 15), (scenes.dubins_scene, 16, 1 << 15),   # through 512, 4,096 and 8,192 slots
    (scenes.di_scene, 4, 128), (scenes.dubins_scene, 2, 256),             # at most 512 slots
    (scenes.dubins_scene, 513, 1 << 14),                                  # never fewer
    (scenes.di_scene, 0, 900), (scenes.di_scene, 0, 1023), (scenes.dubins_scene, 0, 1024), (scenes.di_scene, 0, 5000),
])
@pytest.mark.parametrize("calls", [(1,), (2, 1), (3, 1, 40, 2)])
@pytest.mark.parametrize("many", [False, True])
def test_calls_equal_phase_kernels(make, lam, cap, calls, many):
    prob = make(5, n_obstacles=40, tree_cap=cap, lam=lam)
    fused, plain = kpx.Planner(prob), kpx.Planner(prob, flags=kpx.KPX_FLAG_NO_FUSED)
    if many:  # the graph of the few-iteration calls is built after 64 of them
        for _ in range(70):
            fused.iterate(1)
        fused.reset()
    for i in range(60 // sum(calls) + 1):
        for n in calls:
            fused.iterate(n)
            plain.iterate(n)
        if i % 5 == 0:
            _same(_state(plain, True), _state(fused, True), "%d of %r" % (i, calls))
    _same(_state(plain, True), _state(fused, True), "the end")
    assert fused.header().fused_iterations > 0 and fused.header().graph_pending == 0
    fused.close()
    plain.close()
