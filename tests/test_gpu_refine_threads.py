"""Refinement calls of different sizes from two host threads at once: each
call's launches need another amount of shared memory, and no call may lower
what another one's launch is allowed."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2602_02846_gb300 import refine, scenes  # noqa: E402


def _batch(count, n_boxes):
    prob = scenes.quad_scene(0, clutter=-1)
    rng = np.random.default_rng([count, n_boxes])
    u = np.zeros((count, 2, 4), np.float32)
    u[:, :, 0] = prob.param[0] * prob.param[1] + rng.uniform(-0.8, 0.8, (count, 2))
    x0 = np.tile(np.asarray(prob.start, np.float32), (count, 1))
    c = rng.uniform(0.2, 0.9, (n_boxes, 3))
    obs = np.concatenate([c - 0.01, c + 0.01], 1).astype(np.float32)
    return refine.Batch(prob, x0, u, rng.integers(1, 4, (count, 2)).astype(np.int32), np.full(count, 2, np.int32),
                        obstacles=obs)


def test_two_threads_with_launches_of_different_sizes():
    batches = [_batch(1, 4), _batch(3000, 2500)]
    spec = refine.default_cost(batches[0].prob)

    def both(b, stream):
        J, g = refine.evaluate(b, spec, grad=True, stream=stream)
        return (J, g) + refine.validate(b, stream=stream)

    want = [both(b, torch.cuda.current_stream()) for b in batches]
    torch.cuda.synchronize()
    failures, start = [], threading.Barrier(len(batches))

    def work(i):
        try:
            stream = torch.cuda.Stream()
            start.wait()
            with torch.cuda.stream(stream):
                for _ in range(2500):
                    got = both(batches[i], stream)
            stream.synchronize()
            assert all(torch.equal(a, w) for a, w in zip(got, want[i])), i
        except Exception as e:
            failures.append(repr(e))
    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(batches))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures
