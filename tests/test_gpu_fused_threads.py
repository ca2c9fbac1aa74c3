"""Planners made by several host threads at once as a process's first ones: each
gets the one-cluster kernel, in the form its iterations need."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import threading
import torch
import paper_2602_02846_gb300 as kpx
from paper_2602_02846_gb300 import scenes
torch.zeros(1, device="cuda")
problems = [m(i, lam=lam, tree_cap=1 << 14) for i in range(2) for m in (scenes.di_scene, scenes.dubins_scene)
            for lam in (16, 1024)]
got, start = [None] * len(problems), threading.Barrier(len(problems))

def work(i):
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        start.wait()
        pl = kpx.Planner(problems[i], stream=stream)
        pl.iterate(1)
        stream.synchronize()
        got[i] = pl.header().fused_iterations
        pl.close()
threads = [threading.Thread(target=work, args=(i,)) for i in range(len(problems))]
for t in threads:
    t.start()
for t in threads:
    t.join()
assert got == [1] * len(problems), got
"""


def test_first_planners_of_several_threads():
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
