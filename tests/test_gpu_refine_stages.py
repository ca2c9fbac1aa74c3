"""The adjoint differentiates the trajectory that was integrated: the RK4
stages it records sum to the very state of the forward step, bit for bit, also
where 1 / cos(pitch) is large."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_2602_02846_gb300 import build, scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stages(tmp_path_factory):
    here = os.path.dirname(os.path.abspath(__file__))
    so = str(tmp_path_factory.mktemp("stages") / "libstages.so")
    subprocess.run([build.nvcc(), *build.ARCH, *build.flags_for("kpx_adjoint.cu"), "-shared",
                    os.path.join(here, "refine_stages.cu"), "-o", so], check=True)
    fn = C.CDLL(so).stage_steps
    fn.argtypes = [C.c_int, C.c_float, C.c_float, C.c_float, C.POINTER(C.c_float)] + [C.c_void_p] * 5
    return fn


@pytest.mark.parametrize("inertia", [(1.0, 1.0, 1.0), (1.0, 1.25, 1.75)])
def test_stages_sum_to_the_step(stages, inertia):
    import torch
    n = 1 << 16
    rng = np.random.default_rng(7)
    x = rng.uniform(-1, 1, (n, 12)) * ([1.0] * 3 + [0.8, 0.8, 3.0] + [1.0] * 3 + [3.0] * 3)
    x[: n // 4, 4] = np.pi / 2 - 10.0 ** rng.uniform(-4, -1, n // 4)  # next to cos(pitch) = 0
    mg = scenes.QUAD_MASS * scenes.QUAD_G
    u = np.concatenate([mg + rng.uniform(-0.5, 0.5, (n, 1)), rng.uniform(-1e-3, 1e-3, (n, 3))], axis=1)
    prob = scenes.quad_scene(0, clutter=0, certify=False)
    J = (C.c_float * 3)(*[float(prob.param[2]) * k for k in inertia])
    xd, ud = (torch.as_tensor(a.astype(np.float32), device="cuda") for a in (x, u))
    by_step, by_stage = (torch.empty((n, 6), dtype=torch.float32, device="cuda") for _ in range(2))
    assert stages(n, float(prob.h), float(prob.param[0]), float(prob.param[1]), J, xd.data_ptr(), ud.data_ptr(),
                  by_step.data_ptr(), by_stage.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    a, b = by_step.cpu().numpy(), by_stage.cpu().numpy()
    assert np.isfinite(a).all() and not np.array_equal(a[:, :3], x[:, 3:6].astype(np.float32))
    assert np.array_equal(a.view(np.int32), b.view(np.int32))
