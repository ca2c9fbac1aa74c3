"""The penalty's reciprocals and roots (a hardware approximation and one Newton
step) against CUDA's correctly rounded ones.

reciprocal() and root() are correctly rounded for every mantissa.  The other two
start from approximations of a few units in the last place; the Newton step
squares that error, which leaves the rounding of its last operation (half a unit,
and a little): the result is the correctly rounded value or its neighbour."""
import ctypes as C
import os
import subprocess

import pytest

from paper_2602_02846_gb300 import build

pytestmark = pytest.mark.gpu


def test_against_correctly_rounded(tmp_path):
    import torch
    here = os.path.dirname(os.path.abspath(__file__))
    so = str(tmp_path / "libroots.so")
    subprocess.run([build.nvcc(), *build.ARCH, *build.flags_for("kpx_adjoint.cu"), "-shared",
                    os.path.join(here, "refine_roots.cu"), "-o", so], check=True)
    fn = C.CDLL(so).check_roots
    fn.argtypes = [C.c_void_p, C.c_void_p]
    out = torch.zeros((5, 2), dtype=torch.int64, device="cuda")
    assert fn(out.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    differ, worst = out.cpu().T.tolist()
    print("differ", differ, "worst", worst)
    assert differ[:3] == [0, 0, 0]           # reciprocal, root, the distance
    assert differ[3] <= 4 and worst[3] <= 1  # the distance's reciprocal, of 2^24 values
    assert worst[4] <= 1 and differ[4] <= (6 << 24) // 100
