"""The packed logistic-regression gradient's reciprocal of 1 + e^-|z| is the division's,
bit for bit, on every binary32 value of [1, 2] (so that the packed kernel's results do not
depend on which of the two it uses).  The probe (tests/gpu_src/reciprocal.cu) is compiled
by this test with nvcc."""
import ctypes as C
import os
import subprocess

import pytest
import torch

pytestmark = pytest.mark.gpu

SRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "gpu_src", "reciprocal.cu")


def test_reciprocal_equals_the_division(tmp_path):
    from paper_2601_16696_gb300 import build
    so = str(tmp_path / "libreciprocal.so")
    cmd = [build._nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", SRC, "-o", so]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    lib = C.CDLL(so)
    lib.compare_reciprocal.argtypes = [C.c_void_p, C.c_void_p]
    bad = torch.zeros(1, dtype=torch.int32, device="cuda")
    assert lib.compare_reciprocal(bad.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    assert bad.item() == 0
