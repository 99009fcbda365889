"""The FP64 reciprocal and reciprocal square root that take the place of IEEE
divisions and roots in the FP64 kernels, held to the error stated beside them
(2 ulp) over their whole range, in a small program of its own built around the
library's header."""
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2301_09349_gb300", "csrc")
SRC = os.path.join(ROOT, "tests", "native", "reciprocals_check.cu")


def test_fp64_reciprocals_within_two_ulp(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2301_09349_gb300 import build
    exe = str(tmp_path / "reciprocals_check")
    r = subprocess.run([build.nvcc()] + build.ARCH + ["-O2", "-std=c++17", "-I" + CSRC, SRC, "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    print(r.stdout)
    assert r.returncode == 0, r.stdout + r.stderr
