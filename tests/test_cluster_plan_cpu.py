"""The distribution of a quadrature system's rows over a thread-block cluster,
compiled with the host compiler and checked for every marker count and for
devices that can place clusters of 16, of 8 or none (where the one-CTA solver
serves)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2301_09349_gb300", "csrc")
SRC = os.path.join(ROOT, "tests", "native", "cluster_plan_check.cpp")


def test_cluster_plan_for_every_width(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "cluster_plan_check")
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-I" + CSRC, SRC, "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "cluster plan ok" in r.stdout
