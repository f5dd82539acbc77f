"""Classifier heads of different class counts, launched from two threads: none
lowers the shared-memory limit under the other's launch."""
import os
import subprocess

import pytest

from paper_2504_13850_gb300 import build

pytestmark = pytest.mark.gpu
NATIVE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "native")


def test_two_class_counts_from_two_threads(tmp_path):
    exe = str(tmp_path / "head_threads")
    subprocess.run([build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC,
                    "-I", os.path.join(build.HERE, "..", "include"), os.path.join(NATIVE, "head_threads.cu"),
                    os.path.join(build.CSRC, "k_head.cu"), "-o", exe], check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.split() == ["0", "0"], (r.returncode, r.stdout)
