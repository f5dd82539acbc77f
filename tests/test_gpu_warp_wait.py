"""The bounded waits of the GEMM kernels end alike in all lanes of a warp."""
import os
import re
import subprocess

import pytest

from paper_2504_13850_gb300 import build

NATIVE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "native")


def outside_elected(code):
    """The lines of `code` outside every `if (elect_one()) {` block."""
    out, depth, elected = [], 0, []
    for line in code.split("\n"):
        if not elected:
            out.append(line.strip())
        opened = line.find("if (elect_one()) {")
        for i, ch in enumerate(line):
            if ch == "{":
                depth += 1
                if opened >= 0 and i >= opened and not elected:
                    elected.append(depth)
            elif ch == "}":
                if elected and elected[-1] == depth:
                    elected.pop()
                depth -= 1
    return out


def test_no_lane_decides_for_itself():
    """Lanes that a wait or the abort flag may send different ways never meet in an instruction for the
    whole warp: one elected lane runs the producer's and the MMA issuer's loops, the epilogue votes.
    (The split-K kernel's epilogue warps only note a wait that ran out, and never leave.)"""
    code = re.sub(r"//[^\n]*", "", open(os.path.join(build.CSRC, "tc_gemm_kernels.cuh")).read())
    free = outside_elected(code)
    assert len(free) < code.count("\n")          # some blocks are elected
    assert sorted(x for x in free if re.search(r"\bmbar_wait\(", x)) == [
        "if (!mbar_wait(accum, 0)) atomicExch(p.err, 3);", "if (!mbar_wait(rbar, 0)) atomicExch(p.err, 9);"]
    assert not [x for x in free if re.search(r"(if|for|while) \(.*\*abort_flag", x)]


@pytest.mark.gpu
def test_lanes_agree_when_some_of_them_time_out(tmp_path):
    exe = str(tmp_path / "warp_wait")
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC,
                    os.path.join(NATIVE, "warp_wait.cu"), "-o", exe], check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.split() == ["0", "32", "32", "0", "2"], (r.returncode, r.stdout)
