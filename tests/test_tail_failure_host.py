"""The one-launch cycle reports a kernel that cannot be launched: the launcher's and the cycle
runner's own text, built with g++ against a runtime that refuses the dynamic shared memory. Every
cycle of every solve has to fail, direct or captured, and nothing of the capture may be left."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
MG = os.path.join(os.path.dirname(HERE), "paper_1607_03252_gb300", "csrc", "mg.cu")


def _cut(text, start, end):
    a = text.index(start)
    return text[a:text.index(end, a)]


def test_cycle_reports_a_kernel_that_cannot_be_launched(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    src = open(MG).read()
    launch = _cut(src, "template <typename T, int N0, bool SPLIT, bool P1>\ncudaError_t tail_launch(",
                  "// One level of the V-cycle on colour-split FP32 storage")
    launch = re.sub(r"k_vcycle_tail<T, N0, SPLIT, P1><<<[^>]*>>>\(A\)", "emu_launch(A)", launch)
    assert "emu_launch" in launch
    (tmp_path / "hier.inc").write_text(
        _cut(src, "template <typename T>\nstruct Level {", "template <typename T>\nstruct Hier {")
        + _cut(src, "template <typename T>\nstruct TailLevel {", "// One grid of the tail in a block"))
    (tmp_path / "tail.inc").write_text(
        _cut(src, "inline int tail_coef_arrays(", "template <typename T, int N0, bool SPLIT, bool P1>\n__global__") + launch)
    (tmp_path / "runner.inc").write_text(
        _cut(src, "template <typename T>\nstruct GraphRunner {", "// The vector kernels of flexible CG"))
    exe = tmp_path / "emu"
    res = subprocess.run([gxx, "-std=c++17", "-O1", "-I", str(tmp_path),
                          os.path.join(HERE, "host_emu", "tail_failure_emu.cpp"), "-o", str(exe)],
                         capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-4000:]
    res = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert res.returncode == 0, res.stdout
