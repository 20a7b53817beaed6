"""The integer-pipe remainder of the FP64 to FP32 narrowing (csrc/widen.cuh, its own text built with
g++): bit for bit narrow(d - widen(narrow(d))) for |d| <= 1, zero below 2^-74 as documented."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1607_03252_gb300", "csrc")


def test_remainder_of_the_narrowing(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    src = open(os.path.join(CSRC, "widen.cuh")).read()
    body = src[src.index("__device__ __forceinline__ double widen(float f) {"):src.index("}  // namespace mlmc")]
    (tmp_path / "widen_narrow.inc").write_text(body.replace("__device__ __forceinline__", "static inline"))
    exe = tmp_path / "emu"
    res = subprocess.run([gxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I", str(tmp_path),
                          os.path.join(HERE, "host_emu", "narrow_rest_emu.cpp"), "-o", str(exe)],
                         capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-3000:]
    res = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert res.returncode == 0, res.stdout
