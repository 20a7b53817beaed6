"""The tcgen05 field kernel's issuing thread (its own text, built with g++) leaves nothing in
flight, whichever wait runs out and whether the staging warps take part or have given up: every
copy and every commit's arrival has been waited for when it returns, so the block may free its
tensor memory and its shared memory."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
FIELD = os.path.join(os.path.dirname(HERE), "paper_1607_03252_gb300", "csrc", "field.cu")


def test_issuing_thread_leaves_nothing_in_flight(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    src = open(FIELD).read()
    kernel = src[src.index("k_field_umma(const float4*"):]
    a = kernel.index("bool bad = false;")
    wait = kernel[a:kernel.index("if (warp < SW) {", a)]
    b = kernel.index("} else if (lane == 0) {") + len("} else if (lane == 0) {")
    body = kernel[b:kernel.index("umma::fence_before_sync();\n  __syncthreads();\n  if (warp == 0) umma::dealloc")]
    body = body[:body.rindex("}")]
    text = (wait + body).replace("uint64_t* mb", "Barrier* mb").replace("#pragma unroll\n", "")
    (tmp_path / "issuer.inc").write_text(re.sub(r"\bstatic_assert\b", "// ", text))
    exe = tmp_path / "emu"
    res = subprocess.run([gxx, "-std=c++17", "-O1", "-I", str(tmp_path),
                          os.path.join(HERE, "host_emu", "umma_drain_emu.cpp"), "-o", str(exe)],
                         capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-4000:]
    res = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert res.returncode == 0, res.stdout
