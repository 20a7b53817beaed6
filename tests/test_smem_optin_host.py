"""A kernel's dynamic shared-memory limit belongs to the device it was raised on: csrc/optin.cuh,
built with g++ against a fake runtime, raises it once per kernel and device and reports a failure
on every call, and every kernel takes its limit from there and from nowhere else. A device symbol's
address belongs to its device too: the field's error flag is looked up for each."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1607_03252_gb300", "csrc")

FAKE = """#pragma once
#include <cstddef>
typedef int cudaError_t;
enum { cudaSuccess = 0, cudaFuncAttributeMaxDynamicSharedMemorySize = 8 };
cudaError_t cudaGetDevice(int* device);
cudaError_t fake_set_attribute(const void* f, int attr, int value);
template <class T>
cudaError_t cudaFuncSetAttribute(T* f, int attr, int value) { return fake_set_attribute((const void*)f, attr, value); }
"""


def test_limit_is_per_device_and_failures_are_reported(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    (tmp_path / "cuda_runtime.h").write_text(FAKE)
    exe = tmp_path / "emu"
    res = subprocess.run([gxx, "-std=c++17", "-O1", "-I", str(tmp_path), "-I", CSRC,
                          os.path.join(HERE, "host_emu", "optin_emu.cpp"), "-o", str(exe)],
                         capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-4000:]
    res = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert res.returncode == 0, res.stdout


@pytest.mark.parametrize("name", ["mg.cu", "field.cu", "smooth.cu"])
def test_no_kernel_raises_its_limit_once_per_process(name):
    text = open(os.path.join(CSRC, name)).read()
    assert "cudaFuncSetAttribute" not in text
    for found in re.finditer("cudaGetSymbolAddress", text):  # not in a static's initialiser
        assert "static int* const" not in text[max(0, found.start() - 160):found.start()]
