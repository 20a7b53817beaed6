"""Precision of the Fourier field's two FP64-free steps, from the kernels' own text built with g++.

The complex product of two phasors in double-float is no further from the exact product than the
double-float products and sums it stands for, each renormalised. The last entry of a phasor row (the
faces x, y, z = 1 of the grid, from 9^3 on) is its own sine and cosine: within 2^-52 of each (a library
sincos below one ulp) and, split into two FP32 numbers, within 2^-50 more."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1607_03252_gb300", "csrc")


def _cut(text, start, end):
    a = text.index(start)
    return text[a:text.index(end, a)]


@pytest.fixture(scope="module")
def emu(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    read = lambda name: open(os.path.join(CSRC, name)).read()  # noqa: E731
    text = "\n".join([
        _cut(read("philox.cuh"), "__device__ __forceinline__ void philox10(", "}  // namespace mlmc"),
        _cut(read("widen.cuh"), "__device__ __forceinline__ double widen(float f) {", "}  // namespace mlmc"),
        _cut(read("field.cu"), "__device__ __forceinline__ double u53(", "constexpr int kFieldThreads = 256;")])
    for a, b in (("__host__ __device__ __forceinline__", "static inline"),
                 ("__device__ __forceinline__", "static inline"), ("__device__", "static"), ("__global__", "static"),
                 ("__restrict__", "")):
        text = text.replace(a, b)
    d = tmp_path_factory.mktemp("precision")
    (d / "kernels.inc").write_text(text)
    exe = d / "emu"
    res = subprocess.run([gxx, "-std=c++17", "-O2", "-ffp-contract=off", "-Wno-unknown-pragmas", "-I", str(d), "-I", CSRC,
                          os.path.join(HERE, "host_emu", "field_precision_emu.cpp"), "-o", str(exe)],
                         capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-4000:]
    return str(exe)


def _run(emu, *args):
    res = subprocess.run([emu, *map(str, args)], capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stdout + res.stderr
    return [float(v) for v in res.stdout.split()]


def test_complex_product_is_as_exact_as_its_double_float_steps(emu):
    rms, top, rms_steps, top_steps = _run(emu, "cmul")
    assert rms <= rms_steps and top <= top_steps


@pytest.mark.parametrize("n", [9, 17, 33, 65, 257])
def test_last_phasor_of_a_row_is_its_own_sine_and_cosine(emu, n):
    last, split = _run(emu, "phasors", n, 60, 3)
    assert last <= 2.0 ** -52
    assert split <= 2.0 ** -52 + 2.0 ** -50
