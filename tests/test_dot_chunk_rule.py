"""The rule for the chunks of the GMRES vector kernels, on the CPU: small ones only where they
are few, and fewer in FP32 than in FP64."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"
MAIN = """
#include <cstdio>
#include "%s/paper_1907_13013_gb300/csrc/fpsa_internal.h"
int main() {
    long long n;
    int fp64;
    while (scanf("%%lld %%d", &n, &fp64) == 2) printf("%%d\\n", (int)fpsa::small_dot_chunks(n, fp64 != 0, 152));
}
"""
CASES = [((7, 1), 1), ((125, 0), 1), ((304, 0), 1), ((305, 0), 0), ((600, 0), 0), ((600, 1), 1), ((912, 1), 1),
         ((913, 1), 0), ((1125, 0), 0), ((1125, 1), 0), ((10 ** 12, 1), 0)]


def test_small_dot_chunks(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers are missing")
    src, exe = tmp_path / "rule.cpp", str(tmp_path / "rule")
    src.write_text(MAIN % ROOT)
    subprocess.run([gxx, "-std=c++17", "-I" + CUDA_INC, str(src), "-o", exe], check=True)
    r = subprocess.run([exe], input="\n".join("%d %d" % c for c, _ in CASES), capture_output=True, text=True, check=True)
    assert [int(x) for x in r.stdout.split()] == [want for _, want in CASES]
