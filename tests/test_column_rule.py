"""The rule that chooses the few-column contractions, on the CPU: the fewest columns per
block that leave no SM with two blocks, and never a width at which the 128-column tiles are
the faster form for the order (32 up to N = 32, 64 up to N = 64)."""
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
    int N, K, R;
    while (scanf("%%d %%d %%d", &N, &K, &R) == 3) printf("%%d\\n", fpsa::col_tile(N, K, R, 152));
}
"""
# (N, cells, right-hand sides) -> columns per block on 152 SMs: 16 x 152 / 2 = 1216 cells, 2432, 4864
CASES = [((16, 9, 1), 16), ((16, 1216, 1), 16), ((16, 1217, 1), 0), ((16, 4864, 1), 0), ((32, 1217, 1), 0),
         ((32, 400, 3), 16), ((32, 401, 3), 0), ((48, 2432, 1), 32), ((64, 1216, 1), 16), ((64, 1217, 1), 32),
         ((64, 2432, 1), 32), ((64, 2433, 1), 0), ((80, 2433, 1), 64), ((128, 2432, 1), 32), ((128, 4864, 1), 64),
         ((128, 4865, 1), 0), ((128, 1, 152), 16), ((128, 1, 153), 0), ((128, 1 << 30, 1), 0)]


def test_col_tile(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers are missing")
    src, exe = tmp_path / "rule.cpp", str(tmp_path / "rule")
    src.write_text(MAIN % ROOT)
    subprocess.run([gxx, "-std=c++17", "-I" + CUDA_INC, str(src), "-o", exe], check=True)
    r = subprocess.run([exe], input="\n".join("%d %d %d" % c for c, _ in CASES), capture_output=True, text=True, check=True)
    assert [int(x) for x in r.stdout.split()] == [want for _, want in CASES]
