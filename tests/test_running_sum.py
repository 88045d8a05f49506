"""A thread's FP32 running sum (csrc/running_sum.h) keeps its accuracy over any number of values, compiled for the
host (CPU only).  Bound: two-sum makes each step's rounding error exact, and adding n of them rounds by n 2^-24 of
their sum, itself at most n 2^-24 of the sum of absolute values: n^2 2^-48 of it.  Plain FP32 sums are off by n 2^-24."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1708_03621_gb300", "csrc")

SOURCE = r"""
#include "running_sum.h"
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <initializer_list>
int main() {
    uint64_t x = 88172645463325252ull;
    for (int n : {1, 2, 7, 18, 64, 300}) {
        for (int sign = 0; sign < 2; ++sign) {
            for (int t = 0; t < 200; ++t) {
                jdft::RunningSum<float> s;
                long double exact = 0, abs = 0;
                for (int i = 0; i < n; ++i) {
                    x ^= x << 13; x ^= x >> 7; x ^= x << 17;
                    float a = (float)((double)(x >> 40) * std::exp2(-(double)(x & 31)) + 1e-3);
                    if (sign && (x & 64)) a = -a;
                    s.add(a);
                    exact += a;
                    abs += std::fabs(a);
                }
                const long double bound = (long double)n * n * 0x1p-48L * abs;
                if (std::fabs((long double)s.total() - exact) > bound) { std::printf("%d\n", n); return 1; }
            }
        }
    }
    jdft::RunningSum<float> s;
    s.add(1.f);
    for (int i = 0; i < 17; ++i) s.add(0x1p-25f);
    return s.total() == 1.0 + 17 * 0x1p-25 ? 0 : 2;
}
"""


def test_sum_of_many_values(tmp_path):
    cxx = shutil.which("g++") or pytest.skip("no g++")
    src = tmp_path / "t.cpp"
    src.write_text(SOURCE)
    exe = str(tmp_path / "t")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0


def test_dielectric_sums_use_it():
    """The sums of the conjugate-gradient passes (FP32 among them) are running sums."""
    update = open(os.path.join(CSRC, "field.cu")).read()
    update = update[update.index("pcm_update_kernel("):]
    update = update[:update.index("finish_sum")]
    div = open(os.path.join(CSRC, "field_fast_impl.cuh")).read()
    div = div[div.index("    div_kernel("):]
    div = div[:div.index("finish_sum")]
    assert update.count("RunningSum<T>") == 1 and update.count(".add(") == 2
    assert div.count("RunningSum<T>") == 1 and div.count(".add(") == 1
