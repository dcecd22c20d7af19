"""The arithmetic of the fixed-point recurrences (csrc/fx_site.h) compiled for the host: what the kernel with two
lanes a site (six numbers a lane and spin) and the one with eight (three numbers a lane) do to the same site.
"""
import os
import subprocess

import pytest

from paper_1111_6288_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include <random>
#include "fx_site.h"
using namespace ovl::fx;
int main() {
    std::mt19937_64 rng(1);
    int wrong = 0;
    for (int t = 0; t < 20000; ++t) {
        i64 m[24];
        const int top = (int)(rng() % 62);  // bits of the largest number; 0: only 0 and -1
        for (i64& v : m) v = (i64)(top ? rng() >> (64 - top) : 0) * (rng() & 1 ? 1 : -1) - (i64)(rng() & 1);
        uint64_t o = 0;
        for (i64 v : m) o |= (uint64_t)(v ^ (v >> 63));
        int e6 = 0;
        i64 six[24];
        for (int lane = 0; lane < 2; ++lane) {
            i64 a[6], b[6];
            for (int k = 0; k < 6; ++k) a[k] = m[12 * lane + k], b[k] = m[12 * lane + 6 + k];
            e6 = normalise(a, b, o, -7);
            for (int k = 0; k < 6; ++k) six[12 * lane + k] = a[k], six[12 * lane + 6 + k] = b[k];
        }
        for (int lane = 0; lane < 8; ++lane) {
            i64 a[3] = {m[3 * lane], m[3 * lane + 1], m[3 * lane + 2]};
            const int e3 = normalise(a, o, -7);
            for (int k = 0; k < 3; ++k) wrong += a[k] != six[3 * lane + k] || e3 != e6;
        }
    }
    std::printf("%d\n", wrong);
}
"""


def test_both_normalisations_agree(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("no CUDA toolkit")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", build.CSRC, "-I", cuda, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout == "0\n"
