"""The library's own constants for the exact division of cell indices (magic_div of pic_internal.cuh, compiled here for
the host): every quotient and remainder at the edges of the multiples of n, up to 2^31 - 1, and the two successive
divisions of a 3D cell index by nx and ny, against the integer division."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include "pic_internal.cuh"
#include <cstdio>
#include <random>
using gbpic::magic_div;
static unsigned quotient(unsigned v, unsigned m, int s) { return (unsigned)(((unsigned long long)v * m) >> 32) >> s; }
static long long bad = 0, checked = 0;
static void one(unsigned v, int n, unsigned m, int s)
{
    checked++;
    if (quotient(v, m, s) != v / (unsigned)n) bad++;
}
int main()
{
    std::mt19937 rng(11);
    const unsigned top = 2147483647u;
    for (int n = 3; n < 32768; n += n < 600 ? 1 : 1 + (int)(rng() % 97)) {
        unsigned m;
        int s;
        magic_div(n, m, s);
        for (int t = 0; t < 400; t++) {
            const unsigned q = t < 40 ? (unsigned)t : (t < 80 ? top / n - (unsigned)(t - 40) : rng() % (top / n + 1));
            for (int d = -1; d <= 1; d++) {
                const long long v = (long long)q * n + d;
                if (v >= 0 && v <= (long long)top) one((unsigned)v, n, m, s);
            }
        }
        one(top, n, m, s);
        // 3D: the quotient by nx = n is divided by ny
        const int ny = 3 + (int)(rng() % 32765);
        unsigned my;
        int sy;
        magic_div(ny, my, sy);
        for (int t = 0; t < 200; t++) {
            const unsigned cell = t < 20 ? top - (unsigned)t : rng() % top, q = quotient(cell, m, s), k = quotient(q, my, sy);
            checked++;
            if (q != cell / (unsigned)n || k != cell / (unsigned)n / (unsigned)ny) bad++;
        }
    }
    std::printf("%lld %lld\n", checked, bad);
    return bad != 0;
}
"""


def test_header_constants_divide_exactly(tmp_path):
    cxx = shutil.which("g++")
    cuda = os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))
    if not cxx or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "split.cpp", tmp_path / "split"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", os.path.join(cuda, "include"), "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_1502_07722_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    checked, bad = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert int(checked) > 1_000_000 and int(bad) == 0
