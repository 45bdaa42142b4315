"""The variance of a log-normal draw's field: a thread's sum of squares, held in FP32
numbers, is off by no more than a sum in FP64 (and the last place of its value), for few
and many squares (a draw of 2048^3 cells takes 14000 a thread).  Exact sums: multiples of 2^-20 squared are integers."""
import importlib
import os
import subprocess

import pytest

PROGRAM = r'''
#include <math.h>
#include <stdio.h>
#include "pk_sums.h"

int main() {
    unsigned s = 7u;
    const auto rnd = [&]() { s = s * 1664525u + 1013904223u; return (int)(s >> 8); };       // 24 bits
    int bad = 0;
    for (int n : {1, 2, 6, 52, 430, 8192, 20000}) {
        double worst = 0.0, worst64 = 0.0;
        for (int rep = 0; rep < 50; ++rep) {
            pk::SquareSum q;
            double q64 = 0.0;
            unsigned __int128 exact = 0;
            for (int i = 0; i < n; ++i) {
                const int k = (rnd() + rnd() + rnd() + rnd() - 2 * 16777216) / 8;               // |k| < 2^23
                const float x = (float)k * 9.5367431640625e-07f;
                q.add(x);
                q64 += (double)x * (double)x;
                exact += (unsigned long long)((long long)k * k);
            }
            // differences in units of 2^-40, exactly, by taking the value apart
            const auto off = [&](double value) {
                const double v = value * 1099511627776.0;
                const __int128 whole = (__int128)v;
                return fabs((double)(whole - (__int128)exact) + (v - (double)whole)) / (double)exact;
            };
            worst = fmax(worst, off(q.value()));
            worst64 = fmax(worst64, off(q64));
        }
        printf("%d squares: %.2e, FP64 %.2e\n", n, worst, worst64);
        bad += !(worst <= worst64 + 2.3e-16);
    }
    return bad != 0;
}
'''


def test_square_sums(tmp_path):
    build = importlib.import_module("paper_1712_05834_gb300.build")
    if not os.path.exists(build._nvcc()):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "squares.cu", tmp_path / "squares"
    src.write_text(PROGRAM)
    subprocess.check_call([build._nvcc(), "-O2", "-std=c++17", "-Xcompiler", "-ffp-contract=off", "-I", build.CSRC, str(src),
                           "-o", str(exe)] + build.ARCH)
    out = subprocess.run([str(exe)], stdout=subprocess.PIPE, stderr=subprocess.STDOUT, timeout=120)
    assert out.returncode == 0, out.stdout.decode()
