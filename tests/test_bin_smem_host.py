"""A plan is made for at most 200 KB of histogram and tables per CTA of the bin pass
(sums, one weight and one phase per l with a gap after every fourth, one pair of edges
per k bin, in the mesh precision); whatever it accepts, the kernels' shared memory fits
the 227 KB that a CTA can have, at every mesh size up to 4096.  From the library's own
sizes, without a GPU."""
import importlib
import os
import subprocess

import pytest

PROGRAM = r'''
#include <stdio.h>
#include "pk_internal.h"

static size_t up(size_t x) { return (x + 15) / 16 * 16; }

int main() {
    int bad = 0;
    for (int f64 = 0; f64 < 2; ++f64)
        for (int N = 4; N <= 4096; N += 2)
            for (int nmu = 0; nmu <= 100; nmu += 50) {
                pk::BinGeom g{};
                g.N = N, g.Nh = N / 2 + 1, g.nmu = nmu, g.poles = 1, g.twod = nmu > 0;
                const size_t R = f64 ? 8 : 4, tab = g.Nh + g.Nh / 4 + 1, per = nmu ? nmu : 1;
                // the largest number of k bins within the rule
                const auto rule = [&](size_t nk) { return up(up(up(up(nk * (per + 2) * R) + tab * R) + tab * 2 * R) + nk * 8); };
                size_t nk = 1;
                while (rule(nk + 1) <= 200 * 1024) ++nk;
                g.nk = (int)nk, g.nh = (int)(nk * (per + 2)), g.hbase = (int)(nk * per);
                const size_t got = pk::bin_smem_bytes(g, f64);
                if (got > 227 * 1024 && ++bad < 5) printf("N %d f64 %d nmu %d nk %zu: %zu bytes\n", N, f64, nmu, nk, got);
            }
    printf("%d too large\n", bad);
    return bad != 0;
}
'''


def test_every_accepted_histogram_fits(tmp_path):
    build = importlib.import_module("paper_1712_05834_gb300.build")
    if not os.path.exists(build._nvcc()):
        pytest.skip("no nvcc")
    lib = build.build()
    src, exe = tmp_path / "sizes.cu", tmp_path / "sizes"
    src.write_text(PROGRAM)
    subprocess.check_call([build._nvcc(), "-std=c++17", "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC, str(src),
                           "-o", str(exe), lib, "-Xlinker", "-rpath," + os.path.dirname(lib), "-L", build._cuda_lib_dir(),
                           "-lcufft"] + build.ARCH)
    out = subprocess.run([str(exe)], stdout=subprocess.PIPE, stderr=subprocess.STDOUT, timeout=60)
    assert out.returncode == 0, out.stdout.decode()
