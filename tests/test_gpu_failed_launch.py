"""A compute whose x axis pass could not be launched returns an error, and the next one
is right again: the work counters of the z / y pass before it do not stay behind.  The
failure is an error code from a stand-in for the x pass's launcher (nothing is launched),
put into the plan by a small program linked against the library."""
import importlib
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = r'''
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <vector>
#include "pk.h"
#include "pk_plan.h"

struct Refusing final : pk::ZyxOps {
    const pk::ZyxOps *real;
    mutable int refuse = 1;
    cudaError_t no() const { refuse = 0; return cudaErrorInvalidConfiguration; }
    bool plan_default() const override { return real->plan_default(); }
    int tile_columns() const override { return real->tile_columns(); }
    cudaError_t zy_survey(void *m, int nx, const pk::SurveyRows &sv, int nc, int mc, const void *tw, unsigned *s, int *e,
                          int nsm, cudaStream_t st) const override {
        return real->zy_survey(m, nx, sv, nc, mc, tw, s, e, nsm, st);
    }
    cudaError_t zy(void *m, int p, int nc, int mc, const void *tw, unsigned *s, int *e, int nsm,
                   cudaStream_t st) const override {
        return real->zy(m, p, nc, mc, tw, s, e, nsm, st);
    }
    cudaError_t x(void *m, int n, long long mc, int nc, int mcut, const int *t, int nt, const void *tw, unsigned *s, int ns,
                  cudaStream_t st) const override {
        return refuse ? no() : real->x(m, n, mc, nc, mcut, t, nt, tw, s, ns, st);
    }
};

#define CHECK(e) do { const int r_ = (int)(e); if (r_) { printf("line %d: %d\n", __LINE__, r_); return 1; } } while (0)

int main(int argc, char **argv) {
    pk_config cfg;
    pk_config_default(&cfg);
    cfg.box_size = 100.0;
    cfg.nmesh = atoi(argv[1]);
    cfg.dk = 0.5;
    const int n = 50000;
    std::vector<float> pos(3 * n);
    unsigned s = 12345u;
    for (float &x : pos) { s = s * 1664525u + 1013904223u; x = (float)(s >> 8) * (100.0f / 16777216.0f); }
    pk_plan_t P = nullptr;
    CHECK(pk_plan(&cfg, nullptr, &P));
    std::vector<double> first;
    Refusing fake;
    for (int turn = 0; turn < 4; ++turn) {
        CHECK(pk_paint(P, pos.data(), PK_F32, nullptr, n, 0));
        if (turn == 1) { fake.real = P->zyx; P->zyx = &fake; }
        const pk_status got = pk_compute(P);
        if (turn == 1) {
            if (got == PK_OK) { printf("the refused launch was not reported\n"); return 1; }
            continue;
        }
        CHECK(got);
        pk_result_view v;
        CHECK(pk_result(P, 0, &v));
        if (turn == 0) first.assign(v.pk, v.pk + v.nk);
        for (int b = 0; b < v.nk; ++b)
            if (!(fabs(v.pk[b] - first[b]) <= 1e-5 * (fabs(first[b]) + v.shot_noise))) {
                printf("turn %d bin %d: %g, first %g\n", turn, b, v.pk[b], first[b]);
                return 1;
            }
    }
    P->zyx = fake.real;
    CHECK(pk_destroy(P));
    printf("ok\n");
    return 0;
}
'''


@pytest.mark.parametrize("N", [320, 1024])
def test_compute_after_a_refused_launch(N, tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    build = importlib.import_module("paper_1712_05834_gb300.build")
    lib = build.build()
    src, exe = tmp_path / "refused.cu", tmp_path / "refused"
    src.write_text(PROGRAM)
    subprocess.check_call([build._nvcc(), "-std=c++17", "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC, str(src),
                           "-o", str(exe), lib, "-Xlinker", "-rpath," + os.path.dirname(lib), "-L", build._cuda_lib_dir(),
                           "-lcufft"] + build.ARCH)
    out = subprocess.run([str(exe), str(N)], stdout=subprocess.PIPE, stderr=subprocess.STDOUT, timeout=120)
    assert out.returncode == 0 and b"ok" in out.stdout, out.stdout.decode()
