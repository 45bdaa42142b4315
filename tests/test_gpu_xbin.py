"""The bins of 1024^3 and 2048^3 in the forms that the other tests do not reach: 2048^3
with one mesh, with and without mu bins, and mu bins whose exact rule needs 64-bit
products.  A compute takes z / y, x, bins and results: 4 launches.

A painted delta (weight 1 on node 0, CIC, one mesh, uncompensated) makes every step of
the transform exact in FP32 and every mode's power L^3, so that P(k) and P(k, mu) equal
L^3 to the bit if every mode is in its bin.  Two meshes: against cuFFT on the same
painted meshes, within 1e-5 of the bin's monopole before shot noise.  A displaced lattice,
whose modes differ in power by orders of magnitude: the error of the multipoles against
the FP64 form is at most 1.5 times that of the cuFFT path, which bins the same meshes."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pk():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1712_05834_gb300 as pk
    pk.build()
    pk.load()
    return pk


def _compute(pk, plan):
    before = pk.pk_launch_count(plan)
    pk.pk_compute(plan)
    return pk.pk_launch_count(plan) - before


@pytest.mark.parametrize("N,dk_kf,nmu,launches", [
    (1024, 1.9, 0, 4), (2048, 1.4, 0, 4), (2048, 2.6, 10, 4), (2048, 7.0, 64, 4), (2048, 2.3, 64, 4)])
def test_a_delta_fills_every_bin(pk, N, dk_kf, nmu, launches):
    L = 512.0
    plan = pk.pk_plan(pk.make_config(L, N, "cic", interlaced=False, compensated=False, dk=dk_kf * 2.0 * math.pi / L,
                                     nmu=nmu, subtract_shot=False))
    try:
        pk.pk_paint(plan, np.zeros((1, 3), np.float32))
        assert _compute(pk, plan) == launches
        r = pk.pk_result(plan, 0)
    finally:
        pk.pk_destroy(plan)
    ok = r["modes"] > 0
    assert np.count_nonzero(ok) > 3
    assert np.all(r["power"][ok] == L ** 3)
    if nmu:
        ok2 = r["modes2d"] > 0
        assert np.all(r["power2d"][ok2] == L ** 3)
        assert np.array_equal(r["modes2d"].sum(axis=1), r["modes"])


@pytest.mark.parametrize("nmu,dk_kf,launches", [(64, 7.0, 4), (64, 2.3, 4)])
def test_two_meshes_of_2048_against_cufft(pk, nmu, dk_kf, launches):
    import torch
    N, L, n = 2048, 1000.0, 2_000_000
    pos = (torch.rand((n, 3), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda") ** 1.2 * L).contiguous()
    cfg = pk.make_config(L, N, "cic", interlaced=True, dk=dk_kf * 2.0 * math.pi / L, nmu=nmu, capacity=n)
    out = []
    torch.cuda.empty_cache()
    for own in (True, False):
        plan = pk.pk_plan(cfg)
        try:
            if not own:
                pk.pk_use_own_fft(plan, False)
            pk.pk_paint(plan, pos)
            count = _compute(pk, plan)
            assert not own or count == launches
            out.append(pk.pk_result(plan, 0))
        finally:
            pk.pk_destroy(plan)
    got, ref = out
    assert np.array_equal(got["modes2d"], ref["modes2d"])
    raw = ref["power"] + ref["shot_noise"]
    ok, ok2 = ref["modes"] > 0, ref["modes2d"] > 0
    assert np.all(np.abs(got["power"] - ref["power"])[ok] <= 1e-5 * raw[ok])
    assert np.all(np.abs(got["poles"] - ref["poles"])[:, ok] <= 1e-5 * raw[ok])
    assert np.all(np.abs(got["power2d"] - ref["power2d"])[ok2] <= 1e-5 * np.broadcast_to(raw[:, None], ok2.shape)[ok2])


def test_sums_are_as_exact_as_on_the_cufft_path(pk):
    import synth
    import torch
    n1, L, N = 512, 1000.0, 1024
    pos = synth.zeldovich_lattice(n1, L, synth.seed_for(3), device="cuda")
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    out = {}
    for form in ("f64", "own", "cufft"):
        plan = pk.pk_plan(pk.make_config(L, N, "pcs", interlaced=True, dk=0.005, nmu=10,
                                         precision="f64" if form == "f64" else "f32"))
        try:
            if form == "cufft":
                pk.pk_use_own_fft(plan, False)
            pk.pk_paint(plan, pos)
            pk.pk_compute(plan)
            out[form] = pk.pk_result(plan, 0)
        finally:
            pk.pk_destroy(plan)
            torch.cuda.empty_cache()
    ref = out["f64"]
    ok = ref["modes"] > 0
    raw = (ref["power"] + (L / n1) ** 3)[ok]
    rms = {f: [float(np.sqrt(np.mean(((out[f]["poles"][e] - ref["poles"][e])[ok] / raw) ** 2))) for e in range(3)]
           for f in ("own", "cufft")}
    for a, b in zip(rms["own"], rms["cufft"]):
        assert a <= 1.5 * b, rms
