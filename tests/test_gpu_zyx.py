"""The transform that takes z and y in one pass over device memory and then x
(FP32 meshes of 320^3 to 800^3, 1024^3 and 2048^3), against the cuFFT path on the
same painted meshes: every radix in use (16, 10, 8, 6, 5, 4), k bins up to
and beyond k_N (beyond: the l = N/2 column and rows past the binned sphere
are transformed too), one and two meshes, a batch, cross and projected power
(which read the transform itself), two computes in a row (the pass's work
counters start from zero again) and a captured graph.  Both are FP32
transforms with errors near 1e-7 of a bin's power: they agree within 1e-5 of
the bin's unsubtracted monopole; mode counts are bit-exact."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module")
def pk():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1712_05834_gb300 as pk
    pk.build()
    pk.load()
    return pk


def _close(got, ref, raw):
    assert np.array_equal(got["modes"], ref["modes"])
    ok = ref["modes"] > 0
    for name in ("power", "poles", "power2d"):
        if name in ref:
            lim = TOL * (raw if ref[name].ndim == 1 else raw[None, :] if name == "poles" else raw[:, None])
            d = np.abs(got[name] - ref[name])
            good = ok if ref[name].ndim == 1 else np.broadcast_to(ok if name == "poles" else ok[:, None], d.shape)
            good = good & np.isfinite(ref[name])
            assert np.array_equal(np.isfinite(got[name]), np.isfinite(ref[name])), name
            assert np.all(d[good] <= np.broadcast_to(lim, d.shape)[good]), name


@pytest.mark.parametrize("N,window,interlaced,nmu,beyond", [
    (320, "tsc", True, 5, True), (384, "cic", False, 0, False), (400, "pcs", True, 10, False),
    (480, "tsc", False, 4, True), (500, "cic", False, 0, False), (600, "tsc", False, 0, False),
    (640, "tsc", True, 0, False), (768, "cic", False, 5, False), (800, "cic", False, 0, True),
    (1024, "cic", True, 3, True)])
def test_agrees_with_cufft(pk, N, window, interlaced, nmu, beyond):
    import torch
    L, n = 1000.0, 300_000
    g = torch.Generator(device="cuda").manual_seed(N)
    a = torch.rand((n, 3), generator=g, device="cuda") * L
    pos = torch.cat([a, a[: n // 2] * 0.9]).contiguous()
    offsets = [0, n, n + n // 2] if N <= 500 else [0, n + n // 2]
    items = len(offsets) - 1
    kmax = 1.2 * math.pi * N / L if beyond else None
    cfg = pk.make_config(L, N, window, interlaced=interlaced, dk=0.02, nmu=nmu, kmax=kmax, batch=items,
                         capacity=n + n // 2)
    out = {}
    for own in (True, False):
        plan = pk.pk_plan(cfg)
        try:
            if not own:
                pk.pk_use_own_fft(plan, False)
            for _ in range(2):
                pk.pk_paint_many(plan, pos, offsets)
                pk.pk_compute(plan)
            res = [pk.pk_result(plan, k) for k in range(items)]
            out[own] = (res, pk.pk_cross(plan, 0, items - 1), pk.pk_projected(plan, items - 1, (0, 2)))
        finally:
            pk.pk_destroy(plan)
    raws = [r["power"] + r["shot_noise"] for r in out[False][0]]
    for got, ref, raw in zip(out[True][0], out[False][0], raws):
        _close(got, ref, raw)
    _close(out[True][1], out[False][1], np.sqrt(raws[0] * raws[-1]))
    p, q = out[True][2], out[False][2]
    assert np.array_equal(p["modes"], q["modes"])
    ok = q["modes"] > 0
    assert np.all(np.abs(p["power"] - q["power"])[ok] <= TOL * (np.abs(q["power"][ok]) + q["shot_noise"]))


def test_captured_graph_replays(pk):
    import torch
    L, N, n = 500.0, 320, 100_000
    g = torch.Generator(device="cuda").manual_seed(7)
    pos = torch.rand((n, 3), generator=g, device="cuda") * L
    cfg = pk.make_config(L, N, "tsc", interlaced=True, dk=0.05, capacity=n)
    s = torch.cuda.Stream()
    plan = pk.pk_plan(cfg, s)
    try:
        def step():
            pk.pk_paint(plan, pos)
            pk.pk_compute(plan)
        step()
        ref = pk.pk_result(plan)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s, capture_error_mode="thread_local"):
            step()
        for _ in range(3):
            graph.replay()
        torch.cuda.synchronize()
        got = pk.pk_result(plan)
        _close(got, ref, ref["power"] + ref["shot_noise"])
    finally:
        pk.pk_destroy(plan)


def test_selection_is_accepted_where_it_was(pk):
    plan = pk.pk_plan(pk.make_config(100.0, 400, "cic", dk=0.2))
    try:
        with pytest.raises(pk.PkError) as e:
            pk.pk_use_own_fft(plan, True)
        assert e.value.status == pk.PK_EINVAL
        pk.pk_use_own_fft(plan, False)
    finally:
        pk.pk_destroy(plan)
