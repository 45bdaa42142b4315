"""FP64 meshes: the own transform (every radix from 2 to 16, ragged column tiles,
the smallest size it takes, sizes it leaves to cuFFT) and the FP64 bin pass,
against NumPy on the painted mesh itself.  Both sides are FP64: the transforms
err by some 2e-15 of the rms amplitude (random positions: every bin's power is
near the shot noise) and a bin's sum over at most 1e5 modes by less than 1e-13
of its terms' magnitude, with Legendre factors up to 9: agreement within 1e-12 of
the bin's unsubtracted monopole; mode counts are exact."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 1e-12
ORDER = {"cic": 2, "tsc": 3, "pcs": 4}


@pytest.fixture(scope="module")
def pk():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1712_05834_gb300 as pk
    pk.build()
    pk.load()
    return pk


def _field(meshes, N, p):
    """Compensated transform (interlaced: of the mean of both meshes) of real meshes."""
    f = np.fft.rfftn(meshes[0])
    n1 = np.fft.fftfreq(N, 1.0 / N)
    nz = np.arange(N // 2 + 1)
    s = n1[:, None, None] + n1[None, :, None] + nz[None, None, :]
    if len(meshes) == 2:
        f = 0.5 * (f + np.fft.rfftn(meshes[1]) * np.exp(1j * math.pi * s / N))
    c1, cz = np.sinc(n1 / N) ** -p, np.sinc(nz / N) ** -p
    return f * c1[:, None, None] * c1[None, :, None] * cz[None, None, :]


def _check(got, fa, fb, N, L, nmu, wa, wb, shot):
    n1 = np.rint(np.fft.fftfreq(N, 1.0 / N)).astype(np.int64)
    nz = np.arange(N // 2 + 1)
    m = n1[:, None, None] ** 2 + n1[None, :, None] ** 2 + nz[None, None, :] ** 2
    mult = np.broadcast_to(np.where((nz == 0) | (nz == N // 2), 1, 2), m.shape)
    k = 2 * math.pi / L * np.sqrt(m)
    b = np.searchsorted(got["k_edges"], k, side="right") - 1
    nk = got["nk"]
    use = (b >= 0) & (b < nk) & (m > 0)
    b, m, mult = b[use], m[use], mult[use]
    P = L ** 3 / (wa * wb) * (fa * np.conj(fb)).real[use]
    lz = np.broadcast_to(nz, use.shape)[use]
    mu2 = lz ** 2 / m
    cnt = np.bincount(b, mult, nk)
    assert np.array_equal(cnt.astype(np.int64), got["modes"])
    ok = cnt > 0
    mean = lambda x: np.bincount(b, x * mult, nk)[ok] / cnt[ok]
    raw = mean(np.abs(P))
    assert np.all(np.abs(got["power"][ok] + shot - mean(P)) <= TOL * raw)
    for row, fac, leg in ((1, 5, 1.5 * mu2 - 0.5), (2, 9, (4.375 * mu2 - 3.75) * mu2 + 0.375)):
        assert np.all(np.abs(got["poles"][row][ok] - fac * mean(P * leg)) <= TOL * raw)
    if nmu:
        q = np.minimum(np.array([math.isqrt(nmu * nmu * int(l) ** 2 // int(mm)) for l, mm in zip(lz, m)]), nmu - 1)
        c2 = np.bincount(b * nmu + q, mult, nk * nmu)
        assert np.array_equal(c2.astype(np.int64).reshape(nk, nmu), got["modes2d"])
        p2 = np.bincount(b * nmu + q, P * mult, nk * nmu)
        a2 = np.bincount(b * nmu + q, np.abs(P) * mult, nk * nmu)
        o2 = c2 > 0
        assert np.all(np.abs(got["power2d"].reshape(-1)[o2] + shot - p2[o2] / c2[o2]) <= 3 * TOL * a2[o2] / c2[o2])


@pytest.mark.parametrize("N,window,interlaced,nmu,beyond", [
    (30, "cic", True, 3, True),        # below the smallest own transform
    (32, "tsc", True, 4, True), (34, "cic", False, 0, False),      # 17: cuFFT
    (50, "cic", False, 3, True), (56, "pcs", True, 0, False), (60, "cic", True, 0, True),
    (84, "tsc", False, 2, False), (96, "cic", True, 0, False), (128, "tsc", True, 0, True)])
def test_matches_numpy_on_the_painted_mesh(pk, N, window, interlaced, nmu, beyond):
    L, n = 700.0, 40_000
    r = np.random.default_rng(N)
    pos = np.concatenate([r.uniform(0, L, (n, 3)), r.uniform(0, L, (n // 2, 3))])
    w = np.concatenate([r.uniform(0.5, 1.5, n), r.uniform(0.5, 1.5, n // 2)]).astype(np.float32)
    dk = 1.7 * 2 * math.pi / L
    cfg = pk.make_config(L, N, window, interlaced=interlaced, dk=dk, nmu=nmu, precision="f64", batch=2,
                         kmax=1.3 * math.pi * N / L if beyond else None)
    plan = pk.pk_plan(cfg)
    try:
        pk.pk_paint_many(plan, pos, [0, n, n + n // 2], w)
        fields = [_field([pk.pk_mesh(plan, i, m, N, f64=True).astype(np.float64) for m in range(2 if interlaced else 1)],
                         N, ORDER[window]) for i in range(2)]
        pk.pk_compute(plan)
        res = [pk.pk_result(plan, i) for i in range(2)]
        cross = pk.pk_cross(plan, 0, 1)
    finally:
        pk.pk_destroy(plan)
    for f, got in zip(fields, res):
        _check(got, f, f, N, L, nmu, got["wsum"], got["wsum"], got["shot_noise"])
    _check(cross, fields[0], fields[1], N, L, nmu, res[0]["wsum"], res[1]["wsum"], 0.0)


def test_larger_sizes_and_selection(pk):
    """Own transform against cuFFT on the same meshes where a tile holds four columns
    (above 512) and at the workhorse size; switching off is accepted, on stays refused."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(5)
    L = 1000.0
    pos = torch.rand((200_000, 3), generator=g, device="cuda", dtype=torch.float64) * L
    for N in (256, 540):
        out = []
        for own in (True, False):
            plan = pk.pk_plan(pk.make_config(L, N, "cic", dk=0.03, precision="f64", capacity=len(pos)))
            try:
                if not own:
                    pk.pk_use_own_fft(plan, False)
                    with pytest.raises(pk.PkError):
                        pk.pk_use_own_fft(plan, True)
                for _ in range(2):
                    pk.pk_paint(plan, pos)
                    pk.pk_compute(plan)
                out.append(pk.pk_result(plan))
            finally:
                pk.pk_destroy(plan)
        a, b = out
        ok = b["modes"] > 0
        raw = (b["power"] + b["shot_noise"])[ok]
        assert np.array_equal(a["modes"], b["modes"])
        assert np.all(np.abs(a["power"] - b["power"])[ok] <= TOL * raw)
        assert np.all(np.abs(a["poles"] - b["poles"])[:, ok] <= 2 * TOL * raw)
