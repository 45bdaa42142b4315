"""The mean power that the FP32 transforms give a field of white noise: a gain that is off
by 1e-7 is 1e-5 of a uniform catalog's P(k) once the shot noise is subtracted.  Against the
exact transform (FP64, torch) of the same painted mesh, the own transform's gain is off by
no more than cuFFT's (the other choice of a plan) and 4e-8: a rounding of FP32 is 6e-8,
and the constants and twiddles of some twenty steps average to a few 1e-8."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [320, 384, 400, 480, 500, 600, 640, 768, 800])
def test_gain_of_the_own_transform(N):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1712_05834_gb300 as pk
    pk.build()
    L, n = 1000.0, 3_000_000
    pos = torch.rand((n, 3), generator=torch.Generator(device="cuda").manual_seed(N), device="cuda") * L
    cfg = pk.make_config(L, N, "tsc", compensated=False, dk=math.pi * N / L / 20.5, poles=(0,), subtract_shot=False, capacity=n)
    gain, mesh = {}, None
    for own in (True, False):
        plan = pk.pk_plan(cfg)
        try:
            if not own:
                pk.pk_use_own_fft(plan, False)
            pk.pk_paint(plan, pos)
            if mesh is None:
                mesh = torch.from_numpy(pk.pk_mesh(plan, 0, 0, N)).cuda()
            pk.pk_compute(plan)
            r = pk.pk_result(plan, 0)
        finally:
            pk.pk_destroy(plan)
        gain[own] = float((r["power"] * r["modes"]).sum()) * (n / L ** 1.5) ** 2
    f = torch.fft.rfftn(mesh.double())
    i = torch.fft.fftfreq(N, d=1.0 / N, device="cuda", dtype=torch.float64) ** 2
    l = torch.arange(N // 2 + 1, device="cuda", dtype=torch.float64)
    h = torch.full_like(l, 2.0)
    h[0] = h[-1] = 1.0
    edge = (float(r["k_edges"][-1]) * L / (2.0 * math.pi)) ** 2
    exact, modes = 0.0, 0.0
    for x in range(N):
        m = i[x] + i[:, None] + l[None, :] ** 2
        w = h[None, :] * ((m > 0.0) & (m < edge))
        exact += float((w * (f[x].real ** 2 + f[x].imag ** 2)).sum())
        modes += float(w.sum())
    assert modes == r["modes"].sum()
    off = {own: gain[own] / exact - 1.0 for own in gain}
    assert abs(off[True]) <= abs(off[False]) + 4e-8, off
