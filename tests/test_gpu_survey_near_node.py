"""An observer on a mesh node whose FP32 coordinate there rounds to a few 1e-10 of the box
edge instead of 0 (600 cells of 1100 / 600, the observer three cells from the corner): the
weights Y_lm there stay finite, and the FP32 form's multipoles agree with the FP64
form's to 1e-4 of the monopole before shot noise, as elsewhere.  1300 / 768 likewise."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,L,node,interlaced", [(600, 1100.0, 3, False), (600, 1100.0, 5, True), (768, 1300.0, 3, False)])
def test_multipoles_are_finite(N, L, node, interlaced):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1712_05834_gb300 as pk
    pk.build()
    H, o = np.float32(L / N), np.float32(-node * L / N)
    x = float(np.float64(node) * np.float64(H) + np.float64(o)) / 1024.0       # exact: the node's FP32 coordinate
    assert 0.0 < abs(x) < 1.4e-10, x                                            # the case is what it is meant to be
    g = torch.Generator().manual_seed(N + node)
    dev = lambda n: (200.0 + 0.6 * L * torch.rand((n, 3), generator=g)).cuda()
    data = pk.survey_catalog(dev(40_000), nbar=torch.full((40_000,), 1e-4, device="cuda"))
    rand = pk.survey_catalog(dev(120_000), nbar=torch.full((120_000,), 1e-4, device="cuda"))
    out = []
    for precision in ("f32", "f64"):
        cfg = pk.make_survey_config(L, (-node * L / N,) * 3, N, "tsc", interlaced, dk=0.02, precision=precision)
        with pk.ConvolvedFFTPower(cfg) as power:
            out.append(power.run(data, rand))
    got, ref = out
    ok = ref["modes"] > 0
    assert np.all(np.isfinite(got["poles"][:, ok]))
    raw = np.abs(ref["poles"][0][ok] + ref["shot_noise"])
    for row in range(3):
        err = np.abs(got["poles"][row] - ref["poles"][row])[ok]
        assert np.all(err <= 1e-4 * raw), (row, float(np.max(err / raw)))


def test_observer_very_far_away():
    """2e10 box edges along z, as a program that wants the plane-parallel limit may ask
    for: fourth powers of the distance would leave the FP32 range in units of the box."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1712_05834_gb300 as pk
    pk.build()
    N, L, far = 128, 1000.0, 2.0 ** 44
    g = torch.Generator().manual_seed(3)
    dev = lambda n: (L * torch.rand((n, 3), generator=g, dtype=torch.float64) +
                     torch.tensor([-500.0, -500.0, far], dtype=torch.float64)).cuda()
    data = pk.survey_catalog(dev(40_000), nbar=torch.full((40_000,), 1e-4, device="cuda"))
    rand = pk.survey_catalog(dev(120_000), nbar=torch.full((120_000,), 1e-4, device="cuda"))
    out = []
    for precision in ("f32", "f64"):
        cfg = pk.make_survey_config(L, (-500.0, -500.0, far), N, "tsc", False, dk=0.02, precision=precision)
        with pk.ConvolvedFFTPower(cfg) as power:
            out.append(power.run(data, rand))
    got, ref = out
    ok = ref["modes"] > 0
    raw = np.abs(ref["poles"][0][ok] + ref["shot_noise"])
    for row in range(3):
        err = np.abs(got["poles"][row] - ref["poles"][row])[ok]
        assert np.all(err <= 1e-4 * raw), (row, float(np.max(err / raw)))
