"""Survey multipoles on the library's own transforms (FP32 meshes of the sizes
they exist for): the rows F Y_lm(x^) formed on the way into the z axis, every
batch size and pole set, interlaced and not, an observer on a mesh node, and
k bins beyond k_N.  Reference: the FP64 mesh form (cuFFT and the weighting
kernel), which the oracle pins to 1e-6; the FP32 form is held to 1e-4 of the
bin's monopole before shot noise, as against the oracle, and repeats with the
kept randoms give the same within the FP32 partial sums' order."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 1e-4


@pytest.mark.parametrize("N,window,interlaced,max_batch,poles,beyond", [
    (128, "tsc", True, 0, (0, 2, 4), False), (128, "cic", False, 0, (0, 2, 4), True),
    (192, "pcs", True, 4, (0, 2, 4), False), (256, "cic", False, 3, (0, 4), False),
    (320, "tsc", False, 0, (0, 2), False), (384, "cic", True, 0, (0, 2, 4), True),
    (400, "cic", False, 5, (0, 2, 4), False), (192, "cic", True, 0, (0,), False), (128, "cic", False, 0, (0,), False)])
def test_agrees_with_the_fp64_form(N, window, interlaced, max_batch, poles, beyond):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1712_05834_gb300 as pk
    import synth
    pk.build()
    c = synth.survey_catalogs(30000, 90000, 400.0, synth.seed_for(9, N), ngrid=64)
    L = 1000.0 if N != 128 else 1024.0
    origin = (-300.0, -L / 2, -L / 4)
    if N == 128:
        origin = (-L / 2, -L / 2, -L / 2)          # the observer sits on node (64, 64, 64)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()
    d, r = dev(c["data"]), dev(c["randoms"])
    data = pk.survey_catalog(d, wcomp=dev(c["data_wcomp"]), nbar=dev(c["data_nbar"]))
    rand = pk.survey_catalog(r, nbar=dev(c["rand_nbar"]))
    kmax = 1.15 * math.pi * N / L if beyond else None
    out = {}
    for precision in ("f32", "f64"):
        cfg = pk.make_survey_config(L, origin, N, window, interlaced, dk=0.02, kmax=kmax, poles=poles,
                                    precision=precision, max_batch=max_batch)
        with pk.ConvolvedFFTPower(cfg) as power:
            out[precision] = [power.run(data, rand)]
            if precision == "f32":
                out[precision].append(power.run(data, None))
    ref = out["f64"][0]
    ok = ref["modes"] > 0
    raw = np.abs(ref["poles"][0][ok] + ref["shot_noise"])
    for got in out["f32"]:
        assert np.array_equal(got["modes"], ref["modes"])
        for row, ell in enumerate((0, 2, 4)):
            if ell not in poles:
                assert np.all(np.isnan(got["poles"][row]))
                continue
            err = np.abs(got["poles"][row] - ref["poles"][row])[ok]
            assert np.all(err <= TOL * raw), (ell, float(np.max(err / raw)))
