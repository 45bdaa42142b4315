"""Cross and projected power of 1024^3 read the transform that the compute has written (x
in place, then the bins: 4 launches) and take no axis again; spectra of repeated
passes agree to the FP32 sums' order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("what", ["cross", "projected"])
def test_the_x_axis_is_taken_once(what):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1712_05834_gb300 as pk
    pk.build()
    N, L, n = 1024, 1000.0, 200_000
    pos = (torch.rand((2 * n, 3), generator=torch.Generator().manual_seed(1)) * L).cuda()
    plan = pk.pk_plan(pk.make_config(L, N, "tsc", dk=0.05, batch=2, capacity=2 * n))
    try:
        counts, auto, other = [], [], []
        for _ in range(3):
            pk.pk_paint_many(plan, pos, [0, n, 2 * n])
            a = pk.pk_launch_count(plan)
            pk.pk_compute(plan)
            b = pk.pk_launch_count(plan)
            auto.append([pk.pk_result(plan, k)["power"] for k in range(2)])
            r = pk.pk_cross(plan, 0, 1) if what == "cross" else pk.pk_projected(plan, 1, (0, 1))
            other.append(r["power"])
            counts.append((b - a, pk.pk_launch_count(plan) - b))
    finally:
        pk.pk_destroy(plan)
    assert counts[0] == counts[1] == counts[2] and counts[0][0] == 4, counts
    shot = L ** 3 / n
    for k in (1, 2):
        for x, y in zip(auto[0], auto[k]):
            ok = np.isfinite(x)
            assert np.all(np.abs(x - y)[ok] <= 1e-5 * (np.abs(x[ok]) + shot))
        ok = np.isfinite(other[0])
        scale = np.abs(other[0][ok]).max() + (shot if what == "cross" else 0.0)
        assert np.all(np.abs(other[0] - other[k])[ok] <= 1e-5 * scale)
