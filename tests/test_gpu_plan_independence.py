"""A catalog's painted cells depend on the catalog, the mesh and the window alone: a
plan that reserves its size, one that reserves nothing and grows, and a batch that
holds other catalogs beside it paint the same bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("N,window,interlaced", [(64, "cic", False), (64, "pcs", True), (48, "tsc", True), (24, "tsc", False),
                                                 (72, "tsc", False)])
def test_cells_do_not_depend_on_the_plan(N, window, interlaced, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1712_05834_gb300 as pk
    pk.build()
    n, L = 100_003, 100.0
    g = torch.Generator().manual_seed(N)
    pos = (torch.rand((n, 3), generator=g) * L).cuda()
    both = torch.cat([pos, (torch.rand((n, 3), generator=g) * L).cuda()])
    got = []
    for batch, capacity in ((1, n), (1, 0), (2, 0), (2, 2 * n), (2, 40 * n)):
        plan = pk.pk_plan(pk.make_config(L, N, window, interlaced=interlaced, dk=0.2, precision=precision, batch=batch,
                                         capacity=capacity))
        try:
            if batch == 1:
                pk.pk_paint(plan, pos)
            else:
                pk.pk_paint_many(plan, both, [0, n, 2 * n])
            got.append([pk.pk_mesh(plan, 0, m, N, f64=precision == "f64") for m in range(2 if interlaced else 1)])
        finally:
            pk.pk_destroy(plan)
    for k, other in enumerate(got[1:]):
        for a, b in zip(got[0], other):
            assert np.array_equal(a, b), (k, int((a != b).sum()))
