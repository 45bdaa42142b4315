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


@pytest.mark.parametrize("kind", ["unit", "weighted", "heavy"])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("window,interlaced", [("cic", False), ("cic", True), ("tsc", False), ("tsc", True), ("pcs", False),
                                               ("pcs", True)])
@pytest.mark.parametrize("N", [64, 48, 32, 16])
def test_halves_of_tiles_paint_the_cells_of_whole_ones(N, window, interlaced, dtype, kind):
    """A plan that reserves 1000 objects a tile or more paints small meshes in halves of
    tiles of 16; tiles asked for, and plans that reserve nothing, take whole ones.  Half of
    the objects lie within a few FP32 roundings of cell faces (and so of the halves' seams
    and the tiles' faces), where the cell and the coordinate may round to different sides;
    some lie outside the box, on either side; a clump fills one cell."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1712_05834_gb300 as pk
    pk.build()
    rng = np.random.default_rng(N)
    n, L = max(1000 * (N // 16) ** 3, 20_000), 97.3
    pos = rng.random((n, 3)) * L
    near = np.round(rng.random((n // 2, 3)) * N) * (L / N)
    pos[: n // 2] = near * (1.0 + rng.integers(-4, 5, (n // 2, 3)) * 2.0 ** -24)
    pos[:200] += L * rng.integers(-1, 2, (200, 3))
    pos[-1500:] = np.array([7.9, 8.1, 7.99]) * (L / N) + 0.2 * (L / N) * rng.standard_normal((1500, 3))
    pos = torch.from_numpy(pos.astype(np.float32 if dtype == "f32" else np.float64)).cuda()
    w = {"unit": None, "weighted": rng.normal(0.3, 1.0, n), "heavy": np.exp(3.0 * rng.normal(0.0, 1.0, n))}[kind]
    w = None if w is None else torch.from_numpy(w.astype(np.float32)).cuda()
    got = []
    for capacity, tile in ((n, 0), (n, 16), (0, 0)):
        plan = pk.pk_plan(pk.make_config(L, N, window, interlaced=interlaced, dk=0.3, capacity=capacity, tile=tile))
        try:
            pk.pk_paint(plan, pos, w)
            got.append([pk.pk_mesh(plan, 0, m, N) for m in range(2 if interlaced else 1)])
        finally:
            pk.pk_destroy(plan)
    for a, b, c in zip(*got):
        assert np.array_equal(b, c), int((b != c).sum())
        assert np.array_equal(a, b), int((a != b).sum())
