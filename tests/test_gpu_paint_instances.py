"""An object's deposits do not depend on which instance of the tile paint serves the
call: painted with unit weights or with an array of ones, in tiles of few objects or
many, the cells of the FP64 mesh form (window weights and one rounding per deposit,
summed as integers) are the same bits.  With and without the interlaced mesh a tile
looks at more or fewer candidates, and the split of its deposits into two words may
round one of them the other way: a unit of 2^-32 for each object that reaches a cell."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _cells(pk, pos, w, N, window, interlaced):
    plan = pk.pk_plan(pk.make_config(100.0, N, window, interlaced=interlaced, dk=0.2, precision="f64"))
    try:
        pk.pk_paint(plan, pos, w)
        return [pk.pk_mesh(plan, 0, m, N, f64=True) for m in range(2 if interlaced else 1)]
    finally:
        pk.pk_destroy(plan)


# 96: tiles of 16 known at compile time; 72: of 12.  The counts put some 30, 240 and
# 2000 objects into a tile: staged at once, in batches, and cells of 64 bits.
@pytest.mark.parametrize("window", ["cic", "tsc", "pcs"])
@pytest.mark.parametrize("N,n", [(96, 6001), (96, 200_003), (72, 50_001), (72, 430_001), (48, 100_003)])
def test_ones_and_unit_weights_paint_the_same_cells(window, N, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1712_05834_gb300 as pk
    pk.build()
    pos = (torch.rand((n, 3), generator=torch.Generator().manual_seed(n), dtype=torch.float64) * 100.0).cuda()
    ones = torch.ones(n, device="cuda")
    c = np.floor(pos.cpu().numpy() * (N / 100.0)).astype(int) % N
    count = np.bincount((c[:, 0] * N + c[:, 1]) * N + c[:, 2], minlength=N ** 3).reshape(N, N, N)
    reach = sum(np.roll(count, (i, j, k), (0, 1, 2)) for i in range(-2, 3) for j in range(-2, 3) for k in range(-2, 3))
    first = []
    for interlaced in (True, False):
        unit, weighted = (_cells(pk, pos, w, N, window, interlaced) for w in (None, ones))
        for a, b in zip(unit, weighted):
            assert np.array_equal(a, b), (interlaced, int((a != b).sum()))
        first.append(unit[0])
    assert np.all(np.abs(first[0] - first[1]) <= 2.0 ** -32 * reach)


# FP32 form: deposits of an array of ones are below 2^22, where each is the exact product
# rounded once, as with unit weights; of minus ones, the negative (ties go to even).
@pytest.mark.parametrize("window", ["cic", "tsc", "pcs"])
@pytest.mark.parametrize("N,n", [(96, 6001), (96, 200_003), (72, 50_001), (40, 30_001)])
@pytest.mark.parametrize("interlaced", [False, True])
def test_ones_in_the_fp32_form(window, N, n, interlaced):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1712_05834_gb300 as pk
    pk.build()
    pos = (torch.rand((n, 3), generator=torch.Generator().manual_seed(n)) * 100.0).cuda()
    got = []
    for w in (None, torch.ones(n, device="cuda"), -torch.ones(n, device="cuda")):
        plan = pk.pk_plan(pk.make_config(100.0, N, window, interlaced=interlaced, dk=0.2))
        try:
            pk.pk_paint(plan, pos, w)
            got.append([pk.pk_mesh(plan, 0, m, N) for m in range(2 if interlaced else 1)])
        finally:
            pk.pk_destroy(plan)
    for unit, ones, minus in zip(*got):
        assert np.array_equal(unit, ones), int((unit != ones).sum())
        assert np.array_equal(unit, -minus), int((unit != -minus).sum())


def test_cells_at_the_limit_of_one_word_do_not_depend_on_the_order():
    """A tile whose sum of |W| is at the limit up to which its cells are kept in one word
    (2^22 sum W + n = 4.29e9): whatever order its objects come in, it is painted the same
    way, and its cells are the same bits."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1712_05834_gb300 as pk
    pk.build()
    N, n, light = 64, 1000, 20_000
    rng = np.random.default_rng(7)
    pos = np.concatenate([2.0 + 11.0 * rng.random((n, 3)), 34.0 + 11.0 * rng.random((light, 3))]).astype(np.float32)
    w = np.concatenate([rng.uniform(0.9, 1.1, n), np.full(light, 0.01)]).astype(np.float32)
    w[:n] *= np.float32((4.29e9 - n) / 2.0 ** 22 / w[:n].astype(np.float64).sum())
    w[0] += np.float32((4.29e9 - n) / 2.0 ** 22 - w[:n].astype(np.float64).sum())
    plan = pk.pk_plan(pk.make_config(float(N), N, "cic", dk=0.2))
    try:
        for step in range(-24, 25):
            wk = w.copy()
            wk[0] += np.float32(step * 2.0 ** -15)                # 128 units of 2^-22
            first = None
            for _ in range(4):
                o = rng.permutation(n + light)
                pk.pk_paint(plan, torch.from_numpy(pos[o]).cuda(), torch.from_numpy(wk[o]).cuda())
                cells = pk.pk_mesh(plan, 0, 0, N)
                first = cells if first is None else first
                assert np.array_equal(first, cells), (step, int((first != cells).sum()))
    finally:
        pk.pk_destroy(plan)


@pytest.mark.parametrize("window", ["cic", "tsc", "pcs"])
@pytest.mark.parametrize("N,n,clump", [(96, 100_003, 0), (96, 400_003, 0), (96, 100_003, 3000), (72, 200_003, 2000),
                                       (34, 20_003, 0)])
@pytest.mark.parametrize("kind", ["unit", "positive", "mixed", "heavy"])
def test_fp32_cells_do_not_depend_on_the_way_a_tile_is_painted(window, N, n, clump, kind):
    """One object far from the others and heavier by 1e4 to 1e9 has their tiles painted
    the general way (split into two words, or 64-bit cells) where they are swept with
    one-word cells without it; a cell is the sum of the same integers rounded once."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1712_05834_gb300 as pk
    pk.build()
    rng = np.random.default_rng(n + clump)
    L = float(N)
    pos = rng.random((n, 3)) * L * np.array([0.5, 1.0, 1.0])
    if clump:
        pos[:clump] = np.array([5.3, 6.1, 40.7]) + 0.3 * rng.standard_normal((clump, 3))
    w = {"unit": np.ones(n), "positive": rng.uniform(0.5, 1.5, n), "mixed": rng.normal(0.0, 1.0, n),
         "heavy": rng.uniform(5.0, 40.0, n)}[kind]
    pos = np.concatenate([pos, [[0.75 * L, 0.5 * L, 0.5 * L]]]).astype(np.float32)
    got = []
    for far in (0.0, 1e4, 1e9):
        wk = torch.from_numpy(np.append(w, far).astype(np.float32)).cuda()
        plan = pk.pk_plan(pk.make_config(L, N, window, interlaced=True, dk=0.2))
        try:
            pk.pk_paint(plan, torch.from_numpy(pos).cuda(), wk)
            got.append([pk.pk_mesh(plan, 0, m, N) for m in range(2)])
        finally:
            pk.pk_destroy(plan)
    x = slice(0, N // 2 + 6)                             # without the far object's cells
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert np.array_equal(a[x], b[x]), int((a[x] != b[x]).sum())
