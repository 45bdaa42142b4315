"""Tiles whose candidates in all might overflow one-word cells: counted per block of
cells during the sweep and kept if no 2 x 2 x 2 blocks can fill a cell, else
painted again.  Evenly dense tiles (kept), all of a tile's objects in one cell, on
a cell corner or on a block corner (painted again: more than 1024 units in a cell
wrap a 32-bit word), and counts around the limits; unit, positive, mixed and tiny
weights, every window, several tile edges.

Tolerance: a cell is the sum of its deposits, each rounded to 2^-22 and made of
FP32 window weights; as the sum of |deposits| S of a cell (the oracle's paint of
|W|) bounds both: 2^-23 per deposit of the objects that reach it, 2e-6 S for the
weights, 2^-24 S for the cell.  A wrapped cell is off by 1024 (signed: 512 or more)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,window,interlaced,kind", [
    (32, "cic", False, "unit"), (32, "tsc", True, "unit"), (32, "pcs", True, "unit"), (48, "tsc", False, "positive"),
    (32, "pcs", True, "positive"), (32, "tsc", True, "mixed"), (40, "cic", True, "unit"), (36, "pcs", False, "unit"),
    (46, "tsc", True, "unit"), (54, "cic", True, "tiny")])
@pytest.mark.parametrize("place", ["even", "cell", "corner", "block"])
def test_cells_match_the_oracle(N, window, interlaced, kind, place):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import oracle
    import paper_1712_05834_gb300 as pk
    oracle.build()
    pk.build()
    L = float(N)                                       # cells of 1
    rng = np.random.default_rng(N + len(kind) + len(place))
    even = rng.random((int(0.75 * N ** 3), 3)) * L
    clumps = []
    if place != "even":
        at = {"cell": 5.5, "corner": 6.0, "block": 8.0}[place]
        for k, n in enumerate((700, 1300, 2600, 5200)):
            c = np.array([at, at, at]) + np.array([(0, 0, 0), (16, 0, 0), (0, 16, 0), (16, 16, 16)][k])
            clumps.append(c % N + 0.02 * rng.random((n, 3)))
    pos = (np.concatenate([even] + clumps) % L).astype(np.float32)
    n = len(pos)
    w = {"unit": None, "positive": rng.uniform(0.2, 1.8, n), "mixed": rng.normal(0, 1, n),
         "tiny": np.where(rng.random(n) < 1e-3, 30.0, 1e-4)}[kind]
    w = None if w is None else w.astype(np.float32)
    amp = np.ones(n) if w is None else w.astype(np.float64)
    dev = lambda a: None if a is None else torch.from_numpy(a).cuda()
    plan = pk.pk_plan(pk.make_config(L, N, window, interlaced=interlaced, dk=0.2))
    try:
        pk.pk_paint(plan, dev(pos), dev(w))
        got = [pk.pk_mesh(plan, 0, m, N) for m in range(2 if interlaced else 1)]
    finally:
        pk.pk_destroy(plan)
    p64 = pos.astype(np.float64)
    for m, mesh in enumerate(got):
        ref = oracle.paint(p64, amp, L, N, window, shift=0.5 * m)
        total = oracle.paint(p64, np.abs(amp), L, N, window, shift=0.5 * m)
        count = oracle.paint(p64, None, L, N, "cic", shift=0.5 * m)
        reach = sum(np.roll(count, (i, j, k), (0, 1, 2)) for i in range(-2, 3) for j in range(-2, 3) for k in range(-2, 3))
        tol = 2e-6 * total + 2.0 ** -24 * total + 2.0 ** -23 * reach + 1e-6 * np.abs(amp).max()
        assert np.all(np.abs(mesh - ref) <= tol), np.max(np.abs(mesh - ref) / tol)


@pytest.mark.parametrize("N,window,interlaced,n", [(64, "cic", False, 64_000), (64, "pcs", True, 63_999),
                                                   (48, "tsc", True, 27_000), (24, "pcs", False, 8_000)])
def test_default_tile_of_small_meshes(N, window, interlaced, n):
    """Plans reserved for 1000 objects a tile or more take tiles of 8 where those of 16
    (12 at 24) would leave SMs idle; against both tiles asked for and one object fewer
    reserved.  Tiles hold positions as FP32 offsets below 32, rounded by 2^-20 at most,
    on either side: with window slopes of at most 1 along three axes and deposits
    rounded to 2^-22, 6e-6 for each object that reaches a cell, and 2^-23 of the cell."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1712_05834_gb300 as pk
    pk.build()
    L = 300.0
    pos = (torch.rand((n, 3), generator=torch.Generator().manual_seed(N + n)) * L).cuda()
    got = []
    for capacity, tile in ((n, 0), (n - 1, 0), (n, 8), (n, 12 if N == 24 else 16)):
        plan = pk.pk_plan(pk.make_config(L, N, window, interlaced=interlaced, dk=0.1, capacity=capacity, tile=tile))
        try:
            pk.pk_paint(plan, pos)
            got.append([pk.pk_mesh(plan, 0, m, N) for m in range(2 if interlaced else 1)])
        finally:
            pk.pk_destroy(plan)
    c = np.floor(pos.cpu().numpy().astype(np.float64) * N / L).astype(int) % N
    count = np.bincount((c[:, 0] * N + c[:, 1]) * N + c[:, 2], minlength=N ** 3).reshape(N, N, N)
    reach = sum(np.roll(count, (i, j, k), (0, 1, 2)) for i in range(-2, 3) for j in range(-2, 3) for k in range(-2, 3))
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert np.all(np.abs(a - b) <= 6e-6 * reach + 2.0 ** -23 * np.abs(b))
