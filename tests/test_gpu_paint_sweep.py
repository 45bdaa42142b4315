"""One-word cells of the tile paint for weighted objects: tiles that fit are
painted in one sweep, tiles whose sum of |W V| might pass 2^31 units are painted
again the general way.  A catalog of a uniform background and one tight clump
(both kinds of tile, and tiles right at the limit), positive, mixed-sign and
large weights and painted values, every window, tile edges 16 and others, one
and two meshes: the cells against the oracle's.

Tolerance: a cell is the sum of its deposits, each rounded to 2^-22 and made of
FP32 window weights; the window weights sum to one per object, so the sum of
|deposits| S per cell (the oracle's paint of |W V|) bounds both: the rounding by
2^-23 per deposit and at most k objects, the weights by 2e-6 S, plus the FP32
rounding of the cell, 2^-24 S."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,window,interlaced,kind", [
    (64, "cic", True, "positive"), (64, "tsc", True, "mixed"), (64, "pcs", False, "positive"),
    (48, "pcs", True, "large"), (100, "tsc", False, "values"), (64, "cic", False, "large"), (90, "cic", True, "mixed"),
    (64, "tsc", False, "unit"), (64, "cic", True, "unit"), (100, "pcs", True, "unit")])
def test_cells_match_the_oracle(N, window, interlaced, kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import oracle
    import paper_1712_05834_gb300 as pk
    oracle.build()
    pk.build()
    L = 200.0
    rng = np.random.default_rng(N + len(kind))
    clump = 3 * L / N + rng.random((6000, 3)) * (12 * L / N)           # about 6000 candidates in a tile or two
    edge = L / 2 + rng.random((900, 3)) * (12 * L / N)                 # a few hundred: near the limits
    pos = np.concatenate([rng.random((15000, 3)) * L, clump, edge]).astype(np.float32)
    n = len(pos)
    w = {"positive": rng.uniform(0.5, 1.5, n), "mixed": rng.normal(0, 1, n), "large": rng.uniform(20.0, 90.0, n),
         "values": rng.uniform(0.5, 1.5, n), "unit": None}[kind]
    v = rng.normal(0, 2.0, n).astype(np.float32) if kind == "values" else None
    w = None if w is None else w.astype(np.float32)
    amp = np.ones(n) if w is None else (w if v is None else w * v).astype(np.float64)
    dev = lambda a: None if a is None else torch.from_numpy(a).cuda()
    plan = pk.pk_plan(pk.make_config(L, N, window, interlaced=interlaced, dk=0.05))
    try:
        if v is None:
            pk.pk_paint(plan, dev(pos), dev(w))
        else:
            pk.pk_paint_values(plan, dev(pos), dev(v), weights=dev(w))
        got = [pk.pk_mesh(plan, 0, m, N) for m in range(2 if interlaced else 1)]
    finally:
        pk.pk_destroy(plan)
    p64 = pos.astype(np.float64)
    for m, mesh in enumerate(got):
        ref = oracle.paint(p64, amp, L, N, window, shift=0.5 * m)
        total = oracle.paint(p64, np.abs(amp), L, N, window, shift=0.5 * m)
        count = oracle.paint(p64, None, L, N, "cic", shift=0.5 * m)
        # objects that reach a cell: those of the cells around it
        reach = sum(np.roll(count, (i, j, k), (0, 1, 2)) for i in range(-2, 3) for j in range(-2, 3) for k in range(-2, 3))
        tol = 2e-6 * total + 2.0 ** -24 * total + 2.0 ** -23 * reach + 1e-6 * np.abs(amp).max()
        assert np.all(np.abs(mesh - ref) <= tol), np.max(np.abs(mesh - ref) / tol)
