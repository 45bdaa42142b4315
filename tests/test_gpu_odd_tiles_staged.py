"""The paint's general path on tiles with an odd edge (N = 90 and 150: 15 cells; 54: 9),
whose candidates are staged in shared memory as 16-byte records behind the cells: taken
by every tile of the FP64 mesh form (deposits beyond 23 bits), and in the FP32 form
by tiles with thousands of objects in one cell.  Cells against the oracle's: deposits are
rounded to 2^-32 (2^-22) of a weight unit and made of FP32 window weights, 2e-6 of the sum
of |deposits| of the cell (the oracle's paint of |W|), 2^-24 of it for an FP32 cell, and
1e-6 of the largest weight where a cell is a sliver of a window."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("N,window,interlaced,weighted", [(90, "pcs", True, True), (90, "cic", False, False),
                                                          (150, "tsc", True, True), (54, "cic", True, True),
                                                          (54, "tsc", False, False)])
def test_cells_match_the_oracle(N, window, interlaced, weighted, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import oracle
    import paper_1712_05834_gb300 as pk
    oracle.build()
    pk.build()
    n, L = 40_000, float(N)
    rng = np.random.default_rng(N)
    pos = rng.random((n, 3)) * L
    if precision == "f32":                       # 6000 objects in a cell of each of three tiles
        for k, c in enumerate(([4.5, 4.5, 4.5], [20.5, 4.5, 4.5], [0.5, 0.5, 31.5])):
            pos[6000 * k: 6000 * (k + 1)] = np.array(c) + 0.2 * rng.random((6000, 3))
    pos = pos.astype(np.float32)
    w = rng.uniform(0.5, 1.5, n).astype(np.float32) if weighted else None
    plan = pk.pk_plan(pk.make_config(L, N, window, interlaced=interlaced, dk=0.2, precision=precision))
    try:
        pk.pk_paint(plan, torch.from_numpy(pos).cuda(), None if w is None else torch.from_numpy(w).cuda())
        got = [pk.pk_mesh(plan, 0, m, N, f64=precision == "f64") for m in range(2 if interlaced else 1)]
    finally:
        pk.pk_destroy(plan)
    p64, amp = pos.astype(np.float64), None if w is None else w.astype(np.float64)
    for m, mesh in enumerate(got):
        ref = oracle.paint(p64, amp, L, N, window, shift=0.5 * m)
        count = oracle.paint(p64, None, L, N, "cic", shift=0.5 * m)
        reach = sum(np.roll(count, (i, j, k), (0, 1, 2)) for i in range(-2, 3) for j in range(-2, 3) for k in range(-2, 3))
        tol = (2e-6 + 2.0 ** -24) * ref + 2.0 ** (-32 if precision == "f64" else -22) * reach + 1.5e-6
        assert np.all(np.abs(mesh - ref) <= tol), float(np.max(np.abs(mesh - ref) / tol))
