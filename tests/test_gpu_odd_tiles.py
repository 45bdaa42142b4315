"""Weighted catalogs, and unit-weight CIC, on meshes whose paint tile has an
odd edge (N = 90 and 150: T = 15; N = 54: T = 9): candidates are staged in
shared memory as 16-byte records behind 2 T^3 words of cells, which only an
even edge leaves aligned.  Painted cells against the oracle's mesh: each
deposit is rounded to 2^-22 of a weight unit and the window weights are FP32
(a few 1e-7 of the weight), so a cell of k deposits is within
k (2^-23 + 1e-6) max w of the FP64 value; k is at most the densest cell's
object count times the window's p^3 nodes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,window,interlaced,weighted", [(90, "pcs", True, True), (90, "cic", False, False),
                                                          (150, "tsc", True, True), (54, "cic", True, True)])
def test_staged_candidates_on_odd_tiles(N, window, interlaced, weighted):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import oracle
    import paper_1712_05834_gb300 as pk
    oracle.build()
    pk.build()
    n, L = 40000, 300.0
    rng = np.random.default_rng(N)
    pos = (rng.random((n, 3)) * L).astype(np.float32)
    w = rng.uniform(0.5, 1.5, n).astype(np.float32) if weighted else None
    plan = pk.pk_plan(pk.make_config(L, N, window, interlaced=interlaced, dk=0.05))
    try:
        pk.pk_paint(plan, torch.from_numpy(pos).cuda(), None if w is None else torch.from_numpy(w).cuda())
        got = [pk.pk_mesh(plan, 0, m, N) for m in range(2 if interlaced else 1)]
    finally:
        pk.pk_destroy(plan)
    p = {"cic": 2, "tsc": 3, "pcs": 4}[window]
    per_cell = np.bincount(np.ravel_multi_index(tuple((pos / L * N).astype(int).clip(0, N - 1).T), (N,) * 3)).max()
    tol = per_cell * p ** 3 * (2.0 ** -23 + 1e-6) * 1.5
    for m, mesh in enumerate(got):
        ref = oracle.paint(pos.astype(np.float64), None if w is None else w.astype(np.float64), L, N, window,
                           shift=0.5 * m)
        assert np.abs(mesh - ref).max() <= tol
