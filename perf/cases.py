"""Timed cases: what programs have this library do, through its public calls.

A case names a kind of call and its sizes:

  box     one catalog in a periodic box: paint, compute and read back P(k),
          P(k, mu) and the multipoles with a resident plan (FFTPower.run);
  mocks   a covariance set: new mock catalogs of the sizes a BatchPower was
          made for, evaluated by size class (refill + run);
  cross   the density and the momentum field of one catalog: both auto powers
          and their cross power (pk_paint_values, pk_compute, pk_cross);
  survey  multipoles of survey data and randoms with the local line of sight
          (ConvolvedFFTPower.run);
  draw    a log-normal mock catalog generated on the device
          (LogNormalCatalog.draw).

Spectra of the FP32 mesh form carry FP32 accuracy (bins are summed in FP32
within a block, in an order that can vary between runs), so the programs here
keep them in single precision; k, sums of weights and shot noise, and all of
the FP64 form's results, are kept in double.
"""
import math

import numpy as np
import torch

import paper_1712_05834_gb300 as pk
from paper_1712_05834_gb300 import batch

C_H0 = 2997.92458           # c / H0 in Mpc/h
OMEGA_M = 0.31
SKY_Z = (0.15, 0.7)         # redshift range of the survey samples
ORDER = {"cic": 2, "tsc": 3, "pcs": 4}


def listed():
    box = dict(kind="box", source="lognormal", layout="f32", interlaced=False, nmu=0, precision="f32")
    return [
        # a quick look at a small simulation box: launches and latency are all there is
        dict(box, name="tiny_uniform_64", n=100_000, L=1000.0, nmesh=64, window="cic", dk=0.01, source="uniform",
             layout="f64"),
        # halos with completeness weights on a small mesh whose size is no power of two
        dict(box, name="halos_weighted_100", n=30_011, L=500.0, nmesh=100, window="pcs", dk=0.02, nmu=5,
             interlaced=True, layout="xyzw"),
        # one mock on the mesh that most covariance work uses
        dict(box, name="mock_256", n=2_000_003, L=1000.0, nmesh=256, window="tsc", dk=0.01),
        # a simulation snapshot at the paper's accuracy settings: the headline measurement
        dict(box, name="snapshot_512", n=10_000_000, L=1000.0, nmesh=512, window="tsc", dk=0.005, nmu=10,
             interlaced=True),
        # weighted galaxies in a box, mesh chosen for the cell size (no power of two)
        dict(box, name="galaxies_weighted_400", n=3_000_001, L=1500.0, nmesh=400, window="tsc", dk=0.008, nmu=10,
             interlaced=True, layout="f32+w"),
        # the double-precision form, used where 1e-6 per bin matters
        dict(box, name="precise_256", n=1_000_003, L=1000.0, nmesh=256, window="pcs", dk=0.01, interlaced=True,
             layout="f64+w", precision="f64"),
        # the large job of a P(k) service: a dense snapshot on a fine mesh
        dict(box, name="dense_1024", n=130_000_000, L=1000.0, nmesh=1024, window="tsc", dk=0.01, interlaced=True),
        # particles of an N-body run, still near their lattice order, on the finest mesh
        dict(box, name="particles_2048", n=640 ** 3, L=2000.0, nmesh=2048, window="pcs", dk=0.005,
             source="lattice"),
        # covariance mocks of uneven size, CIC and TSC, over three mesh sizes
        dict(kind="mocks", name="mocks_40", count=40, n_lo=200_000, n_hi=4_000_000, L=1000.0, dk=0.01),
        # density and momentum of one catalog, and their cross power
        dict(kind="cross", name="momentum_256", n=1_500_007, L=1000.0, nmesh=256, window="tsc", dk=0.01,
             interlaced=True),
        # a galaxy survey with ten times as many randoms, sky coordinates and FKP weights
        dict(kind="survey", name="survey_512", n=1_000_000, randoms=10_000_000, nmesh=512, window="tsc",
             interlaced=True, dk=0.005),
        # a mock made on the device, before its power is measured
        dict(kind="draw", name="draw_512", n=10_000_000, L=1000.0, ngrid=512),
    ]


# mesh sizes with small factors whose paint tile (the largest divisor up to 16) has an even edge
MESHES = [64, 72, 80, 96, 100, 108, 112, 128, 140, 144, 160, 192, 200, 216, 224, 240, 250, 256, 280, 288, 320, 336, 350,
          384, 400, 432, 448, 480, 500, 512, 560, 576, 640, 700, 720, 768, 800, 864, 960, 1000, 1024]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _mesh(rng, lo, hi):
    x = _log_uniform(rng, lo, hi)
    return min((m for m in MESHES if lo <= m <= hi), key=lambda m: abs(math.log(m / x)))


def draw(rng):
    kind = rng.choices(["box", "mocks", "cross", "survey", "draw"], [10, 1, 2, 2, 1])[0]
    window = rng.choice(["cic", "tsc", "pcs"])
    if kind == "mocks":
        lo = _log_uniform(rng, 5e4, 4e5)
        return dict(kind=kind, count=rng.randint(6, 40), n_lo=int(lo), n_hi=int(lo * rng.uniform(2.0, 15.0)), L=1000.0,
                    dk=0.01)
    if kind == "draw":
        ng = _mesh(rng, 64, 512)
        return dict(kind=kind, n=int(ng ** 3 * _log_uniform(rng, 0.02, 0.3)) | 1, L=1000.0, ngrid=ng)
    if kind == "survey":
        n = int(_log_uniform(rng, 3e4, 1e6))
        return dict(kind=kind, n=n, randoms=int(n * rng.uniform(2.0, 10.0)) | 1, nmesh=_mesh(rng, 120, 512),
                    window=window, interlaced=rng.random() < 0.5, dk=0.008)
    precision = "f64" if kind == "box" and rng.random() < 0.12 else "f32"
    nmesh = _mesh(rng, 64, 320 if precision == "f64" or kind == "cross" else 1024)
    n = int(min(nmesh ** 3 * _log_uniform(rng, 0.01, 0.5), 1.3e8)) | 1
    L = float(rng.choice([500.0, 1000.0, 1500.0, 2500.0]))
    kf = 2.0 * math.pi / L
    case = dict(kind=kind, n=n, L=L, nmesh=nmesh, window=window, interlaced=rng.random() < 0.6,
                dk=round(kf * rng.uniform(0.8, 3.0), 5))
    if kind == "box":
        case.update(source=rng.choice(["lognormal", "lognormal", "uniform"]), nmu=rng.choice([0, 0, 5, 10]),
                    layout=rng.choice(["f32", "f32", "f32+w", "xyzw", "f64", "f64+w"]), precision=precision)
    return case


# ---- inputs: seeded catalogs made on the GPU ----

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7fffffffffffffff)
    return g


def _kgrid(ng, L):
    kf = 2.0 * math.pi / L
    f = torch.fft.fftfreq(ng, d=1.0 / ng, device="cuda", dtype=torch.float32) * kf
    fz = torch.fft.rfftfreq(ng, d=1.0 / ng, device="cuda", dtype=torch.float32) * kf
    return f[:, None, None], f[None, :, None], fz[None, None, :]


def _gaussian(ng, L, slope, seed):
    """Half-grid transform of a Gaussian field with P(k) ~ k^slope and unit
    variance, and k^2 (1 at k = 0)."""
    wk = torch.fft.rfftn(torch.randn((ng, ng, ng), generator=_gen(seed), device="cuda"))
    kx, ky, kz = _kgrid(ng, L)
    k2 = kx * kx + ky * ky + kz * kz
    k2[0, 0, 0] = 1.0
    wk *= k2 ** (0.25 * slope)
    wk[0, 0, 0] = 0.0
    return wk, k2


def _lognormal(n, L, ng, seed, rsd=0.75):
    """n objects of a log-normal field (in random order), displaced along z."""
    wk, k2 = _gaussian(ng, L, -1.5, seed)
    g = torch.fft.irfftn(wk, s=(ng, ng, ng))
    std = float(g.double().std())
    rho = torch.exp(g * (1.0 / std) - 0.5).mul_(2.0 ** 20).round_().to(torch.int64)
    del g
    cdf = torch.cumsum(rho.reshape(-1), 0)          # integers: the same in any order of summation
    del rho
    gen = _gen(seed + 1)
    pos = torch.empty((n, 3), dtype=torch.float32, device="cuda")
    psi = None
    if rsd:
        psi = torch.fft.irfftn(wk * (1j * (_kgrid(ng, L)[2] / k2)), s=(ng, ng, ng)).reshape(-1) * (rsd / std)
    del wk, k2
    step = 1 << 25
    for a in range(0, n, step):
        m = min(step, n - a)
        u = (torch.rand(m, generator=gen, device="cuda", dtype=torch.float64) * float(cdf[-1])).to(torch.int64)
        cell = torch.searchsorted(cdf, u, right=True).clamp_(max=ng ** 3 - 1)
        off = torch.rand((m, 3), generator=gen, device="cuda")
        x = torch.stack([cell // (ng * ng), (cell // ng) % ng, cell % ng], 1).to(torch.float64).add_(off).mul_(L / ng)
        if psi is not None:
            x[:, 2] += psi[cell]
            x[:, 2] = torch.remainder(x[:, 2], L)
        pos[a:a + m] = x.to(torch.float32)
    return pos.clamp_(min=0.0)


def _lattice(nside, L, seed):
    """A displaced lattice in lattice order (rms displacement 1/4 spacing)."""
    wk, k2 = _gaussian(nside, L, -2.0, seed)
    ks = _kgrid(nside, L)
    q = torch.arange(nside, device="cuda", dtype=torch.float32) * (L / nside)
    pos = torch.empty((nside, nside, nside, 3), dtype=torch.float32, device="cuda")
    for a in range(3):
        psi = torch.fft.irfftn(wk * (1j * (ks[a] / k2)), s=(nside, nside, nside))
        psi *= 0.25 * (L / nside) / float(psi.double().std())
        shape = [1, 1, 1]
        shape[a] = nside
        pos[..., a] = torch.remainder(psi + q.reshape(shape), L)
        del psi
    return pos.reshape(-1, 3)


def _weights(n, seed):
    return torch.rand(n, generator=_gen(seed + 2), device="cuda") * 0.7 + 0.6


def _catalog(case, seed):
    """(positions, weights or None) of a box catalog in its layout."""
    n, L = case["n"], case["L"]
    source, layout = case.get("source", "lognormal"), case.get("layout", "f32")
    if source == "uniform":
        dtype = torch.float64 if layout.startswith("f64") else torch.float32
        pos = torch.rand((n, 3), generator=_gen(seed), device="cuda", dtype=dtype) * L
    elif source == "lattice":
        pos = _lattice(round(n ** (1.0 / 3.0)), L, seed)
    else:
        pos = _lognormal(n, L, min(case["nmesh"], 512), seed)
    if layout.startswith("f64"):
        pos = pos.to(torch.float64)
    w = _weights(n, seed) if layout in ("f32+w", "f64+w", "xyzw") else None
    if layout == "xyzw":
        return torch.cat([pos, w[:, None]], 1).contiguous(), None
    return pos.contiguous(), w


def _mock_specs(case):
    """Sizes of a mock set: fixed by the case, so that a runner's classes are."""
    r = np.random.default_rng(case["count"] * 7919 + case["n_lo"])
    n = np.exp(r.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), case["count"])).astype(np.int64)
    mesh = r.choice([128, 192, 256], case["count"])
    win = r.choice(["cic", "tsc"], case["count"])
    return [(int(n[i]) | 1, int(mesh[i]), str(win[i])) for i in range(case["count"])]


def _mock_catalogs(case, seed):
    return [_lognormal(n, case["L"], mesh, seed * 1009 + i) for i, (n, mesh, _) in enumerate(_mock_specs(case))]


def _chi(z):
    """Comoving distance in Mpc/h of a double tensor of redshifts."""
    x, w = np.polynomial.legendre.leggauss(24)
    chi = torch.zeros_like(z)
    for a, b in zip(x, w):
        t = 1.0 + z * (0.5 * (a + 1.0))
        chi += (0.5 * b) * z / torch.sqrt(OMEGA_M * t ** 3 + (1.0 - OMEGA_M))
    return C_H0 * chi


def _survey_box():
    """Edge and origin of the mesh box: the observer sits near its corner."""
    reach = float(_chi(torch.tensor([SKY_Z[1]], dtype=torch.float64))[0])
    return 1.04 * reach, (-0.02 * reach,) * 3


def _survey_sample(n, seed, clustered):
    """RA, Dec (degrees) and redshift of n objects of the octant shell, their
    number density column and completeness weights (float32)."""
    L, origin = _survey_box()
    zt = torch.linspace(0.0, SKY_Z[1] * 1.001, 4096, dtype=torch.float64, device="cuda")
    ct = _chi(zt)
    lo, hi = _chi(torch.tensor(SKY_Z, dtype=torch.float64)).tolist()
    parts, have, k = [], 0, 0
    while have < n:
        m = int(2.6 * (n - have)) + 4096
        if clustered:
            x = _lognormal(m, L, 128, seed + 31 * k, rsd=0.0).to(torch.float64)
        else:
            x = torch.rand((m, 3), generator=_gen(seed + 31 * k), device="cuda", dtype=torch.float64) * L
        x += origin[0]
        r = x.norm(dim=1)
        keep = (r > lo) & (r < hi) & (x > 0.0).all(1)
        x, r = x[keep], r[keep]
        j = torch.searchsorted(ct, r).clamp_(1, len(zt) - 1)
        z = zt[j - 1] + (zt[j] - zt[j - 1]) * (r - ct[j - 1]) / (ct[j] - ct[j - 1])
        sky = torch.stack([torch.rad2deg(torch.atan2(x[:, 1], x[:, 0])), torch.rad2deg(torch.asin(x[:, 2] / r)), z], 1)
        parts.append(sky[: n - have].to(torch.float32))
        have += len(parts[-1])
        k += 1
    sky = torch.cat(parts).contiguous()
    mid = (sky[:, 2] - SKY_Z[0]) / (SKY_Z[1] - SKY_Z[0])
    nbar = (1e-4 * (2.5 + 1.5 * torch.cos(2.0 * math.pi * mid))).contiguous()
    return sky, nbar, 0.8 + 0.4 * torch.rand(n, generator=_gen(seed + 77), device="cuda")


def _survey(case, seed):
    return _survey_sample(case["n"], seed * 17 + 5, True), _survey_sample(case["randoms"], seed * 17 + 11, False)


def _velocities(n, seed):
    return torch.randn(n, generator=_gen(seed + 9), device="cuda")


# ---- the calls ----

class _Mocks:
    """A batch runner and the catalogs of its next evaluation."""

    def __init__(self, case, seed):
        specs = _mock_specs(case)
        self.cats = [batch.Catalog(p, mesh, win) for p, (_, mesh, win) in zip(_mock_catalogs(case, seed), specs)]
        self.runner = batch.BatchPower(self.cats, case["L"], dk=case["dk"])

    def __del__(self):
        if hasattr(self, "runner"):
            self.runner.close()


def prepare(case, seed):
    kind, stream = case["kind"], torch.cuda.current_stream()
    if kind == "mocks":
        state = {"kind": kind, "mocks": _Mocks(case, seed)}
    elif kind == "draw":
        state = {"kind": kind, "gen": pk.LogNormalCatalog(case["L"], case["ngrid"], stream=stream), "seed": int(seed),
                 "n": case["n"], "out": torch.empty((case["n"], 3), dtype=torch.float32, device="cuda")}
    elif kind == "survey":
        L, origin = _survey_box()
        (d, dn, dw), (r, rn, _) = _survey(case, seed)
        cfg = pk.make_survey_config(L, origin, case["nmesh"], case["window"], case["interlaced"], dk=case["dk"],
                                    omega_m=OMEGA_M, zmax=1.0, p0_fkp=1e4, capacity=len(d) + len(r))
        state = {"kind": kind, "power": pk.ConvolvedFFTPower(cfg, stream),
                 "data": pk.survey_catalog(d, "sky", wcomp=dw, nbar=dn),
                 "randoms": pk.survey_catalog(r, "sky", nbar=rn)}
    else:
        cross = kind == "cross"
        pos, w = _catalog(case, seed)
        cfg = pk.make_config(case["L"], case["nmesh"], case["window"], case["interlaced"], dk=case["dk"],
                             nmu=case.get("nmu", 0), precision=case.get("precision", "f32"), batch=2 if cross else 1,
                             capacity=case["n"] * (2 if cross else 1))
        state = {"kind": kind, "power": pk.FFTPower(cfg, stream), "pos": pos, "weights": w,
                 "double": case.get("precision") == "f64"}
        if cross:
            state["pos"] = torch.cat([pos, pos]).contiguous()
            state["values"] = torch.cat([torch.ones(case["n"], device="cuda"), _velocities(case["n"], seed)])
            state["offsets"] = [0, case["n"], 2 * case["n"]]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()            # plans take their device memory from the driver
    return state


def _kept(res, double=False):
    """What a program keeps of a result (spectra at the form's accuracy)."""
    real = np.float64 if double else np.float32
    out = {"k": res["k"], "modes": res["modes"], "power": res["power"].astype(real),
           "poles": res["poles"].astype(real), "shot_noise": res["shot_noise"], "wsum": res["wsum"],
           "w2sum": res["w2sum"]}
    if res["nmu"]:
        out.update(k2d=res["k2d"], mu2d=res["mu2d"], modes2d=res["modes2d"], power2d=res["power2d"].astype(real))
    return out


def run(state):
    kind = state["kind"]
    if kind == "box":
        return _kept(state["power"].run(state["pos"], state["weights"]), state["double"])
    if kind == "mocks":
        m = state["mocks"]
        m.runner.refill(m.cats)
        res = [_kept(r) for r in m.runner.run()]
        return {name: np.concatenate([np.atleast_1d(r[name]).reshape(-1) for r in res]) for name in res[0]}
    if kind == "cross":
        plan = state["power"].plan
        pk.pk_paint_values(plan, state["pos"], state["values"], state["offsets"])
        pk.pk_compute(plan)
        return {"density": _kept(pk.pk_result(plan, 0)), "momentum": _kept(pk.pk_result(plan, 1)),
                "cross": _kept(pk.pk_cross(plan, 0, 1))}
    if kind == "survey":
        r = state["power"].run(state["data"], state["randoms"])
        out = {name: r[name] for name in ("k", "modes", "alpha", "norm", "shot_noise", "data_wsum", "randoms_wsum",
                                          "data_w2sum", "randoms_w2sum", "randoms_nsum", "n_outside", "n_rejected")}
        out["poles"] = r["poles"].astype(np.float32)
        return out
    return state["gen"].draw(state["seed"], state["n"], out=state["out"])


# ---- what a pass cannot do without ----

def _transform(nmesh, meshes, esz=4):
    """One mesh set that has to be held in memory between its painting and its
    transform (written once, read once), and the transform's arithmetic."""
    cells = nmesh ** 3
    return 2.0 * esz * cells * meshes, 2.5 * cells * math.log2(cells) * meshes


def _bins(case, nmesh):
    return int(math.pi * nmesh / case.get("L", 1800.0) / case["dk"]) + 1


def work(case):
    kind = case["kind"]
    if kind == "mocks":
        total = {"bytes": 0.0, "flops": 0.0}
        for n, mesh, win in _mock_specs(case):
            w = work(dict(kind="box", n=n, L=case["L"], nmesh=mesh, window=win, dk=case["dk"], interlaced=False,
                          layout="f32"))
            total = {k: total[k] + w[k] for k in total}
        return total
    if kind == "draw":
        b, f = _transform(case["ngrid"], 3)
        return {"bytes": b + 12.0 * case["n"], "flops": f + 100.0 * case["n"]}
    p3 = ORDER[case["window"]] ** 3
    nm = 2 if case["interlaced"] else 1
    if kind == "survey":
        n, mesh = case["n"] + case["randoms"], case["nmesh"]
        b, f = _transform(mesh, 15 + (2 * nm + 1 if nm == 2 else 2))
        return {"bytes": b + 20.0 * n + 56.0 * _bins(case, mesh), "flops": f + 2.0 * p3 * nm * n + 60.0 * mesh ** 3}
    items, mesh, n = (2 if kind == "cross" else 1), case["nmesh"], case["n"]
    rec = {"f32": 12, "f32+w": 16, "xyzw": 16, "f64": 24, "f64+w": 28}[case.get("layout", "f32")]
    b, f = _transform(mesh, nm * items, 8 if case.get("precision") == "f64" else 4)
    nk = _bins(case, mesh)
    out = (items + items // 2) * 8.0 * nk * (6 + 4 * case.get("nmu", 0))
    return {"bytes": b + (rec + (4 if items == 2 else 0)) * float(n) * items + out,
            "flops": f + (2.0 * p3 * nm * n + 10.0 * mesh ** 3 * nm) * items}


# ---- the same results in 64 bits, from plain torch ----

def _spline(u, p):
    """First node and per-node weights of the order-p window at u (cells)."""
    if p == 2:
        f0 = torch.floor(u)
        f = u - f0
        return f0, [1.0 - f, f]
    if p == 3:
        f0 = torch.floor(u + 0.5)
        g = u - f0
        return f0 - 1.0, [0.5 * (0.5 - g) ** 2, 0.75 - g ** 2, 0.5 * (0.5 + g) ** 2]
    f0 = torch.floor(u)
    f = u - f0
    r = 1.0 - f
    return f0 - 1.0, [r ** 3 / 6.0, (4.0 - 6.0 * f ** 2 + 3.0 * f ** 3) / 6.0, (4.0 - 6.0 * r ** 2 + 3.0 * r ** 3) / 6.0,
                      f ** 3 / 6.0]


def _paint64(pos, w, L, N, p, shift):
    mesh = torch.zeros(N ** 3, dtype=torch.float64, device="cuda")
    step = 1 << 24
    for a in range(0, len(pos), step):
        x = pos[a:a + step, :3].to(torch.float64) * (N / L) + shift
        ww = None if w is None else w[a:a + step].to(torch.float64)
        ax = [_spline(x[:, d], p) for d in range(3)]
        at = [[torch.remainder(f0 + float(k), N).to(torch.int64) for k in range(p)] for f0, _ in ax]
        for i in range(p):
            wi = ax[0][1][i] if ww is None else ax[0][1][i] * ww
            for j in range(p):
                wij, row = wi * ax[1][1][j], (at[0][i] * N + at[1][j]) * N
                for k in range(p):
                    mesh.index_add_(0, row + at[2][k], wij * ax[2][1][k])
    return mesh.reshape(N, N, N)


def _index(N):
    i = torch.arange(N, device="cuda", dtype=torch.int64)
    return torch.where(i < N // 2, i, i - N)


def _phase(n, N):
    a = n.to(torch.float64) * (math.pi / N)
    return torch.complex(torch.cos(a), torch.sin(a))


def _delta64(pos, w, L, N, p, interlaced):
    """Painted field's transform (interlaced meshes combined), not compensated."""
    fk = torch.fft.rfftn(_paint64(pos, w, L, N, p, 0.0))
    if interlaced:
        gk = torch.fft.rfftn(_paint64(pos, w, L, N, p, 0.5))
        n = _index(N)
        gk *= _phase(n, N)[:, None, None]
        gk *= _phase(n, N)[None, :, None]
        gk *= _phase(torch.arange(N // 2 + 1, device="cuda"), N)[None, None, :]
        fk.add_(gk).mul_(0.5)
    return fk


def _window2(N, p):
    """1 / sinc^2p of the index along one axis (fftfreq order)."""
    return torch.sinc(_index(N).to(torch.float64) / N) ** (-2 * p)


def _slabs(N, L, dk):
    """Per x plane: its index, the integer m = |n|^2, l, k bins (-1: none) and mode weights."""
    kf, nk = 2.0 * math.pi / L, int(math.floor((math.pi * N) / L / dk))
    n, l = _index(N), torch.arange(N // 2 + 1, device="cuda", dtype=torch.int64)
    h = torch.full((N // 2 + 1,), 2.0, dtype=torch.float64, device="cuda")
    h[0] = h[-1] = 1.0
    for i in range(N):
        m = n[i] * n[i] + n[:, None] ** 2 + l[None, :] ** 2
        b = torch.floor(kf * torch.sqrt(m.to(torch.float64)) / dk).to(torch.int64)
        yield i, n, l, m, torch.where((b < nk) & (m > 0), b, torch.full_like(b, -1)), h[None, :].expand(m.shape), nk


def _binned64(fa, fb, wa, wb, L, N, p, dk, nmu, shot, shot2=0.0):
    """power, poles and power2d of Re(fa conj fb), as the library's results hold them."""
    cw = _window2(N, p)
    cl = torch.cat([cw[: N // 2], cw[N // 2: N // 2 + 1]])
    sums = None
    for i, n, l, m, b, h, nk in _slabs(N, L, dk):
        if sums is None:
            sums = torch.zeros((4, nk + 1), dtype=torch.float64, device="cuda")
            s2 = torch.zeros((2, nk * max(nmu, 1) + 1), dtype=torch.float64, device="cuda")
        pw = (fa[i].real * fb[i].real + fa[i].imag * fb[i].imag) * (cw[i] * cw[:, None] * cl[None, :]) * h
        mu2 = (l[None, :] ** 2).to(torch.float64) / m.clamp(min=1).to(torch.float64)
        at = torch.where(b >= 0, b, torch.full_like(b, nk)).reshape(-1)
        for k, v in enumerate((h, pw, pw * (1.5 * mu2 - 0.5), pw * ((4.375 * mu2 - 3.75) * mu2 + 0.375))):
            sums[k] += torch.bincount(at, v.reshape(-1), nk + 1)
        if nmu:
            q = torch.floor(nmu * torch.sqrt(mu2)).to(torch.int64).clamp(0, nmu - 1)
            rhs = nmu * nmu * l[None, :] ** 2
            q = q - ((q > 0) & (q * q * m > rhs)).to(torch.int64)
            q = q + ((q < nmu - 1) & ((q + 1) ** 2 * m <= rhs)).to(torch.int64)
            at2 = torch.where(b >= 0, b * nmu + q, torch.full_like(b, nk * nmu)).reshape(-1)
            s2[0] += torch.bincount(at2, h.reshape(-1), nk * nmu + 1)
            s2[1] += torch.bincount(at2, pw.reshape(-1), nk * nmu + 1)
    norm = L ** 3 / (wa * wb)
    cnt = sums[0, :nk]
    p0 = norm * sums[1, :nk] / cnt - shot
    poles = torch.stack([p0, 5.0 * norm * sums[2, :nk] / cnt, 9.0 * norm * sums[3, :nk] / cnt])
    out = {"power": p0.cpu().numpy(), "poles": poles.cpu().numpy()}
    if nmu:
        out["power2d"] = (norm * s2[1, :-1] / s2[0, :-1] - shot).reshape(nk, nmu).cpu().numpy()
    return out


def _result64(fk, w, wv, n, L, N, p, dk, nmu):
    wsum = float(n) if w is None else float(w.to(torch.float64).sum())
    w2 = float(n) if wv is None else float((wv.to(torch.float64) ** 2).sum())
    shot = L ** 3 * w2 / wsum ** 2
    out = _binned64(fk, fk, wsum, wsum, L, N, p, dk, nmu, shot)
    out.update(k=None, modes=None, shot_noise=shot, wsum=wsum, w2sum=w2)
    if nmu:
        out.update(k2d=None, mu2d=None, modes2d=None)
    return out


def _survey64(case, seed):
    L, origin = _survey_box()
    N, p, dk = case["nmesh"], ORDER[case["window"]], case["dk"]
    field, sums = [], []
    samples = _survey(case, seed)
    for sky, nbar, wc in ((samples[0][0], samples[0][1], samples[0][2]), (samples[1][0], samples[1][1], None)):
        s = sky.to(torch.float64)
        r, ra, dec = _chi(s[:, 2]), torch.deg2rad(s[:, 0]), torch.deg2rad(s[:, 1])
        x = torch.stack([r * torch.cos(dec) * torch.cos(ra), r * torch.cos(dec) * torch.sin(ra), r * torch.sin(dec)], 1)
        x -= torch.tensor(origin, dtype=torch.float64, device="cuda")
        nb = nbar.to(torch.float64)
        wf = 1.0 / (1.0 + nb * 1e4)
        wc = torch.ones_like(nb) if wc is None else wc.to(torch.float64)
        sums.append([float(v.sum()) for v in (wc, (wc * wf) ** 2, nb * wc * wf * wf)])
        field.append((x, wc * wf))
    alpha = sums[0][0] / sums[1][0]
    norm = alpha * sums[1][2]
    shot = (sums[0][1] + alpha ** 2 * sums[1][1]) / norm

    def fkp(shift):
        return _paint64(*field[0], L, N, p, shift) - alpha * _paint64(*field[1], L, N, p, shift)

    F = fkp(0.0)
    n, l = _index(N), torch.arange(N // 2 + 1, device="cuda", dtype=torch.int64)
    if case["interlaced"]:
        G = torch.fft.rfftn(fkp(0.5))
        G *= _phase(n, N)[:, None, None]
        G *= _phase(n, N)[None, :, None]
        G *= _phase(l, N)[None, None, :]
        A0 = (torch.fft.rfftn(F) + G) * 0.5
        A0[N // 2] = 0.0
        A0[:, N // 2] = 0.0
        A0[:, :, N // 2] = 0.0
        F = torch.fft.irfftn(A0, s=(N, N, N))
        del G
    else:
        A0 = torch.fft.rfftn(F)
    H = L / N
    c = torch.arange(N, device="cuda", dtype=torch.float64) * H
    xs = [(c + origin[0])[:, None, None], (c + origin[1])[None, :, None], (c + origin[2])[None, None, :]]
    r2 = xs[0] ** 2 + xs[1] ** 2 + xs[2] ** 2
    away = r2 > 0.0
    inv = torch.where(away, 1.0 / torch.sqrt(torch.where(away, r2, torch.ones_like(r2))), torch.zeros_like(r2))
    del r2, away
    on_los = F * (inv > 0.0)
    ks = [n.to(torch.float64)[:, None, None], n.to(torch.float64)[None, :, None], l.to(torch.float64)[None, None, :]]
    k2 = ks[0] ** 2 + ks[1] ** 2 + ks[2] ** 2
    k2[0, 0, 0] = 1.0
    ik = 1.0 / torch.sqrt(k2)
    A = {}
    for order in (2, 4):            # sum over nodes of F (k^.x^)^order, by its monomials
        total = None
        for a in range(order + 1):
            for b in range(order + 1 - a):
                e = (a, b, order - a - b)
                coef = math.factorial(order) / (math.factorial(e[0]) * math.factorial(e[1]) * math.factorial(e[2]))
                g = on_los * inv ** order
                f = ik ** order * coef
                for d in range(3):
                    if e[d]:
                        g = g * xs[d] ** e[d]
                        f = f * ks[d] ** e[d]
                t = torch.fft.rfftn(g) * f
                total = t if total is None else total.add_(t)
                del g, f, t
        A[order] = total
    B0 = torch.fft.rfftn(on_los)
    A4 = (35.0 * A[4] - 30.0 * A[2] + 3.0 * B0) / 8.0
    A2 = (3.0 * A[2] - B0) / 2.0
    del A, B0, on_los, inv
    cw = _window2(N, p)
    cl = torch.cat([cw[: N // 2], cw[N // 2: N // 2 + 1]])
    sums3 = None
    for i, _, _, _, b, h, nk in _slabs(N, L, dk):
        if sums3 is None:
            sums3 = torch.zeros((4, nk + 1), dtype=torch.float64, device="cuda")
        at = torch.where(b >= 0, b, torch.full_like(b, nk)).reshape(-1)
        g = cw[i] * cw[:, None] * cl[None, :] * h
        sums3[0] += torch.bincount(at, h.reshape(-1), nk + 1)
        for k, X in enumerate((A0, A2, A4)):
            v = (X[i].real * A0[i].real + X[i].imag * A0[i].imag) * g
            sums3[1 + k] += torch.bincount(at, v.reshape(-1), nk + 1)
    cnt = sums3[0, :nk] * norm
    poles = torch.stack([sums3[1, :nk] / cnt - shot, 5.0 * sums3[2, :nk] / cnt, 9.0 * sums3[3, :nk] / cnt])
    return {"k": None, "modes": None, "alpha": alpha, "norm": norm, "shot_noise": shot, "data_wsum": sums[0][0],
            "randoms_wsum": sums[1][0], "data_w2sum": sums[0][1], "randoms_w2sum": sums[1][1],
            "randoms_nsum": sums[1][2], "n_outside": None, "n_rejected": None, "poles": poles.cpu().numpy()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "draw" or case.get("nmesh", 0) > 1024:
        return None             # a random draw has no such value; a 2048^3 transform in 64 bits does not fit
    if kind == "survey":
        return _survey64(case, seed)
    if kind == "mocks":
        res = []
        for pos, (n, mesh, win) in zip(_mock_catalogs(case, seed), _mock_specs(case)):
            fk = _delta64(pos, None, case["L"], mesh, ORDER[win], False)
            res.append(_result64(fk, None, None, n, case["L"], mesh, ORDER[win], case["dk"], 0))
        return {name: None if res[0][name] is None else
                np.concatenate([np.atleast_1d(r[name]).reshape(-1) for r in res]) for name in res[0]}
    n, L, N, p, dk = case["n"], case["L"], case["nmesh"], ORDER[case["window"]], case["dk"]
    pos, w = _catalog(case, seed)
    if case.get("layout") == "xyzw":
        w = pos[:, 3]
    nmu = case.get("nmu", 0)
    fk = _delta64(pos, w, L, N, p, case["interlaced"])
    density = _result64(fk, w, w, n, L, N, p, dk, nmu)
    if kind == "box":
        return density
    v = _velocities(n, seed)
    vk = _delta64(pos, v, L, N, p, case["interlaced"])
    both = _binned64(fk, vk, float(n), float(n), L, N, p, dk, 0, 0.0)
    both.update(k=None, modes=None, shot_noise=0.0, wsum=float(n), w2sum=float(n))
    return {"density": density, "momentum": _result64(vk, None, v, n, L, N, p, dk, 0), "cross": both}
