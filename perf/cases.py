"""Performance cases of the library: what its users have it do, over the range of sizes they do
it at, each through the Python binding (paper_2201_02632_gb300.api).

Every case is one of these kinds (`case["kind"]`):

  records    paste_particles + finalize of particle records: the deposit alone
  cone       a light-cone step: solve, assign, paste_particles, paste_halos, finalize of both
  hp         paste_halos + finalize of a solved catalogue onto one flat map
  hp_batch   a prepared plan over many maps: execute + finalize
  allsky     paste_halos_healpix + finalize of a solved all-sky catalogue
  solve      solve_halos of a catalogue (FP64), or its FP32-gated mode
  hsml       smoothing_lengths of a light-cone's particles
  spectrum   power_spectrum of a map (with or without its compensation plane)
  mlp_train  one training step of the surrogate: forward, loss, backward, Adam
  mlp_infer  features + BF16 inference of the surrogate

The sizes are those of the repository's workloads (bench.py, inputs.py, tests), smaller and
larger ones around them, odd and ragged ones among them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2201_02632_gb300 import _lib as L
from paper_2201_02632_gb300 import api
from paper_2201_02632_gb300 import inputs as I
from paper_2201_02632_gb300.surrogate import feature_norm

DEV = "cuda"
F64, F32, I32 = torch.float64, torch.float32, torch.int32
DEG = math.pi / 180.0


def listed():
    return [
        # a small deposit call: the fine-grained loop of an interactive or per-halo caller
        {"name": "records_20k", "kind": "records", "n": 20_000, "nx": 96, "ny": 96, "hmax": 24.0,
         "select": 0},
        # a ragged rectangular map with a mix of sub-pixel, small and wide kernels
        {"name": "records_1m_ragged", "kind": "records", "n": 1_250_003, "nx": 1333, "ny": 1111,
         "hmax": 40.0, "select": 0},
        # the 4e6-particle light-cone step on 1024^2 maps
        {"name": "cone_4m", "kind": "cone", "n": 4_000_000, "halos": 3000, "side": 2.0,
         "zmax": 1.5, "npix": 1024, "mass": "loguniform", "dt": False},
        # the full-scale light-cone step: 5e8 particles, 2e5 halos, 4096^2 maps
        {"name": "cone_full", "kind": "cone", "n": 500_000_000, "halos": 200_000, "side": 5.0,
         "zmax": 3.0, "npix": 4096, "mass": "powerlaw", "dt": False},
        # the 1000-halo catalogue on one 256^2 map, as temperature maps
        {"name": "hp_1000", "kind": "hp", "n": 1000, "npix": 256, "side": 1.0, "zmin": 0.05,
         "ap": 3.0, "dt": True},
        # a quarter of the batch of 108 maps of 2048^2, about 5e4 halos each
        {"name": "hp_batch_27", "kind": "hp_batch", "maps": 27, "mean": 50_000, "npix": 2048,
         "side": 5.0, "tile": 32},
        # a tenth of the all-sky catalogue of 4.1e7 halos
        {"name": "allsky_4m", "kind": "allsky", "n": 4_100_000, "nside": 4096, "zmin": 0.01,
         "zmax": 3.0, "ap": 0.0},
        # the FP64 solve of a large catalogue
        {"name": "solve_1m", "kind": "solve", "n": 1_000_003, "zmax": 3.0, "gated": False},
        # smoothing lengths of the 4e6-particle light-cone
        {"name": "hsml_4m", "kind": "hsml", "n": 4_000_000, "ngb": 64.0, "guess": False},
        # C_l of a full-scale map with its compensation plane
        {"name": "spectrum_4096", "kind": "spectrum", "nx": 4096, "ny": 4096, "lo": True},
        # one optimisation step of the surrogate at the batch its fit() uses
        {"name": "mlp_train_4096", "kind": "mlp_train", "n": 4096},
        # inference of the surrogate over a catalogue
        {"name": "mlp_infer_3m", "kind": "mlp_infer", "n": 3_000_017},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["records", "cone", "hp", "hp_batch", "allsky", "solve", "hsml", "spectrum",
                       "mlp_train", "mlp_infer"])
    c = {"kind": kind}
    if kind == "records":
        c.update(n=_log_int(rng, 500, 3_000_000), nx=_log_int(rng, 33, 1600),
                 ny=_log_int(rng, 33, 1600), hmax=round(math.exp(rng.uniform(0.7, 4.0)), 2),
                 select=rng.choice([0, 0, 1, 2]))
    elif kind == "cone":
        n = _log_int(rng, 30_000, 200_000_000)
        npix = 1024.0 * (n / 4e6) ** 0.29 * rng.uniform(0.7, 1.4)
        c.update(n=n, halos=max(20, n // rng.randint(1200, 2500)), side=round(rng.uniform(1, 5), 3),
                 zmax=round(rng.uniform(0.5, 3.0), 3), npix=int(min(4096, max(64, npix))),
                 mass=rng.choice(["loguniform", "powerlaw"]), dt=rng.random() < 0.5)
    elif kind == "hp":
        c.update(n=_log_int(rng, 20, 20_000), npix=_log_int(rng, 64, 1024),
                 side=round(rng.uniform(1, 5), 3), zmin=round(rng.uniform(0.05, 0.3), 3),
                 ap=rng.choice([0.0, 2.0, 3.0]), dt=rng.random() < 0.5)
    elif kind == "hp_batch":
        c.update(maps=rng.randint(2, 27), mean=_log_int(rng, 500, 50_000),
                 npix=_log_int(rng, 128, 2048), side=round(rng.uniform(2, 5), 3),
                 tile=rng.choice([32, 64]))
    elif kind == "allsky":
        c.update(n=_log_int(rng, 300, 4_000_000), nside=_log_int(rng, 64, 4096),
                 zmin=round(rng.uniform(0.01, 0.1), 4), zmax=round(rng.uniform(1.0, 3.0), 3),
                 ap=rng.choice([0.0, 0.0, 2.0]))
    elif kind == "solve":
        c.update(n=_log_int(rng, 200, 2_000_000), zmax=round(rng.uniform(0.5, 3.0), 3),
                 gated=rng.random() < 0.25)
    elif kind == "hsml":
        c.update(n=_log_int(rng, 5_000, 4_000_000), ngb=float(rng.choice([32, 64, 64, 100])),
                 guess=rng.random() < 0.5)
    elif kind == "spectrum":
        c.update(nx=1 << rng.randint(7, 12), ny=1 << rng.randint(7, 13), lo=rng.random() < 0.5)
    elif kind == "mlp_train":
        c.update(n=_log_int(rng, 100, 16_384))
    else:
        c.update(n=_log_int(rng, 1000, 10_000_000))
    return c


# ------------------------------------------------------------------ what a program has in hand
_CTX = None


def _ctx():
    """The program's one context (background tables, scratch) on its current stream."""
    global _CTX
    if _CTX is None:
        _CTX = api.Context()
    return _CTX


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _u(g, n, lo=0.0, hi=1.0, dtype=F64):
    return torch.rand(n, generator=g, device=DEV, dtype=dtype) * (hi - lo) + lo


def _randn(g, n, dtype=F32):
    return torch.randn(n, generator=g, device=DEV, dtype=dtype)


def _powerlaw(g, n, mmin=1e12, mmax=1e15, slope=-0.9):
    a, b = mmin ** slope, mmax ** slope
    return (a + _u(g, n) * (b - a)) ** (1.0 / slope)


def _concentration(g, M):
    return 5.0 * (M / 1e14) ** -0.1 * 10.0 ** (0.1 * _randn(g, M.numel(), F64))


def _patch(case, n_maps=1):
    half = 0.5 * case["side"] * DEG
    return half, api.geom(case["npix"], case["npix"], -half, -half, 2 * half / case["npix"], n_maps)


def _catalogue(g, n, half, zr, mass):
    """Halos uniform on a flat patch; mass log-uniform 1e13-1e15 or dN/dlnM ~ M^-0.9."""
    M = 10.0 ** _u(g, n, 13.0, 15.0) if mass == "loguniform" else _powerlaw(g, n)
    return {"M": M, "c": _concentration(g, M), "z": _u(g, n, *zr), "thx": _u(g, n, -half, half),
            "thy": _u(g, n, -half, half), "v": 300.0 * _randn(g, n)}


def _records(case, seed):
    """Deposit records around the map: sub-pixel, small and wide kernels, a few with h = 0, 40%
    field particles (no y), 5% that contribute nothing, signed b."""
    g = _gen(seed)
    n, nx, ny, hmax = case["n"], case["nx"], case["ny"], case["hmax"]
    rec = torch.empty((n, api.ASSIGNED_STRIDE), dtype=F32, device=DEV)
    ints = rec.view(I32)
    for a, side in ((0, nx), (1, ny)):
        p = _u(g, n, -8.0, side + 8.0)
        fl = torch.floor(p)
        f = (p - fl).float()
        up = f >= 1.0
        rec[:, a] = torch.where(up, torch.zeros_like(f), f)
        ints[:, 6 + a] = (fl + up).to(I32)
    u = _u(g, n)
    h = torch.where(u < 0.3, _u(g, n, 0.0, 1.0), _u(g, n, 1.0, min(6.0, hmax)))
    h = torch.where(u < 0.8, h, _u(g, n, min(6.0, 0.5 * hmax), hmax))
    rec[:, 2] = torch.where(_u(g, n) < 0.02, torch.zeros_like(h), h).float()
    kind = (_u(g, n) < 0.4).to(I32)
    kind[_u(g, n) < 0.05] = api.KIND_NONE
    rec[:, 3] = torch.where(kind == api.KIND_HALO, 10.0 ** _u(g, n, -9.0, -6.0),
                            torch.zeros_like(u)).float()
    rec[:, 4] = torch.where(kind == api.KIND_NONE, torch.zeros_like(u),
                            1e-7 * _randn(g, n, F64)).float()
    ints[:, 5] = kind
    return rec


def _cone(case, seed, sample=None):
    return I.lightcone_device(case["n"], case["halos"], side_deg=case["side"],
                              zr=(0.05, case["zmax"]), npix=case["npix"], seed=seed,
                              mass=case["mass"], device=DEV, sample=sample)


def prepare(case, seed):
    kind, ctx = case["kind"], _ctx()
    st = {"kind": kind, "ctx": ctx}
    if kind == "records":
        st["g"] = api.geom(case["nx"], case["ny"], -0.01, -0.01, 2e-5)
        st["rec"], st["select"] = _records(case, seed), case["select"]
        st["maps"] = api.Maps.zeros(st["g"], DEV)
    elif kind == "cone":
        lc = _cone(case, seed)
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
        h = lc.halos
        st.update(parts=lc.parts, Mp=lc.Mp, M=t(h.M), c=t(h.c), z=t(h.z), pos=t(h.pos),
                  thx=t(h.thx), thy=t(h.thy), v=t(h.vlos), dt=case["dt"])
        st["g"] = api.geom(lc.geom.nx, lc.geom.ny, lc.geom.theta0_x, lc.geom.theta0_y,
                           lc.geom.dtheta)
        st["rec"] = torch.empty((case["n"], api.ASSIGNED_STRIDE), dtype=F32, device=DEV)
        st["pp"], st["hp"] = api.Maps.zeros(st["g"], DEV), api.Maps.zeros(st["g"], DEV)
        torch.cuda.empty_cache()
    elif kind == "hp":
        half, st["g"] = _patch(case)
        st.update(_catalogue(_gen(seed), case["n"], half, (case["zmin"], 1.0), "loguniform"))
        st["model"], st["status"] = ctx.solve_halos(st["M"], st["c"], st["z"],
                                                    raise_on_noconv=False)
        st["ap"], st["dt"] = case["ap"], case["dt"]
        st["maps"] = api.Maps.zeros(st["g"], DEV)
    elif kind == "hp_batch":
        g = _gen(seed)
        half, st["g"] = _patch(case, case["maps"])
        cnt = torch.poisson(torch.full((case["maps"],), float(case["mean"]), device=DEV),
                            generator=g).long()
        st.update(_catalogue(g, int(cnt.sum()), half, (0.01, 3.0), "powerlaw"))
        st["mid"] = torch.repeat_interleave(torch.arange(case["maps"], device=DEV, dtype=I32), cnt)
        st["model"], st["status"] = ctx.solve_halos(st["M"], st["c"], st["z"],
                                                    raise_on_noconv=False)
        st["plan"] = ctx.hp_plan(st["thx"], st["thy"], st["model"], st["status"], st["g"], 0.0,
                                 st["mid"], case["tile"])
        st["maps"] = api.Maps.zeros(st["g"], DEV)
    elif kind == "allsky":
        g, n = _gen(seed), case["n"]
        M = _powerlaw(g, n)
        z0, z1 = case["zmin"], case["zmax"]
        st.update(M=M, c=_concentration(g, M),  # denser towards high redshift, as a volume is
                  z=(z0 ** 2 + _u(g, n) * (z1 ** 2 - z0 ** 2)).sqrt(),
                  theta=torch.arccos(_u(g, n, -1.0, 1.0)), phi=_u(g, n, 0.0, 2 * math.pi),
                  v=300.0 * _randn(g, n), nside=case["nside"], ap=case["ap"])
        st["model"], st["status"] = ctx.solve_halos(M, st["c"], st["z"], raise_on_noconv=False)
        st["g"] = api.healpix_geom(case["nside"])
        st["maps"] = api.healpix_maps(case["nside"], DEV)
    elif kind == "solve":
        g, n = _gen(seed), case["n"]
        M = _powerlaw(g, n)
        st.update(M=M, c=_concentration(g, M), z=_u(g, n, 0.01, case["zmax"]), gated=case["gated"])
    elif kind == "hsml":
        lc = _cone({"n": case["n"], "halos": max(25, case["n"] // 1333), "side": 2.0, "zmax": 1.5,
                    "npix": 1024, "mass": "loguniform"}, seed)
        st.update({k: lc.parts[k] for k in "xyz"}, ngb=case["ngb"],
                  guess=lc.parts["hsml"] if case["guess"] else None)
        torch.cuda.empty_cache()
    elif kind == "spectrum":
        g, nx, ny = _gen(seed), case["nx"], case["ny"]
        st["d"] = 5.0 * DEG / max(nx, ny)
        # the y map of a sky: smooth structure over pixel noise
        y = torch.arange(ny, device=DEV, dtype=F32)[:, None] / ny
        x = torch.arange(nx, device=DEV, dtype=F32)[None, :] / nx
        m = 1e-7 * torch.randn((ny, nx), generator=g, device=DEV)
        for k in range(1, 9):
            ph = float(torch.rand(1, generator=g, device=DEV)) * 2 * math.pi
            m += (1e-5 / k) * torch.cos(2 * math.pi * (k * x + (9 - k) * y) + ph)
        st["m"] = m
        st["lo"] = m * 3e-8 * torch.rand((ny, nx), generator=g, device=DEV) if case["lo"] else None
    else:
        g, n = _gen(seed), case["n"]
        p, off = torch.zeros(L.MLP_NPARAMS, device=DEV), 0
        for fin, fout in ((6, 128), (128, 128), (128, 128), (128, 3)):
            lim = math.sqrt(6.0 / (fin + fout))
            p[off:off + fin * fout] = _u(g, fin * fout, -lim, lim, F32)
            off += fin * fout
            p[off:off + fout] = _u(g, fout, -0.1, 0.1, F32)
            off += fout
        st["params"] = p
        if kind == "mlp_train":  # a step in the middle of a run: moments in place
            st["x"], st["t"] = _u(g, (n, 6), -1.0, 1.0, F32), _randn(g, (n, 3))
            st["m"] = 1e-3 * _randn(g, L.MLP_NPARAMS)
            st["v"] = 1e-5 * _u(g, L.MLP_NPARAMS, 0.5, 2.0, F32)
            st["step"] = 1000
            st["cache"] = torch.empty((n, L.MLP_CACHE_PER_ROW), device=DEV)
            st["dy"], st["grad"] = torch.empty((n, 3), device=DEV), torch.empty_like(p)
        else:
            R = I.SURROGATE_RANGES
            fm, fs = feature_norm()
            st["norm"] = torch.from_numpy(np.concatenate([fm, np.zeros(3), fs, np.ones(3)])
                                          .astype(np.float32)).to(DEV)
            M = 10.0 ** _u(g, n, *R["log10_M"])
            st.update(M=M, c=5.0 * (M / 1e14) ** -0.1 * 10.0 ** _u(g, n, *R["dlog10_c"]),
                      z=_u(g, n, *R["z"]),
                      prm=torch.stack([_u(g, n, *R[k]) for k in ("eps_star", "f_star", "eps_dm")]))
            st["wb"] = ctx.mlp_to_bf16(p)
    return st


# ------------------------------------------------------------------ one pass
def _out(st):
    return (api.OUT_DT, 150.0) if st["dt"] else (api.OUT_YB, 0.0)


def run(st):
    kind, ctx = st["kind"], st["ctx"]
    if kind == "records":
        maps = st["maps"].zero_()
        ctx.paste_particles(st["rec"], st["g"], maps, st["select"])
        ctx.finalize(st["g"], maps)
        return maps.y, maps.b
    if kind == "cone":
        pp, hp, g = st["pp"].zero_(), st["hp"].zero_(), st["g"]
        model, status = ctx.solve_halos(st["M"], st["c"], st["z"], raise_on_noconv=False)
        ctx.assign_particles(st["parts"], st["Mp"], st["pos"], model, status, g, out=st["rec"])
        ctx.paste_particles(st["rec"], g, pp)
        ctx.paste_halos(st["thx"], st["thy"], st["v"], model, status, g, hp)
        for m in (pp, hp):
            ctx.finalize(g, m, *_out(st))
        return pp.y, pp.b, hp.y, hp.b
    if kind == "hp":
        maps = st["maps"].zero_()
        ctx.paste_halos(st["thx"], st["thy"], st["v"], st["model"], st["status"], st["g"], maps,
                        ap_r500=st["ap"])
        ctx.finalize(st["g"], maps, *_out(st))
        return maps.y, maps.b
    if kind == "hp_batch":
        maps = st["maps"].zero_()
        st["plan"].execute(st["thx"], st["thy"], st["v"], st["model"], st["status"], maps,
                           st["mid"])
        ctx.finalize(st["g"], maps)
        return maps.y, maps.b
    if kind == "allsky":
        maps = st["maps"].zero_()
        ctx.paste_halos_healpix(st["theta"], st["phi"], st["v"], st["model"], st["status"],
                                st["nside"], maps, ap_r500=st["ap"])
        ctx.finalize(st["g"], maps)
        return maps.y, maps.b
    if kind == "solve":
        if st["gated"]:
            return ctx.solve_halos_ex(st["M"], st["c"], st["z"], gate=1e-4, gated=True,
                                      raise_on_noconv=False)
        return ctx.solve_halos(st["M"], st["c"], st["z"], raise_on_noconv=False)
    if kind == "hsml":
        return ctx.smoothing_lengths(st["x"], st["y"], st["z"], st["ngb"], guess=st["guess"])
    if kind == "spectrum":
        return ctx.power_spectrum(st["m"], st["d"], lo=st["lo"])
    if kind == "mlp_train":
        y, _ = ctx.mlp_forward(st["params"], st["x"], st["cache"])
        ctx.mlp_mse(y, st["t"], st["dy"], want_loss=False)
        ctx.mlp_backward(st["params"], st["x"], st["cache"], st["dy"], st["grad"])
        st["step"] += 1
        ctx.mlp_adam(st["params"], st["grad"], st["m"], st["v"], st["step"], 1e-3)
        return y, st["dy"], st["grad"], st["params"], st["m"], st["v"]
    x = ctx.mlp_features(st["M"], st["c"], st["z"], st["prm"], st["norm"])
    return ctx.mlp_infer_bf16(st["wb"], st["params"], x)


# ------------------------------------------------------------------ work a pass cannot do without
def _footprint(rec, nx, ny, select=0):
    """Sum over the records of pixel updates, both maps: a record's clipped 2h x 2h footprint in
    b, and in y where it carries one."""
    iv = rec.view(I32)
    h, kind = rec[:, 2].double(), iv[:, 5]
    size = []
    for a, n in ((0, nx), (1, ny)):
        p = iv[:, 6 + a].double() + rec[:, a].double()
        lo, hi = torch.floor(p - h).clamp(min=0), torch.floor(p + h).clamp(max=n - 1)
        size.append((hi - lo + 1).clamp(min=0))
    ok = kind != api.KIND_NONE
    if select:
        ok &= kind == (api.KIND_HALO if select == 1 else api.KIND_FIELD)
    upd = size[0] * size[1] * ok
    return float((upd * torch.where(rec[:, 3] != 0, 2.0, 1.0)).sum())


def _apertures(st):
    """Angular aperture radius of every halo [rad]."""
    rf, da = st["model"][api.MF["r_f"]], st["model"][api.MF["D_A"]]
    if st.get("ap", 0.0) > 0:
        rf = torch.minimum(rf, st["ap"] * st["model"][api.MF["r500"]])
    return rf / da


def work(case):
    kind = case["kind"]
    if kind == "records":
        npx = case["nx"] * case["ny"]
        upd = _footprint(_records(case, 0), case["nx"], case["ny"], case["select"])
        return {"bytes": 32 * case["n"] + 8 * npx, "flops": 2 * upd}
    if kind == "cone":
        # footprints from a sample of the cone's own particles, at its smoothing lengths
        f = min(1.0, 2e5 / case["n"])
        lc = _cone(case, 0, None if f == 1.0 else (1.0 if case["halos"] < 400 else max(f, 0.02), f))
        p = lc.parts
        chi = (p["x"].double() ** 2 + p["y"].double() ** 2 + p["z"].double() ** 2).sqrt()
        w = 2.0 * p["hsml"].double() / chi / lc.geom.dtheta + 1.0
        area = w.clamp(max=case["npix"]) ** 2
        halo = p["hid"] >= 0
        upd = 0.6 * 2 * float(area[halo].mean()) + 0.4 * float(area[~halo].mean())
        return {"bytes": 32 * case["n"] + 16 * case["npix"] ** 2, "flops": 2 * upd * case["n"]}
    if kind in ("hp", "hp_batch"):
        st = prepare(case, 0)
        ang, d = _apertures(st), st["g"].dtheta
        side = case["npix"] * d
        fx = ((st["thx"] + ang).clamp(max=side / 2) - (st["thx"] - ang).clamp(min=-side / 2))
        fy = ((st["thy"] + ang).clamp(max=side / 2) - (st["thy"] - ang).clamp(min=-side / 2))
        pix = float(torch.nan_to_num(math.pi / 4 * fx * fy / d ** 2).sum())
        n, npx = st["M"].numel(), case.get("maps", 1) * case["npix"] ** 2
        return {"bytes": n * (16 + 4 + 10 * 8) + 8 * npx, "flops": 20 * pix}
    if kind == "allsky":
        st = prepare(case, 0)
        npx = 12 * case["nside"] ** 2
        pix = float(torch.nan_to_num(_apertures(st) ** 2 * (npx / 4.0)).sum())
        return {"bytes": case["n"] * (16 + 4 + 10 * 8) + 8 * npx, "flops": 60 * pix}
    if kind == "solve":  # two FP64 evaluations of 64-point integrals of the profiles per halo
        return {"bytes": case["n"] * (3 * 8 + 24 * 8 + 4), "flops": case["n"] * 2 * 64 * 60}
    if kind == "hsml":  # three kernel sums over the ~3 N_ngb particles inside h
        return {"bytes": 16 * case["n"], "flops": case["n"] * 3 * 3 * case["ngb"] * 15}
    if kind == "spectrum":  # a real-input transform
        n = case["nx"] * case["ny"]
        return {"bytes": n * (8 if case["lo"] else 4), "flops": 2.5 * n * math.log2(n)}
    nw = 6 * 128 + 2 * 128 * 128 + 3 * 128
    if kind == "mlp_train":
        return {"bytes": 4 * (case["n"] * 12 + 8 * L.MLP_NPARAMS), "flops": 6 * nw * case["n"]}
    return {"bytes": case["n"] * (6 * 8 + 12), "flops": 2 * nw * case["n"]}


# ------------------------------------------------------------------ the same in 64 bits
def _w64(u):
    """The normalised kernel integrated to u = dx / h from the left: 0 at -1, 1 at 1."""
    a = u.abs().clamp(max=1.0)
    wl = torch.where(a < 0.5, 0.5 - 4.0 / 3.0 * a + 8.0 / 3.0 * a ** 3 - 2.0 * a ** 4,
                     2.0 / 3.0 * (1.0 - a) ** 4)
    return torch.where(u < 0, wl, 1.0 - wl)


def _deposit64(rec, nx, ny, select):
    """Both maps of the records in FP64: outer products of the axes' pixel integrals."""
    iv = rec.view(I32)
    kind = iv[:, 5]
    ok = kind != api.KIND_NONE
    if select:
        ok = ok & (kind == (api.KIND_HALO if select == 1 else api.KIND_FIELD))
    rec, iv = rec[ok], iv[ok]
    f = rec[:, :2].double()
    h = rec[:, 2].double()
    cell = iv[:, 6:8].long()
    first = torch.floor(f - h[:, None]).long()  # first covered pixel, relative to the particle's
    wide = (torch.floor(f + h[:, None]).long() - first + 1).amax(1)
    out = torch.zeros((2, ny * nx), dtype=F64, device=DEV)
    size = 2
    while True:
        sel = torch.nonzero((wide <= size) & (wide > (0 if size == 2 else size // 2))).ravel()
        step = max(1, 40_000_000 // (size * size))
        for k in range(0, sel.numel(), step):
            s = sel[k:k + step]
            j = torch.arange(size, device=DEV)
            ws, idx, ins = [], [], []
            for a, n in ((0, nx), (1, ny)):
                rel = first[s, a, None] + j
                lo = rel.double() - f[s, a, None]
                hh = h[s, None]
                w = torch.where(hh > 0, _w64((lo + 1.0) / hh) - _w64(lo / hh),
                                (rel == 0).double())
                p = cell[s, a, None] + rel
                inside = (p >= 0) & (p < n)
                ws.append(torch.where(inside, torch.nan_to_num(w), torch.zeros_like(w)))
                idx.append(p.clamp(0, n - 1))
                ins.append(inside)
            flat = (idx[1][:, :, None] * nx + idx[0][:, None, :]).reshape(-1)
            for m, col in ((0, 3), (1, 4)):
                v = rec[s, col].double()[:, None, None] * ws[1][:, :, None] * ws[0][:, None, :]
                out[m].index_add_(0, flat, v.reshape(-1))
        if size >= int(wide.max()):
            break
        size *= 2
    return out.reshape(2, 1, ny, nx)


# physical constants (CODATA 2018 / IAU 2015), in Msun, Mpc, km/s
_MSUN, _MPC, _C = 1.98840987e30, 3.0856775814913673e22, 299792.458
_G = 6.67430e-11 * _MSUN / (_MPC * 1e6)
_SIG, _MEC2, _MP = 6.6524587321e-29, 8.1871057769e-14, 1.67262192369e-27
_XH, _N, _NNT = 0.76, 5.0, 0.8  # hydrogen fraction, 1 / (Gamma - 1), non-thermal slope


def _line_of_sight64(model, k, rp):
    """y and b / (v / c) of halos k at projected radii rp [Mpc] (inside r_f): the polytrope
    integrated along the line of sight, split at r_vir."""
    m = {n: model[api.MF[n]][k][:, None] for n in ("Mvir", "r_s", "r_vir", "m_c", "Phi0", "r500",
                                                   "T", "rho0", "P0", "r_f", "A_nt", "tau")}
    t, w = np.polynomial.legendre.leggauss(40)
    t = torch.from_numpy(0.5 * (t + 1.0)).to(DEV)
    w = torch.from_numpy(0.5 * w).to(DEV)
    rp = rp[:, None]
    # the non-thermal cut 1 - A_nt (r / r500)^n_nt = 0 is a kink as well
    r_nt = m["r500"] * (1.0 / m["A_nt"]) ** (1.0 / _NNT)
    ends = [(torch.clamp(torch.minimum(r, m["r_f"]) ** 2 - rp ** 2, min=0.0)).sqrt()
            for r in (torch.minimum(m["r_vir"], r_nt), torch.maximum(m["r_vir"], r_nt), m["r_f"])]
    P = torch.zeros_like(rp[:, 0])
    R = torch.zeros_like(P)
    a = torch.zeros_like(rp)
    for b in ends:
        # nodes bunched at the lower end, where the profile is steep for small rp
        q = t[None, :] ** 2
        l = a + (b - a) * q
        r = (l * l + rp * rp).sqrt()
        x = r / m["r_s"]
        n1T = (_N + 1.0) * m["T"]
        inner = 1.0 - _G * m["Mvir"] / (m["m_c"] * m["r_s"] * n1T) * (1.0 - torch.log1p(x) / x)
        outer = 1.0 + m["Phi0"] / n1T + _G * m["Mvir"] / (r * n1T)
        th = torch.where(r <= m["r_vir"], inner, outer).clamp(min=0.0)
        nt = (1.0 - m["A_nt"] * (r / m["r500"]) ** _NNT).clamp(min=0.0)
        jac = (b - a) * 2.0 * t[None, :] * w[None, :]
        P += 2.0 * (jac * th ** (_N + 1.0) * nt).sum(1)
        R += 2.0 * (jac * th ** _N).sum(1)
        a = b
    pe = (2.0 * _XH + 2.0) / (5.0 * _XH + 3.0)
    # pressure Msun (km/s)^2 Mpc^-3 x Mpc, density Msun Mpc^-3 x Mpc
    y = _SIG / _MEC2 * pe * m["P0"][:, 0] * P * _MSUN * 1e6 / _MPC ** 2
    ne = m["rho0"][:, 0] * R * _MSUN / (_MP * 2.0 / (1.0 + _XH)) / _MPC ** 2
    return y, _SIG * ne * torch.exp(-m["tau"][:, 0])


def _halos64(st, npix, n_maps, chunk=400_000):
    """Flat halo maps in FP64: the projected profiles at every pixel centre of every aperture."""
    g, model = st["g"], st["model"]
    rap = model[api.MF["r_f"]]
    if st.get("ap", 0.0) > 0:
        rap = torch.minimum(rap, st["ap"] * model[api.MF["r500"]])
    ok = st["status"] == 0
    r = rap / model[api.MF["D_A"]] / g.dtheta
    cx = (st["thx"] - g.theta0_x) / g.dtheta - 0.5
    cy = (st["thy"] - g.theta0_y) / g.dtheta - 0.5
    box = [torch.floor(cx - r).clamp(min=0), torch.floor(cx + r).clamp(max=npix - 1),
           torch.floor(cy - r).clamp(min=0), torch.floor(cy + r).clamp(max=npix - 1)]
    w = torch.where(ok, (box[1] - box[0] + 1).clamp(min=0), torch.zeros_like(r)).long()
    hgt = torch.where(ok, (box[3] - box[2] + 1).clamp(min=0), torch.zeros_like(r)).long()
    cnt = w * hgt
    total = int(cnt.sum())
    if total > 60_000_000:
        return None
    out = torch.zeros((2, n_maps * npix * npix), dtype=F64, device=DEV)
    start = torch.cumsum(cnt, 0) - cnt
    mid = st.get("mid")
    for a in range(0, total, chunk):
        e = torch.arange(a, min(total, a + chunk), device=DEV)
        k = torch.searchsorted(start + cnt, e, right=True)
        loc = e - start[k]
        i = box[0][k].long() + loc % w[k]
        j = box[2][k].long() + loc // w[k]
        rp = ((i - cx[k]) ** 2 + (j - cy[k]) ** 2).sqrt() * g.dtheta * model[api.MF["D_A"]][k]
        sel = rp < rap[k]
        k, i, j, rp = k[sel], i[sel], j[sel], rp[sel]
        y, b = _line_of_sight64(model, k, rp)
        p = (j if mid is None else mid[k].long() * npix + j) * npix + i
        out[0].index_add_(0, p, y)
        out[1].index_add_(0, p, b * st["v"][k].double() / _C)
    return out.reshape(2, n_maps, npix, npix)


def _to_dt(m, dt):
    if not dt:
        return m[0], m[1]
    x = 6.62607015e-34 * 150e9 / (1.380649e-23 * 2.726)
    return (x / math.tanh(0.5 * x) - 4.0) * m[0], -m[1]


def _ring_centres(nside):
    """Colatitude and longitude of every HEALPix pixel centre, RING order."""
    th, ph = [], []
    for i in range(1, 4 * nside):
        if i < nside or i > 3 * nside:
            q = i if i < nside else 4 * nside - i
            z = 1.0 - q * q / (3.0 * nside * nside)
            z, m, s = (z if i < nside else -z), 4 * q, 0.5
        else:
            z, m = 4.0 / 3.0 - 2.0 * i / (3.0 * nside), 4 * nside
            s = 0.5 if (i - nside) % 2 == 0 else 0.0
        th.append(torch.full((m,), math.acos(z), dtype=F64))
        ph.append((torch.arange(m, dtype=F64) + s) * (2 * math.pi / m))
    return torch.cat(th).to(DEV), torch.cat(ph).to(DEV)


def _allsky64(st, nside):
    npx, n = 12 * nside * nside, st["M"].numel()
    if npx * n > 400_000_000:
        return None
    th, ph = _ring_centres(nside)
    model = st["model"]
    rap = model[api.MF["r_f"]]
    if st["ap"] > 0:
        rap = torch.minimum(rap, st["ap"] * model[api.MF["r500"]])
    out = torch.zeros((2, npx), dtype=F64, device=DEV)
    step = max(1, 20_000_000 // npx)
    for a in range(0, n, step):
        s = slice(a, min(n, a + step))
        t0, p0 = st["theta"][s, None], st["phi"][s, None]
        hav = torch.sin(0.5 * (th - t0)) ** 2 + torch.sin(t0) * torch.sin(th) * torch.sin(
            0.5 * (ph - p0)) ** 2
        rp = 2.0 * torch.asin(hav.clamp(max=1.0).sqrt()) * model[api.MF["D_A"]][s, None]
        k, p = torch.nonzero((rp < rap[s, None]) & (st["status"][s, None] == 0), as_tuple=True)
        for b in range(0, k.numel(), 400_000):
            kk, pp = k[b:b + 400_000], p[b:b + 400_000]
            y, bb = _line_of_sight64(model, kk + a, rp[kk, pp])
            out[0].index_add_(0, pp, y)
            out[1].index_add_(0, pp, bb * st["v"][kk + a].double() / _C)
    return out.reshape(2, 1, nside, 12 * nside)


def _hsml64(st):
    """Smoothing lengths from every distance in FP64, by bisection on the sorted ones."""
    x = torch.stack([st["x"], st["y"], st["z"]], 1).double()
    n, ngb = x.shape[0], st["ngb"]
    if n > 40_000:
        return None
    keep = min(n, 2048)
    out = torch.empty(n, dtype=F64, device=DEV)
    for a in range(0, n, 512):
        d = torch.zeros((min(n, a + 512) - a, n), dtype=F64, device=DEV)
        for q in range(3):
            d += (x[a:a + 512, q, None] - x[None, :, q]) ** 2
        d = torch.topk(d, keep, dim=1, largest=False).values.sqrt()
        lo, hi = torch.zeros_like(d[:, 0]), d[:, -1].clone() if keep < n else d[:, -1] * 64 + 1e-30
        for _ in range(60):
            h = 0.5 * (lo + hi)
            u = d / h[:, None]
            w = torch.where(u < 0.5, 1.0 - 6.0 * u ** 2 + 6.0 * u ** 3, 2.0 * (1.0 - u).clamp(min=0) ** 3)
            big = 32.0 / 3.0 * w.sum(1) >= ngb
            hi = torch.where(big, h, hi)
            lo = torch.where(big, lo, h)
        out[a:a + 512] = 0.5 * (lo + hi)
        if keep < n and bool((hi >= d[:, -1] * (1 - 1e-12)).any()):
            return None  # a clump at a kernel's edge: more neighbours than were kept
    return out


def _spectrum64(st):
    m = st["m"].double() + (st["lo"].double() if st["lo"] is not None else 0.0)
    ny, nx = m.shape
    d = st["d"]
    p = torch.fft.fft2(m).abs() ** 2 * (d * d / (nx * ny))
    ky = torch.fft.fftfreq(ny, 1.0 / ny, device=DEV, dtype=F64)[:, None] * (2 * math.pi / (ny * d))
    kx = torch.fft.fftfreq(nx, 1.0 / nx, device=DEV, dtype=F64)[None, :] * (2 * math.pi / (nx * d))
    e = 10.0 ** np.linspace(2.0, 5.0, 31)
    b = torch.bucketize((kx * kx + ky * ky).reshape(-1), torch.from_numpy(e * e).to(DEV),
                        right=True) - 1
    sums = torch.zeros(32, dtype=F64, device=DEV)
    cnt = torch.zeros(32, dtype=F64, device=DEV)
    b = torch.where((b < 0) | (b > 29), torch.full_like(b, 31), b)
    sums.index_add_(0, b, p.reshape(-1))
    cnt.index_add_(0, b, torch.ones_like(p).reshape(-1))
    return np.sqrt(e[:-1] * e[1:]), (sums / cnt.clamp(min=1.0))[:30], None


def _layers(p):
    out, off = [], 0
    for fin, fout in ((6, 128), (128, 128), (128, 128), (128, 3)):
        w = p[off:off + fin * fout].reshape(fout, fin)
        off += fin * fout
        out.append((w, p[off:off + fout]))
        off += fout
    return out


def _mlp64(layers, x):
    for k, (w, b) in enumerate(layers):
        x = x @ w.T + b
        if k < 3:
            x = 0.5 * x * (1.0 + torch.erf(x / math.sqrt(2.0)))
    return x


def _train64(st):
    p = st["params"].double().clone().requires_grad_(True)
    x, t = st["x"].double(), st["t"].double()
    y = _mlp64(_layers(p), x)
    dy = 2.0 * (y - t) / y.numel()
    (grad,) = torch.autograd.grad((dy.detach() * y).sum(), p)
    k, b1, b2 = st["step"] + 1, 0.9, 0.999
    m = b1 * st["m"].double() + (1 - b1) * grad
    v = b2 * st["v"].double() + (1 - b2) * grad ** 2
    q = p.detach() - 1e-3 * (m / (1 - b1 ** k)) / ((v / (1 - b2 ** k)).sqrt() + 1e-8)
    return y.detach(), dy.detach(), grad, q, m, v


def _infer64(st):
    fm, fs = feature_norm()
    f = torch.stack([torch.log10(st["M"]), torch.log10(st["c"]), st["z"], *st["prm"]], 1)
    norm = st["norm"].double()
    x = (f - norm[:6]) / norm[9:15]
    wb = st["wb"].view(torch.bfloat16).double()
    layers, off = [], 0
    for (w, b) in _layers(st["params"].double()):
        layers.append((wb[off:off + w.numel()].reshape(w.shape), b))
        off += w.numel()
    return torch.cat([_mlp64(layers, q) for q in x.split(500_000)])


def exact(case, seed):
    kind = case["kind"]
    if kind in ("cone", "solve"):
        return None  # a whole step, and a root solve per halo: no short 64-bit form
    if kind == "hsml" and case["n"] > 40_000:
        return None
    if kind == "allsky" and 12 * case["nside"] ** 2 * case["n"] > 400_000_000:
        return None
    if kind == "hp_batch" and case["maps"] * case["mean"] * case["npix"] ** 2 > 3e9:
        return None
    st = prepare(case, seed)
    if kind == "records":
        return tuple(_deposit64(st["rec"], case["nx"], case["ny"], case["select"]))
    if kind in ("hp", "hp_batch"):
        m = _halos64(st, case["npix"], case.get("maps", 1))
        return None if m is None else _to_dt(m, st.get("dt", False))
    if kind == "allsky":
        m = _allsky64(st, case["nside"])
        return None if m is None else (m[0], m[1])
    if kind == "hsml":
        return _hsml64(st)
    if kind == "spectrum":
        return _spectrum64(st)
    if kind == "mlp_train":
        return _train64(st)
    return _infer64(st)
