"""Workloads that stand for the use of this framework, each through its public entry points.

A case is a dict of plain values.  ``kind`` names the entry point:

step      ``casim_step``: one timestep of one domain on the device, in place
tendency  ``casim_step_tendency``: the source terms, the state left unchanged
host      ``casim_step_host``: a state in pinned host memory
batched   ``casim_step_batched``: one call for a list of uneven domains
surrogate ``casim_batch_step_surrogate``: a batch's step with the network's warm-rain rates
train     ``casim_mlp_fit``: minibatch training of that network

``config`` is the scheme's configuration: cold (16 fields), warm, aero (cold with aerosol
mass, 22 fields), warm_aero (19), tri (cold triple-moment, 20) or warm_tri (17).

The inputs follow the recipes of ``synth`` (drawn on the device).  ``exact`` computes the
same step, network and training in 64 bits with plain torch from the published formulas.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2010_14823_gb300 import casim, synth

FLAGS = {"cold": 0, "warm": casim.CASIM_WARM, "aero": casim.CASIM_AEROSOL,
         "warm_aero": casim.CASIM_WARM | casim.CASIM_AEROSOL, "tri": casim.CASIM_THREE_MOMENT,
         "warm_tri": casim.CASIM_WARM | casim.CASIM_THREE_MOMENT}
NFIELDS = {"cold": 16, "warm": 16, "aero": 22, "warm_aero": 19, "tri": 20, "warm_tri": 17}
EXTRA = {"cold": (), "warm": (), "aero": ("ma", "mac", "mar", "mai", "mas", "mag"), "warm_aero": ("ma", "mac", "mar"),
         "tri": ("zr", "zi", "zs", "zg"), "warm_tri": ("zr",)}
PROG = synth.FIELDS[:synth.NPROG]
DEV = "cuda"


def _step(name, ncols, nlev, recipe="deep_convective", precision="mixed", config="cold", dt=1.0, kind="step"):
    return {"name": name, "kind": kind, "ncols": ncols, "nlev": nlev, "recipe": recipe, "precision": precision,
            "config": config, "dt": dt}


def listed():
    return [
        # the smallest domain of the benchmark's recipes: a step that a host model calls for a small patch
        _step("step_16x16x50", 256, 50, "stratus"),
        # the largest domain the paper's port could hold on its GPU
        _step("step_20000x60", 20000, 60),
        # the headline workload: deep convection, a whole GPU's domain
        _step("step_512x512x150", 262144, 150),
        # the plain FP64 form on the broken-stratus domain
        _step("fp64_256x256x100", 65536, 100, "stratus_broken", precision="fp64"),
        # a coarse model's time step: several sedimentation substeps per species and column
        _step("long_dt_256x256x100", 65536, 100, dt=10.0),
        # the liquid-water configuration on stratus
        _step("warm_512x512x150", 262144, 150, "stratus_broken", config="warm"),
        # the triple-moment scheme
        _step("three_moment_256x256x100", 65536, 100, config="tri"),
        # a parent model that integrates the source terms itself
        _step("tendency_256x256x150", 65536, 150, kind="tendency"),
        # the paper's protocol: the state lives on the host, one call per timestep
        _step("host_20000x60", 20000, 60, kind="host"),
        # many independent domains of uneven size in one call
        {"name": "batched_16_domains", "kind": "batched", "ndom": 16, "cols_lo": 1000, "cols_hi": 100000,
         "lev_lo": 40, "lev_hi": 150, "layout": 7, "precision": "mixed", "dt": 1.0},
        # serving the learned warm-rain rates over a batch
        {"name": "surrogate_4_domains", "kind": "surrogate", "ndom": 4, "cols_lo": 8000, "cols_hi": 60000,
         "lev_lo": 60, "lev_hi": 150, "layout": 3, "precision": "mixed", "dt": 1.0},
        # training the network: minibatch Adam on rows of a run
        {"name": "train_8192x32", "kind": "train", "rows": 262144, "batch": 8192, "steps": 32},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 7 + ["tendency", "host", "batched", "surrogate", "train"])
    if kind == "train":
        return {"kind": kind, "rows": _logint(rng, 20000, 400000), "batch": _logint(rng, 500, 12000),
                "steps": rng.randint(4, 32)}
    if kind in ("batched", "surrogate"):
        lo = _logint(rng, 200, 4000)
        return {"kind": kind, "ndom": rng.randint(2, 16 if kind == "batched" else 6), "cols_lo": lo,
                "cols_hi": _logint(rng, 2 * lo, 60000), "lev_lo": rng.randint(20, 60), "lev_hi": rng.randint(61, 150),
                "layout": rng.randint(0, 10 ** 6), "precision": "mixed", "dt": rng.choice([0.5, 1.0, 2.0])}
    fp64 = kind == "step" and rng.random() < 0.3
    nlev = rng.randint(30, 150)
    ncols = _logint(rng, 100, {"host": 60000, "tendency": 150000}.get(kind, 60000 if fp64 else 250000))
    config = rng.choice(["cold"] * 4 + ["warm", "warm", "aero", "tri", "warm_aero", "warm_tri"])
    dt = rng.choice([0.5, 1.0, 1.0, 1.0, 2.0, 5.0, 10.0, 30.0])
    if EXTRA[config]:
        ncols = min(ncols, 10000 if fp64 else 150000)
    if dt > 2.0:
        ncols = min(ncols, 10000 if fp64 else 80000)
    recipe = rng.choice(["stratus", "stratus_broken"] + ["deep_convective"] * 2)
    return {"kind": kind, "ncols": ncols, "nlev": nlev, "recipe": recipe, "precision": "fp64" if fp64 else "mixed",
            "config": config, "dt": dt}


# ------------------------------------------------------------------ inputs
def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


# sphere densities and mass-mean diameter ranges that turn a drawn mass into a number
_DENS = (1000.0, 1000.0, 500.0, 100.0, 400.0)
_DIAM = ((10e-6, 20e-6), (0.3e-3, 1.5e-3), (30e-6, 100e-6), (0.3e-3, 2e-3), (0.5e-3, 3e-3))


def _fields(rc: synth.Recipe, ncols, nlev, dz, config, seed):
    """The recipe's state on the device, [fields][nlev][pitch], padding columns zero (the
    distributions of ``synth.make_state``)."""
    g = _generator(seed)
    f64 = dict(dtype=torch.float64, device=DEV)
    uni = lambda lo, hi, *s: torch.rand(*s, generator=g, **f64) * (hi - lo) + lo  # noqa: E731
    z = np.cumsum(dz) - 0.5 * dz
    tm = rc.T_sfc - rc.lapse * z
    lnp = np.empty(nlev)
    lnp[0] = math.log(1e5) - 9.81 * z[0] / (287.04 * rc.T_sfc)
    for k in range(1, nlev):
        lnp[k] = lnp[k - 1] - 9.81 * (z[k] - z[k - 1]) / (287.04 * 0.5 * (tm[k] + tm[k - 1]))
    zz = torch.tensor(z, **f64)[:, None]
    shape = (nlev, ncols)
    fld = torch.zeros((NFIELDS[config], nlev, synth.pad_columns(ncols)), **f64)
    at = {n: fld[i, :, :ncols] for i, n in enumerate(synth.FIELDS + EXTRA[config])}
    T = at["T"].copy_(torch.tensor(tm, **f64)[:, None] + rc.T_noise * torch.randn(shape, generator=g, **f64))
    p = at["p"].copy_(torch.tensor(np.exp(lnp), **f64)[:, None].expand(shape))
    rho = at["rho"].copy_(p / (287.04 * T))
    cloudy = (torch.rand(ncols, generator=g, **f64) < rc.cloud_frac)[None]
    zb = uni(*rc.base_range, ncols)
    zt = torch.maximum(uni(*rc.top_range, ncols), zb + 200.0)
    inside = cloudy & (zz >= zb) & (zz <= zt)
    tc = T - 273.15
    es = 610.78 * torch.exp(17.27 * tc / (tc + 237.3))
    at["qv"].copy_(torch.where(inside, uni(*rc.rh_cloud, *shape), uni(*rc.rh_clear, *shape)) * 0.622 * es / (p - 0.378 * es))
    masks = (inside, cloudy & (zz <= zt) & (T > 268.15), cloudy & (zz >= zb) & (zz <= zt + 2000.0) & (T < 268.15),
             cloudy & (zz >= zb) & (zz <= zt + 1000.0) & (T < 273.15), cloudy & (zz >= zb) & (zz <= zt) & (T < 275.15))
    for s, x in enumerate("crisg"):
        m = torch.clamp(rc.medians[s] * torch.exp(rc.sigma_ln * torch.randn(shape, generator=g, **f64)), max=rc.q_cap[s])
        q = at["q" + x].copy_(torch.where(masks[s], m, 0.0))
        n = at["n" + x].copy_(q / (math.pi / 6.0 * _DENS[s] * uni(*_DIAM[s], *shape) ** 3))
        if "z" + x in at:   # the sixth moment of a gamma distribution of shape 0..8
            mu = uni(0.0, 8.0, *shape)
            G = (mu + 4) * (mu + 5) * (mu + 6) / ((mu + 1) * (mu + 2) * (mu + 3))
            at["z" + x].copy_(torch.where(q > 1e-14, G * (q / (math.pi / 6.0 * _DENS[s])) ** 2 / n, 0.0))
        if "ma" + x in at:  # aerosol mass held by the species
            at["ma" + x].copy_(q * uni(1e-5, 1e-4, *shape))
    at["na"].copy_(rc.na_cm3 * 1e6 / rho)
    at["w"].copy_(uni(-rc.w_max, rc.w_max, *shape))
    if "ma" in at:
        at["ma"].copy_(uni(1e-9, 5e-9, *shape))
    return fld


def _dz(case):
    return synth.dz_uniform(case["nlev"]) if case["recipe"] == "stratus" else synth.dz_stretched(case["nlev"])


def _domains(case, seed):
    """(recipe, columns, levels, dz, seed) of each domain of a batch; sizes from the case alone."""
    r = np.random.default_rng(case["layout"])
    out = []
    for i in range(case["ndom"]):
        nc = int(round(math.exp(r.uniform(math.log(case["cols_lo"]), math.log(case["cols_hi"])))))
        nl = int(r.integers(case["lev_lo"], case["lev_hi"] + 1))
        if case["kind"] == "surrogate":
            rc = synth.RECIPES["deep_convective"]
        else:
            rc = synth.Recipe(cloud_frac=float(r.uniform(0.05, 0.60)), base_range=(500.0, 2000.0), top_range=(2000.0, 4000.0))
        out.append((rc, nc, nl, synth.dz_stretched(nl), 1000 * seed + i))
    return out


# mean, standard deviation and range of the network's 12 inputs and of its 4 log-rates on
# deep-convection rows (qc, qr, nc, nr, rho, T - T0, p, qv, w, na in the order of the inputs)
_FEAT_MEAN = (-16.2, -15.1, 12.8, 2.6, -0.065, 3.9, 11.22, -5.07, 0.0, 16.8, 0.66, 0.75)
_FEAT_SD = (11.5, 10.1, 9.2, 5.7, 0.21, 13.5, 0.26, 0.72, 5.8, 2.9, 0.47, 0.44)
_RATE_MEAN = (-22.0, -16.0, 7.0, -2.5)
_RATE_SD = (3.0, 1.8, 2.2, 1.7)


def _weights(seed):
    """Xavier-uniform weights and small biases, flat in the header's order."""
    g = torch.Generator().manual_seed(seed)
    parts = []
    for k, n in ((12, 256), (256, 256), (256, 256), (256, 4)):
        a = math.sqrt(6.0 / (k + n))
        parts += [(torch.rand(k * n, generator=g) * 2 - 1) * a, (torch.rand(n, generator=g) * 2 - 1) * 0.1]
    return torch.cat(parts).numpy().astype(np.float32)


def _stats():
    lo = [m - 5.0 * s for m, s in zip(_FEAT_MEAN, _FEAT_SD)]
    hi = [m + 5.0 * s for m, s in zip(_FEAT_MEAN, _FEAT_SD)]
    lo[8], hi[8] = -9.5, 9.5   # updraughts beyond those of the training rows take the scheme's rates
    return np.array(list(_FEAT_MEAN) + list(_FEAT_SD) + list(_RATE_MEAN) + list(_RATE_SD) + lo + hi, dtype=np.float32)


def _rows(case, seed):
    """Training rows: inputs of the ranges above, the scheme's log-rates of them, their masks."""
    g = _generator(seed)
    n = case["rows"]
    f64 = dict(dtype=torch.float64, device=DEV)
    nrm = lambda m, s: m + s * torch.randn(n, generator=g, **f64)  # noqa: E731
    hc = torch.rand(n, generator=g, **f64) < 0.9
    hr = (torch.rand(n, generator=g, **f64) < 0.7) | ~hc
    lqc, lqr = torch.where(hc, nrm(-8.4, 1.0), math.log(1e-14)), torch.where(hr, nrm(-9.3, 1.0), math.log(1e-14))
    lnc, lnr = torch.where(hc, lqc + nrm(26.6, 0.5), 0.0), torch.where(hr, lqr + nrm(15.0, 1.0), math.log(1e-3))
    z = torch.rand(n, generator=g, **f64) * 9.0
    lrho, tc = 0.17 - 0.1 * z, 19.5 - 6.5 * z + 0.5 * torch.randn(n, generator=g, **f64)
    lp, lqv = 11.51 - 0.12 * z, -4.2 - 0.42 * z
    w = torch.rand(n, generator=g, **f64) * 20.0 - 10.0
    lna = nrm(18.0, 0.6)
    X = torch.stack([lqc, lqr, lnc, lnr, lrho, tc, lp, lqv, w, lna, hc.double(), hr.double()], 1).float()
    lncc = torch.clamp(lrho + lnc + math.log(1e-6), min=0.0)
    Y = torch.stack([math.log(1350.0) + 2.47 * lqc - 1.79 * lncc, math.log(67.0) + 1.15 * (lqc + lqr),
                     math.log(9.44e9 * 1.5) + lrho + 2 * lqc, math.log(5.78) + lrho + lnr + lqr], 1)
    M = torch.stack([hc, hc & hr, hc, hr], 1)
    return X.contiguous(), torch.where(M, Y, 0.0).float().contiguous(), M.float().contiguous()


# ------------------------------------------------------------ the program
class _State:
    """What a user's program holds between calls; gives the handles back."""
    ctx = mlp = batch = None

    def __del__(self):
        if self.batch:
            casim.casim_batch_free(self.batch)
        if self.mlp:
            casim.casim_mlp_free(self.mlp)
        if self.ctx:
            casim.casim_free(self.ctx)


def _views(fld, precip, config):
    out = {n: fld[i] for i, n in enumerate(PROG)}
    out.update({n: fld[16 + i] for i, n in enumerate(EXTRA[config])})
    for x in range(precip.shape[0]):
        out["precip%d" % x] = precip[x]
    return out


def _batch_views(doms):
    return [{"T": f[0], "mass": f[1:7], "number": f[7:13], "precip": p} for f, p in doms]


def _nprecip(config):
    return 5 if "aero" in config else 4


def prepare(case, seed):
    s = _State()
    s.case, kind = case, case["kind"]
    if kind == "train":
        s.mlp = casim.casim_mlp_create(seed)
        casim.casim_mlp_set_params(s.mlp, _weights(seed))
        s.X, s.Y, s.M = _rows(case, seed)
        return s
    prec = casim.CASIM_FP64 if case["precision"] == "fp64" else casim.CASIM_MIXED
    config = case.get("config", "cold")
    s.ctx = casim.casim_init(precision=prec, flags=FLAGS[config])
    s.dt = case["dt"]
    if kind in ("batched", "surrogate"):
        s.keep, s.states, s.ncols, s.nlev = [], [], [], []
        for rc, nc, nl, dz, sd in _domains(case, seed):
            fld = _fields(rc, nc, nl, dz, "cold", sd)
            pr, dzt = torch.zeros((4, fld.shape[2]), dtype=torch.float64, device=DEV), torch.tensor(dz, device=DEV)
            s.keep.append((fld, pr, dzt))
            s.states.append(casim.make_state(fld, fld.shape[2], dzt, pr))
            s.ncols.append(nc)
            s.nlev.append(nl)
        s.out = _batch_views([k[:2] for k in s.keep])
        if kind == "surrogate":
            s.mlp = casim.casim_mlp_create(seed)
            casim.casim_mlp_set_params(s.mlp, _weights(seed))
            casim.casim_mlp_set_norm(s.mlp, _stats())
            s.batch = casim.casim_batch_create(s.ctx, s.states, s.ncols, s.nlev)
        return s
    dz = _dz(case)
    fld = _fields(synth.RECIPES[case["recipe"]], case["ncols"], case["nlev"], dz, config, seed)
    s.ncols, s.nlev, pitch = case["ncols"], case["nlev"], fld.shape[2]
    if kind == "host":
        s.fld = torch.empty(fld.shape, dtype=torch.float64, pin_memory=True).copy_(fld)
        s.precip = torch.zeros((_nprecip(config), pitch), dtype=torch.float64, pin_memory=True)
        s.dz = torch.tensor(dz).pin_memory()
    else:
        s.fld, s.dz = fld, torch.tensor(dz, device=DEV)
        s.precip = torch.zeros((_nprecip(config), pitch), dtype=torch.float64, device=DEV)
    s.state = casim.make_state(s.fld, pitch, s.dz, s.precip)
    if kind == "tendency":
        s.tend = torch.zeros((fld.shape[0] - 3,) + tuple(fld.shape[1:]), dtype=torch.float64, device=DEV)
        s.out = {n: s.tend[i] for i, n in enumerate(PROG + EXTRA[config])}
    else:
        s.out = _views(s.fld, s.precip, config)
    return s


def run(s):
    kind = s.case["kind"]
    if kind == "step":
        casim.casim_step(s.ctx, s.state, s.ncols, s.nlev, s.dt)
    elif kind == "tendency":
        casim.casim_step_tendency(s.ctx, s.state, s.ncols, s.nlev, s.dt, s.tend)
    elif kind == "host":
        casim.casim_step_host(s.ctx, s.state, s.ncols, s.nlev, s.dt)
    elif kind == "batched":
        casim.casim_step_batched(s.ctx, s.states, s.ncols, s.nlev, s.dt)
    elif kind == "surrogate":
        casim.casim_batch_step_surrogate(s.ctx, s.batch, s.mlp, s.dt)
    else:
        c = s.case
        loss = casim.casim_mlp_fit(s.mlp, s.X, s.Y, s.M, c["rows"], c["steps"], c["batch"], 1e-3, 11)
        return {"loss": loss, "params": casim.casim_mlp_get_params(s.mlp)}
    return s.out


_NET_FLOP = 2 * (12 * 256 + 2 * 256 * 256 + 256 * 4)   # per row


def work(case):
    kind = case["kind"]
    if kind == "train":
        n = case["batch"] * case["steps"]
        return {"bytes": 20 * 4.0 * n, "flops": 3.0 * _NET_FLOP * n}
    if kind in ("batched", "surrogate"):
        pts = sum(nc * nl for _, nc, nl, _, _ in _domains(case, 0))
        # the network serves about half of the points
        return {"bytes": 232.0 * pts, "flops": 600.0 * pts + (0.5 * _NET_FLOP * pts if kind == "surrogate" else 0.0)}
    pts, extra = case["ncols"] * case["nlev"], len(EXTRA[case["config"]])
    fields = (10 + 7 if case["config"].startswith("warm") else 16 + 13) + 2 * extra
    return {"bytes": 8.0 * fields * pts, "flops": (1200.0 if "tri" in case["config"] else 600.0) * pts}


# ------------------------------------------- the scheme in 64 bits (plain torch)
T0, CP, LV, LF, RD, RV, GRAV, RHOW, RHO0 = 273.15, 1005.0, 2.5e6, 3.34e5, 287.04, 461.5, 9.81, 1000.0, 1.2
LS, EPS, KA, DV, MUAIR, QMIN, TNUC, MI0, RR0 = LV + LF, RD / RV, 2.4e-2, 2.26e-5, 1.72e-5, 1e-14, 268.15, 1e-12, 25e-6
SURFT, MW, MAIR, RGAS, LNS = 0.0761, 0.018015, 0.028965, 8.314, math.log(1.5)
# r, i, s, g: m = a D^3, shape, V = cv D^dv, cap, diameter bounds, capacitance / D
_PI6 = math.pi / 6.0
SPECIES = {"r": (_PI6 * 1000.0, 0.0, 130.0, 0.5, 10.0, 50e-6, 5e-3, 0.5),
           "i": (_PI6 * 500.0, 0.0, 700.0, 1.0, 2.0, 1e-6, 500e-6, 0.5),
           "s": (_PI6 * 100.0, 0.0, 11.72, 0.41, 4.0, 10e-6, 5e-3, 1.0 / math.pi),
           "g": (_PI6 * 400.0, 0.5, 19.3, 0.37, 10.0, 10e-6, 5e-3, 0.5)}


def _es_liq(T):
    return 611.2 * torch.exp(17.67 * (T - T0) / (T - T0 + 243.5))


def _es_ice(T):
    return 610.78 * torch.exp(21.875 * (T - 273.16) / (T - 7.66))


def _qsat(es, p):
    return EPS * es / (p - (1.0 - EPS) * es)


def _gamma_ratio(x, y):
    """Gamma(x) / Gamma(y), for tensors or numbers."""
    if isinstance(x, torch.Tensor):
        return torch.exp(torch.lgamma(x) - torch.lgamma(y))
    return math.gamma(x) / math.gamma(y)


def _lam(x, q, n, mu):
    a, _, _, _, _, dmin, dmax, _ = SPECIES[x]
    lam = (a * _gamma_ratio(mu + 4.0, mu + 1.0) * torch.clamp(n, min=0.0) / q) ** (1.0 / 3.0)
    lo, hi = (mu + 1.0) / dmax, (mu + 1.0) / dmin
    if isinstance(mu, torch.Tensor):
        return torch.minimum(torch.maximum(lam, lo), hi)
    return torch.clamp(lam, lo, hi)


def _moment(x, rho, q, lam, k, mu):
    return rho * q / SPECIES[x][0] * _gamma_ratio(mu + k + 1.0, mu + 4.0) * lam ** (3.0 - k)


def _vent(x, rho, q, lam, mu):
    nu = MUAIR / rho
    vf = SPECIES[x][2] * (RHO0 / rho) ** 0.4
    return 0.78 * _moment(x, rho, q, lam, 1.0, mu) + 0.31 * (nu / DV) ** (1.0 / 3.0) * torch.sqrt(vf / nu) * _moment(
        x, rho, q, lam, 0.5 * (SPECIES[x][3] + 3.0), mu)


def _speed(x, rho, lam, mu, k):
    _, _, cv, dv, vmax, _, _, _ = SPECIES[x]
    return torch.clamp(cv * (RHO0 / rho) ** 0.4 * _gamma_ratio(mu + k + dv + 1.0, mu + k + 1.0) * lam ** -dv, max=vmax)


def _shape(x, q, n, z):
    ok = (q > QMIN) & (n > 0.0) & (z > 0.0)
    G = torch.where(ok, z * n / (q / SPECIES[x][0]) ** 2, 2.0)
    g, lg = G ** (1.0 / 3.0), torch.log(G)
    mu = torch.clamp(torch.where(g > 1.0, (5.0 - 2.0 * g) / (g - 1.0), 20.0), 0.0, 20.0)
    for _ in range(4):
        f = sum(torch.log(mu + j) for j in (4, 5, 6)) - sum(torch.log(mu + j) for j in (1, 2, 3)) - lg
        fp = sum(1.0 / (mu + j) for j in (4, 5, 6)) - sum(1.0 / (mu + j) for j in (1, 2, 3))
        mu = torch.clamp(mu - f / fp, 0.0, 20.0)
    return torch.where(ok, mu, SPECIES[x][1])


def _activated(N, w, T, p):
    es = _es_liq(T)
    alpha = GRAV * MW * LV / (CP * RGAS * T * T) - GRAV * MAIR / (RGAS * T)
    gam = RGAS * T / (es * MW) + MW * LV * LV / (CP * p * MAIR * T)
    G = 1.0 / (RHOW * RGAS * T / (es * DV * MW) + LV * RHOW / (KA * T) * (LV * MW / (RGAS * T) - 1.0))
    A = 2.0 * SURFT * MW / (RHOW * RGAS * T)
    sm = 2.0 / math.sqrt(0.61) * (A / 1.5e-7) ** 1.5
    awg = alpha * w / G
    zeta = 2.0 * A / 3.0 * torch.sqrt(awg)
    eta = awg ** 1.5 / (2.0 * math.pi * RHOW * gam * N)
    total = (0.5 * math.exp(2.5 * LNS * LNS) * (zeta / eta) ** 1.5 + (1.0 + 0.25 * LNS) * (sm * sm / (eta + 3.0 * zeta)) ** 0.75)
    return 0.5 * N * torch.erfc(2.0 * torch.log(sm * torch.sqrt(total / (sm * sm))) / (3.0 * math.sqrt(2.0) * LNS))


def _adjust(v):
    """Saturation adjustment and activation, in place."""
    T, qv, qc, p = v["T"].clone(), v["qv"].clone(), v["qc"].clone(), v["p"]
    on = (qv > _qsat(_es_liq(T), p)) | (qc > QMIN)
    Tn = T.clone()
    for _ in range(4):
        es, tc = _es_liq(Tn), Tn - T0
        den = p - (1.0 - EPS) * es
        slope = EPS * p / (den * den) * es * 17.67 * 243.5 / ((tc + 243.5) * (tc + 243.5))
        Tn = Tn - ((Tn - T) - LV / CP * (qv - _qsat(es, p))) / (1.0 + LV / CP * slope)
    dq = torch.where(on, torch.maximum(CP / LV * (Tn - T), -qc), 0.0)
    v["T"], v["qv"], v["qc"] = T + LV / CP * dq, qv - dq, qc + dq
    N = v["rho"] * (v["na"] + v["nc"])
    on = (v["w"] > 0.0) & (v["qc"] > QMIN) & (N > 0.0)
    act = _activated(torch.where(on, N, 1e8), torch.where(on, v["w"], 1.0), v["T"], p)
    dn = torch.where(on, torch.minimum(torch.clamp(act / v["rho"] - v["nc"], min=0.0), v["na"]), 0.0)
    v["nc"], v["na"] = v["nc"] + dn, v["na"] - dn
    return dn


def _features(v):
    ln = lambda x, lo: torch.log(torch.clamp(x, min=lo))  # noqa: E731
    return torch.stack([ln(v["qc"], QMIN), ln(v["qr"], QMIN), ln(v["nc"], 1.0), ln(v["nr"], 1e-3), torch.log(v["rho"]),
                        v["T"] - T0, torch.log(v["p"]), ln(v["qv"], 1e-10), v["w"], ln(v["na"], 1.0),
                        (v["qc"] > QMIN).double(), (v["qr"] > QMIN).double()], -1)


def _layers(theta):
    at, out = 0, []
    for k, n in ((12, 256), (256, 256), (256, 256), (256, 4)):
        out.append((theta[at:at + k * n].reshape(k, n), theta[at + k * n:at + k * n + n]))
        at += k * n + n
    return out


def _net(layers, X):
    for W, b in layers[:-1]:
        X = torch.tanh(X @ W + b)
    return X @ layers[-1][0] + layers[-1][1]


def _network_rates(v, r, net):
    """The network's four rates where the inputs lie in its box."""
    layers, st = net
    F = _features(v)
    hc, hr = v["qc"] > QMIN, v["qr"] > QMIN
    use = (hc | hr) & ((F >= st[32:44]) & (F <= st[44:56])).all(-1)
    Y = torch.exp(_net(layers, (F[use] - st[:12]) / st[12:24]) * st[28:32] + st[24:28])
    for j, (name, on) in enumerate((("aut", hc), ("acc", hc & hr), ("scc", hc), ("scr", hr))):
        y = torch.zeros_like(v["T"])
        y[use] = Y[:, j]
        r[name] = torch.where(use & on, y, r[name])


def _processes(v, dt, warm, shapes, net=None):
    """Adjustment, activation, rates, limiter and update of every point, in place; returns the
    amounts the aerosol masses and the sixth moments follow."""
    rec = {"qc0": v["qc"].clone(), "na0": v["na"].clone()}
    rec["dn_act"] = _adjust(v)
    T, p, rho, qv, qc, qr, nc, nr = (v[k] for k in ("T", "p", "rho", "qv", "qc", "qr", "nc", "nr"))
    rec["evap"] = torch.clamp(rec["qc0"] - qc, min=0.0)
    rec["qc"], rec["qr"] = qc, qr
    zero = torch.zeros_like(T)
    esl = _es_liq(T)
    Sw = qv / _qsat(esl, p)
    hc, hr = qc > QMIN, qr > QMIN
    q1 = torch.where(hc, qc, 1.0)
    r = {"aut": torch.where(hc, 1350.0 * q1 ** 2.47 * torch.clamp(rho * nc * 1e-6, min=1.0) ** -1.79, zero),
         "scc": torch.where(hc, 9.44e9 * 1.5 * rho * qc * qc, zero),
         "acc": torch.where(hc & hr, 67.0 * (q1 * torch.where(hr, qr, 1.0)) ** 1.15, zero),
         "scr": torch.where(hr, 5.78 * rho * torch.clamp(nr, min=0.0) * qr, zero)}
    safe = torch.where(hr, qr, 1e-5)
    Aw, Bw = LV * LV / (KA * RV * T * T), RV * T / (esl * DV)
    iv = _vent("r", rho, safe, _lam("r", safe, nr, shapes["r"]), shapes["r"])
    r["evr"] = torch.where(hr & (Sw < 1.0), 2.0 * math.pi * (1.0 - Sw) * iv / (rho * (Aw + Bw)), zero)
    ice = () if warm else ("i", "s", "g")
    r["nuc"] = zero
    if not warm:
        esi = _es_ice(T)
        Si = qv / _qsat(esi, p)
        Ai, Bi = LS * LS / (KA * RV * T * T), RV * T / (esi * DV)
        dn = 1e3 * torch.exp(-0.639 + 12.96 * (Si - 1.0)) / rho - v["ni"]
        r["nuc"] = torch.where((T < TNUC) & (Si > 1.0) & (dn > 0.0), dn / dt, zero)
        for x in ice:
            q, has, mu = v["q" + x], v["q" + x] > QMIN, shapes[x]
            safe = torch.where(has, q, 1e-5)
            lam = _lam(x, safe, v["n" + x], mu)
            iv, cap = _vent(x, rho, safe, lam, mu), 4.0 * math.pi * SPECIES[x][7]
            r["dep" + x] = torch.where(has & (T < T0), cap * (Si - 1.0) * iv / (rho * (Ai + Bi)), zero)
            r["mlt" + x] = torch.where(has & (T > T0), cap * KA * (T - T0) * iv / (rho * LF), zero)
            if x != "i":
                vf = SPECIES[x][2] * (RHO0 / rho) ** 0.4
                r["rim" + x] = torch.where(has & (T < T0) & hc, 0.25 * math.pi * qc * vf * _moment(
                    x, rho, safe, lam, 2.0 + SPECIES[x][3], mu), zero)
    if net is not None:
        _network_rates(v, r, net)
    ratio = {x: torch.where(v["q" + x] > QMIN, torch.clamp(v["n" + x], min=0.0) / torch.where(
        v["q" + x] > QMIN, v["q" + x], 1.0), zero) for x in ("c", "r") + ice}
    mr0 = 4.0 / 3.0 * math.pi * RHOW * RR0 ** 3
    # (name, mass rate, from, to, number pool, number sink, number destination, number source, heat)
    tr = [("aut", r["aut"], "qc", "qr", "nc", r["aut"] * ratio["c"], "nr", r["aut"] / mr0, 0.0),
          ("acc", r["acc"], "qc", "qr", "nc", r["acc"] * ratio["c"], None, zero, 0.0),
          ("scc", zero, None, None, "nc", r["scc"], None, zero, 0.0),
          ("scr", zero, None, None, "nr", r["scr"], None, zero, 0.0),
          ("evr", r["evr"], "qr", "qv", "nr", r["evr"] * ratio["r"], None, zero, -LV)]
    if not warm:
        tr.append(("nuc", r["nuc"] * MI0, "qv", "qi", None, zero, "ni", r["nuc"], LS))
        for x in ice:
            d = r["dep" + x]
            tr.append(("dep" + x, torch.clamp(d, min=0.0), "qv", "q" + x, None, zero, None, zero, LS))
            s = torch.clamp(-d, min=0.0)
            tr.append(("sub" + x, s, "q" + x, "qv", "n" + x, s * ratio[x], None, zero, -LS))
        for x in ("s", "g"):
            tr.append(("rim" + x, r["rim" + x], "qc", "qg", "nc", r["rim" + x] * ratio["c"], None, zero, LF))
        for x in ice:
            m = r["mlt" + x]
            tr.append(("mlt" + x, m, "q" + x, "qr", "n" + x, m * ratio[x], "nr", m * ratio[x], -LF))
    sink = {}
    for _, m, src, _, npool, nsink, _, _, _ in tr:
        for pool, s in ((src, m), (npool, nsink)):
            if pool:
                sink[pool] = sink.get(pool, zero) + s
    f = {k: torch.where(s * dt > v[k], torch.clamp(v[k], min=0.0) / torch.where(s > 0.0, s * dt, 1.0), 1.0)
         for k, s in sink.items()}
    for name, m, src, dst, npool, nsink, ndst, nsrc, heat in tr:
        g = torch.ones_like(T)
        if src:
            g = torch.where(m > 0.0, torch.minimum(g, f[src]), g)
        if npool:
            g = torch.where(nsink > 0.0, torch.minimum(g, f[npool]), g)
        tau, nadd = g * m * dt, g * nsrc * dt
        if src:
            v[src], v[dst], v["T"] = v[src] - tau, v[dst] + tau, v["T"] + tau * heat / CP
        if npool:
            v[npool] = v[npool] - g * nsink * dt
        if ndst:
            v[ndst] = v[ndst] + nadd
        rec[name], rec["n_" + name] = tau, nadd
    return rec


def _aerosol(v, rec, q0, warm):
    """Aerosol mass moves with the water."""
    frac = lambda s, q: torch.where((s > 0.0) & (q > 0.0), torch.clamp(s / torch.where(q > 0.0, q, 1.0), max=1.0), 0.0)  # noqa: E731

    def move(src, amount, *to):
        v[src] = v[src] - amount
        for dst, share in to:
            v[dst] = v[dst] + amount * share

    move("mac", v["mac"] * frac(rec["evap"], rec["qc0"]), ("ma", 1.0))
    move("ma", v["ma"] * frac(rec["dn_act"], rec["na0"]), ("mac", 1.0))
    rain = rec["aut"] + rec["acc"]
    if warm:
        move("mac", v["mac"] * frac(rain, rec["qc"]), ("mar", 1.0))
    else:
        rim = rec["rims"] + rec["rimg"]
        share = rim / torch.where(rain + rim > 0.0, rain + rim, 1.0)
        move("mac", v["mac"] * frac(rain + rim, rec["qc"]), ("mag", share), ("mar", 1.0 - share))
    move("mar", v["mar"] * frac(rec["evr"], rec["qr"]), ("ma", 1.0))
    if not warm:
        for x in ("i", "s", "g"):
            s = rec["sub" + x] + rec["mlt" + x]
            share = rec["mlt" + x] / torch.where(s > 0.0, s, 1.0)
            move("ma" + x, v["ma" + x] * frac(s, q0["q" + x]), ("mar", share), ("ma", 1.0 - share))


def _sixth_moments(v, rec, q0, warm, active):
    """Processes keep a species' shape, sources add their own sixth moment."""
    def kept(x, q, n):
        a, b, z = q0["q" + x], q0["n" + x], q0["z" + x]
        ok = (a > QMIN) & (b > 0.0) & (q > 0.0) & (n > 0.0)
        return torch.where(ok, z * (q / torch.where(ok, a, 1.0)) ** 2 * (b / torch.where(ok, n, 1.0)), 0.0)

    q, n, src = v["qr"] - rec["aut"], v["nr"] - rec["n_aut"], rec["n_aut"] * (2.0 * RR0) ** 6
    for x in () if warm else ("i", "s", "g"):
        m, nm = rec["mlt" + x], rec["n_mlt" + x]
        q, n = q - m, n - nm
        has = (m > 0.0) & (q0["q" + x] > QMIN)
        src = src + torch.where(has, (SPECIES[x][0] / SPECIES["r"][0]) ** 2 * m / torch.where(has, q0["q" + x], 1.0), 0.0) * q0["z" + x]
        first = x == "i"
        z = kept(x, v["q" + x] - (rec["nuc"] if first else 0.0), v["n" + x] - (rec["n_nuc"] if first else 0.0))
        v["z" + x] = torch.where(active, z + (rec["n_nuc"] * (MI0 / SPECIES["i"][0]) ** 2 if first else 0.0), q0["z" + x])
    v["zr"] = torch.where(active, kept("r", q, n) + src, q0["zr"])


def _sediment(v, dz, dt, species, aero, tri):
    """First-order upwind sedimentation in CFL substeps per column and species; surface fluxes."""
    rho, fall = v["rho"], []
    down = lambda F: torch.cat([F[1:], torch.zeros_like(F[:1])])  # noqa: E731
    aerosol = torch.zeros_like(rho[0])
    for x in species:
        def speeds(limit):
            q, n = v["q" + x], v["n" + x]
            has = q > QMIN
            safe = torch.where(has, q, 1e-5)
            mu = _shape(x, q, n, v["z" + x]) if tri else SPECIES[x][1]
            lam = _lam(x, safe, n, mu)
            return [torch.where(has, torch.minimum(_speed(x, rho, lam, mu, k), limit), 0.0) for k in ((3.0, 0.0, 6.0) if tri else (3.0, 0.0))]
        cmax = (speeds(torch.full_like(rho, 1e30))[0] * dt / dz).amax(0)
        ns = torch.clamp(torch.ceil(cmax), 1, 64)
        dts = dt / ns
        total = torch.zeros_like(rho[0])
        for st in range(int(ns.max())):
            on = (st < ns).double() * dts
            V = speeds(dz / dts)
            moved = [("q" + x, V[0]), ("n" + x, V[1])] + ([("z" + x, V[2])] if tri else []) + ([("ma" + x, V[0])] if aero else [])
            for name, speed in moved:
                X = v[name] if name[0] in "qm" else torch.clamp(v[name], min=0.0)
                F = rho * X * speed
                v[name] = v[name] + on * (down(F) - F) / (rho * dz)
                if name == "q" + x:
                    total += on * F[0]
                elif name[0] == "m":
                    aerosol += on * F[0]
        fall.append(total)
    return fall + [torch.zeros_like(aerosol)] * (4 - len(fall)) + ([aerosol] if aero else [])


def _exact_step(fld, dz, ncols, dt, config, net=None):
    """One step of the state in 64 bits: (new fields, surface rows), in chunks of columns."""
    warm, aero, tri = config.startswith("warm"), "aero" in config, "tri" in config
    out = fld.clone()
    precip = torch.zeros((_nprecip(config), fld.shape[2]), dtype=torch.float64, device=DEV)
    dzc = torch.tensor(dz, dtype=torch.float64, device=DEV)[:, None]
    names = synth.FIELDS + EXTRA[config]
    for c in range(0, ncols, 32768):
        cs = slice(c, min(ncols, c + 32768))
        v = {n: fld[i, :, cs].clone() for i, n in enumerate(names)}
        if warm:
            for n in ("qi", "qs", "qg", "ni", "ns", "ng"):
                v[n] = torch.zeros_like(v["T"])
        q0 = dict(v)
        active = (v["qc"] > QMIN) | (v["qr"] > QMIN) | (v["qv"] > _qsat(_es_liq(v["T"]), v["p"]))
        if not warm:
            active |= (v["qi"] > QMIN) | (v["qs"] > QMIN) | (v["qg"] > QMIN)
            active |= (v["T"] < TNUC) & (v["qv"] > _qsat(_es_ice(v["T"]), v["p"]))
        sed = ("r",) if warm else ("r", "i", "s", "g")
        shapes = {x: _shape(x, v["q" + x], v["n" + x], v["z" + x]) if tri and x in sed else SPECIES[x][1] for x in SPECIES}
        rec = _processes(v, dt, warm, shapes, net)
        if aero:
            _aerosol(v, rec, q0, warm)
        if tri:
            _sixth_moments(v, rec, q0, warm, active)
        for x, row in enumerate(_sediment(v, dzc, dt, sed, aero, tri)):
            precip[x, cs] = row
        for i, n in enumerate(names):
            if not (warm and n in ("qi", "qs", "qg", "ni", "ns", "ng")):
                out[i, :, cs] = v[n]
    return out, precip


def _mix64(z):
    z = z + np.uint64(0x9e3779b97f4a7c15)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xbf58476d1ce4e5b9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94d049bb133111eb)
    return z ^ (z >> np.uint64(31))


def _exact_training(case, seed):
    """The same minibatches and Adam steps in 64 bits."""
    X, Y, M = (t.double() for t in _rows(case, seed))
    theta = torch.tensor(_weights(seed), dtype=torch.float64, device=DEV)
    mu, sd = X.mean(0), X.var(0, unbiased=False).clamp(min=1e-12).sqrt()
    cnt = M.sum(0).clamp(min=1.0)
    muy = (Y * M).sum(0) / cnt
    sdy = ((Y * Y * M).sum(0) / cnt - muy * muy).clamp(min=1e-12).sqrt()
    m1, m2, losses = torch.zeros_like(theta), torch.zeros_like(theta), []
    rows = np.arange(case["batch"], dtype=np.uint64)
    for s in range(case["steps"]):
        with np.errstate(over="ignore"):
            h = _mix64(np.uint64(11) ^ _mix64(np.uint64(s) * np.uint64(0x100000001b3) + rows))
        at = torch.tensor((h % np.uint64(case["rows"])).astype(np.int64), device=DEV)
        x, m = (X[at] - mu) / sd, M[at]
        t = torch.where(m > 0.0, (Y[at] - muy) / sdy, 0.0)
        th = theta.clone().requires_grad_()
        loss = (((_net(_layers(th), x) - t) * m) ** 2).sum() / m.sum().clamp(min=1.0)
        g, = torch.autograd.grad(loss, th)
        losses.append(loss.detach())
        m1, m2 = 0.9 * m1 + 0.1 * g, 0.999 * m2 + 0.001 * g * g
        theta = theta - 1e-3 * (m1 / (1.0 - 0.9 ** (s + 1))) / (torch.sqrt(m2 / (1.0 - 0.999 ** (s + 1))) + 1e-8)
    return {"loss": torch.stack(losses), "params": theta}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_training(case, seed)
    if kind in ("batched", "surrogate"):
        net = None
        if kind == "surrogate":
            f64 = dict(dtype=torch.float64, device=DEV)
            net = _layers(torch.tensor(_weights(seed), **f64)), torch.tensor(_stats(), **f64)
        return _batch_views([_exact_step(_fields(rc, nc, nl, dz, "cold", sd), dz, nc, case["dt"], "cold", net)
                             for rc, nc, nl, dz, sd in _domains(case, seed)])
    dz, config = _dz(case), case["config"]
    fld = _fields(synth.RECIPES[case["recipe"]], case["ncols"], case["nlev"], dz, config, seed)
    out, precip = _exact_step(fld, dz, case["ncols"], case["dt"], config)
    if kind == "tendency":
        d = (out - fld) / case["dt"]
        return {n: d[i if i < 13 else i + 3] for i, n in enumerate(PROG + EXTRA[config])}
    return _views(out, precip, config)
