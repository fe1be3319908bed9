"""Measured cases: calls of the SED library as fitting programs make them.

A program that fits galaxies loads a stellar-population grid once, creates a
model per galaxy (filters, spectrum, data, options) and then evaluates batches
of parameter rows: log-likelihoods for a nested sampler's live points,
gradients for a gradient-based sampler, model fluxes for predictions, or a
whole nested-sampling run.  A case is one such call.  The grids are seeded
synthetic ones of the sizes the framework is used with; the galaxy (true row,
data) and the parameter rows follow from the seed alone.

exact() restates the model in plain 64-bit torch: SFH weights, contraction,
dust, nebular emission, photometry, spectrum, likelihood; gradients by
autograd.
"""
import math
import random
import types
import weakref

import numpy as np
import torch

from paper_2609_30145_gb300 import Context

DEV = "cuda"
LSUN, HPL, C_AA, C_KMS = 3.839e33, 6.62607015e-27, 2.99792458e18, 299792.458
AB, PC, MPC_KM, YR = 3.631e-20, 3.0856775814913673e18, 3.0856775814913673e19, 3.15576e7
H0, OM, FWHM = 67.66, 0.3097, 2.3548200450309493
FLOPS_NNZ = 1.45   # non-zero weights per (age node + SFH bin) with one [Fe/H] per bin

GRIDS = {
    # 16 ages x 4 [Fe/H] x 512 wavelengths, no nebular emission
    "tiny": dict(n_age=16, age=(6.0, 10.1), feh=(-2.0, 0.2), n_feh=4, afe=(0.0,), n_lam=512, lam=(1e3, 5e4), neb=0, zf=10.0),
    # 107 x 12 x 6000 with a 7 x 12 nebular continuum and 30 emission lines
    "paper": dict(n_age=107, age=(5.5, 10.8), feh=(-2.5, 0.5), n_feh=12, afe=(0.0,), n_lam=6000, lam=(1e2, 6e4), neb=1, zf=30.0),
    # 107 x 12 x 5 [alpha/Fe] x 6000
    "alpha": dict(n_age=107, age=(5.5, 10.8), feh=(-2.5, 0.5), n_feh=12, afe=(-0.2, 0.0, 0.2, 0.4, 0.6), n_lam=6000,
                  lam=(1e2, 6e4), neb=0, zf=30.0),
}


def _case(op, grid, rows, prec="fp32", n_sfh=120, zmode=0, n_filt=20, n_pix=0, z_lo=0.0, z_hi=12.0, sgal=False,
          calib=False, lines=False, name=None):
    c = dict(op=op, grid=grid, rows=rows, prec=prec, n_sfh=n_sfh, zmode=zmode, n_filt=n_filt, n_pix=n_pix, z_lo=z_lo,
             z_hi=z_hi, sgal=sgal, calib=calib, lines=lines)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: a 64-row step of a toy photometric fit (8 bins, 8 bands), latency alone
        _case("loglike", "tiny", 64, n_sfh=8, n_filt=8, z_lo=0.5, z_hi=8.0, name="tiny_loglike_64"),
        # one replacement round of a nested sampler on a paper-scale photometric fit, late in the run (z constrained)
        _case("loglike", "paper", 64, z_lo=1.8, z_hi=2.2, name="phot_loglike_64"),
        # the ordinary batch: 1024 prior draws of the paper-scale photometric fit
        _case("loglike", "paper", 1024, name="phot_loglike_1024"),
        # the same call from page-locked host arrays: a sampler that runs on the CPU
        _case("host", "paper", 1000, name="phot_host_1000"),
        # large live sets with the reduced-precision contractions
        _case("loglike", "paper", 4096, prec="bf16", name="phot_loglike_4096_bf16"),
        _case("loglike", "paper", 2500, prec="fp8", n_filt=15, name="phot_loglike_2500_fp8"),
        # posterior predictions of a spectro-photometric fit with [alpha/Fe]: odd numbers of rows and pixels
        _case("forward", "alpha", 301, zmode=1, n_pix=1111, z_lo=0.9, z_hi=1.3, name="spec_forward_301"),
        # gradients of the full spectro-photometric batch (prior draws), and of the chains of a gradient-based
        # sampler near the mode of a photometric fit with one [Fe/H] per bin
        _case("grad", "alpha", 2048, zmode=1, n_pix=1500, name="spec_grad_2048"),
        _case("grad", "paper", 200, n_sfh=40, z_lo=2.9, z_hi=3.1, name="phot_grad_200"),
        # a spectrum with the grid's emission lines on pixels and bands, sampled gas dispersion
        _case("loglike", "paper", 1024, n_pix=1500, lines=True, name="lines_loglike_1024"),
        # sampled stellar dispersion and a 13-term marginalised calibration polynomial, BF16 contraction
        _case("loglike", "alpha", 512, prec="bf16", zmode=1, n_pix=1500, sgal=True, calib=True, z_lo=3.0, z_hi=7.0,
              name="calib_loglike_512_bf16"),
        # two iterations of nested slice sampling on the device: 15 bands, 22 line fluxes, 8 bins, z known
        _case("nss", "paper", 300, n_sfh=8, zmode=1, n_filt=15, lines=True, z_lo=5.0, z_hi=5.0, name="nss_300"),
    ]


def draw(rng):
    def loguni(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    grid = rng.choice(["tiny", "paper", "paper", "paper", "alpha", "alpha"])
    op = rng.choice(["loglike", "loglike", "loglike", "forward", "grad", "grad", "host"])
    if grid == "tiny":
        return _case(op, grid, loguni(16, 1024), n_sfh=rng.randint(4, 30), n_filt=rng.randint(4, 12), zmode=rng.randint(0, 1),
                     z_lo=0.5, z_hi=rng.uniform(1.0, 8.0))
    n_pix = rng.choice([0, 0, loguni(200, 3000)])
    prec = "fp32" if op == "grad" else rng.choice(["fp32", "fp32", "bf16", "fp8"])
    rows = loguni(32, 1024 if n_pix or op == "grad" else 4096)
    z = rng.uniform(0.0, 11.0)
    dz = rng.choice([0.2, 2.0, 12.0])
    return _case(op, grid, rows, prec=prec, n_sfh=rng.randint(10, 120), zmode=1 if grid == "alpha" else rng.randint(0, 1),
                 n_filt=rng.randint(8, 30), n_pix=n_pix, z_lo=max(0.0, z - dz), z_hi=min(12.0, z + dz),
                 sgal=n_pix > 0 and rng.random() < 0.4, calib=n_pix > 0 and rng.random() < 0.3,
                 lines=n_pix > 0 and grid == "paper" and rng.random() < 0.4)


# ---------------------------------------------------------------- grids (made once per process, as a program loads them)
_made, _loaded = {}, {}


def _grid(kind):
    """Blackbody-like spectra times lognormal amplitudes over six decades with absorption dips; nebular tables."""
    if kind in _made:
        return _made[kind]
    k = GRIDS[kind]
    rng = np.random.Generator(np.random.PCG64(1))
    g = types.SimpleNamespace(zf=k["zf"])
    g.log_age_yr, g.feh = np.linspace(*k["age"], k["n_age"]), np.linspace(*k["feh"], k["n_feh"])
    g.afe, g.lam_aa = np.array(k["afe"]), np.geomspace(*k["lam"], k["n_lam"])
    shape = (g.afe.size, k["n_feh"], k["n_age"])
    t = lambda a: torch.from_numpy(np.asarray(a, dtype=np.float64)).to(DEV)  # noqa: E731
    lam, ll = t(g.lam_aa), t(np.log(g.lam_aa))
    af, fe, ag = (t(a) for a in np.meshgrid(g.afe, g.feh, g.log_age_yr, indexing="ij"))
    temp = 3e4 * 10 ** (-0.35 * (ag - 6.0)) * (1 + 0.05 * fe) * (1 - 0.03 * af)
    frac = (ag - g.log_age_yr[0]) / (g.log_age_yr[-1] - g.log_age_yr[0])
    amp = 1e-11 * 10 ** (-6.0 * frac + 0.1 * t(rng.standard_normal(shape)))
    dc, dd, dw = (t(rng.random(shape + (6,))) for _ in range(3))
    flux = torch.empty(shape + (lam.numel(),), dtype=torch.float64, device=DEV)
    for n in range(shape[0]):
        for m in range(shape[1]):
            x = (HPL / 1.380649e-16) * (C_AA / lam) / temp[n, m, :, None]
            b = x ** 3 * torch.exp(-x) / -torch.expm1(-x)
            b = b / b.amax(1, keepdim=True) * amp[n, m, :, None]
            for i in range(6):
                c = torch.exp(ll[0] + (0.15 + 0.7 * dc[n, m, :, i, None]) * (ll[-1] - ll[0]))
                d = (0.05 + 0.15 * dd[n, m, :, i, None]) * (1 + 0.5 * g.afe[n])
                b = b * (1 - d * torch.exp(-0.5 * ((lam - c) / (5.0 + 45.0 * dw[n, m, :, i, None])) ** 2))
            flux[n, m] = b
    g.flux = flux.cpu().numpy()
    if k["neb"]:
        g.neb_logu, g.neb_logz = np.linspace(-4.0, -1.0, 7), np.linspace(-1.3, 0.3, 12)
        u, z = g.neb_logu[:, None, None], g.neb_logz[None, :, None]
        g.neb_tab = -60.3 - 0.4 * (np.log10(g.lam_aa) - 3.7) + np.log10(1.0 + 0.05 * (u + 2.5) - 0.04 * z)
        g.neb_tab[:, :, g.lam_aa < 912.0] = -99.0
        n = 30
        g.line_lam = np.sort(np.exp(np.log(1e3) + rng.random(n) * np.log(22.0)))
        g.line_tab = (-46.0 + np.log10(0.1 + 2.9 * rng.random(n)) + 0.3 * (rng.random(n) - 0.5) * (u + 2.5)
                      + 0.4 * (rng.random(n) - 0.5) * (z + 0.5))
        g.t_neb, g.t_line, g.t_line_lam = t(g.neb_tab), t(g.line_tab), t(g.line_lam)
        g.t_logu, g.t_logz = t(g.neb_logu), t(g.neb_logz)
    # the same in 64-bit torch, for the reference
    g.t_lam, g.t_ll, g.t_flux, g.t_feh, g.t_afe = lam, ll, flux, t(g.feh), t(g.afe)
    g.t_young = t(g.log_age_yr <= 7.03) > 0
    below = lam < 912.0
    kl = int(below.sum())
    if kl:
        f, x = flux[..., : kl + 1], lam[: kl + 1].clone()
        fe_ = f[..., -2] + (f[..., -1] - f[..., -2]) * (912.0 - x[-2]) / (x[-1] - x[-2])
        f = torch.cat([f[..., :-1], fe_[..., None]], -1)
        x[-1] = 912.0
        y = f / x
        g.t_q = LSUN / HPL * (0.5 * (y[..., 1:] + y[..., :-1]) * (x[1:] - x[:-1])).sum(-1)
    age = t(10.0 ** g.log_age_yr)
    mid = 0.5 * (age[1:] + age[:-1])
    g.t_cm = torch.cat([mid.new_zeros(1), mid])
    g.t_cp = torch.cat([mid, mid.new_full((1,), math.inf)])
    lum = lam * 1e-4
    red = 2.659 * (-1.857 + 1.040 / lum) + 4.05
    uv = 2.659 * (-2.156 + 1.509 / lum - 0.198 / lum ** 2 + 0.011 / lum ** 3) + 4.05
    g.t_kp = torch.where(lum >= 0.63, red, uv).clamp_min(0.0)
    g.lnf = math.log(k["lam"][1] / k["lam"][0])
    _made[kind] = g
    return g


def _context(kind):
    if "ctx" not in _loaded:
        _loaded["ctx"] = Context(0)
    if kind not in _loaded:
        _loaded[kind] = _loaded["ctx"].load_grid(_grid(kind))
    return _loaded["ctx"], _loaded[kind]


# ---------------------------------------------------------------- one galaxy and its parameter rows
def _columns(case):
    """Column ranges of a parameter row in the library's key order."""
    widths = [("sfh", case["n_sfh"]), ("logzsol", 1 if case["zmode"] else case["n_sfh"]), ("afe", 1), ("logmass", 1),
              ("zred", 1), ("tau_pow", 1), ("alpha_pow", 1), ("diffuse_tau_kc", 1), ("diffuse_dust_index", 1),
              ("gas_logz", 1), ("gas_logu", 1)]
    if case["sgal"]:
        widths.append(("sigma_gal", 1))
    if case["lines"] and case["n_pix"]:
        widths.append(("sigma_gas", 1))
    cols, at = {}, 0
    for k, w in widths:
        cols[k] = slice(at, at + w)
        at += w
    return cols, at


def _rows(case, n, rng, z=None):
    g, tiny = _grid(case["grid"]), case["grid"] == "tiny"
    cols, width = _columns(case)
    th = np.zeros((n, width))
    u = lambda lo, hi, w=1: lo + (hi - lo) * rng.random((n, w))  # noqa: E731
    e = -np.log1p(-rng.random((n, case["n_sfh"])))
    th[:, cols["sfh"]] = e / e.sum(1, keepdims=True)
    th[:, cols["logzsol"]] = u(g.feh[0], g.feh[-1], cols["logzsol"].stop - cols["logzsol"].start)
    th[:, cols["afe"]] = u(-0.2, 0.6) if case["grid"] == "alpha" else 0.0
    th[:, cols["logmass"]] = u(8.0, 11.0)
    th[:, cols["zred"]] = u(max(case["z_lo"], 0.02), case["z_hi"]) if z is None else z
    th[:, cols["diffuse_tau_kc"]] = u(0.0, 2.0)
    th[:, cols["tau_pow"]] = th[:, cols["diffuse_tau_kc"]] if tiny else u(0.0, 2.0)
    th[:, cols["alpha_pow"]] = -1.0
    th[:, cols["diffuse_dust_index"]] = -0.7 if tiny else u(-1.0, 0.4)
    th[:, cols["gas_logz"]], th[:, cols["gas_logu"]] = (u(-1.3, 0.3), u(-4.0, -1.0)) if hasattr(g, "neb_tab") else (0.0, -2.0)
    if "sigma_gal" in cols:
        th[:, cols["sigma_gal"]] = u(50.0, 500.0)
    if "sigma_gas" in cols:
        th[:, cols["sigma_gas"]] = u(50.0, 400.0)
    return th.astype(np.float32)


def _filters(n):
    """Flat-topped broad (R ~ 4) and medium (R ~ 10) bands over 0.6-5 um, 200 samples each."""
    wide = (2 * n) // 5
    cw, cm = np.geomspace(7.5e3, 5e4 / 1.15, wide), np.geomspace(6.48e3, 5e4 / 1.06, n - wide)
    out = []
    for i, (c, r) in enumerate([(c, 4.0) for c in cw] + [(c, 10.0) for c in cm]):
        h = 0.5 * c / r
        lam = np.linspace(c - 1.6 * h, c + 1.6 * h, 200)
        x = (lam - c) / h
        tr = np.clip(np.exp(-0.5 * x ** 8) * (0.85 + 0.03 * np.sin(9 * x + i)) - 1e-12, 0.0, None)
        tr[0] = tr[-1] = 0.0
        out.append((lam, tr))
    return out


def _galaxy(case, seed):
    """What the program has observed (bands, pixels, data) and the rows it evaluates."""
    rng = np.random.Generator(np.random.PCG64([int(seed), 7]))
    o = types.SimpleNamespace(filters=_filters(case["n_filt"]), spec_lam=None, lcat=None)
    if case["n_pix"]:
        o.spec_lam = np.geomspace(6e3, 5.3e4, case["n_pix"])
        o.spec_r = np.linspace(100.0, 1000.0, case["n_pix"])
    z_true = 0.5 * (case["z_lo"] + case["z_hi"])
    if case["z_hi"] - case["z_lo"] > 6.0:
        z_true = 1.0 + 2.0 * rng.random()
    truth = torch.from_numpy(_rows(case, 1, rng, z=z_true)).to(DEV).double()
    with torch.no_grad():
        m = _model64(case, o, truth)

    def noisy(a, snr):   # errors of a constant signal-to-noise ratio down to the survey's depth
        err = np.hypot(np.abs(a) / snr, 0.01 * np.median(np.abs(a)))
        return a + err * rng.standard_normal(a.shape), err

    o.phot_d, o.phot_s = noisy(m["phot"][0].cpu().numpy(), 20.0)
    if case["n_pix"]:
        sp = m["spec"][0].cpu().numpy()
        seen = m["valid"][0].cpu().numpy()
        o.spec_mask = seen.astype(np.uint8)
        sp = np.where(seen, sp, np.median(np.abs(sp[seen])))
        x = np.linspace(-1.0, 1.0, sp.size)
        o.spec_d, o.spec_s = noisy(sp, 20.0)
        if case["calib"]:
            o.spec_d = o.spec_d * (1 + 0.08 * x - 0.05 * (2 * x * x - 1))
    if case["op"] == "nss":
        o.blends = [[i] for i in range(19)] + [[19, 20], [21, 22, 23], [24, 25]]
        fl = m["lines"][0].cpu().numpy()
        o.lcat = noisy(np.array([fl[b].sum() for b in o.blends]), 10.0)
    o.theta = _rows(case, case["rows"], rng)
    return o


# ---------------------------------------------------------------- the calls
class _State:
    pass


def prepare(case, seed):
    ctx, gid = _context(case["grid"])
    g, o = _grid(case["grid"]), _galaxy(case, seed)
    tiny = case["grid"] == "tiny"
    kw = dict(use_afe=int(case["grid"] == "alpha"), use_nebular=int(hasattr(g, "neb_tab")), dust_law=0 if tiny else 1,
              filters=(np.array([f[0].size for f in o.filters]), np.concatenate([f[0] for f in o.filters]),
                       np.concatenate([f[1] for f in o.filters])), phot_d=o.phot_d, phot_sigma=o.phot_s)
    if case["n_pix"]:
        kw.update(spec_lam=o.spec_lam, spec_d=o.spec_d, spec_sigma=o.spec_s, spec_mask=o.spec_mask, lsf_mode=0,
                  lsf_value=o.spec_r, sigma_gal_kms=300.0, z_ref=0.5 * (case["z_lo"] + case["z_hi"]))
        if case["sgal"]:
            kw.update(sample_sigma_gal=1, sigma_gal_max_kms=600.0)
        if case["calib"]:
            kw.update(calib_sigma=np.array([0.2] + [0.1] * 12))
    if case["lines"]:
        kw.update(use_lines=1, gas_sigma_mode=2 if case["n_pix"] else 0, sigma_gas_max_kms=600.0)
    if case["op"] == "nss":
        kw.update(lcat=(o.blends, o.lcat[0], o.lcat[1], None, None),
                  fixed={"afe": 0.0, "zred": case["z_lo"], "alpha_pow": -1.0})
    s = _State()
    s.op, s.prec, s.seed, s.rows = case["op"], case["prec"], int(seed), case["rows"]
    s.model = ctx.create_model(gid, case["n_sfh"], g.zf, case["zmode"], **kw)
    weakref.finalize(s, _close, s.model)
    if s.op == "nss":   # box prior of the 15 sampled columns
        s.lo = np.array([0.0] * 8 + [-2.0, 7.0, 0.0, 0.0, -1.0, -1.3, -4.0])
        s.hi = np.array([1.0] * 8 + [0.3, 12.0, 2.0, 2.0, 0.4, 0.3, -1.0])
    elif s.op == "host":
        s.theta = torch.from_numpy(o.theta).pin_memory()
        s.lnl = torch.empty(case["rows"], dtype=torch.float64).pin_memory()
        s.status = torch.empty(case["rows"], dtype=torch.int32).pin_memory()
    else:
        s.theta = torch.from_numpy(o.theta).to(DEV)
    return s


def _close(model):
    torch.cuda.synchronize()
    model.close()


def run(s):
    if s.op == "loglike":
        return s.model.loglike(s.theta, s.prec)
    if s.op == "grad":
        return s.model.loglike_grad(s.theta, s.prec)
    if s.op == "forward":
        return s.model.forward(s.theta, s.prec)
    if s.op == "host":
        return s.model.loglike_host(s.theta, s.prec, out=s.lnl, status=s.status)
    r = s.model.nss(s.lo, s.hi, n_live=s.rows, n_replace=64, n_slice_steps=40, max_iter=2, seed=100 + s.seed,
                    precision=s.prec)
    return {k: r[k] for k in ("lnz", "info_h", "n_like", "theta", "lnl", "logw", "ins_rank")}


def work(case):
    """Bytes: rows, results and, once, the part of the grid that the batch's redshifts reach.  Operations: the products
    of the non-zero weights with the nodes each row reaches (twice for a gradient), and for a spectrum its response."""
    k, g = GRIDS[case["grid"]], GRIDS[case["grid"]]
    n, lnf = case["rows"], math.log(g["lam"][1] / g["lam"][0])
    lo, hi = (6e3, 5.3e4) if case["n_pix"] else (5.4e3, 5.4e4)
    one = min(1.0, math.log(hi / lo) / lnf)
    union = min(1.0, one + math.log((1 + case["z_hi"]) / (1 + case["z_lo"])) / lnf)
    kz = k["n_feh"] * k["n_age"]
    if case["zmode"]:
        nnz = k["n_age"] * 2 * (2 if len(k["afe"]) > 1 else 1)
    else:
        nnz = min(kz, FLOPS_NNZ * (k["n_age"] + case["n_sfh"]))
    calls = 1
    if case["op"] == "nss":   # proposals of two iterations: 64 chains x 40 steps x about 5 evaluations
        n, calls = 64, 400
    per = 2.0 * nnz * one * k["n_lam"] * (2 if case["op"] == "grad" else 1) + 100.0 * case["n_pix"] + 10.0 * one * k["n_lam"]
    width = _columns(case)[1]
    size = {"fp32": 4, "bf16": 2, "fp8": 1}[case["prec"]]
    grid_bytes = union * k["n_lam"] * (min(kz * len(k["afe"]), n * nnz)) * size
    out = 12 + (4 * width if case["op"] == "grad" else 4 * (case["n_filt"] + case["n_pix"]) if case["op"] == "forward" else 0)
    return {"bytes": grid_bytes + calls * n * (4 * width + out), "flops": float(calls * n * per)}


# ---------------------------------------------------------------- 64-bit reference
def _bracket(x, v):
    """Left node and weight of the right node, clamped to the axis."""
    if x.numel() == 1:
        return torch.zeros_like(v, dtype=torch.long), torch.zeros_like(v)
    j = (torch.searchsorted(x, v.detach().contiguous(), right=True) - 1).clamp(0, x.numel() - 2)
    return j, ((v - x[j]) / (x[j + 1] - x[j])).clamp(0.0, 1.0)


def _hat(x, v):
    """Linear interpolation weights [..., n] of v on the nodes x."""
    j, t = _bracket(x, v)
    w = v.new_zeros(v.shape + (x.numel(),))
    if x.numel() == 1:
        return w + 1.0
    return w.scatter(-1, j[..., None], (1 - t)[..., None]) + w.scatter(-1, j[..., None] + 1, t[..., None])


def _age_of(z):
    """Cosmic time (yr) in a flat universe of matter and a constant."""
    return MPC_KM / H0 / YR * 2.0 / (3.0 * math.sqrt(1 - OM)) * torch.asinh(math.sqrt((1 - OM) / OM) * (1 + z) ** -1.5)


def _dust(lam, kp, tau, index, law):
    p = (lam / 5500.0) ** index[:, None]
    if law == 0:
        return tau[:, None] * p
    x2, d = (lam * 350.0) ** 2, lam * lam - 2175.0 ** 2
    drude = (0.85 - 1.9 * index)[:, None] * (x2 / (d * d + x2))
    return tau[:, None] * (kp + drude) / 4.05 * p


def _neb(g, tab, th):
    wu, wz = _hat(g.t_logu, th["gas_logu"]), _hat(g.t_logz, th["gas_logz"])
    return 10.0 ** torch.einsum("nu,nz,uzk->nk", wu, wz, tab)


def _model64(case, o, theta):
    g = _grid(case["grid"])
    cols, _ = _columns(case)
    th = {k: theta[:, c] if k in ("sfh", "logzsol") else theta[:, c.start] for k, c in cols.items()}
    nt, z = case["n_sfh"], th["zred"]
    lam, ll, zp = g.t_lam, g.t_ll, 1 + th["zred"]
    # luminosity distance by Gauss-Legendre in ln(1+z); SFH edges from the age of the universe
    xs, ws = (torch.from_numpy(a).to(theta) for a in np.polynomial.legendre.leggauss(48))
    half = 0.5 * torch.log1p(z)[:, None]
    zz = torch.exp(half * (1 + xs))
    dc = C_KMS / H0 * 1e6 * PC * (half * ws * zz / torch.sqrt(OM * zz ** 3 + 1 - OM)).sum(1)
    dl = (zp * dc).clamp_min(10.0 * PC)
    tmax = _age_of(z) - _age_of(torch.tensor(float(g.zf), dtype=torch.float64, device=theta.device))
    i = torch.arange(3, nt + 1, device=theta.device)
    edges = torch.cat([tmax.new_tensor([0.0, 5e6, 1e7]).expand(z.numel(), 3),
                       1e7 * (tmax / 1e7)[:, None] ** ((i - 2) / (nt - 2.0))], 1)
    t0, t1 = edges[:, :-1, None], edges[:, 1:, None]
    part = (torch.minimum(t1, g.t_cp) - torch.maximum(t0, g.t_cm)).clamp_min(0.0) / (t1 - t0) * th["sfh"][..., None]
    w = torch.einsum("nta,ntz->nza", part, _hat(g.t_feh, th["logzsol"]).expand(-1, nt, -1))
    w = _hat(g.t_afe, th["afe"])[:, :, None, None] * w[:, None] if case["grid"] == "alpha" else w[:, None]
    neb = hasattr(g, "neb_tab")
    yf = lambda f: f[:, :, g.t_young].reshape(-1, lam.numel())  # noqa: E731
    young = w[..., g.t_young].flatten(1) @ yf(g.t_flux)
    old = w[..., ~g.t_young].flatten(1) @ g.t_flux[:, :, ~g.t_young].reshape(-1, lam.numel())
    if neb:
        qy = (w[..., g.t_young] * g.t_q[..., g.t_young]).flatten(1).sum(1)
        young = torch.where(lam < 912.0, torch.zeros_like(young), young) + qy[:, None] * _neb(g, g.t_neb, th)
    law = 0 if case["grid"] == "tiny" else 1
    bc = lambda x: th["tau_pow"][:, None] * (x / 5500.0) ** th["alpha_pow"][:, None]  # noqa: E731
    f = torch.exp(-_dust(lam, g.t_kp, th["diffuse_tau_kc"], th["diffuse_dust_index"], law)) * (torch.exp(-bc(lam)) * young + old)
    base = 10.0 ** th["logmass"] * LSUN / (4 * math.pi * dl * dl)
    fnu = (base * zp)[:, None] * f
    out = {}
    if case["lines"]:
        x = g.t_line_lam
        lum = x * 1e-4
        kp = torch.where(lum >= 0.63, 2.659 * (-1.857 + 1.040 / lum) + 4.05,
                         2.659 * (-2.156 + 1.509 / lum - 0.198 / lum ** 2 + 0.011 / lum ** 3) + 4.05).clamp_min(0.0)
        lf = (qy * base)[:, None] * _neb(g, g.t_line, th) * torch.exp(
            -_dust(x, kp, th["diffuse_tau_kc"], th["diffuse_dust_index"], law) - bc(x))
        xo = x * zp[:, None]
        out["lines"] = lf
    # photometry: linear in observed wavelength between the redshifted nodes
    flam = C_AA * fnu / (zp[:, None] * lam) ** 2
    phot = []
    for fl, tr in o.filters:
        dlam = np.gradient(fl)
        dlam[0], dlam[-1] = 0.5 * (fl[1] - fl[0]), 0.5 * (fl[-1] - fl[-2])
        y = tr * C_AA * AB / fl
        zb = float((0.5 * (y[1:] + y[:-1]) * np.diff(fl)).sum())
        wl = torch.from_numpy(tr * fl * dlam / zb).to(theta)
        xr = torch.from_numpy(fl).to(theta) / zp[:, None]
        j = (torch.searchsorted(lam, xr.detach().contiguous(), right=True) - 1).clamp(0, lam.numel() - 2)
        t = (xr - lam[j]) / (lam[j + 1] - lam[j])
        v = flam.gather(1, j) * (1 - t) + flam.gather(1, j + 1) * t
        m = (wl * v * ((xr >= lam[0]) & (xr <= lam[-1]))).sum(1)
        if case["lines"]:
            gx, gr = torch.from_numpy(fl).to(theta), torch.from_numpy(tr).to(theta)
            q = (torch.searchsorted(gx, xo.detach().contiguous(), right=True) - 1).clamp(0, fl.size - 2)
            r = gr[q] + (gr[q + 1] - gr[q]) * (xo - gx[q]) / (gx[q + 1] - gx[q])
            m = m + (lf * r * xo / zb * ((xo >= gx[0]) & (xo <= gx[-1]))).sum(1)
        phot.append(m)
    out["phot"] = torch.stack(phot, 1)
    if case["n_pix"]:
        pix = torch.from_numpy(o.spec_lam).to(theta)
        inst = torch.from_numpy(C_KMS / (FWHM * o.spec_r)).to(theta)
        gap = torch.cat([(lam[1:2] - lam[:1]), 0.5 * (lam[2:] - lam[:-2]), lam[-1:] - lam[-2:-1]])
        lib = C_KMS / FWHM * 2.0 * gap / lam
        zr = 1 + 0.5 * (case["z_lo"] + case["z_hi"])
        j, t = _bracket(lam, pix / zr)
        fix2 = (inst ** 2 - (lib[j] + (lib[j + 1] - lib[j]) * t) ** 2).clamp_min(0.0)
        sg = th["sigma_gal"] if case["sgal"] else torch.full_like(z, 300.0)
        s = torch.sqrt(fix2 + sg[:, None] ** 2) / C_KMS
        x = torch.log(pix) - torch.log(zp)[:, None]
        valid = (x >= ll[0]) & (x <= ll[-1])
        k = (torch.searchsorted(ll, x.detach().contiguous(), right=True) - 1).clamp(0, ll.numel() - 2)
        t = (x - ll[k]) / (ll[k + 1] - ll[k])
        lin = fnu.gather(1, k) * (1 - t) + fnu.gather(1, k + 1) * t
        wide = int(5.0 * float(s.max()) / float((ll[1:] - ll[:-1]).min())) + 2
        idx = k[..., None] + torch.arange(-wide, wide + 2, device=theta.device)
        inside = (idx >= 0) & (idx < ll.numel())
        idx = idx.clamp(0, ll.numel() - 1)
        u = (ll[idx] - x[..., None]) / s[..., None]
        gw = torch.exp(-0.5 * u * u) * (inside & (u.abs() <= 5.0))
        v = (gw * fnu.gather(1, idx.flatten(1)).view(idx.shape)).sum(-1) / gw.sum(-1).clamp_min(1e-300)
        sp = torch.where(s < 0.5 * (ll[k + 1] - ll[k]), lin, v) * valid
        if case["lines"]:
            q = (torch.searchsorted(pix, xo.detach().contiguous(), right=True) - 1).clamp(0, pix.numel() - 2)
            ti = ((xo - pix[q]) / (pix[q + 1] - pix[q])).clamp(0.0, 1.0)
            si = inst[q] + (inst[q + 1] - inst[q]) * ti
            gas = th["sigma_gas"] if "sigma_gas" in th else torch.full_like(z, 300.0)
            sl = torch.sqrt(gas[:, None] ** 2 + si ** 2) / C_KMS
            u = (torch.log(pix)[:, None] - torch.log(xo)[:, None, :]) / sl[:, None, :]
            pr = torch.exp(-0.5 * u * u) * (u.abs() <= 5.0) / (math.sqrt(2 * math.pi) * sl)[:, None, :]
            sp = sp + (pr * lf[:, None, :]).sum(-1) * (pix / C_AA)
        out["spec"], out["valid"] = sp, valid
    return out


def _lnl64(case, o, m):
    t = lambda a: torch.from_numpy(np.asarray(a, dtype=np.float64)).to(DEV)  # noqa: E731
    s = t(o.phot_s)
    lnl = (-0.5 * ((t(o.phot_d) - m["phot"]) / s) ** 2 - 0.5 * torch.log(2 * math.pi * s * s)).sum(1)
    if case["n_pix"]:
        s, d = t(o.spec_s), t(o.spec_d)
        inc = m["valid"] & (t(o.spec_mask) > 0)
        r = (d - m["spec"]) / s
        lnl = lnl + ((-0.5 * r * r - 0.5 * (math.log(2 * math.pi) + 2 * torch.log(s))) * inc).sum(1)
        if case["calib"]:
            lam = t(o.spec_lam)
            x = (2 * lam - (lam[0] + lam[-1])) / (lam[-1] - lam[0])
            cheb = torch.cos(torch.arange(13, device=x.device)[:, None] * torch.acos(x.clamp(-1.0, 1.0)))
            a = cheb * (m["spec"] / s * inc)[:, None, :]
            sig = t([0.2] + [0.1] * 12)
            mat = a @ a.transpose(1, 2) + torch.diag(sig ** -2)
            b = (a * r[:, None, :]).sum(-1)
            chol = torch.linalg.cholesky(mat)
            y = torch.linalg.solve_triangular(chol, b[..., None], upper=False)[..., 0]
            lnl = lnl + 0.5 * (y * y).sum(1) - torch.log(torch.diagonal(chol, dim1=1, dim2=2)).sum(1) - torch.log(sig).sum()
    return lnl


def exact(case, seed):
    if case["op"] == "nss":   # a stochastic run: its points follow from every comparison on the way
        return None
    o = _galaxy(case, seed)
    got = []
    for at in range(0, case["rows"], 128):
        th = torch.from_numpy(o.theta[at:at + 128]).to(DEV).double()
        with torch.set_grad_enabled(case["op"] == "grad"):
            th.requires_grad_(case["op"] == "grad")
            m = _model64(case, o, th)
            if case["op"] == "forward":
                got.append((m["phot"], m["spec"]) if case["n_pix"] else (m["phot"],))
                continue
            lnl = _lnl64(case, o, m)
            got.append((lnl.detach(), torch.autograd.grad(lnl.sum(), th)[0]) if case["op"] == "grad" else (lnl,))
    parts = [torch.cat(p) for p in zip(*got)]
    if case["op"] == "forward":
        return (parts[0], parts[1] if case["n_pix"] else None)
    return tuple(parts) + (None,)
