"""The workloads this library is measured on, each one pass through its public entry points.

Kinds of case (the "kind" of a case's dict):
  star     one star: new geometry, new local spectra, spectra of the active star at every phase
           and their radial velocities (the whole path of a forward model)
  batch    many configurations of one star type in one call, spectra or residuals, with or without RVs
  ccf      RVs of spectra that exist already (an observed or simulated series)
  local    line bisectors put into local spectra, the quiet star integrated at instrument resolution
  train    one epoch of surrogate training from given weights
  query    surrogate queries answered with residual spectra
  project  residual spectra projected onto the surrogate's PCA basis

Sizes are those of the library's own workloads (disk 50 x 50 at 4,096 px to disk 300 x 300 at
205,800 px; batches at 150 x 150 and 16,834 px; queries of 16,834 px) and odd ones between them.
Spectra are Gaussian-line spectra on the log-uniform grid, one line per slot of equal width so
that they are built on the GPU from the seed alone, with the line depths, widths and convective
shifts of `synth`.
"""
import math

import numpy as np
import torch

from paper_2301_04259_gb300 import soap as S
from paper_2301_04259_gb300 import synth

C_KMS = 299792.458
HCK = 6.62607015e-34 * 299792458.0 / 1.380649e-23 * 1e10        # h c / k_B, Angstrom Kelvin
PX_KMS = C_KMS / (3 * 115000.0)                                 # 3 pixels per R = 115000 element
U1, U2, T_QUIET, LAM0 = 0.29, 0.34, 5778.0, 3800.0
MASK_WIDTH, V_STEP, V_MARGIN = 0.82, 0.25, 20.0
LSF_R = 115000.0
DEV = "cuda"
N_COEF, HIDDEN = 128, 256


# ---------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest forward model a user runs, e.g. inside a fit's loop: launches and latency
        {"name": "star_small", "kind": "star", "precision": "fp32", "grid_n": 50, "n_px": 4096, "px_kms": 0.122,
         "line_px": 136.5, "n_mu": 11, "n_phases": 25, "spots": 1, "faculae": 0, "vsini": 2.0, "lsf": False,
         "limb": False},
        # the headline: full visible range, 100 phases, CCF on the tensor cores
        {"name": "star_full", "kind": "star", "precision": "fp32tc", "grid_n": 300, "n_px": 205800, "px_kms": PX_KMS,
         "line_px": 10.29, "n_mu": 20, "n_phases": 100, "spots": 2, "faculae": 1, "vsini": 2.0, "lsf": False,
         "limb": False},
        # the same star in FP64 (reference runs)
        {"name": "star_fp64", "kind": "star", "precision": "fp64", "grid_n": 300, "n_px": 205800, "px_kms": PX_KMS,
         "line_px": 10.29, "n_mu": 20, "n_phases": 100, "spots": 2, "faculae": 1, "vsini": 2.0, "lsf": False,
         "limb": False},
        # an odd-sized faster rotator with every option on: facula limb brightening, instrument resolution
        {"name": "star_options", "kind": "star", "precision": "fp32", "grid_n": 211, "n_px": 61747, "px_kms": PX_KMS,
         "line_px": 10.29, "n_mu": 17, "n_phases": 37, "spots": 3, "faculae": 2, "vsini": 5.3, "lsf": True,
         "limb": True},
        # a library of configurations with the RV of every spectrum
        {"name": "batch_rv", "kind": "batch", "n_items": 512, "phases_lo": 10, "phases_hi": 200, "n_px": 16834,
         "grid_n": 150, "residual": False, "rv": True, "tc": True},
        # training data of the surrogate: one phase per configuration, residual spectra
        {"name": "batch_residual", "kind": "batch", "n_items": 3001, "phases_lo": 1, "phases_hi": 1, "n_px": 16834,
         "grid_n": 150, "residual": True, "rv": False, "tc": False},
        # RVs of a series of spectra with the default (FP32) CCF
        {"name": "ccf_series", "kind": "ccf", "precision": "fp32", "n_spec": 317, "n_px": 102901, "px_kms": PX_KMS,
         "line_px": 10.29, "vsini": 3.0},
        # local spectra prepared for a run: bisectors, quiet star, instrument resolution (FP64)
        {"name": "local_bisectors", "kind": "local", "n_mu": 20, "n_px": 205800, "n_depth": 11, "grid_n": 300,
         "vsini": 2.0},
        # surrogate training: 16 batches of 4,096 (a ragged data set)
        {"name": "train_epoch", "kind": "train", "rows": 66003, "batch": 4096},
        # surrogate queries: one interactive handful, and a large ensemble
        {"name": "query_few", "kind": "query", "n": 7, "n_px": 16834},
        {"name": "query_many", "kind": "query", "n": 40000, "n_px": 16834},
        # coefficients of plain-method residuals (training, and queries the surrogate declines)
        {"name": "project", "kind": "project", "n": 20011, "n_px": 16834},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["star", "star", "star", "batch", "batch", "ccf", "local", "train", "query", "project"])
    if kind == "star":
        precision = rng.choice(["fp32", "fp32tc", "bf16x3", "fp64"])
        fine = rng.random() < 0.25                          # a short, finely sampled range
        n_px = int(_log(rng, 4096, 20000 if fine else 60000 if precision == "fp64" else 205800))
        return {"kind": kind, "precision": precision, "grid_n": int(_log(rng, 50, 300)), "n_px": n_px,
                "px_kms": _log(rng, 0.122, 0.4) if fine else PX_KMS, "line_px": 136.5 if fine else 10.29,
                "n_mu": rng.randint(8, 24), "n_phases": rng.randint(1, 100), "spots": rng.randint(1, 4),
                "faculae": rng.randint(0, 2), "vsini": rng.uniform(1.0, 5.0 if fine else 8.0),
                "lsf": rng.random() < 0.3, "limb": rng.random() < 0.3}
    if kind == "batch":
        single = rng.random() < 0.4
        rv = not single and rng.random() < 0.6
        lo = 1 if single else rng.randint(2, 30)
        return {"kind": kind, "n_items": int(_log(rng, 100, 3500)) if single else int(_log(rng, 8, 400)),
                "phases_lo": lo, "phases_hi": lo if single else rng.randint(lo, 200),
                "n_px": int(_log(rng, 4096, 16834)), "grid_n": rng.randint(80, 150),
                "residual": not rv and rng.random() < 0.6, "rv": rv, "tc": rng.random() < 0.5}
    if kind == "ccf":
        return {"kind": kind, "precision": rng.choice(["fp32", "fp32tc", "fp64"]), "n_spec": int(_log(rng, 1, 200)),
                "n_px": int(_log(rng, 8000, 102901)), "px_kms": PX_KMS, "line_px": 10.29,
                "vsini": rng.uniform(1.0, 8.0)}
    if kind == "local":
        return {"kind": kind, "n_mu": rng.randint(8, 24), "n_px": int(_log(rng, 8000, 205800)),
                "n_depth": rng.randint(2, 101), "grid_n": rng.randint(100, 300), "vsini": rng.uniform(1.0, 8.0)}
    if kind == "train":
        batch = 128 * int(_log(rng, 4, 32))
        return {"kind": kind, "rows": batch * rng.randint(1, 16) + rng.randint(0, 127), "batch": batch}
    if kind == "query":
        return {"kind": kind, "n": int(_log(rng, 1, 40000)), "n_px": int(_log(rng, 4096, 16834))}
    return {"kind": "project", "n": int(_log(rng, 300, 20011)), "n_px": int(_log(rng, 4096, 16834))}


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------
def _grid(case):
    delta = case.get("px_kms", PX_KMS) / C_KMS
    lam1 = LAM0 * math.exp((case["n_px"] - 1) * delta)
    return lam1, math.log1p((lam1 - LAM0) / LAM0) / (case["n_px"] - 1)


def _line_rows(n_px, slot, n_slots, centre, depth, sigma, mus, shift_px, depth_scale):
    """[n_mu, n_px] product of (1 - d g) over lines, line s inside slot s of `slot` pixels."""
    n = torch.arange(n_px, dtype=torch.float64, device=DEV)
    home = (n / slot).to(torch.int64)
    reach = int(math.ceil(5.0 * float(sigma.max()) / slot)) + 1
    c, d, s = (torch.from_numpy(a).to(DEV) for a in (centre, depth * depth_scale, sigma))
    mu = torch.from_numpy(mus).to(DEV)[:, None]
    out = torch.ones((len(mus), n_px), dtype=torch.float64, device=DEV)
    for q in range(-reach, reach + 1):
        k = home + q
        ok = (k >= 0) & (k < n_slots)
        k = k.clamp(0, n_slots - 1)
        z = (n - c[k] - shift_px * mu) / s[k]
        dep = torch.clamp(d[k] * (0.8 + 0.2 * mu), max=0.99) * ok
        out *= 1.0 - dep * torch.exp(-0.5 * z * z)
    return out


def _spectra(case, seed, mus, line_px):
    """Quiet and active local spectra (float64 on the GPU) and the CCF mask (host)."""
    rng = np.random.default_rng(seed)
    n_px = case["n_px"]
    _, delta = _grid(case)
    px = C_KMS * delta

    def lines(slot, lo, hi, law):
        m = max(1, int(n_px / slot))
        cen = (np.arange(m) + rng.uniform(0.05, 0.95, m)) * slot
        dep = np.exp(rng.uniform(np.log(lo), np.log(hi), m)) if law == "log" else rng.uniform(lo, hi, m)
        return m, cen, dep, rng.uniform(1.5, 4.0, m) / px

    m, cen, dep, sig = lines(line_px, 0.01, 0.9, "log") if line_px < 50 else lines(line_px, 0.1, 0.8, "uniform")
    m2, cen2, dep2, sig2 = lines(3 * line_px, 0.01, 0.1, "uniform")
    quiet = _line_rows(n_px, line_px, m, cen, dep, sig, mus, -0.3 / px, 1.0)
    active = _line_rows(n_px, line_px, m, cen, dep, sig, mus, 0.0, 1.2)
    active *= _line_rows(n_px, 3 * line_px, m2, cen2, dep2, sig2, mus, 0.0, 1.0)
    keep = dep > 0.05
    return quiet, active, LAM0 * np.exp(cen[keep] * delta), dep[keep].copy()


def _star(case, mus, vsini, incl):
    lam1, _ = _grid(case)
    return synth.Star(grid_n=case["grid_n"], vsini_kms=vsini, incl_deg=incl, u1=U1, u2=U2, lambda_start_A=LAM0,
                      lambda_end_A=lam1, n_px=case["n_px"], mu_values=mus, t_quiet_K=T_QUIET)


def _mus(n):
    return (np.arange(n) + 0.5) / n


def _velocities(vsini):
    half = vsini + V_MARGIN
    return -half, V_STEP, int(math.floor(2 * half / V_STEP + 1e-9)) + 1


def _star_inputs(case, seed):
    rng = np.random.default_rng(seed + 1)
    mus = 0.1 + 0.09 * np.arange(11) if case["n_mu"] == 11 else _mus(case["n_mu"])
    regions = [(synth.FACULA, rng.uniform(-60, 60), rng.uniform(0, 360), 0.15, 6100.0) for _ in range(case["faculae"])]
    for k in range(case["spots"]):
        lat, lon = rng.uniform(-60, 60), rng.uniform(0, 360)
        if k == 0 and regions:
            lat, lon = regions[0][1], regions[0][2]          # a spot inside the first facula
        regions.append((synth.SPOT, lat, lon, rng.uniform(0.05, 0.1), 4800.0))
    incl = 90.0 if case["vsini"] == 2.0 else rng.uniform(50.0, 90.0)
    quiet, active, ml, mw = _spectra(case, seed, mus, case["line_px"])
    if case["precision"] != "fp64":
        quiet, active = quiet.float(), active.float()
    phases = np.arange(case["n_phases"], dtype=np.float64) / case["n_phases"]
    return mus, regions, incl, quiet, active, ml, mw, phases


def _batch_inputs(case, seed):
    """Item, region and phase columns: 1-4 spots per configuration, or for single-phase items the
    surrogate's query parameters (a facula around one spot of its own temperature)."""
    rng = np.random.default_rng(seed + 2)
    n = case["n_items"]
    single = case["phases_hi"] == 1
    # phase counts go with the case, so that every seed has the same number of spectra
    n_ph = np.random.default_rng(n).integers(case["phases_lo"], case["phases_hi"] + 1, n)
    vsini, incl = rng.uniform(1, 10, n), rng.uniform(30, 90, n)
    regs, first, count, phases = [], [], [], []
    for i in range(n):
        first.append(len(regs))
        if single:
            lat, lon, r, fill = rng.uniform(-60, 60), rng.uniform(0, 360), rng.uniform(0.01, 0.2), rng.uniform(0, 3)
            regs.append((synth.FACULA, lat, lon, min(1.0, r * math.sqrt(1.0 + fill)), 6100.0))
            regs.append((synth.SPOT, lat, lon, r, rng.uniform(3800.0, 5600.0)))
            phases.append(np.array([rng.uniform(0, 1)]))
        else:
            for _ in range(int(rng.integers(1, 5))):
                regs.append((synth.SPOT, rng.uniform(-60, 60), rng.uniform(0, 360), rng.uniform(0.01, 0.2), 4800.0))
            phases.append(np.arange(n_ph[i]) / n_ph[i])
        count.append(len(regs) - first[-1])
    t, lat, lon, rad, temp = (np.array(c) for c in zip(*regs))
    cols = dict(vsini=vsini, incl=incl, first_region=np.array(first, np.int32), n_regions=np.array(count, np.int32),
                first_phase=np.concatenate([[0], np.cumsum(n_ph)[:-1]]).astype(np.int32),
                n_phases=n_ph.astype(np.int32), type=t.astype(np.int32), lat=lat, lon=lon, radius=rad, temp=temp,
                phases=np.concatenate(phases))
    return cols


def _ccf_inputs(case, seed):
    """Disk-integrated-looking spectra: one quiet row, each spectrum moved by its own sub-pixel shift."""
    rng = np.random.default_rng(seed + 3)
    base, _, ml, mw = _spectra(case, seed, np.array([0.6]), case["line_px"])
    base = base[0]
    shift = torch.from_numpy(rng.normal(0.0, 0.05, case["n_spec"])).to(DEV)
    lo, hi = torch.roll(base, 1), torch.roll(base, -1)
    slope = 0.5 * (hi - lo)
    slope[0] = slope[-1] = 0.0
    spectra = 0.25 * (lo + 2 * base + hi)[None, :] - shift[:, None] * slope[None, :]
    gain = torch.from_numpy(rng.uniform(1.5, 3.0, case["n_spec"])).to(DEV)
    spectra *= gain[:, None]
    return (spectra if case["precision"] == "fp64" else spectra.float()), ml, mw


def _local_inputs(case, seed):
    rng = np.random.default_rng(seed + 4)
    mus = _mus(case["n_mu"])
    quiet, _, _, _ = _spectra(case, seed, mus, 10.29)
    d = np.linspace(0.0, 1.0, case["n_depth"])
    a, b, c = rng.uniform(-1, 1, (3, case["n_mu"], 1)) * np.array([0.05, 0.25, 0.25])[:, None, None]
    return mus, quiet, a + b * d + c * d * d, np.zeros(case["n_depth"])


# network inputs: region centre in the observer frame (y, x, z), radius, temperature, vsini x, vsini, filling
NET_LO = np.array([-1.0, -1.0, 0.01, 3800.0, -1.0, -10.0, 1.0, 0.0])
NET_HI = np.array([1.0, 1.0, 0.2, 5600.0, 1.0, 10.0, 10.0, 3.0])
QUERY_LO = np.array([-60.0, 0.0, 0.01, 3800.0, 0.0, 30.0, 1.0, 0.0])
QUERY_HI = np.array([60.0, 360.0, 0.2, 5600.0, 1.0, 90.0, 10.0, 3.0])
SHAPES = ((HIDDEN, 8), (HIDDEN, HIDDEN), (HIDDEN, HIDDEN), (HIDDEN, HIDDEN), (N_COEF + 1, HIDDEN))


def _network(rng):
    parts = []
    for l, (o, i) in enumerate(SHAPES):
        parts += [rng.normal(0.0, math.sqrt((1.0 if l == len(SHAPES) - 1 else 2.0) / i), o * i),
                  rng.normal(0.0, 0.01, o)]
    return np.concatenate(parts).astype(np.float32)


def _queries(rng, n):
    return (QUERY_LO + (QUERY_HI - QUERY_LO) * rng.uniform(size=(n, 8))).astype(np.float32)


def _basis(seed, n_px):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed + 5)
    mean = 0.01 * torch.randn(n_px, generator=g, device=DEV)
    basis = torch.randn((N_COEF, n_px), generator=g, device=DEV) / math.sqrt(n_px)
    return mean, basis


def _query_inputs(case, seed):
    rng = np.random.default_rng(seed + 6)
    params = torch.from_numpy(_queries(rng, case["n"])).to(DEV)
    nets = _network(rng), _network(rng)
    std = (0.5 * 0.95 ** np.arange(N_COEF)).astype(np.float32)
    return params, nets, rng.normal(0.0, 0.01, N_COEF).astype(np.float32), std, _basis(seed, case["n_px"])


def _train_inputs(case, seed):
    rng = np.random.default_rng(seed + 7)
    params = torch.from_numpy(_queries(rng, case["rows"])).to(DEV)
    w = torch.from_numpy(rng.normal(0.0, 1.0, (8, N_COEF + 1)).astype(np.float32)).to(DEV)
    lo, hi = (torch.from_numpy(a.astype(np.float32)).to(DEV) for a in (QUERY_LO, QUERY_HI))
    z = (params - lo) / (hi - lo) * 2 - 1
    target = torch.zeros((case["rows"], N_COEF + 1), device=DEV)
    for i in range(8):                                        # a smooth map, one term at a time (fixed order)
        target += torch.sin(2.0 * z[:, i:i + 1] + w[i][None, :])
    target *= 0.5
    target[:, N_COEF] = 0.0
    loss_w = np.full(N_COEF + 1, 1.0 / N_COEF, np.float32)
    loss_w[N_COEF] = 0.0
    return params, target.contiguous(), loss_w, _network(rng)


def _project_inputs(case, seed):
    mean, basis = _basis(seed, case["n_px"])
    g = torch.Generator(device=DEV)
    g.manual_seed(seed + 8)
    x = torch.randn((case["n"], case["n_px"]), generator=g, device=DEV)
    x *= 0.02
    return x + mean, mean, basis


# ---------------------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------------------
class _Net:
    """A surrogate handle that frees itself."""

    def __init__(self, batch, params):
        self.h = S.soap_surrogate_create(NET_LO, NET_HI, batch, torch.cuda.current_stream())
        S.soap_surrogate_set_params(self.h, params)

    def __del__(self):
        try:
            S.soap_surrogate_free(self.h)
        except Exception:
            pass


PRECISION = {"fp64": S.SOAP_FP64, "fp32": S.SOAP_FP32, "fp32tc": S.SOAP_FP32, "bf16x3": S.SOAP_BF16X3}


def prepare(case, seed):
    st = {"case": case}
    kind = case["kind"]
    stream = torch.cuda.current_stream()
    if kind == "star":
        mus, regions, incl, quiet, active, ml, mw, phases = _star_inputs(case, seed)
        star = _star(case, mus, case["vsini"], incl)
        disk = S.Disk(star, quiet.double(), stream=stream)
        S.soap_set_ccf_tensor_cores(disk.ctx, case["precision"] == "fp32tc")
        S.soap_set_facula_limb_brightening(disk.ctx, case["limb"])
        S.soap_set_instrument_resolution(disk.ctx, LSF_R if case["lsf"] else 0.0)
        out = torch.empty((case["n_phases"], case["n_px"]), dtype=quiet.dtype, device=DEV)
        st.update(disk=disk, star=star, quiet=quiet, active=active, mask=(ml, mw), phases=phases, out=out,
                  regions=[synth.Region(*r) for r in regions], grid=_velocities(case["vsini"]),
                  rv=torch.empty(case["n_phases"], dtype=torch.float64, device=DEV))
    elif kind == "batch":
        mus = _mus(20)
        quiet, active, ml, mw = _spectra(case, seed, mus, 8.7)
        disk = S.Disk(_star(case, mus, 10.0, 90.0), quiet, {S.SOAP_SPOT: active}, stream=stream)
        if case["rv"]:
            lo, step, nv = _velocities(10.0)
            S.soap_batch_set_rv(disk.ctx, ml, mw, MASK_WIDTH, lo, step, nv, V_MARGIN, tensor_cores=case["tc"])
        arrays = S.batch_columns_arrays(_batch_inputs(case, seed))
        n = len(arrays[2])
        st.update(disk=disk, arrays=arrays, out=torch.empty((n, case["n_px"]), dtype=torch.float32, device=DEV),
                  rv=torch.empty(n, dtype=torch.float64, device=DEV) if case["rv"] else None)
    elif kind == "ccf":
        spectra, ml, mw = _ccf_inputs(case, seed)
        star = _star(dict(case, grid_n=50), np.array([1.0]), case["vsini"], 90.0)
        disk = S.Disk(star, spectra[:1].double().contiguous(), stream=stream)
        grid = _velocities(case["vsini"])
        f64 = dict(dtype=torch.float64, device=DEV)
        st.update(disk=disk, spectra=spectra, mask=(ml, mw), grid=grid, rv=torch.empty(case["n_spec"], **f64),
                  fit=torch.empty((case["n_spec"], 4), **f64), ccf=torch.empty((case["n_spec"], grid[2]), **f64))
    elif kind == "local":
        mus, quiet, bis, orig = _local_inputs(case, seed)
        disk = S.Disk(_star(case, mus, case["vsini"], 90.0), quiet, stream=stream)
        S.soap_set_instrument_resolution(disk.ctx, LSF_R)
        st.update(disk=disk, quiet=quiet, bis=bis, orig=orig, rows=torch.empty_like(quiet),
                  flux=torch.empty(case["n_px"], dtype=torch.float64, device=DEV))
    elif kind == "train":
        params, target, loss_w, net = _train_inputs(case, seed)
        x = torch.empty_like(params)
        S.soap_surrogate_encode(params, x, stream)
        st.update(net=_Net(case["batch"], net), weights=net, x=x, target=target, loss_w=loss_w, seed=seed)
    elif kind == "query":
        params, nets, mean, std, (mu, basis) = _query_inputs(case, seed)
        main, err = _Net(128, nets[0]), _Net(128, nets[1])
        S.soap_surrogate_set_scaling(main.h, mean, std)
        S.soap_surrogate_set_basis(main.h, mu, basis)
        S.soap_surrogate_set_error_net(main.h, err.h)
        n = case["n"]
        st.update(net=main, err=err, params=params, x=torch.empty_like(params),
                  out=torch.empty((n, case["n_px"]), device=DEV), pred=torch.empty(n, device=DEV),
                  accepted=torch.empty(n, dtype=torch.uint8, device=DEV))
    else:
        x, mean, basis = _project_inputs(case, seed)
        st.update(x=x, mean=mean, basis=basis, coef=torch.empty((case["n"], N_COEF), device=DEV))
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    stream = torch.cuda.current_stream()
    if kind == "star":
        ctx = st["disk"].ctx
        S.soap_update_star(ctx, st["star"])
        S.soap_set_quiet_spectrum(ctx, st["quiet"])
        S.soap_set_active_spectrum(ctx, S.SOAP_SPOT, st["active"])
        S.soap_active_rv(ctx, st["regions"], st["phases"], S.SOAP_EFFECT_TOT, PRECISION[case["precision"]], *st["mask"],
                         MASK_WIDTH, *st["grid"], st["out"], st["rv"])
        # RVs of float32 spectra are kept in float32 beside them, the results' own precision
        return st["out"], st["rv"].to(st["out"].dtype)
    if kind == "batch":
        items, regions, phases = st["arrays"]
        S.soap_active_batch_arrays(st["disk"].ctx, items, regions, phases, st["out"],
                                   output=S.SOAP_BATCH_RESIDUAL if case["residual"] else S.SOAP_BATCH_SPECTRUM,
                                   rv_out=st["rv"])
        return (st["out"], st["rv"].float()) if case["rv"] else (st["out"],)
    if kind == "ccf":
        S.soap_rv_ccf(st["disk"].ctx, st["spectra"], *st["mask"], MASK_WIDTH, *st["grid"], st["rv"], st["fit"],
                      st["ccf"], tensor_cores=case["precision"] == "fp32tc")
        return tuple(st[k].to(st["spectra"].dtype) for k in ("rv", "fit", "ccf"))
    if kind == "local":
        ctx = st["disk"].ctx
        S.soap_inject_bisectors(ctx, st["quiet"], st["rows"], st["bis"], st["orig"])
        S.soap_set_quiet_spectrum(ctx, st["rows"])
        S.soap_quiet_spectrum(ctx, S.SOAP_FORM_TOEPLITZ, S.SOAP_FP64, st["flux"])
        return st["rows"], st["flux"]
    if kind == "train":
        S.soap_surrogate_set_params(st["net"].h, st["weights"])
        loss = S.soap_surrogate_train(st["net"].h, st["x"], st["target"], 1, 3e-3, st["loss_w"], stage=0,
                                      seed=st["seed"])
        return S.soap_surrogate_get_params(st["net"].h), loss
    if kind == "query":
        S.soap_surrogate_encode(st["params"], st["x"], stream)
        S.soap_surrogate_query(st["net"].h, st["x"], 10.0, st["out"], st["accepted"], st["pred"])
        return st["out"], st["pred"], st["accepted"]
    S.soap_pca_project(st["x"], st["mean"], st["basis"], st["coef"], stream)
    return (st["coef"],)


# ---------------------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------------------
def _ccf_flops(n_px, line_px, vsini, n_spec):
    """One multiply-add per mask line, pixel the velocity grid sweeps and spectrum."""
    lines = 0.65 * n_px / line_px
    return 2.0 * lines * (2 * (vsini + V_MARGIN) / PX_KMS + 2) * n_spec


def work(case):
    kind, n_px = case["kind"], case.get("n_px", 0)
    if kind == "star":
        size = 8 if case["precision"] == "fp64" else 4
        taps = 2 * case["vsini"] / case["px_kms"] + 2
        per_px = 2.0 * (case["n_mu"] * taps + case["n_phases"] * 4 * (case["spots"] + case["faculae"]))
        return {"bytes": size * n_px * (2 * case["n_mu"] + case["n_phases"]),
                "flops": per_px * n_px + _ccf_flops(n_px, case["line_px"], case["vsini"], case["n_phases"])}
    if kind == "batch":
        n = case["n_items"] * 0.5 * (case["phases_lo"] + case["phases_hi"])
        return {"bytes": 4 * n_px * n + 320 * n_px,
                "flops": 2.0 * 20 * n_px * n + (_ccf_flops(n_px, 8.7, 10.0, n) if case["rv"] else 0.0)}
    if kind == "ccf":
        size = 8 if case["precision"] == "fp64" else 4
        return {"bytes": size * n_px * case["n_spec"], "flops": _ccf_flops(n_px, case["line_px"], case["vsini"],
                                                                          case["n_spec"])}
    if kind == "local":
        taps = 2 * case["vsini"] / PX_KMS + 2
        return {"bytes": 16 * n_px * case["n_mu"] + 8 * n_px, "flops": n_px * case["n_mu"] * (30.0 + 2 * taps)}
    weights = sum(o * i for o, i in SHAPES)
    if kind == "train":
        rows = case["rows"] // case["batch"] * case["batch"]
        return {"bytes": rows * 4 * (8 + N_COEF + 1) + 8 * weights, "flops": 6.0 * weights * rows}
    if kind == "query":
        n = case["n"]
        return {"bytes": 4 * n * (8 + n_px) + 4 * N_COEF * n_px, "flops": n * (4.0 * weights + 2.0 * N_COEF * n_px)}
    return {"bytes": 4 * n_px * (case["n"] + N_COEF), "flops": 2.0 * N_COEF * n_px * case["n"]}


# ---------------------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------------------
def _t(a):
    return torch.as_tensor(np.asarray(a, np.float64), device=DEV)


def _cells(n):
    c = (2.0 * torch.arange(n, dtype=torch.float64, device=DEV) + 1 - n) / n
    y, x = torch.meshgrid(c, c, indexing="ij")
    vis = x * x + y * y < 1
    x, y = x[vis], y[vis]
    mu = torch.sqrt(1 - x * x - y * y)
    weight = (2.0 / n) ** 2 * (1 - U1 * (1 - mu) - U2 * (1 - mu) ** 2)
    return x, y, mu, weight


def _taps(x, vsini, delta):
    s = torch.atanh(vsini * x / C_KMS) / delta
    j = torch.ceil(s)
    return j.to(torch.int64), torch.expm1((j - s) * delta) / math.expm1(delta)


def _shifted(rows, taps):
    """[n_mu, n_taps, n_px]: rows moved by each tap, end values repeating."""
    n_px = rows.shape[1]
    m = torch.arange(n_px, device=DEV)
    return torch.stack([rows[:, (m - k).clamp(0, n_px - 1)] for k in taps], 1)


def _owners(x, y, mu, regions, incl, phases):
    """[n_phases, n_cells] index of the region that owns each cell (the last one in the list), or -1."""
    si, ci = math.sin(math.radians(incl)), math.cos(math.radians(incl))
    own = torch.full((len(phases), len(x)), -1, dtype=torch.int64, device=DEV)
    p = _t(phases)[:, None]
    for q, (_, lat, lon, rad, _) in enumerate(regions):
        la, lo = math.radians(lat), torch.deg2rad(lon + 360.0 * p)
        px, pc, ps = math.cos(la) * torch.sin(lo), math.cos(la) * torch.cos(lo), math.sin(la)
        dot = x * px + y * (ps * si - pc * ci) + mu * (ps * ci + pc * si)
        own[dot >= math.sqrt(1 - rad * rad)] = q
    return own


def _kernels(own, member, col0, n_col, weight, w):
    """[n_phases, n_col] two-tap sums of the cells that regions in `member` own."""
    on = torch.zeros(own.shape, dtype=torch.bool, device=DEV)
    for q in member:
        on |= own == q
    k = torch.zeros((own.shape[0], n_col), dtype=torch.float64, device=DEV)
    idx = col0[None, :].expand(own.shape[0], -1)
    k.scatter_add_(1, idx, on * (weight * (1 - w)))
    k.scatter_add_(1, idx - 1, on * (weight * w))
    return k


def _planck(lam, temp):
    return 1.0 / torch.expm1(HCK / (lam * temp))


def _lsf(rows, delta):
    sigma = 1.0 / (LSF_R * delta * 2.0 * math.sqrt(2.0 * math.log(2.0)))
    reach = int(math.ceil(6.0 * sigma)) + 1
    g = np.array([0.5 * (math.erfc((abs(k) - 0.5) / (sigma * math.sqrt(2))) -
                         math.erfc((abs(k) + 0.5) / (sigma * math.sqrt(2)))) for k in range(-reach, reach + 1)])
    g /= g.sum()
    m = torch.arange(rows.shape[1], device=DEV)
    out = torch.zeros_like(rows)
    for k in range(-reach, reach + 1):
        out += g[k + reach] * rows[:, (m - k).clamp(0, rows.shape[1] - 1)]
    return out


def _mask_matrix(n_px, delta, ml, mw, grid):
    """[n_px, n_v] overlap of the mask's boxes with the pixels at every velocity."""
    lo, step, nv = grid
    u = torch.log(_t(ml) / LAM0) / delta
    s = torch.atanh((lo + step * torch.arange(nv, dtype=torch.float64, device=DEV)) / C_KMS) / delta
    h = MASK_WIDTH / (2 * C_KMS * delta)
    ok = (u + s[0] - h >= -0.5) & (u + s[-1] + h <= n_px - 0.5)
    u, w = u[ok], _t(mw)[ok]
    a = u[:, None] + s[None, :] - h + 0.5                    # box start, pixel n covering [n, n + 1)
    n0 = torch.floor(a)
    col = torch.arange(nv, device=DEV)[None, :].expand_as(a)
    m = torch.zeros((n_px, nv), dtype=torch.float64, device=DEV)
    for i in range(int(math.ceil(2 * h)) + 1):
        n = n0 + i
        part = (torch.minimum(a + 2 * h, n + 1) - torch.maximum(a, n)).clamp(min=0) * w[:, None]
        m.index_put_((n.to(torch.int64).clamp(0, n_px - 1), col), part, accumulate=True)
    return m


def _fit(ccf, grid, half=None):
    """Least-squares Gaussians (A, B, mu, s) of CCFs [n, n_v]; half: per row, fit |v| <= half only."""
    lo, step, nv = grid
    v = lo + step * torch.arange(nv, dtype=torch.float64, device=DEV)[None, :]
    on = torch.ones_like(ccf) if half is None else (v.abs() <= half[:, None] + 1e-9).to(ccf.dtype)
    inf = torch.full_like(ccf, math.inf)
    top = torch.where(on > 0, ccf, -inf).amax(1, keepdim=True)
    low, at = torch.where(on > 0, ccf, inf).min(1, keepdim=True)
    y = ccf / top.abs()
    top, low, scale = top / top.abs(), low / top.abs(), top.abs()
    s0 = ((top - y) * on).sum(1, keepdim=True) * step / ((low - top).abs() * math.sqrt(2 * math.pi))
    s0, c0 = s0.clamp(min=step), lo + step * at
    t = (v - c0) / s0
    p = torch.cat([top, low - top, torch.zeros_like(top), torch.ones_like(top)], 1)

    def model(p):
        d = (t - p[:, 2:3]) / p[:, 3:4]
        g = torch.exp(-0.5 * d * d)
        r = (p[:, 0:1] + p[:, 1:2] * g - y) * on
        b = p[:, 1:2] * g / p[:, 3:4]
        return r, d, g, torch.stack([on, g * on, b * d * on, b * d * d * on], 2)

    lam = torch.full((len(y), 1, 1), 1e-3, dtype=torch.float64, device=DEV)
    r, d, g, jac = model(p)
    for _ in range(60):
        h = jac.transpose(1, 2) @ jac
        grad = jac.transpose(1, 2) @ r[:, :, None]
        hd = h + lam * torch.diag_embed(torch.diagonal(h, dim1=1, dim2=2))
        q = p - torch.linalg.solve(hd, grad)[:, :, 0]
        r2, d2, g2, jac2 = model(q)
        better = (r2 * r2).sum(1) <= (r * r).sum(1)
        p = torch.where(better[:, None], q, p)
        lam = torch.where(better[:, None, None], lam * 0.1, lam * 10).clamp(1e-12, 1e6)
        r, jac = torch.where(better[:, None], r2, r), torch.where(better[:, None, None], jac2, jac)
    for _ in range(6):                                        # Newton on the exact Hessian
        r, d, g, jac = model(p)
        h = jac.transpose(1, 2) @ jac
        w, b = p[:, 3], p[:, 1]
        m = [(r * g * d ** k).sum(1) for k in range(5)]
        h[:, 1, 2] += m[1] / w
        h[:, 1, 3] += m[2] / w
        h[:, 2, 2] += b / w ** 2 * (m[2] - m[0])
        h[:, 2, 3] += b / w ** 2 * (m[3] - 2 * m[1])
        h[:, 3, 3] += b / w ** 2 * (m[4] - 3 * m[2])
        for i, k in ((2, 1), (3, 1), (3, 2)):
            h[:, i, k] = h[:, k, i]
        p = p - torch.linalg.solve(h, jac.transpose(1, 2) @ r[:, :, None])[:, :, 0]
    mu, wid = p[:, 2] * s0[:, 0] + c0[:, 0], p[:, 3].abs() * s0[:, 0]
    return torch.stack([p[:, 0] * scale[:, 0], p[:, 1] * scale[:, 0], mu, wid], 1)


def _exact_star(case, seed):
    mus, regions, incl, quiet, active, ml, mw, phases = _star_inputs(case, seed)
    quiet, active = quiet.double(), active.double()
    n_px, n_mu = case["n_px"], len(mus)
    _, delta = _grid(case)
    x, y, mu, weight = _cells(case["grid_n"])
    bins = (mu[:, None] - _t(mus)[None, :]).abs().argmin(1)
    j, w = _taps(x, case["vsini"], delta)
    k0, k1 = int(j.min()) - 1, int(j.max())
    taps = list(range(k0, k1 + 1))
    col0, n_col = bins * len(taps) + (j - k0), n_mu * len(taps)
    kq = torch.zeros(n_col, dtype=torch.float64, device=DEV)
    kq.index_add_(0, col0, weight * (1 - w))
    kq.index_add_(0, col0 - 1, weight * w)
    lam = LAM0 * torch.exp(delta * torch.arange(n_px, dtype=torch.float64, device=DEV))
    own = _owners(x, y, mu, regions, incl, phases)
    classes = {}
    for q, r in enumerate(regions):
        classes.setdefault((r[0], r[4]), []).append(q)
    ker = {c: _kernels(own, q, col0, n_col, weight, w) for c, q in classes.items()}
    flux = torch.zeros((len(phases), n_px), dtype=torch.float64, device=DEV)
    for b in range(n_mu):
        cols = slice(b * len(taps), (b + 1) * len(taps))
        sq = _shifted(quiet[b:b + 1], taps)[0]
        sa = _shifted(active[b:b + 1], taps)[0]
        flux += kq[cols] @ sq
        for (kind, temp), k in ker.items():
            if case["limb"] and kind == synth.FACULA:
                temp = T_QUIET + 250.9 - 407.7 * mus[b] + 190.9 * mus[b] ** 2
            flux += (k[:, cols] @ sa) * (_planck(lam, temp) / _planck(lam, T_QUIET)) - k[:, cols] @ sq
    if case["lsf"]:
        flux = _lsf(flux, delta)
    grid = _velocities(case["vsini"])
    return flux, _fit(flux @ _mask_matrix(n_px, delta, ml, mw, grid), grid)[:, 2]


def _exact_batch(case, seed):
    mus = _mus(20)
    quiet, active, ml, mw = _spectra(case, seed, mus, 8.7)
    cols = _batch_inputs(case, seed)
    n_px = case["n_px"]
    _, delta = _grid(case)
    x, y, mu, weight = _cells(case["grid_n"])
    bins = (mu[:, None] - _t(mus)[None, :]).abs().argmin(1)
    reach = int(math.ceil(math.atanh(10.0 / C_KMS) / delta)) + 1
    taps = list(range(-reach, reach + 1))
    n_col = 20 * len(taps)
    sq, sa = (_shifted(r, taps).reshape(n_col, n_px) for r in (quiet, active))
    lam = LAM0 * torch.exp(delta * torch.arange(n_px, dtype=torch.float64, device=DEV))
    out = torch.empty((len(cols["phases"]), n_px), dtype=torch.float64, device=DEV)
    for i in range(case["n_items"]):
        r0, p0 = int(cols["first_region"][i]), int(cols["first_phase"][i])
        rs, ps = slice(r0, r0 + int(cols["n_regions"][i])), slice(p0, p0 + int(cols["n_phases"][i]))
        regions = list(zip(*(cols[k][rs] for k in ("type", "lat", "lon", "radius", "temp"))))
        j, w = _taps(x, float(cols["vsini"][i]), delta)
        col0 = bins * len(taps) + (j + reach)
        own = _owners(x, y, mu, regions, float(cols["incl"][i]), cols["phases"][ps])
        total = torch.zeros((own.shape[0], n_col), dtype=torch.float64, device=DEV)
        flux = torch.zeros((own.shape[0], n_px), dtype=torch.float64, device=DEV)
        for temp in sorted({r[4] for r in regions}):
            k = _kernels(own, [q for q, r in enumerate(regions) if r[4] == temp], col0, n_col, weight, w)
            total -= k
            used = k.abs().amax(0) > 0
            flux += (k[:, used] @ sa[used]) * (_planck(lam, float(temp)) / _planck(lam, T_QUIET))
        if not case["residual"]:
            total.index_add_(1, col0, (weight * (1 - w)).expand(len(total), -1))
            total.index_add_(1, col0 - 1, (weight * w).expand(len(total), -1))
        used = total.abs().amax(0) > 0
        out[ps] = flux + total[:, used] @ sq[used]
    if not case["rv"]:
        return (out,)
    grid = _velocities(10.0)
    half = _t(np.repeat(np.abs(cols["vsini"]) + V_MARGIN, cols["n_phases"]))
    m = _mask_matrix(n_px, delta, ml, mw, grid)
    rv = [_fit(out[a:a + 8192] @ m, grid, half[a:a + 8192])[:, 2] for a in range(0, len(out), 8192)]
    return out, torch.cat(rv)


def _exact_local(case, seed):
    mus, quiet, bis, orig = _local_inputs(case, seed)
    n_px = case["n_px"]
    _, delta = _grid(case)
    n = torch.arange(n_px, dtype=torch.float64, device=DEV)
    rows = torch.empty_like(quiet)
    for b in range(case["n_mu"]):
        f = quiet[b]
        tab = _t(bis[b] - orig)
        pos = (1 - f).clamp(0, 1) * (case["n_depth"] - 1)
        i = pos.to(torch.int64).clamp(max=case["n_depth"] - 2)
        v = tab[i] + (pos - i) * (tab[i + 1] - tab[i])
        u = n + torch.atanh(v / C_KMS) / delta
        k = torch.searchsorted(u, n, right=True) - 1
        kc = k.clamp(0, n_px - 2)
        w = torch.expm1((n - u[kc]) * delta) / torch.expm1((u[kc + 1] - u[kc]) * delta)
        val = f[kc] + w * (f[kc + 1] - f[kc])
        rows[b] = torch.where(k < 0, f[0], torch.where(k >= n_px - 1, f[-1], val))
    x, _, mu, weight = _cells(case["grid_n"])
    bins = (mu[:, None] - _t(mus)[None, :]).abs().argmin(1)
    j, w = _taps(x, case["vsini"], delta)
    k0 = int(j.min()) - 1
    taps = list(range(k0, int(j.max()) + 1))
    kq = torch.zeros(case["n_mu"] * len(taps), dtype=torch.float64, device=DEV)
    col0 = bins * len(taps) + (j - k0)
    kq.index_add_(0, col0, weight * (1 - w))
    kq.index_add_(0, col0 - 1, weight * w)
    flux = torch.zeros(n_px, dtype=torch.float64, device=DEV)
    for b in range(case["n_mu"]):
        flux += kq[b * len(taps):(b + 1) * len(taps)] @ _shifted(rows[b:b + 1], taps)[0]
    return rows, _lsf(flux[None, :], delta)[0]


def _encode(params):
    q = params.double()
    lat, lon, inc = torch.deg2rad(q[:, 0]), torch.deg2rad(q[:, 1] + 360 * q[:, 4]), torch.deg2rad(q[:, 5])
    px, ps, pc = torch.cos(lat) * torch.sin(lon), torch.sin(lat), torch.cos(lat) * torch.cos(lon)
    return torch.stack([ps * torch.sin(inc) - pc * torch.cos(inc), px, q[:, 2], q[:, 3],
                        ps * torch.cos(inc) + pc * torch.sin(inc), q[:, 6] * px, q[:, 6], q[:, 7]], 1)


def _forward(flat, x):
    a = 2 * (x - _t(NET_LO)) / _t(NET_HI - NET_LO) - 1
    at = 0
    for l, (o, i) in enumerate(SHAPES):
        w, b = _t(flat[at:at + o * i]).reshape(o, i), _t(flat[at + o * i:at + o * i + o])
        at += o * i + o
        a = a @ w.T + b
        if l < len(SHAPES) - 1:
            a = 0.5 * a * (1 + torch.erf(a / math.sqrt(2)))
    return a


def exact(case, seed):
    kind = case["kind"]
    if kind == "star":
        return _exact_star(case, seed)
    if kind == "batch":
        return _exact_batch(case, seed)
    if kind == "ccf":
        spectra, ml, mw = _ccf_inputs(case, seed)
        grid = _velocities(case["vsini"])
        ccf = spectra.double() @ _mask_matrix(case["n_px"], _grid(case)[1], ml, mw, grid)
        fit = _fit(ccf, grid)
        return fit[:, 2], fit, ccf
    if kind == "local":
        return _exact_local(case, seed)
    if kind == "query":
        params, nets, mean, std, (mu, basis) = _query_inputs(case, seed)
        x = _encode(params)
        coef = _forward(nets[0], x)[:, :N_COEF] * _t(std) + _t(mean)
        return mu.double() + coef @ basis.double(), 10.0 ** _forward(nets[1], x)[:, N_COEF], None
    if kind == "project":
        x, mean, basis = _project_inputs(case, seed)
        coef = torch.empty((case["n"], N_COEF), dtype=torch.float64, device=DEV)
        for a in range(0, case["n"], 4096):
            coef[a:a + 4096] = (x[a:a + 4096].double() - mean.double()) @ basis.double().T
        return (coef,)
    # train: the weights after many BF16-operand steps depend on the library's own shuffle of the rows
    return None
