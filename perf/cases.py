"""Performance cases: the calls that a user of this framework spends time in, at the sizes met
in use, each through an entry point of `fitcore` or `warmstart`.

Kinds of case (`kind`):
  eval      fit_model_eval: -2lnL and its gradient of `batch` parameter vectors (what a minimiser,
            a sampler or an autograd program outside the library calls)
  expect    fit_model_expected_tc, split-TF32 fold: expected counts of `batch` parameter vectors
            (pseudo-experiment and training-set generation)
  events    fit_mc_spectrum: `events` simulated events reweighted for `sets` parameter sets
  train     one AdamW step of the warm-start network on `batch` samples
  starts    start points of `batch` fits: linearised best fit plus the network's corrections
  fit       fit_batch from a cold start on `batch` pseudo-experiments
  scan      fit_profile_scan of one oscillation parameter over `points` held values

Models are the ones of `synth`: c0 (one detector, 25 parameters), c1 (three datasets, 291), c1s
(c1 with the 3+1 formula, 293), c2 (53 km, 460 parameters, 2000 true bins); `spline` selects the
paper's area-conserving energy correction instead of the overlap rule. `masks` "mixed": every
pseudo-experiment of c1 fits one of the dataset subsets of `synth.C1_MASKS`, as the uneven
ensemble does.

Fits are measured on c2 and on the spline models. With the overlap rule on the coarse grids of c0
and c1 the likelihood has creases with separate minima on them, and which one a fit ends in
turns on the last bit of an evaluation, so best fits there cannot be compared one by one (the
evaluations themselves can, and c1 with the overlap rule is an `eval` case). Of a fit the best
point and -2lnL there are returned; iteration counts and the last EDM say how the minimiser got
there, to rounding.

Everything the library computes, it computes in FP32 (doubles carry parameter vectors, sums and
results across the boundary). A double output is therefore returned as the FP32 number whose
digits it has.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2502_15253_gb300 import fitcore, synth, warmstart

K_OSC = 1.266932679815373   # dm2[eV^2] L[m] / (4 E[MeV]) in radians
DEV = "cuda"


# ---- cases ---------------------------------------------------------------------------------
def listed():
    return [
        # one step of an external minimiser on the Double Chooz-like fit: latency
        {"name": "eval c1 x1", "kind": "eval", "model": "c1", "spline": False, "batch": 1, "masks": "all"},
        # a generation of sampler walkers or finite differences around a best fit, dataset subsets mixed
        {"name": "eval c1 x4096", "kind": "eval", "model": "c1", "spline": False, "batch": 4096, "masks": "mixed"},
        # the 53 km model, the largest of the configurations
        {"name": "eval c2 x2048", "kind": "eval", "model": "c2", "spline": False, "batch": 2048, "masks": "all"},
        # the sterile search with the paper's spline correction, an odd batch
        {"name": "eval c1s spline x509", "kind": "eval", "model": "c1s", "spline": True, "batch": 509, "masks": "all"},
        # spectra for pseudo-experiments and for training
        {"name": "expect c2 x4096", "kind": "expect", "model": "c2", "spline": False, "batch": 4096},
        # the paper's event-level step: a full simulation sample at one parameter set
        {"name": "events dc 12M x1", "kind": "events", "geometry": "dc_fd", "events": 12_000_000, "sets": 1},
        # the same for the medium baseline, many parameter sets per pass
        {"name": "events juno 1.5M x24", "kind": "events", "geometry": "juno_fd", "events": 1_500_001, "sets": 24},
        # a training step at the trainer's default batch
        {"name": "train x4096", "kind": "train", "batch": 4096},
        # start points for an ensemble
        {"name": "starts c1 x3001", "kind": "starts", "model": "c1", "batch": 3001, "masks": "mixed"},
        # ensembles of fits: the main path
        {"name": "fit c2 x1000", "kind": "fit", "model": "c2", "spline": False, "batch": 1000, "masks": "all"},
        {"name": "fit c1 spline x2500", "kind": "fit", "model": "c1", "spline": True, "batch": 2500, "masks": "mixed"},
        # a profile of one mass splitting (the ordering study): few, long fits
        {"name": "scan c2 x41", "kind": "scan", "model": "c2", "spline": False, "param": "dm2_31", "points": 41},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["eval", "eval", "eval", "eval", "expect", "events", "events", "train", "starts", "fit", "fit", "scan"])
    if kind == "eval":
        model = rng.choice(["c0", "c1", "c1", "c1s", "c2", "c2"])
        spline = rng.random() < 0.3
        top = 2048 if model == "c2" else 4096
        return {"kind": kind, "model": model, "spline": spline, "batch": size(1, top),
                "masks": "mixed" if model == "c1" and rng.random() < 0.5 else "all"}
    if kind == "expect":
        model = rng.choice(["c1", "c2"])
        return {"kind": kind, "model": model, "spline": rng.random() < 0.3, "batch": size(64, 4096)}
    if kind == "events":
        if rng.random() < 0.5:
            return {"kind": kind, "geometry": "dc_fd", "events": size(100_000, 12_000_000), "sets": 1}
        return {"kind": kind, "geometry": rng.choice(["dc_fd", "juno_fd"]), "events": size(100_000, 1_500_000),
                "sets": size(2, 64)}
    if kind == "train":
        return {"kind": kind, "batch": size(512, 16384)}
    if kind == "starts":
        model = rng.choice(["c1", "c2"])
        return {"kind": kind, "model": model, "batch": size(64, 4096), "masks": "mixed" if model == "c1" else "all"}
    if kind == "fit":
        model = rng.choice(["c0", "c1", "c2"])
        if model == "c2":
            return {"kind": kind, "model": model, "spline": False, "batch": size(16, 1000), "masks": "all"}
        return {"kind": kind, "model": model, "spline": True, "batch": size(16, 2500),
                "masks": rng.choice(["all", "mixed"]) if model == "c1" else "all"}
    model = rng.choice(["c1", "c2"])
    return {"kind": "scan", "model": model, "spline": model == "c1", "param": "sin2_2th13" if model == "c1" else "dm2_31",
            "points": size(11, 101)}


# ---- models and inputs -----------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _spec(model, spline):
    return synth.make_model(model, remap=1 if spline else 0)


@functools.lru_cache(maxsize=None)
def _model(model, spline):
    """The model handle, created once and kept as a user's program keeps it."""
    return fitcore.Model(_spec(model, spline))


def _whitened(spec, z):
    """theta0 + J z for rows of z [B, P]: prior widths, step scales, Cholesky factors of the blocks."""
    s = np.where(spec.prior_sigma > 0, spec.prior_sigma, spec.scale)
    th = spec.theta0 + s * z
    for ix, cov in spec.cov_blocks:
        th[:, ix] = spec.theta0[ix] + z[:, ix] @ np.linalg.cholesky(cov).T
    return th


def _thetas(spec, batch, rng):
    """Points a minimiser or sampler visits: about half a prior width around nominal."""
    th = _whitened(spec, 0.5 * rng.standard_normal((batch, spec.n_params)))
    if spec.osc_mode == synth.OSC_STERILE4:   # sterile mixing and splitting over the search range
        th[:, spec.index("sin2_2th14")] = rng.uniform(0.005, 0.2, batch)
        th[:, spec.index("dm2_41")] = np.exp(rng.uniform(math.log(2e-3), math.log(0.5), batch))
    return th


def _masks(case, spec, batch, rng):
    if case.get("masks") == "mixed":
        return np.array(synth.C1_MASKS, np.uint32)[rng.integers(len(synth.C1_MASKS), size=batch)]
    return np.full(batch, spec.all_mask(), np.uint32)


def _pseudo_data(spec, batch, rng):
    """Poisson counts around the expectations of 16 true points within +-3 widths of nominal."""
    th = np.tile(spec.theta0, (16, 1))
    if spec.name in synth.TRUE_DRAW_SIGMA:
        th = np.array([synth.draw_theta_true(spec, rng) for _ in range(16)])
    with torch.no_grad():
        mu = _expected64(spec, torch.tensor(th, device=DEV)).cpu().numpy()
    return rng.poisson(mu[rng.integers(16, size=batch)]).astype(np.float32)


def _events(case, seed):
    """Simulated events as synth.make_mc_events describes them, drawn on the GPU: energies by
    inverse CDF, a core in proportion to L^-2, smeared into reco bins, sorted by bin."""
    far = case["geometry"] == "dc_fd"
    n = case["events"]
    L = np.array([950.0, 1150.0]) if far else np.linspace(52_000.0, 53_500.0, 10)
    res, lo, hi, n_bins = (0.08, 1.0, 8.6, 38) if far else (0.03, 1.018, 7.218, 400)
    grid = np.linspace(1.8, 10.0, 20_001)
    mid = 0.5 * (grid[:-1] + grid[1:])
    x = np.clip(np.minimum(mid - 1.8, 10.0 - mid) / synth.SPECTRUM_TAPER_MEV, 0.0, 1.0)
    cdf = np.concatenate([[0.0], np.cumsum(synth.flux_xsec(mid) * x * x * (3.0 - 2.0 * x))])
    cdf = torch.tensor(cdf / cdf[-1], device=DEV)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    m = int(1.1 * n) + 1000
    u = torch.rand(m, generator=gen, device=DEV, dtype=torch.float64)
    cell = (torch.searchsorted(cdf, u, right=True) - 1).clamp(0, len(mid) - 1)
    e = 1.8 + (cell + (u - cdf[cell]) / (cdf[cell + 1] - cdf[cell]).clamp_min(1e-300)) * (grid[1] - grid[0])
    w = torch.tensor(L ** -2.0, device=DEV)
    core = torch.searchsorted(torch.cumsum(w / w.sum(), 0), torch.rand(m, generator=gen, device=DEV, dtype=torch.float64))
    vis = (e - synth.PROMPT_SHIFT_MEV).clamp_min(1e-3)
    rec = vis + res * vis.sqrt() * torch.randn(m, generator=gen, device=DEV, dtype=torch.float64)
    b = torch.floor((rec - lo) / ((hi - lo) / n_bins)).long()
    keep = torch.nonzero((b >= 0) & (b < n_bins)).flatten()[:n]
    keep = keep[torch.sort(b[keep], stable=True).indices]
    mode = synth.OSC_EQ1 if far else synth.OSC_VACUUM3
    nominal = np.array([0.09, 2.5e-3, 0.851, 7.53e-5] if far else [0.307, 0.022, 7.5e-5, 2.5e-3])
    n_exp = 40_000.0 if far else 100_000.0
    return synth.McEvents(energy=e[keep].float().cpu().numpy(), core=core[keep].clamp(0, len(L) - 1).byte().cpu().numpy(),
                          weight=np.full(len(keep), 0.9 * n_exp / n, np.float32), bin=b[keep].int().cpu().numpy(),
                          n_bins=n_bins, core_L=L, osc_mode=mode, osc_nominal=nominal)


def _event_params(case, rng):
    far = case["geometry"] == "dc_fd"
    nominal = np.array([0.09, 2.5e-3, 0.851, 7.53e-5] if far else [0.307, 0.022, 7.5e-5, 2.5e-3])
    width = np.array([0.016, 1e-4, 0.02, 1.8e-6] if far else [0.013, 7e-4, 2e-6, 1e-5])
    return nominal + width * rng.uniform(-3.0, 3.0, (case["sets"], 4))


def _training_batch(batch, seed):
    """Standardised counts and targets as the trainer forms them: log-normalised spectra scatter by
    about their relative Poisson error, targets by a fraction of a width."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    x = torch.randn((batch, warmstart.N_IN), generator=gen, device=DEV) * 0.03
    y = torch.randn((batch, warmstart.N_OUT), generator=gen, device=DEV) * 0.5
    return x, y


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    st = {"case": case}
    if kind == "events":
        ev = _events(case, seed)
        st["mc"] = fitcore.McEventSet(ev)
        st["params"] = torch.tensor(_event_params(case, rng), device=DEV)
        st["out"] = torch.zeros((case["sets"], ev.n_bins), dtype=torch.float64, device=DEV)
        return st
    if kind == "train":
        st["net"] = warmstart.network(seed)
        st["x"], st["y"] = _training_batch(case["batch"], seed)
        st["loss"] = torch.zeros(1, dtype=torch.float64, device=DEV)
        st["grads"] = [(torch.empty(st["net"].layer_shape(k), device=DEV), torch.empty(st["net"].layer_shape(k)[0], device=DEV))
                       for k in range(st["net"].n_layers)]
        return st
    spline = bool(case.get("spline", False))
    spec, model = _spec(case["model"], spline), _model(case["model"], spline)
    P, D = spec.n_params, spec.n_bins
    st["model"], st["spec"] = model, spec
    if kind == "scan":
        lim = synth.TRUE_DRAW_SIGMA[case["model"]][case["param"]] * 3.0
        i = spec.index(case["param"])
        st["index"] = i
        st["points"] = spec.theta0[i] + np.linspace(-lim, lim, case["points"])
        st["data"] = torch.tensor(_pseudo_data(spec, 1, rng), device=DEV)
        return st
    B = case["batch"]
    if kind == "expect":
        st["theta"] = torch.tensor(_thetas(spec, B, rng), device=DEV)
        st["mu"] = torch.empty((B, D), device=DEV)
        st["status"] = torch.empty(B, dtype=torch.int32, device=DEV)
        return st
    masks = _masks(case, spec, B, rng)
    st["data"] = torch.tensor(_pseudo_data(spec, B, rng), device=DEV)
    if kind == "eval":
        st["theta"] = torch.tensor(_thetas(spec, B, rng), device=DEV)
        st["masks"] = torch.tensor(masks.astype(np.int32), device=DEV) if case["masks"] == "mixed" else None
        st["nll"] = torch.empty(B, dtype=torch.float64, device=DEV)
        st["grad"] = torch.empty((B, P), device=DEV)
        st["status"] = torch.empty(B, dtype=torch.int32, device=DEV)
    elif kind == "starts":
        st["net"] = warmstart.network(seed)
        st["masks"] = torch.tensor(masks.astype(np.int32), device=DEV)
        st["theta"] = torch.empty((B, P), dtype=torch.float64, device=DEV)
    else:
        inst = np.zeros(B, fitcore.INSTANCE_DTYPE)
        inst["mask"] = masks
        inst["data_off"] = np.arange(B) * D
        inst["param_off"] = np.arange(B) * P
        st["inst"] = inst
        st["best"] = torch.empty(B * P, dtype=torch.float64, device=DEV)
        st["results"] = torch.empty(B * fitcore.RESULT_DTYPE.itemsize, dtype=torch.uint8, device=DEV)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "eval":
        fitcore.fit_model_eval(st["model"], case["batch"], st["theta"], st["data"], st["masks"], st["nll"], st["grad"],
                               st["status"])
        return {"nll": st["nll"].float(), "grad": st["grad"], "status": st["status"]}
    if kind == "expect":
        fitcore.fit_model_expected_tc(st["model"], case["batch"], st["theta"], st["mu"], st["status"], precision=1)
        return {"mu": st["mu"], "status": st["status"]}
    if kind == "events":
        st["mc"].spectrum(case["sets"], st["params"], st["out"])
        return {"spectrum": st["out"].float()}
    if kind == "train":
        net = st["net"]
        net.train_step(case["batch"], st["x"], st["y"], 1e-3, 1e-4, st["loss"])
        lib = fitcore.load()
        for k, (gw, gb) in enumerate(st["grads"]):
            assert lib.fit_mlp_get_layer(net.handle, k, None, None, gw.data_ptr(), gb.data_ptr()) == 0
        return {"loss": st["loss"].float(), "grads": [list(g) for g in st["grads"]]}
    if kind == "starts":
        warmstart.predict_starts(st["net"], st["model"], st["spec"], case["batch"], st["data"], st["masks"], st["theta"])
        return {"theta": st["theta"].float()}
    if kind == "fit":
        fitcore.fit_batch([st["model"]], st["inst"], st["data"], None, st["best"], st["results"])
        nll = st["results"].view(torch.float64).view(case["batch"], -1)[:, 0]
        return {"best": st["best"].float(), "nll_min": nll.float()}
    r = fitcore.fit_profile_scan(st["model"], st["data"], st["spec"].all_mask(), [st["index"]], st["points"])
    return {"dchi2": r["dchi2"].astype(np.float32), "theta": r["theta"].astype(np.float32)}


# ---- what one pass cannot do without -----------------------------------------------------------
def _eval_flops(spec, grad):
    """Arithmetic of one expectation (and gradient): survival per true bin and core, energy map,
    banded fold, backgrounds, priors."""
    ph = {synth.OSC_EQ1: 2, synth.OSC_VACUUM3: 2, synth.OSC_STERILE4: 3}[spec.osc_mode]
    tot = 0.0
    for ds in spec.datasets:
        R = spec.detectors[ds.det].response
        nnz = float(np.count_nonzero(R))
        tot += spec.n_true * (spec.n_cores * (20 * ph + 10) + 30) + 2 * nnz + R.shape[0] * (10 + 6 * len(ds.backgrounds))
        if grad:
            tot += spec.n_true * (spec.n_cores * (8 * ph + 6) + 30) + 2 * nnz + R.shape[0] * (10 + 6 * len(ds.backgrounds))
    if grad:
        tot += sum(2.0 * len(ix) ** 2 for ix, _ in spec.cov_blocks) + 6 * spec.n_params
    return tot


def _table_bytes(spec):
    n = sum(2.0 * np.count_nonzero(d.response) * 4 for d in spec.detectors) + sum(4.0 * len(ix) ** 2 for ix, _ in spec.cov_blocks)
    return n + 16.0 * spec.n_true * len(spec.datasets)


def work(case):
    kind = case["kind"]
    if kind == "events":
        ph = 2 if case["geometry"] == "dc_fd" else 3
        return {"bytes": 13.0 * case["events"], "flops": case["events"] * (8.0 + case["sets"] * (26.0 * ph + 2))}
    if kind == "train":
        d = [warmstart.N_IN] + [warmstart.N_HIDDEN] * warmstart.N_HIDDEN_LAYERS + [warmstart.N_OUT]
        n = sum(a * b for a, b in zip(d, d[1:]))
        return {"bytes": 4.0 * case["batch"] * (d[0] + d[-1]) + 28.0 * n, "flops": 2.0 * case["batch"] * (3 * n - d[0] * d[1])}
    spec = _spec(case["model"], bool(case.get("spline", False)))
    P, D = spec.n_params, spec.n_bins
    if kind == "scan":   # at least eight evaluations per fit from a cold start
        n = case["points"] + 1
        return {"bytes": _table_bytes(spec) + 4.0 * D + 8.0 * n * P, "flops": 8.0 * n * _eval_flops(spec, True)}
    B = case["batch"]
    if kind == "eval":
        return {"bytes": _table_bytes(spec) + B * (12.0 * P + 4.0 * D + 12), "flops": B * _eval_flops(spec, True)}
    if kind == "expect":
        return {"bytes": _table_bytes(spec) + B * (8.0 * P + 4.0 * D), "flops": B * _eval_flops(spec, False)}
    if kind == "starts":
        d = [warmstart.N_IN] + [warmstart.N_HIDDEN] * warmstart.N_HIDDEN_LAYERS + [warmstart.N_OUT]
        n = sum(a * b for a, b in zip(d, d[1:]))
        return {"bytes": B * (4.0 * D + 8.0 * P) + 4.0 * P * D + 4.0 * n, "flops": 2.0 * B * (P * D + n)}
    return {"bytes": _table_bytes(spec) + B * (8.0 * P + 4.0 * D), "flops": 8.0 * B * _eval_flops(spec, True)}


# ---- the same in 64 bits ---------------------------------------------------------------------
def _survival64(mode, eta, x):
    """P(L, E) with eta [B, n] columns and x = K L / E [C, N]; returns [B, C, N]."""
    e = [eta[:, i, None, None] for i in range(eta.shape[1])]

    def s2(dm):
        return torch.sin(dm * x) ** 2

    if mode == synth.OSC_EQ1:
        c2 = 0.5 * (1.0 + torch.sqrt(1.0 - e[0]))
        return 1.0 - e[0] * s2(e[1]) - c2 * c2 * e[2] * s2(e[3])
    c12, c13 = 1.0 - e[0], 1.0 - e[1]
    inner = (4.0 * e[0] * c12 * c13 * c13 * s2(e[2])
             + 4.0 * e[1] * c13 * (c12 * s2(e[3]) + e[0] * s2(e[3] - e[2])))
    if mode == synth.OSC_VACUUM3:
        return 1.0 - inner
    c14 = 0.5 * (1.0 + torch.sqrt(1.0 - e[4]))
    return (1.0 - c14 * c14 * inner
            - e[4] * (c13 * (c12 * s2(e[5]) + e[0] * s2(e[5] - e[2])) + e[1] * s2(e[5] - e[3])))


def _remap64(spec, u, a0, a1, a2):
    """Corrected spectrum of u [B, N] under E' = a0 + a1 E + a2 E^2 (coefficients [B, 1])."""
    N, de = spec.n_true, (spec.e_hi - spec.e_lo) / spec.n_true
    B = u.shape[0]
    edges = torch.linspace(spec.e_lo, spec.e_hi, N + 1, dtype=torch.float64, device=u.device).expand(B, N + 1)
    zero = u.new_zeros(B, 1)
    cum = torch.cat([zero, torch.cumsum(u, 1)], 1)
    if not spec.remap:   # cumulative content, linear between the mapped edges, at the grid edges
        y = a0 + a1 * edges + a2 * edges * edges
        k = (torch.searchsorted(y.detach().contiguous(), edges.contiguous(), right=True) - 1).clamp(0, N - 1)
        y0, y1 = y.gather(1, k), y.gather(1, k + 1)
        t = ((edges - y0) / (y1 - y0)).clamp(0.0, 1.0)
        F = cum.gather(1, k) + t * u.gather(1, k)
    else:                # cubic Hermite cumulative at the inverse-mapped grid edges
        x = 2.0 * (edges - a0) / (a1 + torch.sqrt(a1 * a1 + 4.0 * a2 * (edges - a0)))
        g = (x - spec.e_lo) / de
        k = torch.floor(g.detach()).long().clamp(0, N - 1)
        t = (g - k).clamp(0.0, 1.0)
        S = torch.cat([u[:, :1], 0.5 * (u[:, 1:] + u[:, :-1]), u[:, -1:]], 1)
        h01, h10, h11 = t * t * (3.0 - 2.0 * t), t * (1.0 - t) ** 2, t * t * (t - 1.0)
        F = cum.gather(1, k) + u.gather(1, k) * h01 + S.gather(1, k) * h10 + S.gather(1, k + 1) * h11
    return F[:, 1:] - F[:, :-1]


def _expected64(spec, theta):
    """Expected counts [B, n_data] of theta [B, P] (float64), differentiable."""
    dev = theta.device
    t64 = functools.partial(torch.tensor, dtype=torch.float64, device=dev)
    edges = spec.true_edges
    ec = t64(0.5 * (edges[:-1] + edges[1:]))

    def par(i, default):
        return theta[:, int(i), None] if int(i) >= 0 else theta.new_full((theta.shape[0], 1), default)

    eta = torch.cat([par(i, v) for i, v in zip(spec.osc_idx, spec.osc_val)], 1)
    ones = theta.new_ones(theta.shape[0], 1)
    out = []
    for ds in spec.datasets:
        P = _survival64(spec.osc_mode, eta, K_OSC * t64(ds.baseline)[:, None] / ec[None, :])
        power = torch.cat([par(i, 1.0) for i in spec.core_power_idx], 1) * t64(ds.weight)
        shape_idx = torch.tensor(np.where(ds.shape_idx >= 0, ds.shape_idx, spec.n_params), dtype=torch.long, device=dev)
        u = t64(ds.t) * par(ds.norm_idx, 1.0) * torch.cat([theta, ones], 1)[:, shape_idx] * (power[:, :, None] * P).sum(1)
        v = _remap64(spec, u, *(par(i, d) for i, d in zip(ds.escale_idx, (0.0, 1.0, 0.0))))
        mu = par(ds.eff_idx, 1.0) * (v @ t64(spec.detectors[ds.det].response).T)
        for b in ds.backgrounds:
            d = torch.tensor(np.where(b.shape_idx >= 0, b.shape_idx, spec.n_params), dtype=torch.long, device=dev)
            mu = mu + par(b.rate_idx, 1.0) * t64(b.template) * (1.0 + torch.cat([theta, 0.0 * ones], 1)[:, d])
        out.append(mu)
    return torch.cat(out, 1)


def _nll64(spec, theta, data, masks):
    mu = _expected64(spec, theta)
    used = torch.repeat_interleave((masks[:, None] >> torch.arange(len(spec.datasets), device=theta.device)) & 1,
                                   torch.tensor(spec.reco_sizes(), device=theta.device), dim=1).bool()
    dev = 2.0 * (mu - data + torch.xlogy(data, data) - data * torch.log(mu))
    d = theta - torch.tensor(spec.theta0, device=theta.device)
    s = torch.tensor(np.where(spec.prior_sigma > 0, 1.0 / np.where(spec.prior_sigma > 0, spec.prior_sigma, 1.0), 0.0),
                     device=theta.device)
    nll = torch.where(used, dev, 0.0).sum(1) + ((d * s) ** 2).sum(1)
    for ix, cov in spec.cov_blocks:
        q = d[:, torch.tensor(ix, dtype=torch.long, device=theta.device)]
        nll = nll + (q @ torch.tensor(np.linalg.inv(cov), device=theta.device) * q).sum(1)
    return nll


def _mlp64(weights, x):
    for k, (w, b) in enumerate(weights):
        x = x @ w.T + b
        if k + 1 < len(weights):
            x = torch.nn.functional.gelu(x)
    return x


def _initial_weights(net):
    return [[torch.tensor(a, dtype=torch.float64, device=DEV, requires_grad=True) for a in net.get_layer(k)[:2]]
            for k in range(net.n_layers)]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("fit", "scan", "starts"):   # minima of the exact likelihood: no closed form, minutes by quasi-Newton
        return None
    rng = np.random.default_rng(seed)
    if kind == "events":
        ev, par = _events(case, seed), torch.tensor(_event_params(case, rng), device=DEV)
        E = torch.tensor(ev.energy, device=DEV).double()
        x = K_OSC * torch.tensor(ev.core_L, device=DEV)[torch.tensor(ev.core, device=DEV).long()] / E
        w, b = torch.tensor(ev.weight, device=DEV).double(), torch.tensor(ev.bin, device=DEV).long()
        out = torch.zeros((case["sets"], ev.n_bins), dtype=torch.float64, device=DEV)
        for k in range(case["sets"]):
            out[k].index_add_(0, b, w * _survival64(ev.osc_mode, par[k:k + 1], x[None])[0, 0])
        return {"spectrum": out}
    if kind == "train":
        weights = _initial_weights(warmstart.network(seed))
        x, y = _training_batch(case["batch"], seed)
        loss = ((_mlp64(weights, x.double()) - y.double()) ** 2).mean()
        loss.backward()
        return {"loss": loss.detach().reshape(1), "grads": [[w.grad, b.grad] for w, b in weights]}
    spec = _spec(case["model"], bool(case["spline"]))
    B = case["batch"]
    step = max(1, (1 << 19) // (spec.n_true * spec.n_cores))
    if kind == "expect":
        theta = torch.tensor(_thetas(spec, B, rng), device=DEV)
        with torch.no_grad():
            mu = torch.cat([_expected64(spec, theta[i:i + step]) for i in range(0, B, step)])
        return {"mu": mu, "status": None}
    masks = torch.tensor(_masks(case, spec, B, rng).astype(np.int64), device=DEV)
    data = torch.tensor(_pseudo_data(spec, B, rng), device=DEV).double()
    theta = torch.tensor(_thetas(spec, B, rng), device=DEV).requires_grad_()
    nll = []
    for i in range(0, B, step):
        f = _nll64(spec, theta[i:i + step], data[i:i + step], masks[i:i + step])
        f.sum().backward()
        nll.append(f.detach())
    return {"nll": torch.cat(nll), "grad": theta.grad, "status": None}
