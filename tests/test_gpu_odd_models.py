"""Expectation, -2lnL, gradient, tensor-core expectation and fits on models of awkward form, against
the FP64 oracle: true and reco sizes that are no multiple of four or of a warp, one reco bin, odd
numbers of cores with a core that a dataset does not see, parameters that play several roles or
serve several datasets, interleaved shape groups, interleaved and large covariance blocks, models
whose datasets do not fit into one group, and each block size that the sizes select.

Tolerances: expectation and -2lnL as in the parity tests on the named models (2e-5 per bin; 1e-3 near
the minimum plus 2e-7 (|nll| + sum |mu - n|)). Gradient: with J = d mu / d theta (central differences
of the oracle, to which the bar is proportional) and w = 2 (1 - n / mu), a component is sum_j J_j w_j
plus its prior term. J has the relative error of an expectation, 2e-5; w moves by 2 (n / mu) times
the relative error of mu, at most 2e-6 (a survival error of 2e-7 where P >= 0.1); the prior term
2 W^T W d, W the inverse Cholesky factor of a block, is two FP32 products, whose terms |W|^T |W| |d|
are each exact to 1e-6 (FP32 rounding over at most a few hundred of them).
"""
import numpy as np
import pytest

import oracle
from paper_2502_15253_gb300 import fitcore, synth

pytestmark = pytest.mark.gpu

EQ1, VAC3, STERILE = synth.OSC_EQ1, synth.OSC_VACUUM3, synth.OSC_STERILE4
#        n_true, reco sizes, datasets, cores, formula, remap, shape groups, covariance of all shapes in one block
FORMS = {
    "tiny": (13, (1,), 1, 1, EQ1, 0, 3, True),
    "one warp": (33, (5, 31), 2, 3, VAC3, 1, 7, True),
    "128 threads": (203, (37, 61), 2, 3, VAC3, 0, 29, False),
    "256 threads": (402, (41, 6), 3, 5, EQ1, 1, 33, True),
    "512 threads": (1601, (130, 39), 1, 16, STERILE, 0, 150, True),
    "eight datasets": (301, (23, 64, 9), 8, 2, STERILE, 1, 11, False),
    "two groups": (1999, (77, 250), 3, 7, VAC3, 0, 211, True),
    "many shapes": (997, (333,), 2, 4, EQ1, 0, 300, True),
}


def make(form, seed=5):
    n_true, recos, n_ds, C, mode, remap, groups, joint = FORMS[form]
    rng = np.random.default_rng(seed)
    e_lo, e_hi = 1.8, 9.0
    edges = np.linspace(e_lo, e_hi, n_true + 1)
    p = synth._Params()
    if mode == EQ1:
        osc, val = [p.add("s13", 0.09, 0.0, 0.02), p.add("dmee", 2.5e-3, 1e-4), -1, -1], [0.09, 2.5e-3, 0.851, 7.53e-5]
    elif mode == VAC3:
        osc = [p.add("s12", 0.307, 0.013), p.add("s13", 0.022, 0.001), p.add("dm21", 7.5e-5, 2e-6),
               p.add("dm31", 2.5e-3, 5e-5)]
        val = [0.307, 0.022, 7.5e-5, 2.5e-3]
    else:
        osc = [-1, p.add("s13", 0.022, 0.001), p.add("dm21", 7.5e-5, 2e-6), p.add("dm31", 2.5e-3, 5e-5),
               p.add("s14", 0.05, 0.01), p.add("dm41", 0.1, 2e-3)]
        val = [0.307, 0.022, 7.5e-5, 2.5e-3, 0.05, 0.1]
    power = [p.add(f"power{c}", 1.0, 0.01) for c in range((C + 1) // 2)]   # two cores share a parameter
    a = [np.array([p.add(f"a0{d}", 0.0, 0.01), p.add(f"a1{d}", 1.0, 0.004), -1 if d else p.add("a2", 0.0, 0.001)],
                  np.int32) for d in range(min(n_ds, 2))]
    both = p.add("norm and efficiency", 1.0, 0.02)
    rate = [p.add(f"rate{b}", 1.0, 0.1) for b in range(2)]
    shp = p.add_block("shape", groups * n_ds, 1.0, 0.02)
    bsh = p.add_block("bshape", recos[0], 0.0, 0.05)
    names, th0, sig, scl = p.arrays()
    if joint:   # every second shape parameter first: not consecutive
        order = np.concatenate([shp[::2], shp[1::2]]) if len(shp) > 1 else shp
        blocks = [(order.astype(np.int32), 0.02 ** 2 * synth.shape_correlation(len(shp), rng))]
    else:
        blocks = [(shp[d::n_ds].astype(np.int32), 0.02 ** 2 * synth.shape_correlation(groups, rng)) for d in range(n_ds)]
    dets = [synth.Detector(f"D{i}", np.linspace(1.0, 8.0, n + 1),
                           synth.gaussian_response(edges, np.linspace(1.0, 8.0, n + 1), 0.05)) for i, n in enumerate(recos)]
    ds = []
    for d in range(n_ds):
        base = np.linspace(400.0 + 300 * d, 1500.0, C) if mode != VAC3 else np.linspace(50000.0, 53000.0 + d, C)
        w = synth._core_weights(base)
        if d and C > 1:
            w = w.copy()
            w[C // 2] = 0.0
            w /= w.sum()
        nr = recos[d % len(recos)]
        none = np.full(nr, -1, np.int32)
        redges = dets[d % len(recos)].reco_edges
        bk = [synth.Background("s", synth._template_flat(redges, 200.0 * nr), rate[0],
                               bsh.copy() if nr == recos[0] else none),
              synth.Background("t", synth._template_exp(redges, 100.0 * nr, 2.0), rate[0] if d == 0 else rate[1], none)]
        group = (np.arange(n_true) * 7) % groups                     # interleaved groups
        if d % 2 == 0:
            group = np.minimum(np.arange(n_true) * groups // n_true, groups - 1)   # and runs
        idx = shp[d * groups + group].astype(np.int32)
        idx[::11] = -1
        ds.append(synth.Dataset(f"S{d}", d % len(recos), synth.signal_spectrum(edges, 3000.0 * nr), base, w,
                                both if d == 0 else -1, both if d != 1 else -1, a[min(d, len(a) - 1)], idx,
                                bk if d != 2 else []))
    core = np.array([power[c // 2] for c in range(C)], np.int32)
    if C > 2:
        core[-1] = both
    return synth.ModelSpec("odd", names, th0, sig, scl, blocks, mode, np.array(osc, np.int32), np.array(val), core,
                           n_true, e_lo, e_hi, dets, ds, remap=remap)


@pytest.fixture(scope="module", params=list(FORMS))
def odd(request):
    spec = make(request.param)
    om = oracle.OracleModel(spec)
    rng = np.random.default_rng(8)
    th = np.stack([om.theta_of_z(0.4 * rng.standard_normal(spec.n_params)) for _ in range(3)])
    return spec, om, fitcore.Model(spec), th


def test_expectation_both_paths(odd):
    spec, om, gm, th = odd
    mu, st = fitcore.expected_numpy(gm, th)
    tc, stc = np.zeros_like(mu), np.zeros(len(th), np.int32)
    fitcore.fit_model_expected_tc(gm, len(th), th, tc, stc, 1)
    assert not st.any() and not stc.any()
    for b in range(len(th)):
        ref = om.expected(th[b])
        np.testing.assert_allclose(mu[b], ref, rtol=2e-5, atol=1e-6 * ref.max())
        np.testing.assert_allclose(tc[b], ref, rtol=2e-5, atol=1e-6 * ref.max())


def test_nll_and_gradient(odd):
    spec, om, gm, th = odd
    data = synth.poisson_data(om.expected(spec.theta0), 3)
    data[::9] = 0.0
    n_ds = len(spec.datasets)
    masks = np.array([spec.all_mask(), 1 << (n_ds - 1), spec.all_mask() & 0b10101010 or 1], np.uint32)
    nll, g, st = fitcore.eval_numpy(gm, th, np.tile(data, (3, 1)), masks)
    assert not st.any()
    offs = spec.data_offsets()
    h = 1e-4 * np.where(spec.prior_sigma > 0, spec.prior_sigma, spec.scale)
    for b in range(3):
        ref, gref = om.nll(th[b], data, mask=int(masks[b]), grad=True)
        use = np.zeros(len(data), bool)
        for d in range(n_ds):
            if (int(masks[b]) >> d) & 1:
                use[offs[d]:offs[d + 1]] = True
        mu = om.expected(th[b])
        assert abs(nll[b] - ref) <= 1e-3 + 2e-7 * (abs(ref) + np.abs(mu - data)[use].sum())
        w = np.where(use, 2 * (1 - data / mu), 0.0)
        prior = np.zeros(spec.n_params)
        own = spec.prior_sigma > 0
        prior[own] = 2 * np.abs(th[b] - spec.theta0)[own] / spec.prior_sigma[own] ** 2
        for idx, cov in spec.cov_blocks:
            W = np.abs(np.linalg.inv(np.linalg.cholesky(cov)))
            prior[idx] += 2 * W.T @ (W @ np.abs(th[b] - spec.theta0)[idx])
        for p in range(spec.n_params):
            t1, t2 = th[b].copy(), th[b].copy()
            t1[p] += h[p]
            t2[p] -= h[p]
            J = (om.expected(t1) - om.expected(t2)) / (2 * h[p])
            bar = np.sum(np.abs(J) * use * (2e-5 * np.abs(w) + 4e-6 * data / mu)) + 1e-6 * prior[p]
            assert abs(g[b, p] - gref[p]) <= bar + 1e-10 / h[p], (b, spec.param_names[p], g[b, p], gref[p], bar)


@pytest.mark.parametrize("form", ["tiny", "one warp", "128 threads", "256 threads", "eight datasets", "two groups"])
def test_fit_reaches_the_oracle_minimum(form):
    """Under the launch that the sizes select and the spline energy correction (smooth, so one minimum):
    -2lnL at the minimum within 1e-3 of the oracle's."""
    spec = make(form)
    spec.remap = 1
    om = oracle.OracleModel(spec)
    data = synth.poisson_data(om.expected(spec.theta0), 4)
    inst = np.zeros(1, fitcore.INSTANCE_DTYPE)
    inst["mask"] = spec.all_mask()
    _, res = fitcore.fit_numpy([fitcore.Model(spec)], inst, data)
    ref = om.fit(data)
    assert res["status"][0] == 0 and abs(res["nll_min"][0] - ref["nll"]) <= 1e-3
