"""The overlap-length energy correction far from nominal, against the FP64 oracle: slopes of 0.3 to 3.5
at either end of the grid, with the displacement of thousands of bins that goes with them, in both
expectations, -2lnL and gradient.

Tolerance: a mapped edge is k + D(e_k), D a polynomial of three terms in FP32, so it is off by at most
delta = 4 * 2^-24 of the sum of the terms' sizes (three roundings and that of the sum with k). A
source bin's overlaps then add up to its content to 2 delta / slope, coherently over the bins at
worst. An expectation therefore has the relative bar eps = 2e-5 (that of the parity tests) + 2 delta
/ smallest slope. With w = 2 (1 - n / mu) and J = d mu / d theta, -2lnL moves by sum |w| mu eps +
n eps^2 and a gradient component by sum |J| (|w| + 2 n / mu) eps.

A mapped edge Y adds (u / slope) (mean of gv over its source - gv[floor Y]) dY to -2lnL, gv = R^T w. That
has no derivative where Y is a whole number, as it is on a part of the edges when the slope is
a round number and the map leaves a grid edge in place, so the gradient is compared at other
maps. The energy coefficients' bar there has two more terms per edge: the jump |gv[t] - gv[t - 1]|
of the edges within delta of a grid edge, and 8 * 2^-24 of the largest |gv| for the difference.
"""
import numpy as np
import pytest

import oracle
from paper_2502_15253_gb300 import fitcore, synth

pytestmark = pytest.mark.gpu

E_LO, E_HI = 1.8, 9.0
SLOPES = [(0.3, 0.3), (0.6, 0.9), (0.84, 0.84), (1.2, 1.2), (1.5, 1.1), (3.5, 3.5), (0.3, 3.5), (3.5, 0.3)]


def make(n_true):
    edges, redges = np.linspace(E_LO, E_HI, n_true + 1), np.linspace(1.0, 8.0, 31)
    p = synth._Params()
    osc = [p.add("s13", 0.09, 0.0, 0.02), p.add("dmee", 2.5e-3, 1e-4), -1, -1]
    a = np.array([p.add("a0", 0.0, 5.0), p.add("a1", 1.0, 2.0), p.add("a2", 0.0, 0.5)], np.int32)
    norm, rate = p.add("norm", 1.0, 0.05), p.add("rate", 1.0, 0.1)
    shape = p.add_block("shape", 7, 1.0, 0.05)
    names, th0, sig, scl = p.arrays()
    base = np.array([950.0, 1150.0])
    det = synth.Detector("D", redges, synth.gaussian_response(edges, redges, 0.08))
    ds = synth.Dataset("S", 0, synth.signal_spectrum(edges, 90000.0), base, synth._core_weights(base), norm, -1, a,
                       shape[np.arange(n_true) * 7 // n_true].astype(np.int32),
                       [synth.Background("b", synth._template_flat(redges, 6000.0), rate, np.full(30, -1, np.int32))])
    return synth.ModelSpec("wide", names, th0, sig, scl, [(shape.astype(np.int32), 0.05 ** 2 * np.eye(7))], synth.OSC_EQ1,
                           np.array(osc, np.int32), np.array([0.09, 2.5e-3, 0.851, 7.53e-5]), np.full(2, -1, np.int32),
                           n_true, E_LO, E_HI, [det], [ds], remap=0)


def points(spec, off):
    """theta at every pair of slopes (off: added to both) and fixed point of the map, with delta and eps."""
    i0 = spec.index("a0")
    th, delta, eps = [], [], []
    for s_lo, s_hi in SLOPES:
        for fixed_point in (E_LO, 0.5 * (E_LO + E_HI), E_HI):
            x = fixed_point + 0.3 * off
            a2 = (s_hi - s_lo) / (2 * (E_HI - E_LO))
            a1 = s_lo + off - 2 * a2 * E_LO
            t = spec.theta0.copy()
            t[i0:i0 + 3] = x - a1 * x - a2 * x ** 2, a1, a2
            th.append(t)
            size = (abs(t[i0]) + abs(a1 - 1.0) * E_HI + abs(a2) * E_HI ** 2) * spec.n_true / (E_HI - E_LO)
            delta.append(4 * 2.0 ** -24 * size)
            eps.append(2e-5 + 2 * delta[-1] / (min(s_lo, s_hi) + off))
    return np.array(th), np.array(delta), np.array(eps)


@pytest.mark.parametrize("n_true", [400, 2000, 4096])
def test_expectations_and_nll(n_true):
    spec = make(n_true)
    om, gm = oracle.OracleModel(spec), fitcore.Model(spec)
    th, delta, eps = points(spec, 0.0)
    ref = np.array([om.expected(t) for t in th])
    data = np.array([synth.poisson_data(m, 5 + b) for b, m in enumerate(ref)])
    mu, st = fitcore.expected_numpy(gm, th)
    tc, stc = np.zeros_like(mu), np.zeros(len(th), np.int32)
    fitcore.fit_model_expected_tc(gm, len(th), th, tc, stc, 1)
    nll, _, stn = fitcore.eval_numpy(gm, th, data)
    assert not st.any() and not stc.any() and not stn.any()
    for b, t in enumerate(th):
        for m in (mu[b], tc[b]):
            assert np.all(np.abs(m - ref[b]) <= eps[b] * ref[b]), (b, np.abs(m / ref[b] - 1).max(), eps[b])
        r = om.nll(t, data[b])
        w = np.abs(2 * (1 - data[b] / ref[b]))
        assert abs(nll[b] - r) <= 1e-3 + 2e-7 * abs(r) + np.sum(w * ref[b] * eps[b] + data[b] * eps[b] ** 2), (b, nll[b], r)


@pytest.mark.parametrize("n_true", [400, 2000, 4096])
def test_gradient(n_true):
    spec = make(n_true)
    om, gm = oracle.OracleModel(spec), fitcore.Model(spec)
    i0 = spec.index("a0")
    th, delta, eps = points(spec, 0.01 * np.sqrt(2.0))
    edges = np.linspace(E_LO, E_HI, n_true + 1)
    e, de = 0.5 * (edges[1:] + edges[:-1]), (E_HI - E_LO) / n_true
    ds = spec.datasets[0]
    x = 1.266932679815373 * ds.baseline[:, None] / e
    c4 = (0.5 * (1 + np.sqrt(1 - 0.09))) ** 2
    u = ds.t * (ds.weight @ (1 - 0.09 * np.sin(2.5e-3 * x) ** 2 - c4 * 0.851 * np.sin(7.53e-5 * x) ** 2))
    h = 1e-4 * np.where(spec.prior_sigma > 0, spec.prior_sigma, spec.scale)
    ref = np.array([om.expected(t) for t in th])
    data = np.array([synth.poisson_data(m, 5 + b) for b, m in enumerate(ref)])
    _, g, st = fitcore.eval_numpy(gm, th, data)
    assert not st.any()
    for b, t in enumerate(th):
        _, gr = om.nll(t, data[b], grad=True)
        w = 2 * (1 - data[b] / ref[b])
        gv = np.concatenate([[0.0], w @ spec.detectors[0].response, [0.0]])   # by target bin + 1
        a0, a1, a2 = t[i0:i0 + 3]
        Y = (a0 + a1 * edges + a2 * edges ** 2 - E_LO) / de
        per_width = u / np.diff(Y)
        at = np.rint(Y)
        on = np.clip(at.astype(int), 0, n_true)                # the jump at grid edge m: gv[m] - gv[m - 1]
        jump = np.where((np.abs(Y - at) <= delta[b]) & (at == on), np.abs(gv[on + 1] - gv[on]), 0.0)
        slip = np.where((Y >= -1) & (Y <= n_true + 1), 8 * 2.0 ** -24 * np.abs(gv).max(), 0.0)
        per_edge = (np.concatenate([per_width, [0.0]]) + np.concatenate([[0.0], per_width])) * (jump + slip) / de
        for p in range(spec.n_params):
            t1, t2 = t.copy(), t.copy()
            t1[p] += h[p]
            t2[p] -= h[p]
            J = np.abs(om.expected(t1) - om.expected(t2)) / (2 * h[p])
            bar = np.sum(J * (np.abs(w) + 2 * data[b] / ref[b])) * eps[b]
            if i0 <= p < i0 + 3:
                bar += np.sum(per_edge * edges ** (p - i0))
            own = 2 * abs(t[p] - spec.theta0[p]) / spec.prior_sigma[p] ** 2 if spec.prior_sigma[p] > 0 else 0.0
            assert abs(g[b, p] - gr[p]) <= bar + 1e-6 * own + 1e-10 / h[p], (b, spec.param_names[p], g[b, p], gr[p], bar)
