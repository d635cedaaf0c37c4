"""A fit's result does not depend on the models that are fitted, or only passed, beside it: each model
alone against a call with all of them (blocks of 128, 256 and 512 threads, the general and the plain
build), their instances interleaved, plainly and through CUDA graphs, bit for bit."""
import numpy as np
import pytest

from paper_2502_15253_gb300 import fitcore, synth

pytestmark = pytest.mark.gpu
FORMS = [("c0", 0, 23), ("c1", 0, 17), ("c2", 0, 9), ("c1", 1, 12), ("c0", 1, 5)]


@pytest.fixture(scope="module")
def work():
    specs = [synth.make_model(n, remap=r) for n, r, _ in FORMS]
    models = [fitcore.Model(s) for s in specs]
    kind = np.concatenate([np.full(n, k) for k, (_, _, n) in enumerate(FORMS)])
    kind = kind[np.random.default_rng(6).permutation(len(kind))]
    D, P = max(s.n_bins for s in specs), max(s.n_params for s in specs)
    data = np.zeros((len(kind), D), np.float32)
    for k, (s, m) in enumerate(zip(specs, models)):
        mu, _ = fitcore.expected_numpy(m, s.theta0[None])
        rows = np.flatnonzero(kind == k)
        data[rows, :s.n_bins] = np.random.default_rng(k).poisson(np.tile(mu.astype(np.float64), (len(rows), 1)))
    inst = np.zeros(len(kind), fitcore.INSTANCE_DTYPE)
    inst["model"], inst["mask"] = kind, [specs[k].all_mask() for k in kind]
    inst["data_off"], inst["param_off"] = np.arange(len(kind)) * D, np.arange(len(kind)) * P
    return specs, models, kind, inst, data, P


def _fit(models, inst, data, P, **kw):
    o = fitcore.fit_batch_default_opts()
    for k, v in kw.items():
        setattr(o, k, v)
    best, res = np.zeros(len(data) * P), np.zeros(len(inst), fitcore.RESULT_DTYPE)
    fitcore.fit_batch(models, inst, data.ravel(), None, best, res, o)
    return best.reshape(len(data), P), res


@pytest.mark.parametrize("graph", [0, 1])
def test_alone_and_together(work, graph):
    specs, models, kind, inst, data, P = work
    best, res = _fit(models, inst, data, P, use_graph=graph)
    assert np.all((res["status"] == 0) | (res["status"] == 7))
    for k in range(len(models)):
        rows = np.flatnonzero(kind == k)
        own = inst[rows].copy()
        for passed in ([models[k]], [models[k]] + models):   # alone, and with models that nothing fits
            own["model"] = 0
            b, r = _fit(passed, own, data, P)
            np.testing.assert_array_equal(b[rows], best[rows])
            for f in ("nll_min", "iters", "n_evals", "status"):
                np.testing.assert_array_equal(r[f], res[f][rows])


def test_two_models_in_order(work):
    """Instances that are sorted by launch already."""
    specs, models, kind, inst, data, P = work
    rows = np.concatenate([np.flatnonzero(kind == 2), np.flatnonzero(kind == 1), np.flatnonzero(kind == 0)])
    best, res = _fit(models, inst[rows], data, P)
    every, ref = _fit(models, inst, data, P)
    np.testing.assert_array_equal(best[rows], every[rows])
    np.testing.assert_array_equal(res["nll_min"], ref["nll_min"][rows])


def test_budget_of_a_mixed_call(work):
    specs, models, kind, inst, data, P = work
    _, res = _fit(models, inst, data, P, time_budget_s=1e-9)
    assert np.all(res["status"] == 6)
