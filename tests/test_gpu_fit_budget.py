"""Fits under clock budgets that end at any point of a launch, also between two fits of a block: every
fit of the call converges or says that its time ran out, and the same call with time enough gives
the results it gave before."""
import numpy as np
import pytest

from paper_2502_15253_gb300 import fitcore, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,threads", [("c0", 0), ("c1", 0), ("c1", 64)])
def test_budget_runs_out(name, threads):
    spec = synth.make_model(name, remap=1)
    gm = fitcore.Model(spec)
    n = 2000
    mu, _ = fitcore.expected_numpy(gm, spec.theta0[None])
    data = np.random.default_rng(3).poisson(np.tile(mu.astype(np.float64), (n, 1))).astype(np.float32)
    inst = np.zeros(n, fitcore.INSTANCE_DTYPE)
    inst["mask"] = spec.all_mask()
    inst["data_off"] = np.arange(n) * spec.n_bins
    inst["param_off"] = np.arange(n) * spec.n_params

    def fit(budget):
        o = fitcore.fit_batch_default_opts()
        o.threads, o.time_budget_s = threads, budget
        return fitcore.fit_numpy([gm], inst, data, opts=o)
    best, res = fit(0.0)
    assert np.all(res["status"] == 0)
    seen = 0
    for budget in np.geomspace(1e-6, 3e-2, 60):
        b, r = fit(budget)
        late = r["status"] == 6
        seen += int(late.any() and not late.all())
        assert np.all(late | (r["status"] == 0))
        np.testing.assert_array_equal(r["nll_min"][~late], res["nll_min"][~late])
        assert np.all(np.isfinite(b))
    assert seen > 0
    again, _ = fit(0.0)
    np.testing.assert_array_equal(again, best)
