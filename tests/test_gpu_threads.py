"""Calls for a small and for a large model from two threads at once, each on a stream of its own: the
kernels' shared-memory limit, which the threads share, is never lowered under the larger one."""
import threading

import numpy as np
import pytest

from paper_2502_15253_gb300 import fitcore, synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _both(work):
    """work(k) on two threads; raises what either raised."""
    failed = []

    def body(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                work(k)
        except Exception as e:   # reported below, in the test's own thread
            failed.append(e)
    ts = [threading.Thread(target=body, args=(k,)) for k in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    if failed:
        raise failed[0]


def test_expectations():
    specs = [synth.make_model("c0"), synth.make_model("c2", remap=1)]
    models = [fitcore.Model(s) for s in specs]
    theta = [torch.tensor(np.tile(s.theta0, (3, 1)), device="cuda") for s in specs]
    want = [fitcore.expected_numpy(m, s.theta0[None])[0][0] for m, s in zip(models, specs)]
    torch.cuda.synchronize()

    def work(k):
        stream = torch.cuda.current_stream()
        mu = torch.zeros((3, specs[k].n_bins), device="cuda")
        st = torch.zeros(3, dtype=torch.int32, device="cuda")
        for _ in range(1000):
            fitcore.fit_model_expected_tc(models[k], 3, theta[k], mu, st, 1, stream)
        stream.synchronize()
        assert not st.any()
        np.testing.assert_allclose(mu[1].cpu().numpy(), want[k], rtol=2e-5, atol=1e-6 * want[k].max())
    _both(work)


def test_rows_of_the_linear_start():
    """Every thread makes its models anew, so that each call forms the rows."""
    specs = [synth.make_model("c0"), synth.make_model("c1")]
    specs[0].remap = 1

    def starts(k):
        s = specs[k]
        data = torch.full((2, s.n_bins), 80.0, device="cuda")
        theta = torch.zeros((2, s.n_params), dtype=torch.float64, device="cuda")
        fitcore.fit_linear_start(fitcore.Model(s), 2, data, None, theta, torch.cuda.current_stream())
        torch.cuda.current_stream().synchronize()
        return theta.cpu().numpy()
    want = [starts(0), starts(1)]

    def work(k):
        for _ in range(40 if k == 0 else 6):
            np.testing.assert_array_equal(starts(k), want[k])
    _both(work)
