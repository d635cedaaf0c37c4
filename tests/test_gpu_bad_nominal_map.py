"""Start points of a model whose energy map turns invalid next to the nominal point, in the second of
three datasets only: the rows of its Jacobian stop there (every warp of a block at the same dataset)
and the call reports it, the same on every fresh model, and another model's starts are what they
were before."""
import numpy as np
import pytest

from paper_2502_15253_gb300 import fitcore, synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _starts(spec):
    model = fitcore.Model(spec)
    data = torch.full((5, spec.n_bins), 90.0, device="cuda")
    theta = torch.zeros((5, spec.n_params), dtype=torch.float64, device="cuda")
    fitcore.fit_linear_start(model, 5, data, None, theta)
    torch.cuda.synchronize()
    return theta.cpu().numpy()


def test_invalid_map_in_one_dataset():
    before = _starts(synth.make_model("c1"))
    bad = synth.make_model("c1")
    bad.theta0 = bad.theta0.copy()
    bad.theta0[bad.index("a1[1]")] = 4.0 - 1e-5   # slopes of 4 are refused; the rows step by 5e-5
    for _ in range(10):
        with pytest.raises(fitcore.FitError, match="near theta0"):
            _starts(bad)
    np.testing.assert_array_equal(_starts(synth.make_model("c1")), before)
