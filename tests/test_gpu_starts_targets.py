"""Network starts where the targets repeat, are one, or are many, at sample counts around a block.

theta = linear start + sum of out_t scale_t over a parameter's targets, in FP64 from the same FP32 network
outputs: exact to FP64 rounding of a few terms (1e-12 of their size)."""
import numpy as np
import pytest

from paper_2502_15253_gb300 import fitcore, synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("B", [1, 85, 257])
@pytest.mark.parametrize("targets", [[24], [3, 0, 3, 3, 7, 0], list(range(15, -1, -1))])
def test_targets(B, targets):
    spec = synth.make_model("c0")
    model = fitcore.Model(spec)
    net = fitcore.Mlp(64, 64, 1, 16, seed=4)
    rng = np.random.default_rng(B)
    d = torch.tensor(rng.poisson(200.0, (B, spec.n_bins)).astype(np.float32), device="cuda")
    scale = rng.uniform(0.01, 0.1, len(targets))
    x = torch.zeros((B, 64), dtype=torch.float32, device="cuda")
    y = torch.zeros((B, 16), dtype=torch.float32, device="cuda")
    base = torch.zeros((B, spec.n_params), dtype=torch.float64, device="cuda")
    got = torch.zeros_like(base)
    fitcore.fit_warmstart_features(model, B, d, None, 64, 0, 60, x)
    net.forward(B, x, y)
    fitcore.fit_linear_start(model, B, d, None, base)
    fitcore.fit_warmstart_predict(net, model, B, d, None, 0, 60, targets, scale, got)
    torch.cuda.synchronize()
    ref, out = base.cpu().numpy(), y.cpu().numpy().astype(np.float64)
    size = 1 + np.abs(ref)
    for t, i in enumerate(targets):
        ref[:, i] += out[:, t] * scale[t]
        size[:, i] += np.abs(out[:, t] * scale[t])
    assert np.all(np.abs(got.cpu().numpy() - ref) <= 1e-12 * size)
