"""Training steps of the warm-start network give the same bits on every run: losses, gradients and
weights of two networks from one seed over twenty AdamW steps, at batches whose weight gradients are
one product (33), split over K into a few shares with a ragged last one (777, 4097) and into many
(9001), and for layer sizes that are no multiple of four."""
import numpy as np
import pytest

from paper_2502_15253_gb300 import fitcore

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _run(dims, batches):
    net = fitcore.Mlp(*dims, seed=4)
    gen = torch.Generator(device="cuda").manual_seed(2)
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    out = []
    for k in range(20):
        B = batches[k % len(batches)]
        x = torch.randn((B, dims[0]), generator=gen, device="cuda")
        y = torch.randn((B, dims[3]), generator=gen, device="cuda")
        net.train_step(B, x, y, 1e-3, 1e-4, loss)
        out.append(loss.cpu().numpy().copy())
    for layer in range(net.n_layers):
        out += list(net.get_layer(layer))
    return out


@pytest.mark.parametrize("dims,batches", [((438, 512, 3, 12), (4097,)), ((438, 512, 3, 12), (9001, 777)),
                                          ((70, 97, 2, 5), (33, 2050)), ((5, 16, 0, 3), (700,))])
def test_steps_are_the_same_bits(dims, batches):
    first = _run(dims, batches)
    assert all(np.all(np.isfinite(a)) for a in first)
    for _ in range(3):
        for a, b in zip(_run(dims, batches), first):
            np.testing.assert_array_equal(a, b)
