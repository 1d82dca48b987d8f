"""Surrogate loss and gradient at the edges of the training kernels' tiles: 128-row tiles of
the batch, 64-row chunks of the weight gradients, 64-column tiles of the hidden layers,
8-column chunks of the output layer.

Bars as for the surrogate's other gradient test (BF16 operands, 8 significant bits, over
four layers): loss 2e-2, gradient 5e-2 normwise per parameter block against the FP64 oracle
at the same parameters.  The sums are formed in a fixed order, so a second call gives the
same bits.
"""
import numpy as np
import pytest

from oracle import metrics, surrogate

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NORM = (np.log(1000.0), 1.0, np.log(100.0), 1.2, 1.0, 0.2)


def f32(x):
    return np.asarray(x).astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("hidden,rank,batch", [(64, 32, 1), (64, 3, 127), (128, 8, 128), (128, 20, 1409),
                                               (256, 32, 129), (256, 17, 4096)])
def test_loss_gradient_at_tile_edges(hidden, rank, batch):
    import paper_1904_13244_gb300 as mr
    rng = np.random.default_rng([hidden, rank, batch])
    theta = []
    for o, i in surrogate.layer_shapes(hidden, rank):
        lim = np.sqrt(6.0 / (o + i))
        theta += [rng.uniform(-lim, lim, o * i), rng.uniform(-0.1, 0.1, o)]
    theta = f32(np.concatenate(theta))
    scale = f32(np.linspace(1.0, 0.2, rank))
    x = f32(np.stack([rng.uniform(np.log(100), np.log(6000), batch), rng.uniform(np.log(10), np.log(3000), batch),
                      rng.uniform(0.8, 1.2, batch)]))
    target = f32(rng.standard_normal((3, rank, batch)) * scale[None, :, None])
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda")  # noqa: E731
    with mr.Surrogate(hidden, rank, NORM, 0.3, seed=0) as net:
        net.set_params(theta)
        net.set_output_scale(scale)
        grads, losses = [], []
        for n in (2 * batch + 5, batch, batch):  # a larger batch first: the buffers are then shared
            idx = np.arange(n) % batch
            g = torch.full((net.num_params,), float("nan"), device="cuda")
            losses.append(net.loss_grad(dev(x[:2, idx]), dev(target[:, :, idx]), b1=dev(x[2, idx]), grad=g))
            grads.append(g)
    assert losses[1] == losses[2] and torch.equal(grads[1], grads[2])
    L, ref = surrogate.loss_grad(theta, x, tuple(target), NORM, scale, hidden, rank, 0.3)
    assert abs(losses[1] - L) / L < 2e-2
    g, k = grads[1].cpu().numpy().astype(np.float64), 0
    for o, i in surrogate.layer_shapes(hidden, rank):
        for n in (o * i, o):
            assert metrics.relerr(g[k:k + n], ref[k:k + n]) < 5e-2, (k, n)
            k += n
