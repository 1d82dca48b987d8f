"""Scalars that are sums over a whole batch or parameter vector keep float64's precision and
range.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [1e12, 1e20])
@pytest.mark.parametrize("rank,batch", [(32, 4096), (20, 700), (3, 1)])
def test_training_loss_is_summed_in_float64(rank, batch, size):
    """Targets so large that a prediction vanishes beside them in float32: the residuals are
    then the targets, and the loss is their known sum of squares (past float32's range at
    1e20).  A term is rounded three times and goes through at most 24 additions in its thread,
    9 in its warp and block and some 40 over the blocks: 76 x 2^-53 = 8.5e-15, bar 1e-14."""
    import paper_1904_13244_gb300 as mr
    rng = np.random.default_rng([rank, batch])
    x = np.stack([rng.uniform(np.log(100), np.log(6000), batch), rng.uniform(np.log(10), np.log(3000), batch)])
    t = (size * rng.uniform(0.5, 2, (3, rank, batch)) * rng.choice([-1, 1], (3, rank, batch))).astype(np.float32)
    lam = 0.3
    with mr.Surrogate(64, rank, (np.log(1000.0), 1.0, np.log(100.0), 1.2, 1.0, 0.2), lam, seed=0) as net:
        loss = net.loss_grad(torch.tensor(x, dtype=torch.float32, device="cuda"), torch.tensor(t, device="cuda"))
    sq = np.sum(t.astype(np.longdouble) ** 2, axis=(1, 2))
    want = (sq[0] + np.longdouble(np.float32(lam)) * (sq[1] + sq[2])) / batch
    assert abs(loss - want) / want < 1e-14, (loss, float(want))
