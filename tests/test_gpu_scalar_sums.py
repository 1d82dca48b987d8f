"""Scalars that are sums over a whole batch or parameter vector keep float64's precision and
range.
"""
import numpy as np
import pytest

import synth

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


def worst_constant(n=16):
    """A float32 c whose squares, added n times in a float32 chain, drift furthest from n c^2."""
    c = np.float32(1) + np.arange(1 << 16, dtype=np.float32) / np.float32(1 << 16)
    s = np.zeros_like(c)
    for _ in range(n):  # one rounding per step, as a fused multiply-add
        s = (c.astype(np.float64) ** 2 + s).astype(np.float32)
    exact = n * c.astype(np.float64) ** 2
    return float(c[np.argmax(np.abs(s / exact - 1))])


def test_cg_inner_products_of_the_exact_model():
    """The first CG step from a constant right-hand side r: x = a r with a = <r, r> / <r, B r>.
    a and x are rounded to float32 once each, 2 x 6e-8; float32 sums of four squares of this r
    are exact, and the roundings of sums of four terms of <r, B r> average out over 1900 of
    them.  Bar 1.4e-7; a float32 chain of sixteen squares is off by 2.7e-7."""
    import paper_1904_13244_gb300 as mr
    seq = synth.make_sequence(64, 30, 1, 7.6, 3.8, seed=2)  # one segment: the longest chains
    rng = np.random.default_rng(5)
    alpha = np.stack([rng.uniform(np.log(300), np.log(3000), seq.nv), rng.uniform(np.log(30), np.log(300), seq.nv),
                      rng.uniform(0.5, 1, seq.nv), rng.uniform(0.5, 1, seq.nv)])
    r = torch.full((4, seq.nv), worst_constant(), device="cuda")
    with mr.Plan(seq) as plan:
        plan.linearize(torch.tensor(alpha, dtype=torch.float32, device="cuda"))
        h = plan.jhjv(r)
        x = plan.cg_fixed(r, 1)
    a = float((r.double() ** 2).sum() / (r.double() * h.double()).sum())
    got = float((x.double() / r.double()).mean())
    assert abs(got / a - 1) < 1.4e-7, got / a - 1
