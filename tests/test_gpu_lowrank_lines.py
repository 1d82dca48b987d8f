"""Low-rank products on shapes at the edges of the by-line kernels (4 and 8 phase-encode lines
per block, 32 readout samples, TR slots of 8, 16 and 32 and beyond): uneven TR counts per
line, lines without a TR, image sizes that fill no tile, every rank class.

J.v, Re(J^H w) and Re(J^H J) v against the oracle's projected model at the split-BF16 bar of
the low-rank products, 3e-5 normwise."""
import dataclasses

import numpy as np
import pytest

import synth
from oracle import metrics, model

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nkx,most,rank", [(33, 9, 33, 8, 8), (7, 35, 7, 9, 16), (40, 12, 40, 16, 32),
                                                 (13, 20, 13, 17, 24), (31, 6, 31, 33, 32), (10, 11, 23, 5, 24)])
def test_products_match_projected_model(nx, ny, nkx, most, rank):
    import paper_1904_13244_gb300 as mr
    rng = np.random.default_rng([nx, ny, most])
    counts = rng.integers(0, most + 1, ny)
    counts[rng.integers(ny)] = most  # the slot class of the test
    counts[(np.argmax(counts) + 1) % ny] = 0
    ky = np.repeat(np.arange(ny) - ny // 2, counts).astype(np.int32)
    rng.shuffle(ky)
    ntr = len(ky)
    flips = synth.flip_train(ntr, 3, 1).astype(np.float32).astype(np.float64)
    seq = dataclasses.replace(synth.make_sequence(nx, ny, 1, 7.6, 3.8, nkx=nkx), flip_rad=flips, ky=ky)
    f32 = lambda x: np.asarray(x).astype(np.float32).astype(np.float64)  # noqa: E731
    alpha = f32(np.stack([rng.uniform(np.log(300), np.log(3000), seq.nv), rng.uniform(np.log(30), np.log(300), seq.nv),
                          rng.uniform(-1, 1, seq.nv), rng.uniform(-1, 1, seq.nv)]))
    mask = rng.random(seq.nv) < 0.9
    train = np.stack([rng.uniform(np.log(100), np.log(6000), 200), rng.uniform(np.log(10), np.log(3000), 200)])
    U, _ = model.time_basis(seq, np.exp(train[0]), np.exp(train[1]), rank)
    U = f32(U)
    lin = model.project_onto_basis(model.linearize(seq, alpha, mask=mask), U)
    v, w = synth.random_params(seq.nv, 3), synth.random_kspace(ntr, nkx, 4)
    dev = lambda a, t=torch.float32: torch.tensor(np.ascontiguousarray(a), dtype=t, device="cuda")  # noqa: E731
    with mr.Plan(seq) as plan:
        plan.lowrank_set_basis(dev(U))
        plan.lowrank_linearize(dev(alpha), mask=dev(mask.astype(np.uint8), torch.uint8))
        jv = plan.jvp(dev(v)).cpu().numpy()
        g = plan.jhw(dev(w, torch.complex64)).cpu().numpy()
        h = plan.jhjv(dev(v)).cpu().numpy()
        plan.check()
    assert metrics.relerr(jv, model.jvp(lin, v)) < 3e-5
    assert metrics.relerr(g, model.jhw(lin, w)) < 3e-5
    assert metrics.relerr(h, model.gauss_newton_product(lin, v)) < 3e-5
