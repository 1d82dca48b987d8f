"""With nkx == nx an image column of Re(J^H J) v depends on no other column of v: a non-finite
value in one column leaves the others bit for bit as they were, also where the column tiles
of four and the row groups of 32 are not full.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("nx,ny,ntr", [(13, 9, 40), (8, 32, 64), (5, 97, 300)])
def test_columns_are_independent(nx, ny, ntr, value):
    import paper_1904_13244_gb300 as mr
    seq = synth.make_sequence(nx, ny, 1, 7.6, 3.8, seed=nx, extra_trs=ntr - ny)
    rng = np.random.default_rng([nx, ny])
    alpha = np.stack([rng.uniform(np.log(300), np.log(3000), seq.nv), rng.uniform(np.log(30), np.log(300), seq.nv),
                      rng.uniform(0.5, 1, seq.nv), rng.uniform(-1, 1, seq.nv)])
    v = torch.tensor(rng.standard_normal((4, ny, nx)), dtype=torch.float32, device="cuda")
    with mr.Plan(seq) as plan:
        plan.linearize(torch.tensor(alpha, dtype=torch.float32, device="cuda"))
        ref = plan.jhjv(v.view(4, -1)).view(4, ny, nx)
        for col in (0, nx - 1):
            bad = v.clone()
            bad[:, 0, col] = value
            got = plan.jhjv(bad.view(4, -1)).view(4, ny, nx)
            rest = [i for i in range(nx) if i != col]
            assert torch.equal(got[:, :, rest], ref[:, :, rest])
