"""The mirrored-pair slice recursion for every pair count (1, 2, 4 and 8 lanes per voxel),
with voxels that do not fill a warp, a mask that empties whole warps and TR counts that are
not a multiple of the staged chunk: time courses and the forward signal against the oracle's
recursion over all isochromats.

Bar 1e-5 normwise, the FP32 bar of the slice model's other tests."""
import numpy as np
import pytest

import synth
from oracle import encoding, metrics, slice_profile as sp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_iso,nx,ny,fills,extra", [(4, 7, 11, 3, 2), (16, 13, 9, 2, 0), (32, 5, 6, 3, 1), (8, 17, 8, 4, 3),
                                                     (1, 3, 5, 3, 0), (2, 33, 4, 5, 1)])
def test_pairs_match_oracle(n_iso, nx, ny, fills, extra):
    import paper_1904_13244_gb300 as mr
    seq = synth.make_sequence(nx, ny, fills, 7.8, 3.4, seed=n_iso, extra_trs=extra)
    rng = np.random.default_rng([n_iso, nx])
    nv = seq.nv
    alpha = np.stack([rng.uniform(np.log(200), np.log(3000), nv), rng.uniform(np.log(20), np.log(300), nv),
                      rng.uniform(0.5, 1, nv), rng.uniform(-1, 1, nv)]).astype(np.float32)
    mask = (rng.random(nv) < 0.7).astype(np.uint8)
    mask[nv // 3: nv // 3 + 2 * 32] = 0
    mask[0] = 1
    prof = sp.SliceProfile(n_iso=n_iso, n_sub=6)
    ref = sp.simulate(seq, np.exp(alpha[0].astype(np.float64)), np.exp(alpha[1].astype(np.float64)), prof)
    on = mask.astype(bool)
    a, mk = torch.tensor(alpha, device="cuda"), torch.tensor(mask, device="cuda")
    with mr.Plan(seq) as plan:
        plan.set_slice_profile(prof.n_iso, prof.n_sub, prof.sigma, prof.tbw, prof.extent)
        plan.linearize(a, mask=mk)
        for c, key in enumerate(("m", "dm_dlnT1", "dm_dlnT2")):
            got = plan.timecourses(c).cpu().numpy().astype(np.float64)
            assert metrics.relerr(got[:, on], ref[key].imag[:, on]) < 1e-5, key
            assert not got[:, ~on].any()
        s = plan.forward(a, mask=mk).cpu().numpy()
    rho = (alpha[2] + 1j * alpha[3]).astype(np.complex128) * on
    want = np.stack([encoding.phase_matrix(seq, int(seq.ky[n])) @ (rho * ref["m"][n]) for n in range(seq.ntr)])
    assert metrics.relerr(s, want) < 1e-5
