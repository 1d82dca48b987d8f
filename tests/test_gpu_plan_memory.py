"""Device memory of the recomputed exact form: its products run on a few floats per voxel and
segment, so neither a linearisation nor a solve depends on room for the time courses.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def maps(seq, seed=3):
    rng = np.random.default_rng(seed)
    return torch.tensor(np.stack([rng.uniform(np.log(300), np.log(3000), seq.nv),
                                  rng.uniform(np.log(30), np.log(300), seq.nv), rng.uniform(0.5, 1, seq.nv),
                                  rng.uniform(-1, 1, seq.nv)]), dtype=torch.float32, device="cuda")


def test_linearisation_whose_time_courses_exceed_the_device():
    """1700 x 256 voxels and 65536 TRs: 342 GB of time courses, 0.1 GB of states."""
    import paper_1904_13244_gb300 as mr
    seq = synth.make_sequence(1700, 256, 256, 7.6, 3.8, nkx=2)
    d_bytes = 12 * seq.ntr * seq.nv
    if torch.cuda.mem_get_info()[1] >= d_bytes:
        pytest.skip("the time courses fit this device")
    rng = np.random.default_rng(1)
    v = torch.tensor(rng.standard_normal((4, seq.nv)), dtype=torch.float32, device="cuda")
    with mr.Plan(seq) as plan:
        plan.linearize(maps(seq))
        info = plan.info()
        assert info["timecourse_bytes"] == 0 and info["device_bytes"] < 1e10
        jv = plan.jvp(v)
        h = plan.jhjv(v)
        # <v, J^H J v> = <J v, J v>, at the bar of the inner-product tests
        a, b = float((v.double() * h.double()).sum()), float(jv.abs().double().square().sum())
        assert abs(a - b) < 1e-4 * b, (a, b)


def test_solve_needs_no_time_courses():
    import paper_1904_13244_gb300 as mr
    seq = synth.make_sequence(48, 40, 16, 7.6, 3.8, seed=4)
    truth = maps(seq)
    with mr.Plan(seq) as plan:
        d = plan.forward(truth)
        a = truth + 0.05
        plan.gn_solve(d, a, outer_iters=2, inner_iters=4, rho_init_exact=1)
        assert plan.info()["timecourse_bytes"] == 0
        got = [plan.timecourses(c) for c in range(3)]  # of the solution, filled on demand
        plan.linearize(a)
        ref = [plan.timecourses(c) for c in range(3)]
        n = plan.info()["device_bytes"]
        plan.linearize(a)
        plan.timecourses(0)
        assert plan.info()["device_bytes"] == n
    assert all(torch.equal(x, y) for x, y in zip(got, ref)) and float(ref[0].abs().max()) > 0


def test_checkpoint_intervals_share_one_allocation():
    """Longer and shorter intervals in turn: the states are allocated again only for more of them."""
    import paper_1904_13244_gb300 as mr
    seq = synth.make_sequence(20, 24, 30, 7.6, 3.8, seed=6)
    a, w = maps(seq), torch.tensor(synth.random_kspace(seq.ntr, seq.nkx, 2), dtype=torch.complex64, device="cuda")
    with mr.Plan(seq) as plan:
        plan.linearize(a)
        s, g = plan.forward(a), plan.jhw(w)
        sizes = []
        for interval in (720, 12, 720, 12):
            sc, gc = plan.forward_ckpt(a, interval=interval), plan.jhw_ckpt(w)
            assert float((sc - s).abs().max()) < 1e-4 * float(s.abs().max())
            assert float((gc - g).abs().max()) < 1e-4 * float(g.abs().max())
            sizes.append(plan.info()["device_bytes"])
        assert sizes[0] < sizes[1] == sizes[2] == sizes[3]
