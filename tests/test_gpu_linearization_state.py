"""A plan whose linearisation is gone says so: a product then is an error, not a launch on
buffers that were never filled.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def setup():
    import paper_1904_13244_gb300 as mr
    seq = synth.make_sequence(12, 10, 4, 7.6, 3.8, seed=1)
    rng = np.random.default_rng(1)
    alpha = np.stack([rng.uniform(np.log(300), np.log(3000), seq.nv), rng.uniform(np.log(30), np.log(300), seq.nv),
                      rng.uniform(0.5, 1, seq.nv), rng.uniform(-1, 1, seq.nv)])
    U = torch.linalg.qr(torch.randn((seq.ntr, 8), generator=torch.Generator().manual_seed(3)))[0].contiguous().cuda()
    dev = lambda a, t=torch.float32: torch.tensor(a, dtype=t, device="cuda")  # noqa: E731
    return (mr, mr.Plan(seq), dev(alpha), U, dev(synth.random_params(seq.nv, 1)),
            dev(synth.random_kspace(seq.ntr, seq.nkx, 2), torch.complex64))


def refused(mr, plan, v, w):
    for call in (lambda: plan.jvp(v), lambda: plan.jhw(w), lambda: plan.jhjv(v), lambda: plan.cg_fixed(v, 2),
                 lambda: plan.timecourses(0)):
        with pytest.raises(mr.MrstatError, match="(?i)lineari"):
            call()


def test_another_basis_drops_the_lowrank_linearisation():
    mr, plan, a, U, v, w = setup()
    with plan:
        plan.lowrank_set_basis(U)
        plan.lowrank_linearize(a)
        plan.jvp(v)
        plan.lowrank_set_basis(U)
        refused(mr, plan, v, w)
        plan.linearize(a)  # an exact linearisation stays when the basis changes
        ref = plan.jhjv(v)
        plan.lowrank_set_basis(U)
        assert torch.equal(plan.jhjv(v), ref)


def test_failed_solve_leaves_no_linearisation():
    mr, plan, a, U, v, w = setup()
    with plan:
        plan.linearize(a)
        ref = plan.jhjv(v)
        with pytest.raises(mr.MrstatError, match="finite"):
            plan.gn_solve(torch.full_like(w, float("nan")), a.clone(), outer_iters=1, inner_iters=2)
        refused(mr, plan, v, w)
        plan.linearize(a)
        assert torch.equal(plan.jhjv(v), ref)


def test_captured_calls_follow_the_linearisation():
    """A captured product or time course reads the plan's linearisation when it is replayed, and a
    captured linearisation serves the calls after its replay."""
    mr, plan, a, U, v, w = setup()
    b = a + 0.2
    with plan:
        def calls():
            return [plan.timecourses(c) for c in range(3)] + [plan.jvp(v), plan.jhw(w), plan.jhjv(v)]

        plan.linearize(b)
        ref = calls()
        x = a.clone()
        plan.linearize(x)
        old = calls()
        torch.cuda.synchronize()
        reads, lin = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
        with torch.cuda.graph(reads):
            out = calls()
        with torch.cuda.graph(lin):
            plan.linearize(x)
        plan.linearize(b)
        reads.replay()
        assert all(torch.equal(p, q) for p, q in zip(out, ref))
        lin.replay()
        assert all(torch.equal(p, q) for p, q in zip(calls(), old))
        x.copy_(b)
        lin.replay()
        assert all(torch.equal(p, q) for p, q in zip(calls(), ref))


def test_captured_lowrank_calls_follow_the_coefficients():
    """The same for the low-rank form, whose column kernels read a reordered copy of the
    coefficients: whatever was captured, a product sees those of the last linearisation."""
    import paper_1904_13244_gb300 as mr
    seq = synth.make_sequence(20, 64, 3, 7.6, 3.8, seed=1)
    rng = np.random.default_rng(1)
    a, b = (torch.tensor(np.stack([rng.uniform(np.log(300), np.log(3000), seq.nv),
                                   rng.uniform(np.log(30), np.log(300), seq.nv), rng.uniform(0.5, 1, seq.nv),
                                   rng.uniform(-1, 1, seq.nv)]), dtype=torch.float32, device="cuda") for _ in range(2))
    U = torch.linalg.qr(torch.randn((seq.ntr, 16), generator=torch.Generator().manual_seed(3)))[0].contiguous().cuda()
    v = torch.tensor(synth.random_params(seq.nv, 1), dtype=torch.float32, device="cuda")
    with mr.Plan(seq) as plan:
        plan.lowrank_set_basis(U)

        def calls():
            return [plan.jhjv(v), plan.jvp(v)]

        ref, coef = [], []
        for x in (a, b):
            plan.lowrank_linearize(x)
            coef.append(plan.lowrank_coefficients())
            ref.append(calls())
        assert not torch.equal(ref[0][0], ref[1][0])
        x = a.clone()
        torch.cuda.synchronize()
        reads, proj, both = (torch.cuda.CUDAGraph() for _ in range(3))
        with torch.cuda.graph(reads):
            out = calls()
        with torch.cuda.graph(proj):
            plan.lowrank_linearize(x)
        with torch.cuda.graph(both):
            plan.lowrank_linearize(x, coef=coef[0])
            out_both = calls()

        def same(got, k):
            return all(torch.equal(p, q) for p, q in zip(got, ref[k]))

        plan.lowrank_linearize(a)
        reads.replay()
        assert same(out, 0)
        plan.lowrank_linearize(b, coef=coef[1])
        reads.replay()
        assert same(out, 1)
        proj.replay()  # an adopted linearisation, then a replayed projection (rho stays b's or x's)
        assert same(calls(), 0)
        x.copy_(b)
        proj.replay()
        assert same(calls(), 1)
        reads.replay()
        assert same(out, 1)
        x.copy_(a)
        both.replay()
        assert same(out_both, 0) and same(calls(), 0)
