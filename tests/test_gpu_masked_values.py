"""Parameters outside the mask do not count, whatever they hold: NaN, or the -inf that the log
of a map leaves where the map is zero.  Every output is bit for bit the one with finite
parameters there.  The masks leave warps and blocks partly and wholly empty.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BAD = [float("nan"), float("-inf")]


def make(nx, ny, fills, extra=0, npar=4):
    rng = np.random.default_rng([nx, ny])
    seq = synth.make_sequence(nx, ny, fills, 7.8, 3.4, seed=nx, extra_trs=extra)
    nv = seq.nv
    alpha = [rng.uniform(np.log(200), np.log(3000), nv), rng.uniform(np.log(20), np.log(300), nv),
             rng.uniform(0.5, 1, nv), rng.uniform(-1, 1, nv), rng.uniform(0.8, 1.2, nv)][:npar]
    mask = (rng.random(nv) < 0.7).astype(np.uint8)
    mask[nv // 3: nv // 3 + nv // 4] = 0
    mask[-1], mask[0] = 0, 1
    dev = lambda a, t=torch.float32: torch.tensor(np.ascontiguousarray(a), dtype=t, device="cuda")  # noqa: E731
    v = rng.standard_normal((npar, nv))
    return (seq, dev(np.stack(alpha)), dev(mask, torch.uint8), dev(v),
            dev(synth.random_kspace(seq.ntr, seq.nkx, 2), torch.complex64))


def spoil(x, mask, value, rows=slice(None)):
    x = x.clone()
    x[rows, mask == 0] = value
    return x


def all_equal(got, ref):
    return all(bool(torch.isfinite(torch.view_as_real(r) if r.is_complex() else r).all()) for r in ref) and \
        all(torch.equal(g, r) for g, r in zip(got, ref))


def exact_calls(plan, a, mask, v, w, b1=None):
    plan.linearize(a, b1=b1, mask=mask)
    out = [plan.jvp(v), plan.jhw(w), plan.jhjv(v), plan.forward(a, b1=b1, mask=mask)]
    return out + [plan.timecourses(c) for c in range(a.shape[0] - 1)]


# 13 x 9: a lane per voxel in the forward kernel; 144 x 136: four of them
@pytest.mark.parametrize("value", BAD)
@pytest.mark.parametrize("nx,ny,fills", [(13, 9, 3), (144, 136, 1)])
@pytest.mark.parametrize("n_iso", [1, 8, 32])
def test_slice_profile_relaxation_times(n_iso, nx, ny, fills, value):
    import paper_1904_13244_gb300 as mr
    seq, a, mask, v, w = make(nx, ny, fills, extra=2)
    bad = spoil(a, mask, value, slice(0, 2))
    with mr.Plan(seq) as plan:
        plan.set_slice_profile(n_iso, 6, 0.2, 4.0, 2.0)
        ref = exact_calls(plan, a, mask, v, w)
        got = exact_calls(plan, bad, mask, v, w)
    assert all_equal(got, ref)
    assert not any(t[:, mask == 0].any() for t in got[4:])


@pytest.mark.parametrize("value", BAD)
def test_slice_profile_solve(value):
    import paper_1904_13244_gb300 as mr
    seq, a, mask, _, _ = make(24, 20, 5)
    with mr.Plan(seq) as plan:
        plan.set_slice_profile(8, 6, 0.2, 4.0, 2.0)
        d = plan.forward(a, mask=mask)
        outs = []
        for x in (a, spoil(a, mask, value, slice(0, 2))):
            x = x.clone()
            x[:2, mask != 0] += 0.1
            rep = plan.gn_solve(d, x, mask=mask, outer_iters=2, inner_iters=4)
            outs.append((x[:, mask != 0], rep["f"], rep["f_final"]))
    assert np.isfinite(outs[0][2])
    assert torch.equal(outs[0][0], outs[1][0]) and outs[0][1:] == outs[1][1:]


# 64 x 40: columns of 32 N rows; 33 x 20: the DFTs as GEMMs
@pytest.mark.parametrize("value", BAD)
@pytest.mark.parametrize("nx,ny,rank", [(40, 64, 32), (33, 20, 8)])
@pytest.mark.parametrize("with_b1", [False, True])
def test_lowrank_projection(with_b1, nx, ny, rank, value):
    import paper_1904_13244_gb300 as mr
    seq, a, mask, v, w = make(nx, ny, 4, extra=1)
    U = torch.linalg.qr(torch.randn((seq.ntr, rank), generator=torch.Generator().manual_seed(3)))[0].cuda()
    b1 = 0.9 + 0.2 * torch.rand(seq.nv, device="cuda") if with_b1 else None
    bad, bad_b1 = spoil(a, mask, value, slice(0, 2)), spoil(b1[None], mask, value)[0] if with_b1 else None
    with mr.Plan(seq) as plan:
        plan.lowrank_set_basis(U.contiguous())
        outs = []
        for x, b in ((a, b1), (bad, bad_b1)):
            plan.lowrank_linearize(x, b1=b, mask=mask)
            outs.append([plan.lowrank_coefficients(), plan.jvp(v), plan.jhw(w), plan.jhjv(v), plan.cg_fixed(v, 3)])
    assert all_equal(outs[1], outs[0])
    assert not outs[1][0][..., mask == 0].any()


@pytest.mark.parametrize("value", BAD)
@pytest.mark.parametrize("rows", [slice(2, 4), slice(None)], ids=["rho", "every row"])
@pytest.mark.parametrize("model", ["slice", "b1", "estimated b1", "checkpointed b1", "recompute"])
def test_proton_density(model, rows, value):
    import paper_1904_13244_gb300 as mr
    seq, a, mask, v, w = make(29, 21, 4, extra=3, npar=5 if model == "estimated b1" else 4)
    b1 = 0.9 + 0.2 * torch.rand(seq.nv, device="cuda") if model in ("b1", "checkpointed b1") else None
    bad = spoil(a, mask, value, rows)
    bad_b1 = spoil(b1[None], mask, value)[0] if b1 is not None and rows == slice(None) else b1
    with mr.Plan(seq, estimate_b1=model == "estimated b1") as plan:
        if model == "slice":
            plan.set_slice_profile(16, 6, 0.2, 4.0, 2.0)
        if model == "recompute":
            plan.set_recompute(32)
        outs = []
        for x, b in ((a, b1), (bad, bad_b1)):
            if model == "checkpointed b1":
                outs.append([plan.forward_ckpt(x, b1=b, mask=mask, interval=16), plan.jhw_ckpt(w)])
            elif model == "recompute":
                plan.linearize(x, mask=mask)
                outs.append([plan.jvp(v), plan.jhw(w), plan.jhjv(v)])
            else:
                outs.append(exact_calls(plan, x, mask, v, w, b1=b))
    assert all_equal(outs[1], outs[0])


@pytest.mark.parametrize("value", BAD)
@pytest.mark.parametrize("with_b1", [False, True])
def test_recompute_form(with_b1, value):
    import paper_1904_13244_gb300 as mr
    seq, a, mask, v, w = make(29, 21, 4, extra=3)
    b1 = 0.9 + 0.2 * torch.rand(seq.nv, device="cuda") if with_b1 else None
    bad, bad_b1 = spoil(a, mask, value), spoil(b1[None], mask, value)[0] if with_b1 else None
    outs = []
    with mr.Plan(seq) as plan:
        plan.set_recompute(32)
        for x, b in ((a, b1), (bad, bad_b1)):
            plan.linearize(x, b1=b, mask=mask)
            outs.append([plan.jvp(v), plan.jhw(w), plan.jhjv(v)])
    assert all_equal(outs[1], outs[0])
