"""The exact model by recomputation (the path of hard-pulse plans without a B1 map, ny <= 256)
against the stored time courses, which the same plan takes when a B1 map of ones is given.

Both are FP32 evaluations of one model; each is within 1e-5 of the oracle (the other parity
tests), most of it the recursion's rounding over the train.  Bar 1e-5 normwise per output and
parameter row.  Shapes at the edges of the kernels: one row, odd rows, a row count that fills
the last warp (256) and the first that does not apply (257); columns that do not fill a tile;
trains that are not a multiple of the chunk, span several pulse tables and segments; ky orders
that are shuffled or leave lines out; masks that empty warps and whole columns.
"""
import dataclasses

import numpy as np
import pytest

import synth
from oracle import metrics

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 1e-5

# nx, ny, nkx, ntr, ky order, mask
SHAPES = [(1, 1, 1, 5, "linear", False), (3, 2, 3, 7, "linear", False), (5, 31, 5, 130, "shuffled", True),
          (6, 33, 9, 129, "linear", False), (4, 64, 4, 1031, "random", True), (13, 97, 13, 300, "shuffled", True),
          (9, 224, 9, 449, "linear", True), (7, 255, 11, 260, "random", False), (6, 256, 6, 513, "linear", True),
          (5, 257, 5, 260, "linear", False), (130, 16, 130, 64, "linear", True)]


def make(nx, ny, nkx, ntr, order, masked):
    rng = np.random.default_rng([nx, ny, ntr])
    seq = synth.make_sequence(nx, ny, 1, 7.6, 3.3, seed=ny, nkx=nkx, extra_trs=max(0, ntr - ny))
    ky = seq.ky[:ntr].copy()
    if order == "shuffled":
        rng.shuffle(ky)
    elif order == "random":
        ky = (rng.integers(0, ny, ntr) - ny // 2).astype(np.int32)
    seq = dataclasses.replace(seq, flip_rad=synth.flip_train(ntr, 3, 5).astype(np.float32).astype(np.float64), ky=ky)
    nv = nx * ny
    alpha = np.stack([rng.uniform(np.log(200), np.log(4000), nv), rng.uniform(np.log(20), np.log(400), nv),
                      rng.uniform(-1, 1, nv), rng.uniform(-1, 1, nv)]).astype(np.float32)
    mask = None
    if masked:
        mask = (rng.random((ny, nx)) < 0.8)
        mask[ny // 4: ny // 4 + max(1, ny // 2)] = False
        mask[:, nx // 2] = False
        mask = mask.astype(np.uint8).ravel()
    dev = lambda a, t=torch.float32: torch.tensor(np.ascontiguousarray(a), dtype=t, device="cuda")  # noqa: E731
    return (seq, dev(alpha), None if mask is None else dev(mask, torch.uint8), dev(synth.random_params(nv, 1)),
            dev(synth.random_kspace(ntr, nkx, 2), torch.complex64), torch.ones(nv, device="cuda"))


def close(got, ref, what):
    got, ref = got.cpu().numpy(), ref.cpu().numpy()
    for k in range(len(ref)) if what in ("g", "h", "gc") else [slice(None)]:
        if np.linalg.norm(ref[k]) > 0:
            assert metrics.relerr(got[k], ref[k]) < TOL, (what, k, metrics.relerr(got[k], ref[k]))
        else:
            assert not np.any(got[k]), (what, k)


@pytest.mark.parametrize("shape", SHAPES)
def test_products_match_stored_time_courses(shape):
    import paper_1904_13244_gb300 as mr
    seq, a, mask, v, w, ones = make(*shape)
    out = {}
    with mr.Plan(seq) as plan:
        for b1 in (None, ones):
            plan.linearize(a, b1=b1, mask=mask)
            r = dict(jv=plan.jvp(v), g=plan.jhw(w), h=plan.jhjv(v), s=plan.forward(a, b1=b1, mask=mask))
            r.update({f"t{c}": plan.timecourses(c) for c in range(3)})
            r["h2"] = plan.jhjv(v)  # timecourses leave the linearisation as it was
            r["sc"] = plan.forward_ckpt(a, b1=b1, mask=mask, interval=12)
            r["gc"] = plan.jhw_ckpt(w)
            r["jv2"] = plan.jvp(v)  # and so does a checkpointed forward
            out[b1 is None] = r
        plan.check()
    for k, ref in out[False].items():
        close(out[True][k], ref, k)
    assert torch.equal(out[True]["h"], out[True]["h2"]) and torch.equal(out[True]["jv"], out[True]["jv2"])


def test_parameters_outside_the_mask_do_not_count():
    import paper_1904_13244_gb300 as mr
    seq, a, mask, v, w, _ = make(13, 97, 13, 300, "linear", True)
    bad = a.clone()
    bad[:, mask == 0] = float("nan")
    with mr.Plan(seq) as plan:
        plan.linearize(a, mask=mask)
        ref = [plan.jvp(v), plan.jhw(w), plan.jhjv(v), plan.forward(a, mask=mask)]
        plan.linearize(bad, mask=mask)
        got = [plan.jvp(v), plan.jhw(w), plan.jhjv(v), plan.forward(bad, mask=mask)]
    assert all(torch.equal(x, y) for x, y in zip(got, ref))


def test_solves_in_a_row_on_one_plan_agree():
    import paper_1904_13244_gb300 as mr
    seq, ph = synth.config("quad16")
    rho = np.stack([ph.rho.real.ravel(), ph.rho.imag.ravel()])
    truth = np.concatenate([np.log([ph.t1_ms.ravel(), ph.t2_ms.ravel()]), rho])
    with mr.Plan(seq) as plan:
        d = plan.forward(torch.tensor(truth, dtype=torch.float32, device="cuda"))
        runs = []
        for _ in range(3):
            a = torch.zeros((4, seq.nv), device="cuda")
            mask = torch.zeros(seq.nv, dtype=torch.uint8, device="cuda")
            rep = plan.gn_solve(d, a, mask=mask, outer_iters=3, inner_iters=5, rho_init_exact=1, mask_threshold=0.1)
            runs.append((a, rep["f"]))
            plan.timecourses(0)
        assert sum(rep["accepted"]) >= 1
    assert all(torch.equal(r[0], runs[0][0]) and r[1] == runs[0][1] for r in runs)
