"""Performance cases: the work a user of the framework has it do, through its public entry points.

The framework evaluates the MR-STAT signal model and its Jacobian products over parameter
maps.  A user builds a plan for a pulse sequence, linearises at a parameter map and applies
J v, Re(J^H w) and Re(J^H J) v inside CG; trains and runs a surrogate; differentiates the
signal with autograd; or hands the whole Gauss-Newton reconstruction to the library.  The
cases cover each of these over the sizes of the repository's own workloads (16 ... 256
voxels per side, 3 ... 16 k-space fills), with ragged sizes beside the round ones.

Kinds and their ``calls`` (made in this order by one pass):
  exact      the exact model: linearize, forward, jvp, jhw, jhjv (linearised in prepare() when
             ``linearize`` is not among the calls: the products of an inner CG solve)
  autograd   loss 1/2 ||s - d||^2 through the checkpointed torch.autograd form, and its gradient
  lowrank    the compressed form: linearize (exact projection) or infer (surrogate), then
             jvp, jhw, jhjv or cg (a fixed-count CG)
  train      loss and parameter gradient of the surrogate on one batch
  recon      a whole Gauss-Newton reconstruction
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_1904_13244_gb300 as mr
from paper_1904_13244_gb300.autograd import signal

TBW, EXTENT, SIGMA = 4.0, 2.0, 0.2  # slice profile (the library's defaults)
NORM = (math.log(1000.0), 1.0, math.log(100.0), 1.2, 1.0, 0.2)  # surrogate input normalisation


def listed():
    base = dict(form=0, extra=0, b1=False, mask=False, est_b1=False, n_iso=0, n_sub=0)
    return [
        # one outer step's products on a small grid: the smallest calls, where launches count
        dict(base, name="exact_64", kind="exact", nx=64, ny=64, nkx=64, fills=5, calls="linearize jvp jhw jhjv"),
        # a ragged acquisition: odd grid, oversampled readout, a partial last fill, a known
        # transmit map and a mask
        dict(base, name="exact_ragged_b1", kind="exact", nx=97, ny=81, nkx=128, fills=6, extra=5, b1=True, mask=True,
             calls="linearize forward jvp jhw jhjv"),
        # B1 estimated as the fifth unknown
        dict(base, name="exact_estimate_b1_128", kind="exact", nx=128, ny=128, nkx=128, fills=5, est_b1=True,
             calls="linearize jvp jhw jhjv"),
        # the products of the inner CG solve of a full-size slice, at a cached linearisation
        dict(base, name="exact_products_224", kind="exact", nx=224, ny=224, nkx=224, fills=5, calls="jvp jhw jhjv"),
        # the outer iteration's share at full size: model, linearisation and gradient, with the
        # readout DFT on the tensor cores
        dict(base, name="exact_outer_224_split", kind="exact", nx=224, ny=224, nkx=224, fills=5, form=1, mask=True,
             calls="linearize forward jhw"),
        # the slice-profile model at full size (the largest case)
        dict(base, name="slice_profile_224", kind="exact", nx=224, ny=224, nkx=224, fills=5, n_iso=32, n_sub=16,
             calls="linearize jhw forward"),
        # differentiation at full size: forward and backward with checkpoints every 64 TRs
        dict(base, name="autograd_224", kind="autograd", nx=224, ny=224, nkx=224, fills=5, interval=64),
        # the compressed model of a masked slice: projection of the exact recursion and CG
        dict(base, name="compressed_cg_224", kind="lowrank", nx=224, ny=224, nkx=224, fills=5, mask=True, rank=32,
             calls="linearize cg", iters=6),
        # the learned model with a transmit map: inference, adoption and CG
        dict(base, name="surrogate_cg_256_b1", kind="lowrank", nx=256, ny=256, nkx=256, fills=5, b1=True, rank=32,
             calls="infer cg", iters=6, hidden=256),
        # the compressed model on the constant-flip scan's grid (no multiple of 32): DFTs as GEMMs
        dict(base, name="compressed_112x88", kind="lowrank", nx=112, ny=88, nkx=112, fills=16, rank=32,
             calls="jvp jhw jhjv"),
        # a batch of surrogate training
        dict(base, name="train_4096", kind="train", nx=64, ny=64, nkx=64, fills=5, rank=32, hidden=256, batch=4096),
        # a whole reconstruction of a small slice
        dict(base, name="recon_64", kind="recon", nx=64, ny=64, nkx=64, fills=5, outer=3, inner=6),
    ]


def draw(rng):
    def size(lo, hi, step=1):
        return max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)) * step)

    base = dict(form=0, extra=0, b1=False, mask=rng.random() < 0.5, est_b1=False, n_iso=0, n_sub=0)
    kind = rng.choice(["exact", "exact", "exact", "autograd", "lowrank", "lowrank", "train", "recon", "slice"])
    nx, ny, fills = size(40, 240), size(40, 240), rng.randint(3, 8)
    nkx = rng.choice([nx, nx, nx, 2 * nx, nx + rng.randint(1, 30)])
    if kind == "exact":
        est = rng.random() < 0.25
        calls = rng.choice(["linearize jvp jhw jhjv", "jvp jhw jhjv", "linearize forward jhw", "linearize jhjv forward"])
        return dict(base, kind="exact", nx=nx, ny=ny, nkx=nkx, fills=fills, extra=rng.randint(0, 9), calls=calls,
                    form=rng.choice([0, 0, 1]), est_b1=est, b1=not est and rng.random() < 0.4)
    if kind == "slice":
        return dict(base, kind="exact", nx=size(40, 160), ny=size(40, 160), nkx=nx, fills=3, calls="linearize jhw forward",
                    n_iso=rng.choice([8, 16, 32]), n_sub=rng.choice([8, 16, 32]))
    if kind == "autograd":
        return dict(base, kind="autograd", nx=nx, ny=ny, nkx=nkx, fills=fills, extra=rng.randint(0, 9),
                    interval=rng.choice([32, 64, 128]), b1=rng.random() < 0.4)
    if kind == "lowrank":
        if rng.random() < 0.6:
            ny = 32 * rng.randint(2, 8)
        first = rng.choice(["linearize", "linearize", "infer", ""])
        then = rng.choice(["cg", "jhjv", "jvp jhw jhjv"])
        return dict(base, kind="lowrank", nx=nx, ny=ny, nkx=nx, fills=fills, rank=rng.choice([16, 24, 32, 32]),
                    calls=(first + " " + then).strip(), iters=rng.randint(2, 6), hidden=rng.choice([128, 256]),
                    b1=rng.random() < 0.4)
    if kind == "train":
        return dict(base, kind="train", nx=64, ny=64, nkx=64, fills=fills, rank=rng.choice([16, 24, 32]),
                    hidden=rng.choice([64, 128, 256]), batch=size(700, 16384))
    return dict(base, kind="recon", nx=size(32, 96), ny=size(32, 96), nkx=nx, fills=fills + 1, outer=rng.randint(1, 3),
                inner=rng.randint(2, 6), mask=False)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _sequence(case, rng):
    """Smooth flip train (three sinusoids, 0 ... 60 degrees), linear Cartesian order, inversion."""
    nx, ny, fills = case["nx"], case["ny"], case["fills"]
    nkx = case["nkx"] if case["kind"] in ("exact", "autograd") and not case["n_iso"] else nx
    ntr = fills * ny + case["extra"]
    n = np.arange(ntr) / ntr
    a, f, p = rng.uniform(0.5, 1, 3), rng.uniform(1, 2 * fills, 3), rng.uniform(0, 2 * np.pi, 3)
    raw = sum(a[i] * np.sin(2 * np.pi * f[i] * n + p[i]) for i in range(3))
    flips = (np.deg2rad(60.0) * (raw - raw.min()) / (raw.max() - raw.min())).astype(np.float32)
    return SimpleNamespace(nx=nx, ny=ny, nkx=nkx, ntr=ntr, nv=nx * ny, tr_ms=7.6, te_ms=3.8, inversion=True,
                           alternate_phase=True, flip_rad=flips, ky=(np.arange(ntr) % ny - ny // 2).astype(np.int32))


def _smooth(nx, ny, rng, terms=6):
    """Zero-mean unit-deviation smooth field [ny, nx]."""
    x, y = np.linspace(0, 1, nx), np.linspace(0, 1, ny)
    out = np.zeros((ny, nx))
    for _ in range(terms):
        kx, ky, px, py = rng.uniform(0.5, 4), rng.uniform(0.5, 4), *rng.uniform(0, 2 * np.pi, 2)
        out += rng.normal() * np.cos(2 * np.pi * ky * y + py)[:, None] * np.cos(2 * np.pi * kx * x + px)[None, :]
    return (out - out.mean()) / max(out.std(), 1e-9)


def _maps(case, seq, rng):
    """A head-like slice: four tissue classes with 10 % texture, smooth proton-density phase,
    about half of the field of view empty.  (alpha [4 or 5, nv], b1, mask) in float32 / uint8."""
    nx, ny = seq.nx, seq.ny
    u, v = np.linspace(-1, 1, nx)[None, :], np.linspace(-1, 1, ny)[:, None]
    r = (u / 0.78) ** 2 + (v / 0.86) ** 2
    inside = r <= 1
    label = np.digitize(_smooth(nx, ny, rng), [-0.6, 0.5, 1.4])
    label = np.where(r > 0.85, 3, label)
    t1 = np.array([800.0, 1300.0, 4000.0, 350.0])[label] * (1 + 0.1 * np.clip(_smooth(nx, ny, rng), -2.5, 2.5))
    t2 = np.array([70.0, 90.0, 2000.0, 80.0])[label] * (1 + 0.1 * np.clip(_smooth(nx, ny, rng), -2.5, 2.5))
    t1, t2 = np.where(inside, t1, 1000.0), np.where(inside, t2, 100.0)
    rho = np.where(inside, np.array([0.65, 0.8, 1.0, 0.9])[label], 0.0) * np.exp(1j * _smooth(nx, ny, rng))
    b1 = np.clip(1 + 0.1 * _smooth(nx, ny, rng), 0.8, 1.2).astype(np.float32).ravel()
    rows = [np.log(t1), np.log(t2), rho.real, rho.imag]
    alpha = np.stack([x.ravel() for x in rows] + ([b1] if case["est_b1"] else [])).astype(np.float32)
    return alpha, b1 if case["b1"] else None, inside.ravel().astype(np.uint8) if case["mask"] else None


def _basis(seq, rank, rng):
    """Leading left singular vectors of simulated time courses and tangents, float32 [ntr, rank]."""
    n = 160
    x = np.stack([rng.uniform(math.log(100), math.log(6000), n), rng.uniform(math.log(10), math.log(3000), n)])
    Y = _courses(seq, x[0], x[1], rng.uniform(0.8, 1.2, n), 3, np)
    Y = np.concatenate(list(Y), axis=1)
    w, V = np.linalg.eigh(Y.T @ Y)
    Q, _ = np.linalg.qr(Y @ V[:, ::-1][:, :rank])
    return Q.astype(np.float32)


def _surrogate(seq, U, hidden, rank, rng):
    """Parameters of a network that follows the compressed model: random tanh features and a
    least-squares output layer on values and both tangents.  (theta, output scale) float32."""
    n = 768
    x = np.stack([rng.uniform(math.log(100), math.log(6000), n), rng.uniform(math.log(10), math.log(3000), n),
                  rng.uniform(0.8, 1.2, n)])
    tgt = U.astype(np.float64).T @ _courses(seq, x[0], x[1], x[2], 3, np)  # [3, rank, n]
    scale = np.maximum(np.abs(tgt[0]).max(axis=1), 1e-6).astype(np.float32)
    layers = [(rng.normal(size=(hidden, 3)) * 0.6, rng.normal(size=hidden) * 0.5)]
    layers += [(rng.normal(size=(hidden, hidden)) * (1.2 / math.sqrt(hidden)), rng.normal(size=hidden) * 0.2)
               for _ in range(2)]
    layers.append((np.zeros((rank, hidden)), np.zeros(rank)))
    feats = _mlp(torch.tensor(x), layers, True)[:3]
    F = np.concatenate([np.concatenate([feats[0].numpy(), np.ones((1, n))]),
                        *[np.concatenate([f.numpy(), np.zeros((1, n))]) for f in feats[1:]]], axis=1)
    T = np.concatenate(list(tgt), axis=1) / scale[:, None]
    G = F @ F.T
    W = np.linalg.solve(G + 1e-6 * np.trace(G) / len(G) * np.eye(len(G)), F @ T.T).T
    layers[3] = (W[:, :hidden], W[:, hidden])
    return np.concatenate([np.concatenate([w.ravel(), b]) for w, b in layers]).astype(np.float32), scale


def _inputs(case, seed):
    """Everything a pass reads, on the host or the device, without the framework."""
    rng = np.random.default_rng([int(seed), 41])
    s = SimpleNamespace(seq=_sequence(case, rng))
    seq, dev = s.seq, "cuda"
    s.alpha_h, s.b1_h, s.mask_h = _maps(case, seq, rng)
    npar = len(s.alpha_h)
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    s.alpha = torch.tensor(s.alpha_h, device=dev)
    s.b1 = None if s.b1_h is None else torch.tensor(s.b1_h, device=dev)
    s.mask = None if s.mask_h is None else torch.tensor(s.mask_h, device=dev)
    s.v = torch.randn((npar, seq.nv), generator=gen, device=dev)
    s.w = torch.randn((seq.ntr, seq.nkx), generator=gen, device=dev, dtype=torch.complex64)
    if case["kind"] in ("lowrank", "train"):
        s.U_h = _basis(seq, case["rank"], rng)
        s.U = torch.tensor(s.U_h, device=dev)
        if case["kind"] == "train" or "infer" in case["calls"]:
            s.theta, s.scale = _surrogate(seq, s.U_h, case["hidden"], case["rank"], rng)
    if case["kind"] == "train":
        n = case["batch"]
        x = np.stack([rng.uniform(math.log(100), math.log(6000), n), rng.uniform(math.log(10), math.log(3000), n)])
        s.x = torch.tensor(x, dtype=torch.float32, device=dev)
        s.xb = torch.tensor(rng.uniform(0.8, 1.2, n), dtype=torch.float32, device=dev)
        Y = _courses(seq, s.x[0].double(), s.x[1].double(), s.xb.double(), 3, torch)
        s.target = torch.matmul(s.U.double().T, Y).float().contiguous()
        # weights somewhere in the middle of a training: off the fitted ones
        s.theta = (s.theta * (1 + 0.05 * rng.normal(size=len(s.theta)))).astype(np.float32)
    if "cg" in case.get("calls", ""):
        # a Gauss-Newton right-hand side: Re(J^H w) scaled to unit RMS
        g = _jhw(_model(case, s), s.w)
        s.rhs = (g / g.square().mean().sqrt()).float().contiguous()
    if case["kind"] in ("autograd", "recon"):
        # noisy data of the true maps; the gradient is taken at a point beside them
        d = _forward(_model(case, s))
        noise = torch.randn(d.shape, generator=gen, device=dev, dtype=torch.complex64)
        s.d = (d + noise * (torch.linalg.vector_norm(d) / (30 * torch.linalg.vector_norm(noise)))).to(torch.complex64)
        s.alpha = s.alpha + 0.1 * torch.tensor(np.stack([_smooth(seq.nx, seq.ny, rng).ravel() for _ in range(4)]),
                                               dtype=torch.float32, device=dev) * (s.alpha[2:3] != 0)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s.case = case
    if case["kind"] == "train" or "infer" in case.get("calls", ""):
        s.net = mr.Surrogate(case["hidden"], case["rank"], NORM, 0.5, seed=1)
        s.net.set_output_scale(s.scale)
        s.net.set_params(s.theta)
    if case["kind"] == "train":
        s.grad = torch.empty(s.net.num_params, dtype=torch.float32, device="cuda")
        return s
    s.plan = mr.Plan(s.seq, form=case["form"], estimate_b1=case["est_b1"])
    if case["n_iso"]:
        s.plan.set_slice_profile(n_iso=case["n_iso"], n_sub=case["n_sub"], sigma=SIGMA, tbw=TBW, extent=EXTENT)
    if case["kind"] == "autograd":
        s.alpha.requires_grad_(True)
    if case["kind"] == "lowrank":
        s.plan.lowrank_set_basis(s.U)
        if "linearize" not in case["calls"] and "infer" not in case["calls"]:
            s.plan.lowrank_linearize(s.alpha, b1=s.b1, mask=s.mask)
    if case["kind"] == "exact" and "linearize" not in case["calls"]:
        s.plan.linearize(s.alpha, b1=s.b1, mask=s.mask)
    return s


def run(s):
    case = s.case
    if case["kind"] == "train":
        loss = s.net.loss_grad(s.x, s.target, b1=s.xb, grad=s.grad)
        return {"loss": loss, "grad": s.grad}
    if case["kind"] == "autograd":
        sig = signal(s.alpha, s.plan, s.b1, s.mask, case["interval"])
        loss = 0.5 * torch.sum(torch.abs(sig - s.d) ** 2)
        (grad,) = torch.autograd.grad(loss, s.alpha)
        return {"loss": loss.detach(), "s": sig.detach(), "grad": grad}
    if case["kind"] == "recon":
        alpha = s.alpha.clone()
        mask = torch.zeros(s.seq.nv, dtype=torch.uint8, device="cuda")
        rep = s.plan.gn_solve(s.d, alpha, mask=mask, outer_iters=case["outer"], inner_iters=case["inner"],
                              rho_init_exact=1, mask_threshold=0.1)
        return {"alpha": alpha, "f": rep["f_final"]}
    plan, out = s.plan, {}
    for c in case["calls"].split():
        if c == "linearize":
            (plan.linearize if case["kind"] == "exact" else plan.lowrank_linearize)(s.alpha, b1=s.b1, mask=s.mask)
        elif c == "infer":
            out["coef"] = s.net.infer(s.alpha[:2], b1=s.b1)
            plan.lowrank_linearize(s.alpha, b1=s.b1, mask=s.mask, coef=out["coef"])
        elif c == "forward":
            out["s"] = plan.forward(s.alpha, b1=s.b1, mask=s.mask)
        elif c == "jvp":
            out["jv"] = plan.jvp(s.v)
        elif c == "jhw":
            out["g"] = plan.jhw(s.w)
        elif c == "jhjv":
            out["h"] = plan.jhjv(s.v)
        elif c == "cg":
            out["x"] = plan.cg_fixed(s.rhs, case["iters"])
    return out


def work(case):
    seq = _sequence(case, np.random.default_rng(0))
    nv, ntr, npar = seq.nv, seq.ntr, 5 if case["est_b1"] else 4
    ks, par, vt = 8.0 * ntr * seq.nkx, 4.0 * npar * nv, float(nv) * ntr
    dft = 8.0 * ntr * seq.nx * seq.nkx
    nch = npar - 1
    if case["kind"] == "train":
        h, r, n = case["hidden"], case["rank"], case["batch"]
        return {"bytes": 4.0 * n * (3 + 3 * r) + 8.0 * (2 * h * h + h * r), "flops": 3 * 2.0 * 3 * n * (2 * h * h + h * (r + 1))}
    if case["kind"] == "autograd":
        return {"bytes": 2 * par + 2 * ks, "flops": vt * (40 + 12 + 60 + 20) + 2 * dft}
    if case["kind"] == "recon":
        k = case["outer"] * case["inner"]
        return {"bytes": ks + 2 * par, "flops": vt * (60 * (case["outer"] + 1) + 44 * k) + dft * (2 * case["outer"] + 1)}
    byts = flops = 0.0
    if case["kind"] == "lowrank":
        r = case["rank"]
        coef = 12.0 * r * nv
        # 2D DFTs of r images (5 N log2 N) and the sums over the basis
        fft = r * nv * 5.0 * (math.log2(seq.ny) + math.log2(seq.nx))
        colfft = r * nv * 5.0 * math.log2(seq.ny)
        for c in case["calls"].split():
            if c == "linearize":
                byts, flops = byts + par, flops + vt * (60 + 6 * r)
            elif c == "infer":
                h = case["hidden"]
                byts, flops = byts + par + coef, flops + 2.0 * 3 * nv * (2 * h * h + h * (r + 1))
            elif c in ("jvp", "jhw"):
                byts, flops = byts + ks + par + coef, flops + 10.0 * r * nv + fft + 4.0 * r * ntr * seq.nkx
            else:
                k = case["iters"] if c == "cg" else 1
                byts += 2 * par + coef
                flops += k * (20.0 * r * nv + 2 * colfft + 8.0 * r * ntr * seq.nx)
        return {"bytes": byts, "flops": flops}
    cached = "linearize" not in case["calls"]
    iso = max(1, case["n_iso"])
    sim = 95.0 * iso if case["n_iso"] else 20.0 * nch
    for c in case["calls"].split():
        if c == "linearize":
            byts, flops = byts + par, flops + vt * sim
        elif c == "forward":
            byts, flops = byts + par + ks, flops + vt * (sim / 3 + 12) + dft
        else:
            byts += {"jvp": par + ks, "jhw": par + ks, "jhjv": 2 * par}[c] + (4.0 * nch * vt if cached else 0.0)
            flops += {"jvp": 20 * vt + dft, "jhw": 20 * vt + dft, "jhjv": 40 * vt}[c]
    return {"bytes": byts, "flops": flops}


# ---------------------------------------------------------------------------
# the same results in 64 bits, in plain numpy / torch
# ---------------------------------------------------------------------------
def _courses(seq, lnt1, lnt2, b1, nch, xp, profile=None):
    """Echo values of m_y and its tangents (ln T1, ln T2[, B1]), [nch, ntr, n], of the Bloch
    recursion: rotation by the signed flip, relaxation over TE, echo, relaxation over TR - TE."""
    exp = np.exp if xp is np else torch.exp
    t1, t2 = exp(lnt1), exp(lnt2)
    n, ntr = len(t1), seq.ntr
    sign = np.where(np.arange(ntr) % 2 == 1, -1.0, 1.0) if seq.alternate_phase else np.ones(ntr)
    phi = seq.flip_rad.astype(np.float64) * sign
    zeros = (lambda *d: np.zeros(d)) if xp is np else (lambda *d: torch.zeros(d, dtype=torch.float64, device=t1.device))
    if profile is not None:
        return _slice_courses(seq, t1, t2, phi, profile)
    y, z, out = zeros(nch, n), zeros(nch, n), zeros(nch, ntr, n)
    z[0] = -1.0 if seq.inversion else 1.0
    steps = []
    for dt in (seq.te_ms, seq.tr_ms - seq.te_ms):
        e1, e2 = exp(-dt / t1), exp(-dt / t2)
        steps.append((e1, e2, dt / t1 * e1, dt / t2 * e2))
    if b1 is not None:
        cos, sin = (np.cos, np.sin) if xp is np else (torch.cos, torch.sin)
    for k in range(ntr):
        if b1 is None:
            c, s = math.cos(phi[k]), math.sin(phi[k])
        else:
            c, s = cos(phi[k] * b1), sin(phi[k] * b1)
        y, z = c * y + s * z, c * z - s * y
        if nch > 3:
            y[3] += phi[k] * z[0]
            z[3] -= phi[k] * y[0]
        for i, (e1, e2, d1, d2) in enumerate(steps):
            add1, add2 = d1 * (z[0] - 1), d2 * y[0]
            y, z = e2 * y, e1 * z
            z[0] += 1 - e1
            if nch > 1:
                z[1] += add1
                y[2] += add2
            if i == 0:
                out[:, k] = y
    return out


def _slice_courses(seq, t1, t2, phi, profile):
    """The slice-profile model: isochromats across the slice, Gaussian sub-pulses against a
    balanced slice-select gradient, the echo their mean."""
    n_iso, n_sub = profile
    u = EXTENT * ((np.arange(n_iso) + 0.5) / n_iso - 0.5)
    wt = np.exp(-(((np.arange(n_sub) + 0.5) / n_sub - 0.5) ** 2) / (2 * SIGMA ** 2))
    wt /= wt.sum()
    beta = 2 * np.pi * TBW * u / n_sub

    def about_z(a):
        o = np.zeros((n_iso, 3, 3))
        o[:, 0, 0] = o[:, 1, 1] = np.cos(a)
        o[:, 0, 1], o[:, 1, 0], o[:, 2, 2] = -np.sin(a), np.sin(a), 1
        return o

    wind, grad = about_z(-0.5 * n_sub * beta), about_z(beta)
    n, ntr, dev = len(t1), seq.ntr, t1.device
    m = torch.zeros((n_iso, 3, 3 * n), dtype=torch.float64, device=dev)  # [iso, xyz, (value, d1, d2) x n]
    m[:, 2, :n] = -1.0 if seq.inversion else 1.0
    out = torch.zeros((3, ntr, n), dtype=torch.float64, device=dev)
    for k in range(ntr):
        rot = wind
        for s in range(n_sub):
            a = phi[k] * wt[s]
            rx = np.array([[1, 0, 0], [0, math.cos(a), math.sin(a)], [0, -math.sin(a), math.cos(a)]])
            rot = grad @ (rx @ rot)
        m = torch.matmul(torch.tensor(wind @ rot, device=dev), m)
        for i, dt in enumerate((seq.te_ms, seq.tr_ms - seq.te_ms)):
            e1, e2 = torch.exp(-dt / t1), torch.exp(-dt / t2)
            add1 = (dt / t1 * e1) * (m[:, 2, :n] - 1)
            add2 = (dt / t2 * e2) * m[:, :2, :n]
            m[:, :2] *= e2.repeat(3)
            m[:, 2] *= e1.repeat(3)
            m[:, 2, :n] += 1 - e1
            m[:, 2, n:2 * n] += add1
            m[:, :2, 2 * n:] += add2
            if i == 0:
                out[:, k] = m[:, 1].mean(0).view(3, n)
    return out


def _model(case, s, alpha=None, courses=None):
    """Time courses, phases and masked proton density of the linearised model in 64 bits."""
    seq, dev = s.seq, "cuda"
    a = (s.alpha if alpha is None else alpha).detach().double()
    npar = a.shape[0]
    b1 = a[4] if npar == 5 else None if s.b1 is None else s.b1.double()
    if courses is None:
        prof = (case["n_iso"], case["n_sub"]) if case["n_iso"] else None
        courses = _courses(seq, a[0], a[1], b1, npar - 1, torch, prof)
    k = torch.arange(seq.nkx, device=dev, dtype=torch.float64) - seq.nkx // 2
    ix, iy = torch.arange(seq.nx, device=dev).double(), torch.arange(seq.ny, device=dev).double()
    F = torch.exp(-2j * np.pi * torch.remainder(k[:, None] * ix[None], seq.nx) / seq.nx)  # [nkx, nx]
    E = torch.exp(-2j * np.pi * torch.remainder(torch.tensor(seq.ky, device=dev).double()[:, None] * iy[None], seq.ny) / seq.ny)
    m = torch.ones(seq.nv, device=dev, dtype=torch.float64) if s.mask is None else (s.mask != 0).double()
    return SimpleNamespace(seq=seq, Y=courses, F=F, E=E, m=m, rho=torch.complex(a[2], a[3]) * m, npar=npar)


def _encode(M, coef):
    """s = sum over voxels of i sum_c coef_c y_c exp(-i k.r), coef [nch, nv] complex."""
    seq, out = M.seq, []
    for a in range(0, seq.ntr, 64):
        q = sum(c * y for c, y in zip(coef, M.Y[:, a:a + 64]))
        q = (1j * q).view(-1, seq.ny, seq.nx)
        out.append(torch.matmul(torch.matmul(M.E[a:a + 64, None, :], q)[:, 0], M.F.T))
    return torch.cat(out)


def _forward(M):
    return _encode(M, [M.rho])


def _jvp(M, v):
    v = v.double()
    return _encode(M, [torch.complex(v[2], v[3]) * M.m, M.rho * v[0], M.rho * v[1]] + [M.rho * v[k] for k in range(4, M.npar)])


def _jhw(M, w):
    seq = M.seq
    wt = torch.matmul(w.to(torch.complex128), M.F.conj())  # [ntr, nx]
    Z = torch.zeros((len(M.Y), seq.nv), dtype=torch.complex128, device=wt.device)
    for a in range(0, seq.ntr, 64):
        b = (M.E[a:a + 64].conj()[:, :, None] * wt[a:a + 64, None, :]).view(-1, seq.nv)
        for c in range(len(M.Y)):
            Z[c] += (M.Y[c, a:a + 64] * b).sum(0)
    Z = -1j * Z  # conj(i)
    r = M.rho.conj()
    rows = [(r * Z[1]).real, (r * Z[2]).real, Z[0].real * M.m, (-1j * Z[0]).real * M.m]
    return torch.stack(rows + [(r * Z[k - 1]).real for k in range(4, M.npar)])


def _mlp(x, layers, features=False):
    """Values and ln T1 / ln T2 tangents of the network; x: [3, n] float64 tensor."""
    mu, sd = x.new_tensor(NORM[0::2])[:, None], x.new_tensor(NORM[1::2])[:, None]
    a = (x - mu) / sd
    t = [torch.zeros_like(a), torch.zeros_like(a)]
    t[0][0], t[1][1] = 1 / sd[0], 1 / sd[1]
    for i, (W, b) in enumerate(layers):
        if features and i == 3:
            break
        W, b = torch.as_tensor(W, dtype=x.dtype, device=x.device), torch.as_tensor(b, dtype=x.dtype, device=x.device)
        z, t = W @ a + b[:, None], [W @ q for q in t]
        a = z
        if i < 3:
            a = torch.tanh(z)
            t = [(1 - a * a) * q for q in t]
    return a, t[0], t[1]


def _layers(theta, hidden, rank):
    out, k = [], 0
    for o, i in ((hidden, 3), (hidden, hidden), (hidden, hidden), (rank, hidden)):
        out.append((theta[k:k + o * i].view(o, i), theta[k + o * i:k + o * i + o]))
        k += o * i + o
    return out


def exact(case, seed):
    if case["kind"] == "recon":
        return None
    s = _inputs(case, seed)
    seq = s.seq
    if case["kind"] == "train":
        theta = torch.tensor(s.theta, dtype=torch.float64, device="cuda", requires_grad=True)
        x = torch.cat([s.x.double(), s.xb.double()[None]])
        pred = _mlp(x, _layers(theta, case["hidden"], case["rank"]))
        sc = torch.tensor(s.scale, device="cuda").double()[:, None]
        res = [p - t.double() / sc for p, t in zip(pred, s.target)]
        loss = (res[0].square().sum() + 0.5 * (res[1].square().sum() + res[2].square().sum())) / case["batch"]
        (grad,) = torch.autograd.grad(loss, theta)
        return {"loss": float(loss), "grad": grad}
    if case["kind"] == "autograd":
        M = _model(case, s)
        sig = _forward(M)
        res = sig - s.d.to(torch.complex128)
        return {"loss": 0.5 * res.abs().square().sum(), "s": sig, "grad": _jhw(M, res)}
    out = {}
    if case["kind"] == "exact":
        M = _model(case, s)
    else:
        U = s.U.double()
        if "infer" in case["calls"]:
            b1 = torch.ones_like(s.alpha[0]) if s.b1 is None else s.b1
            layers = _layers(torch.tensor(s.theta, device="cuda").double(), case["hidden"], case["rank"])
            sc = torch.tensor(s.scale, device="cuda").double()[:, None]
            coef = torch.stack([sc * c for c in _mlp(torch.cat([s.alpha[:2], b1[None]]).double(), layers)])
            out["coef"] = coef
            M = _model(case, s, courses=torch.matmul(U, coef))
        else:
            M = _model(case, s)
            M.Y = torch.matmul(U, torch.matmul(U.T, M.Y))
    for c in case["calls"].split():
        if c == "forward":
            out["s"] = _forward(M)
        elif c == "jvp":
            out["jv"] = _jvp(M, s.v)
        elif c == "jhw":
            out["g"] = _jhw(M, s.w)
        elif c == "jhjv":
            out["h"] = _jhw(M, _jvp(M, s.v))
        elif c == "cg":
            r = s.rhs.double()
            x, p, rr = torch.zeros_like(r), r.clone(), (r * r).sum()
            for _ in range(case["iters"]):
                q = _jhw(M, _jvp(M, p))
                al = rr / (p * q).sum()
                x, r = x + al * p, r - al * q
                new = (r * r).sum()
                p, rr = r + new / rr * p, new
            out["x"] = x
    return out
