"""What the simulator is timed on: the calls a user's program makes, over the range of sizes,
storages and directions it makes them at.

A case names one operation on one plan.  `op`:
  forward    Plan.forward: images of a batch of scenes
  sparse     Plan.forward(skip_zeros=True): images of scenes that are mostly empty
  adjoint    Plan.adjoint: A^T g for a batch of image-space residuals
  gradient   RingProblem.loss_and_grad: one step of a ring retrieval (loss, its gradient)
  build      Plan(...): the interpolated PSF library A itself
  multi      MultiForward.enqueue: scenes of several sizes and scales in one launch
`n` / `N` are the image and scene sides in pixels, `s` / `S` their scales in lambda/D, `n_r` the
number of library radii from 0 to `r_last` lambda/D, `B` the batch, `storage` and `interp` those
of Plan.  Libraries are synthetic Lyot-coronagraph PSFs, scenes are synthetic exozodiacal rings
with planets, residuals are noise at the level of a fit: all from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2106_09122_gb300.fit import RingProblem
from paper_2106_09122_gb300.plan import Plan
from paper_2106_09122_gb300.serve import MultiForward

DEV = torch.device("cuda")
F64 = torch.float64
FIELD = 32.0  # lambda/D across the image and the scene: the pixel scales follow from the sizes
SIGMA = 1e-11  # image noise of the retrieval cases
BYTES = {"fp32": 4, "fp32_sym": 4, "split_bf16": 4, "split_bf16_sym": 4, "bf16": 2}
SYMMETRIC = ("fp32_sym", "split_bf16_sym", "fused")  # an even scene side is needed


def _case(op, storage, n, N, n_r, B=1, r_last=12.0, s=None, S=None, interp="linear", scene="ring", name=None):
    c = {"op": op, "storage": storage, "n": n, "N": N, "s": s or FIELD / n, "S": S or FIELD / max(N, 1), "n_r": n_r,
         "r_last": r_last, "B": B, "interp": interp, "scene": scene}
    return dict(c, name=name) if name else c


def listed():
    mas = 575e-9 / 2.3631 * 180.0 / math.pi * 3600e3  # one lambda/D at 575 nm, D = 2.3631 m
    return [
        # One scene through a small plan: an interactive look, or one sample of a sampler's chain.
        _case("forward", "fp32", 64, 64, 20, 1, 9.5, scene="ring+planets", name="forward_64_one"),
        # A small batch of candidate scenes against plain FP32 storage (an odd batch).
        _case("forward", "fp32", 128, 128, 40, 11, name="forward_128_fp32_batch"),
        # Nothing a multiple of anything: a detector crop and an odd scene in the half-size storage.
        _case("forward", "bf16", 100, 85, 33, 23, name="forward_ragged_bf16"),
        # A ring masked beyond the outer working angle: most scene pixels are zero.
        _case("sparse", "fp32", 128, 128, 40, 1, scene="narrow", name="sparse_128_ring"),
        # One step of the ring retrieval, on the plain and on the compact storage.
        _case("gradient", "fp32", 128, 128, 40, name="gradient_128"),
        _case("gradient", "fp32_sym", 128, 128, 40, name="gradient_128_sym"),
        # Residuals of several images pulled back to their scenes.
        _case("adjoint", "split_bf16", 128, 128, 40, 8, name="adjoint_128_split_batch"),
        # A wave of 50 scenes of mixed sizes and scales, as a server runs it.
        dict(_case("multi", "split_bf16", 128, 0, 60, 50, name="multi_uneven"),
             buckets="64:0.3,64:0.5,96:0.3,96:0.5,128:0.3,128:0.5,192:0.3,192:0.5,256:0.3,256:0.5"),
        # 64 scenes at one wavelength of the 256 x 256 instrument, compact storage.
        _case("forward", "split_bf16_sym", 256, 256, 60, 64, scene="ring+planets", name="forward_256_split_sym"),
        # The library of one wavelength of that instrument, dense.
        _case("build", "split_bf16", 256, 256, 60, name="build_256_split"),
        # The paper's own geometry: 128 x 128 PSFs at 0.2 lambda/D onto a 256 x 256 scene at 3.529 mas.
        _case("build", "fp32", 128, 256, 86, r_last=11.0, s=0.2, S=3.529 / mas, name="build_paper_fp32"),
        # A scene whose A does not fit in memory: A is regenerated on chip for 32 scenes.
        _case("forward", "fused", 512, 512, 80, 32, scene="two_rings", name="fused_512"),
    ]


def _spread(rng, lo, hi):
    """A whole number between lo and hi, spread over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["forward", "forward", "forward", "sparse", "adjoint", "gradient", "build", "multi", "fused"])
    interp = rng.choice(["linear", "linear", "linear", "nearest"])
    n_r, r_last = rng.randint(16, 90), rng.uniform(6.0, 14.0)
    if op == "multi":
        k = rng.randint(2, 8)
        buckets = ",".join("%d:%.2f" % (_spread(rng, 48, 192), rng.uniform(0.2, 0.6)) for _ in range(k))
        return dict(_case("multi", rng.choice(["split_bf16", "bf16"]), _spread(rng, 64, 128), 0, n_r,
                          rng.randint(k, 8 * k), r_last, s=0.25, S=0.25, interp=interp), buckets=buckets)
    if op == "fused":
        n, N, B = _spread(rng, 96, 480), _spread(rng, 96, 480) // 2 * 2, _spread(rng, 1, 32)
        return _case("forward", "fused", n, N, n_r, B, r_last, interp=interp, scene="two_rings")
    storage = {"forward": ["fp32", "split_bf16", "bf16", "fp32_sym", "split_bf16_sym"], "sparse": ["fp32"],
               "adjoint": ["fp32", "split_bf16", "bf16", "fp32_sym", "split_bf16_sym"],
               "gradient": ["fp32", "fp32_sym"], "build": ["fp32", "split_bf16", "bf16"]}[op]
    storage = rng.choice(storage)
    top = 160 if storage.startswith("fp32") and op != "build" else 256
    top = 160 if op == "adjoint" else top
    n, N = _spread(rng, 48, top), _spread(rng, 48, top)
    if storage in SYMMETRIC:
        N = N // 2 * 2
    B = {"forward": _spread(rng, 1, 16 if storage.startswith("fp32") else 64), "sparse": _spread(rng, 1, 8),
         "adjoint": _spread(rng, 1, 16), "gradient": 1, "build": 1}[op]
    scene = rng.choice(["points", "narrow"]) if op == "sparse" else rng.choice(["ring", "ring+planets"])
    return _case(op, storage, n, N, n_r, B, r_last, interp=interp, scene=scene)


# ---------------------------------------------------------------- inputs


def _radii(case):
    if case["n_r"] == 86 and case["r_last"] == 11.0:  # the paper's sampling of its library
        return np.unique(np.round(np.concatenate([np.arange(0.0, 4.0, 0.06), np.arange(4.0, 9.0, 0.5),
                                                  np.arange(9.0, 11.0001, 0.25)]), 6))
    return np.linspace(0.0, case["r_last"], case["n_r"])


def _rng(seed, what):
    return np.random.default_rng([int(seed), what])


def _library(case, seed):
    """Off-axis PSFs of a Lyot coronagraph by matrix Fourier transforms: a circular pupil with a
    seeded low-order phase, a focal occulter 1 - exp(-(rho/2.5)^4), a 0.9 Lyot stop; float32
    [n_r, n, n] in units of the unocculted peak."""
    n, s, radii = case["n"], case["s"], torch.from_numpy(_radii(case)).to(DEV)
    P = 48
    u = ((torch.arange(P, dtype=F64, device=DEV) + 0.5) / P - 0.5)
    X, Y = u.view(1, -1), u.view(-1, 1)
    rho, th = 2.0 * torch.hypot(X, Y), torch.atan2(Y.expand(P, P), X.expand(P, P))
    pupil = (rho <= 1.0).to(F64)
    c = _rng(seed, 1).standard_normal(6) * 0.03
    phase = c[0] * (2 * rho**2 - 1) + c[1] * rho**2 * torch.cos(2 * th) + c[2] * rho**2 * torch.sin(2 * th) \
        + c[3] * (3 * rho**3 - 2 * rho) * torch.cos(th) + c[4] * (3 * rho**3 - 2 * rho) * torch.sin(th) \
        + c[5] * (6 * rho**4 - 6 * rho**2 + 1)
    field = (pupil * torch.exp(2j * math.pi * phase)).to(torch.complex128)
    tilt = torch.exp(2j * math.pi * radii.view(-1, 1, 1) * X)

    def kernel(coords):  # focal coordinates (lambda/D) x pupil coordinates
        return torch.exp(-2j * math.pi * coords.view(-1, 1) * u.view(1, -1)) / P

    f = (torch.arange(64, dtype=F64, device=DEV) - 31.5) * 0.25
    Ff = kernel(f)
    block = torch.exp(-(torch.hypot(f.view(1, -1), f.view(-1, 1)) / 2.5) ** 4).to(torch.complex128)
    E = field * tilt
    Ef = (Ff @ E @ Ff.t()) * block
    E = E - (Ff.conj().t() @ Ef @ Ff.conj()) * (P * 0.25) ** 2  # the part that the occulter removes
    E = E * (rho <= 0.9)
    Fi = kernel((torch.arange(n, dtype=F64, device=DEV) - 0.5 * (n - 1)) * s)
    psf = (Fi @ E @ Fi.t()).abs() ** 2
    return (psf / float((pupil.sum() / P**2) ** 2)).float().contiguous()


def _pixels(N, S):
    a = (torch.arange(N, dtype=F64, device=DEV) - 0.5 * (N - 1)) * S
    return a.view(1, -1), a.view(-1, 1)


def _ring(theta, x, y, r_max):
    R, w, inc, g, b = theta
    ci, si = torch.cos(inc), torch.sin(inc)
    yd = y / ci
    rd = torch.sqrt(x * x + yd * yd)
    mu = torch.where(rd > 0, si * yd / rd.clamp_min(1e-300), torch.zeros_like(rd))
    h = ((1 + g * g) / (1 + g * g - 2 * g * mu)) ** 1.5
    z = b * torch.exp(-4 * math.log(2.0) * (rd - R) ** 2 / w**2) * h
    return torch.where(torch.sqrt(x * x + y * y) <= r_max, z, torch.zeros_like(z))


def _scenes(N, S, B, kind, r_last, seed):
    """float32 [B, N*N]: inclined rings (one or two), planets on single pixels, or planets alone."""
    x, y = _pixels(N, S)
    rng, out = _rng(seed, 2), torch.zeros((B, N, N), dtype=F64, device=DEV)
    half = 0.5 * (N - 1) * S
    reach = min(r_last, half)
    for b in range(B):
        R, inc, g = rng.uniform(0.25, 0.7) * reach, rng.uniform(0.0, 1.3), rng.uniform(0.0, 0.6)
        if kind != "points":
            th = torch.tensor([R, 1.0, inc, g, 1e-9], dtype=F64)
            out[b] = _ring(th, x, y, r_last)
            if kind == "two_rings":
                out[b] += _ring(torch.tensor([2 * R, 1.0, inc, g, 0.3e-9], dtype=F64), x, y, r_last)
            if kind == "narrow":
                out[b][out[b] < 1e-12] = 0.0
        if kind in ("points", "ring+planets"):
            for _ in range(int(rng.integers(1, 5)) if kind != "points" else 10):
                rp, tp = rng.uniform(0.2, 0.9) * reach, rng.uniform(-math.pi, math.pi)
                ix = int(round(rp * math.cos(tp) / S + 0.5 * (N - 1)))
                iy = int(round(rp * math.sin(tp) / S + 0.5 * (N - 1)))
                out[b, min(max(iy, 0), N - 1), min(max(ix, 0), N - 1)] += 10 ** rng.uniform(-9, -7)
    return out.view(B, N * N).float().contiguous()


def _buckets(case):
    return [(int(a), float(b)) for a, b in (t.split(":") for t in case["buckets"].split(","))]


def _multi_counts(case, seed):
    nb = len(_buckets(case))
    pick = _rng(seed, 3).integers(0, nb, case["B"])
    return np.minimum(np.bincount(pick, minlength=nb), 16).astype(np.int32)


def _truth_and_guess(case, seed):
    rng = _rng(seed, 4)
    reach = min(case["r_last"], 0.5 * case["N"] * case["S"])
    t = np.array([0.42 * reach, 1.0, math.radians(60.0), 0.3, 1e-9])
    g = t * np.array([rng.uniform(0.93, 1.07), rng.uniform(0.8, 1.25), 1.0, 1.0, rng.uniform(0.7, 1.4)])
    g[2] += math.radians(rng.uniform(-6.0, 6.0))
    g[3] += rng.uniform(-0.1, 0.1)
    return t, g


def _target(case, seed, lib):
    """The noisy image a retrieval is given: the true ring through the library, plus noise."""
    x, y = _pixels(case["N"], case["S"])
    truth = torch.from_numpy(_truth_and_guess(case, seed)[0])
    z = _ring(truth, x, y, case["r_last"]).view(1, -1)
    img = torch.zeros((1, case["n"] ** 2), dtype=F64, device=DEV)
    for j, a in _columns(lib, case, case["N"], case["S"]):
        img += z[:, j] @ a
    noise = _rng(seed, 5).standard_normal(case["n"] ** 2) * SIGMA
    return (img[0] + torch.from_numpy(noise).to(DEV)).float().contiguous()


def _plan(case, lib, N, S):
    return Plan(lib, _radii(case), case["s"], N=N, S=S, storage=case["storage"], interp=case["interp"])


def prepare(case, seed):
    lib = _library(case, seed)
    st = {"case": case, "lib": lib}
    op = case["op"]
    if op == "build":
        st["radii"] = _radii(case)
        return st
    if op == "multi":
        counts = _multi_counts(case, seed)
        plans = [_plan(case, lib, N, S) for N, S in _buckets(case)]
        mf = MultiForward(plans, [16] * len(plans))
        for i, (N, S) in enumerate(_buckets(case)):
            if counts[i]:
                mf.x[i][:counts[i]] = _scenes(N, S, int(counts[i]), "ring", case["r_last"], seed + 100 * i)
        mf.count.copy_(torch.from_numpy(counts))
        return dict(st, mf=mf)
    plan = st["plan"] = _plan(case, lib, case["N"], case["S"])
    if op in ("forward", "sparse"):
        st["x"] = _scenes(case["N"], case["S"], case["B"], case["scene"], case["r_last"], seed)
    elif op == "adjoint":
        g = _rng(seed, 6).standard_normal((case["B"], case["n"] ** 2), dtype=np.float32) / SIGMA
        st["g"] = torch.from_numpy(g.astype(np.float32)).to(DEV)
    else:
        st["theta"] = _truth_and_guess(case, seed)[1]
        st["problem"] = RingProblem(plan, case["N"], case["S"], case["r_last"], _target(case, seed, lib), SIGMA)
    return st


# ---------------------------------------------------------------- one pass


def run(st):
    case = st["case"]
    op = case["op"]
    if op == "forward":
        return st["plan"].forward(st["x"])
    if op == "sparse":
        return st["plan"].forward(st["x"], skip_zeros=True)
    if op == "adjoint":
        return st["plan"].adjoint(st["g"])
    if op == "multi":
        st["mf"].enqueue()
        return list(st["mf"].y)
    if op == "gradient":  # the optimiser's parameters, and so their gradient, are float32
        p = st["problem"]
        loss, grad = p.loss_and_grad(st["theta"])
        return {"loss": loss, "grad": grad.astype(np.float32), "image": p.y, "scene_grad": p.gz}
    plan = Plan(st["lib"], st["radii"], case["s"], N=case["N"], S=case["S"], storage=case["storage"],
                interp=case["interp"])
    if case["storage"] == "fp32":
        return plan.A_fp32().t()
    hi, lo, scale = plan.A_split()
    return [None if t is None else t[:plan.M, :plan.K] for t in (hi, lo)] + [scale[:plan.K]]


# ---------------------------------------------------------------- what a pass cannot do without


def _inside(case, N, S):
    """Scene pixels inside the last library radius (the others' PSFs are zero)."""
    a = (np.arange(N) - 0.5 * (N - 1)) * S
    return int((np.hypot(a.reshape(1, -1), a.reshape(-1, 1)) <= _radii(case)[-1]).sum())


def work(case):
    M, op, B = case["n"] ** 2, case["op"], case["B"]
    if op == "multi":
        nbytes, flops = 0.0, 0.0
        b = B / len(_buckets(case))
        for N, S in _buckets(case):
            k = _inside(case, N, S)
            nbytes += M * k * BYTES[case["storage"]] + 4 * b * (M + N * N)
            flops += 2.0 * M * k * b
        return {"bytes": nbytes, "flops": flops}
    N, K, lib = case["N"], case["N"] ** 2, 4.0 * len(_radii(case)) * M
    inside = _inside(case, N, case["S"])
    if op == "build":  # every element of A once; 8 taps an element of a quarter of the columns
        return {"bytes": lib + M * K * BYTES[case["storage"]], "flops": 16.0 * M * inside / (4 if N % 2 == 0 else 1)}
    if case["storage"] == "fused":
        return {"bytes": lib + 4.0 * B * (M + K), "flops": 2.0 * M * inside * B}
    stored = M * inside * BYTES[case["storage"]] / (4 if case["storage"] in SYMMETRIC else 1)
    if op == "sparse":  # the columns of the pixels that hold flux: a narrow ring's share, or ten a scene
        frac = 0.17 * K if case["scene"] == "narrow" else min(10.0 * B, K)
        return {"bytes": 4.0 * M * min(frac, inside) + 4.0 * B * (M + K), "flops": 2.0 * M * min(frac, inside) * B}
    if op == "gradient":
        return {"bytes": stored + 4.0 * (4 * M + 8 * K), "flops": 4.0 * M * inside}
    return {"bytes": stored + 4.0 * B * (M + K), "flops": 2.0 * M * inside * B}


# ---------------------------------------------------------------- the same in 64 bits


def _columns(lib, case, N, S, most=1 << 27):
    """(column indices, [columns, M] float64) of A for the N x N scene, in blocks of one radial
    bracket; columns beyond the last radius (zero) are left out."""
    n, radii = case["n"], _radii(case)
    L = lib.double()
    x, y = (t.expand(N, N).reshape(-1) for t in _pixels(N, S))
    r = torch.sqrt(x * x + y * y)
    rad = torch.from_numpy(radii).to(DEV)
    k = (torch.searchsorted(rad, r, right=True) - 1).clamp(0, len(radii) - 2)
    w = ((r - rad[k]) / (rad[k + 1] - rad[k])).clamp_min(0.0)
    if case["interp"] == "nearest":
        w = (w > 0.5).to(F64)
    cos, sin = torch.where(r > 0, x / r, torch.ones_like(r)), torch.where(r > 0, y / r, torch.zeros_like(r))
    c = (torch.arange(n, dtype=F64, device=DEV) - 0.5 * (n - 1))
    Q, P = c.view(1, 1, -1), c.view(1, -1, 1)
    inside = r <= rad[-1]
    step = max(1, most // (n * n))
    for b in range(len(radii) - 1):
        idx = torch.nonzero(inside & (k == b)).view(-1)
        for j in idx.split(step):
            cj, sj = cos[j].view(-1, 1, 1), sin[j].view(-1, 1, 1)
            grid = torch.stack((cj * Q + sj * P, cj * P - sj * Q), -1).view(1, -1, n, 2) / (0.5 * (n - 1))
            v = torch.nn.functional.grid_sample(L[b:b + 2].unsqueeze(0), grid, mode="bilinear",
                                                padding_mode="zeros", align_corners=True)
            v = v.view(2, len(j), n * n)
            wj = w[j].view(-1, 1)
            yield j, torch.addcmul((1 - wj) * v[0], wj, v[1])


def exact(case, seed):
    op = case["op"]
    if case["storage"] == "fused" and case["n"] > 320 and case["N"] > 320:
        most = 1 << 28
    else:
        most = 1 << 27
    lib = _library(case, seed)
    if op == "multi":
        out, counts = [], _multi_counts(case, seed)
        for i, (N, S) in enumerate(_buckets(case)):
            y = torch.zeros((16, case["n"] ** 2), dtype=F64, device=DEV)
            if counts[i]:
                z = _scenes(N, S, int(counts[i]), "ring", case["r_last"], seed + 100 * i).double()
                for j, a in _columns(lib, case, N, S):
                    y[:counts[i]] += z[:, j] @ a
            out.append(y)
        return out
    N, S, M, B = case["N"], case["S"], case["n"] ** 2, case["B"]
    if op in ("forward", "sparse"):
        z = _scenes(N, S, B, case["scene"], case["r_last"], seed).double()
        y = torch.zeros((B, M), dtype=F64, device=DEV)
        for j, a in _columns(lib, case, N, S, most):
            y.addmm_(z[:, j], a)
        return y
    if op == "adjoint":
        g = _rng(seed, 6).standard_normal((B, M), dtype=np.float32) / SIGMA
        g = torch.from_numpy(g.astype(np.float32)).to(DEV).double()
        gx = torch.zeros((B, N * N), dtype=F64, device=DEV)
        for j, a in _columns(lib, case, N, S):
            gx[:, j] = g @ a.t()
        return gx
    if op == "gradient":
        x, y = _pixels(N, S)
        theta = torch.from_numpy(_truth_and_guess(case, seed)[1]).requires_grad_(True)
        z = _ring(theta, x, y, case["r_last"]).view(1, -1)
        img = torch.zeros((1, M), dtype=F64, device=DEV)
        for j, a in _columns(lib, case, N, S):
            img += z.detach()[:, j] @ a
        res = (img - _target(case, seed, lib).double()) / SIGMA**2
        gz = torch.zeros((1, N * N), dtype=F64, device=DEV)
        for j, a in _columns(lib, case, N, S):
            gz[:, j] = res @ a.t()
        (z * gz).sum().backward()
        loss = 0.5 * float((res * res).sum()) * SIGMA**2
        return {"loss": torch.tensor(loss, dtype=F64), "grad": theta.grad, "image": img[0], "scene_grad": gz[0]}
    A = torch.zeros((N * N, M), dtype=F64, device=DEV)
    for j, a in _columns(lib, case, N, S):
        A[j] = a
    if case["storage"] == "fp32":
        return A
    # split storage: hi holds A over a power of two per column, to 8 bits; lo what hi leaves
    top = lib.double().abs().amax((1, 2))
    radii = torch.from_numpy(_radii(case)).to(DEV)
    x, y = (t.expand(N, N).reshape(-1) for t in _pixels(N, S))
    r = torch.sqrt(x * x + y * y)
    k = (torch.searchsorted(radii, r, right=True) - 1).clamp(0, len(radii) - 2)
    sigma = torch.exp2(torch.ceil(torch.log2(torch.maximum(top[k], top[k + 1]))))
    sigma = torch.where(r <= radii[-1], sigma, torch.ones_like(sigma))
    A /= sigma.view(-1, 1)
    return [A.t(), None, sigma]
