"""What is timed of this framework, as a user's program calls it: translations of a tree's levels
(uniform, periodic, adaptive, batched, from host memory), a gradient through them, the whole FMM
potential, the gradient of a far-field objective, and the fast Gauss transform by Taylor series and by
Hermite evaluation.

``listed()`` names the cases, ``draw(rng)`` makes one more of the same ranges, ``prepare`` makes a
case's inputs and the handles a program keeps, ``run`` is one pass through the public entry points, and
``exact`` is the same result in 64 bits, in plain torch.  Sizes are those of the repository's
configurations (``workloads.CONFIGS``) and of its tests, and sizes between them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1009_3457_gb300 import farfield, fmmgb, pipeline
from paper_1009_3457_gb300.autograd import m2l_levels

PRECS = {"fp32": fmmgb.FMM_FP32, "bf16x3": fmmgb.FMM_TC_BF16X3, "tf32x3": fmmgb.FMM_TC_TF32X3}
NCUT = 10  # FGT neighbourhood half-width in boxes
DEV = "cuda"
C64, F64 = torch.complex128, torch.float64


# ---------------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest call a program makes: the small tree, one launch, where latency counts
        dict(name="m2l_level4_p8", kind="m2l", level=4, p=8, prec="fp32", periodic=False),
        # the M2L stage of a 2^22-point uniform tree, the benchmark's headline workload
        dict(name="m2l_level8_p16", kind="m2l", level=8, p=16, prec="fp32", periodic=False),
        # the same tree at the order of the precision study, on the tensor cores
        dict(name="m2l_level8_p24_bf16x3", kind="m2l", level=8, p=24, prec="bf16x3", periodic=False),
        # M2L inside a PyTorch model: forward and backward over the V-lists of a clustered tree
        dict(name="m2l_autograd_adaptive", kind="m2l_autograd", n=1 << 20, cap=64, level=9, p=16),
        # many trees of unlike depth and order translated together, the plan kept (a solver's batch)
        dict(name="m2l_batched_40", kind="batched", nprob=40, lmin=4, lmax=9),
        # problems that live in host memory, served one after another through the overlapped pipeline
        dict(name="host_stream_level8_p16", kind="host", level=8, p=16, prec="fp32", steps=4),
        # the whole potential of 2^22 points at themselves, bins and buffers kept (an iterative solver)
        dict(name="potential_4m", kind="potential", n=1 << 22, m=0, level=8, p=16, prec="fp32", rebuild=False),
        # the whole potential of a small set at other points, new positions each call (a time step)
        dict(name="potential_50k_rebuilt", kind="potential", n=50021, m=30011, level=5, p=8, prec="fp32",
             rebuild=True),
        # gradient of a far-field objective with respect to a million clustered positions
        dict(name="far_field_gradient_1m", kind="gradient", n=1 << 20, m=4096, cap=64, level=9, p=16),
        # the fast Gauss transform by Taylor series, a million clustered sources, new points each call
        dict(name="fgt_taylor_1m", kind="fgt_taylor", n=1 << 20, m=1 << 20, sigma=0.05, p=16, prec="fp32",
             uniform_targets=True),
        # the transform by Hermite evaluation at a million clustered targets, in FP32
        dict(name="fgt_hermite_1m", kind="fgt_hermite", n=1 << 20, m=1 << 20, sigma=0.05, p=16, prec="fp32",
             uniform_targets=False),
        # the same on the tensor cores, wider Gaussian, ragged sizes
        dict(name="fgt_hermite_300k_bf16x3", kind="fgt_hermite", n=200003, m=300007, sigma=0.1, p=16, prec="bf16x3",
             uniform_targets=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["m2l", "m2l", "m2l_autograd", "batched", "host", "potential", "potential", "gradient",
                       "fgt_taylor", "fgt_hermite", "fgt_hermite"])
    if kind == "m2l":
        prec = rng.choice(["fp32", "fp32", "bf16x3", "tf32x3"])
        p = {"fp32": rng.choice([6, 8, 12, 16, 24]), "bf16x3": rng.choice([16, 24]), "tf32x3": 16}[prec]
        return dict(kind=kind, level=rng.randint(3, 9), p=p, prec=prec, periodic=rng.random() < 0.3)
    if kind == "m2l_autograd":
        return dict(kind=kind, n=_log_int(rng, 10_000, 1 << 20), cap=rng.choice([16, 32, 64, 100]),
                    level=rng.randint(6, 9), p=rng.choice([8, 12, 16]))
    if kind == "batched":
        lo = rng.randint(3, 5)
        return dict(kind=kind, nprob=_log_int(rng, 3, 40), lmin=lo, lmax=rng.randint(lo + 1, 9))
    if kind == "host":
        return dict(kind=kind, level=rng.randint(5, 8), p=rng.choice([8, 12, 16]), prec="fp32", steps=rng.randint(2, 4))
    if kind == "potential":
        n = _log_int(rng, 5_000, 1 << 21)
        level = max(3, min(8, int(round(math.log(n / rng.uniform(16, 64), 4)))))
        return dict(kind=kind, n=n, m=rng.choice([0, _log_int(rng, 5_000, 1 << 21)]), level=level,
                    p=rng.choice([8, 12, 16, 24]), prec="fp32", rebuild=rng.random() < 0.5)
    if kind == "gradient":
        return dict(kind=kind, n=_log_int(rng, 20_000, 1 << 20), m=_log_int(rng, 500, 20_000),
                    cap=rng.choice([32, 64, 100]), level=rng.randint(6, 9), p=rng.choice([8, 12, 16]))
    sigma = round(math.exp(rng.uniform(math.log(0.03), math.log(0.25))), 4)
    n, m = _log_int(rng, 20_000, 1 << 20), _log_int(rng, 20_000, 1 << 20)
    if kind == "fgt_taylor":
        return dict(kind=kind, n=n, m=m, sigma=sigma, p=rng.choice([8, 12, 16]), prec="fp32",
                    uniform_targets=rng.random() < 0.5)
    prec = rng.choice(["fp32", "fp32", "bf16x3"])
    return dict(kind=kind, n=n, m=m, sigma=sigma, p=16 if prec != "fp32" else rng.choice([8, 12, 16]), prec=prec,
                uniform_targets=rng.random() < 0.5)


# ---------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------
def _gen(seed, salt=0):
    return torch.Generator(device=DEV).manual_seed(1_000_003 * int(seed) + salt)


def _uniform(n, g):
    return torch.rand((n, 2), dtype=F64, device=DEV, generator=g)


def _mixture(n, g, ncomp=16):
    """n points of an equal-weight Gaussian mixture (16 components, sigma 0.01..0.05) inside [0, 1)^2."""
    means = 0.1 + 0.8 * torch.rand((ncomp, 2), dtype=F64, device=DEV, generator=g)
    sig = 0.01 + 0.04 * torch.rand(ncomp, dtype=F64, device=DEV, generator=g)
    got = []
    left = n
    while left > 0:
        k = 2 * left + 64
        comp = torch.randint(0, ncomp, (k,), device=DEV, generator=g)
        pts = means[comp] + sig[comp, None] * torch.randn((k, 2), dtype=F64, device=DEV, generator=g)
        pts = pts[((pts >= 0) & (pts < 1)).all(1)][:left]
        got.append(pts)
        left -= pts.shape[0]
    return torch.cat(got).contiguous()


def _strengths(n, g):
    return 2 * torch.rand(n, dtype=F64, device=DEV, generator=g) - 1


def _moments(p):
    """E|d|^2k for d uniform in a unit box about its centre, k < p."""
    t = (np.arange(400) + 0.5) / 400 - 0.5
    r2 = t[:, None] ** 2 + t[None, :] ** 2
    return np.array([np.mean(r2**k) for k in range(p)])


def _expansions(level, leaf_level, p, g):
    """Random radius-scaled MEs with the magnitudes that 64 points per leaf of strength U[-1, 1] give."""
    sd = np.sqrt(64.0 * 4.0 ** (leaf_level - level) / 3.0 * _moments(p) / 2)
    x = torch.randn((4**level, p, 2), dtype=torch.float32, device=DEV, generator=g)
    x *= torch.from_numpy(sd).to(DEV, torch.float32)[None, :, None]
    return torch.view_as_complex(x)


def _batch_shapes(case, seed):
    rng = np.random.default_rng(7919 + int(seed))
    return [(int(rng.integers(case["lmin"], case["lmax"] + 1)), int(rng.choice([6, 8, 12, 16])))
            for _ in range(case["nprob"])]


def _grid_log2(sigma):
    return int(math.ceil(math.log2(math.sqrt(2.0) / sigma)))


def _inputs(case, seed):
    """The arrays of a case, from the seed alone."""
    kind, g = case["kind"], _gen(seed)
    if kind == "m2l":
        return [_expansions(l, case["level"], case["p"], g) for l in range(2, case["level"] + 1)]
    if kind == "m2l_autograd":
        pts = _mixture(case["n"], g)
        lv = range(2, case["level"] + 1)
        Ms = [_expansions(l, case["level"], case["p"], g) for l in lv]
        return pts, Ms, [_expansions(l, case["level"], case["p"], g) for l in lv]
    if kind == "batched":
        # the shapes of a batch are the program's, the same for every seed of a case
        return [(L, p, [_expansions(l, L, p, g) for l in range(2, L + 1)]) for L, p in _batch_shapes(case, 0)]
    if kind == "host":
        return [torch.cat([_expansions(l, case["level"], case["p"], g).reshape(-1) for l in range(2, case["level"] + 1)])
                for _ in range(case["steps"])]
    if kind == "potential":
        xy, c = _uniform(case["n"], g), _strengths(case["n"], g)
        return xy, c, _uniform(case["m"], g) if case["m"] else xy
    if kind == "gradient":
        xy, c = _mixture(case["n"], g), _strengths(case["n"], g)
        return xy, c, _uniform(case["m"], g), _strengths(case["m"], g)
    x, q = _mixture(case["n"], g), _strengths(case["n"], g)
    return x, q, _uniform(case["m"], g) if case["uniform_targets"] else _mixture(case["m"], g)


def prepare(case, seed):
    kind, p, s = case["kind"], case.get("p"), {"case": dict(case)}
    data = _inputs(case, seed)
    prec = PRECS[case.get("prec", "fp32")]
    if kind == "m2l":
        s.update(tree=fmmgb.fmm_build_lists(None, case["level"], periodic=case["periodic"]), Ms=data,
                 Ls=[torch.empty_like(m) for m in data])
        fmmgb.fmm_prepare(p, prec)
    elif kind == "m2l_autograd":
        pts, Ms, Ws = data
        s.update(tree=fmmgb.fmm_build_lists(pts.cpu().numpy(), case["level"], leaf_cap=case["cap"]),
                 Ms=[m.requires_grad_(True) for m in Ms], Ws=Ws)
    elif kind == "batched":
        trees = [fmmgb.fmm_build_lists(None, L) for L, _, _ in data]
        Ms = [m for _, _, m in data]
        flat = torch.empty(sum(x.numel() for m in Ms for x in m), dtype=torch.complex64, device=DEV)
        Ls, at = [], 0
        for m in Ms:
            Ls.append([])
            for x in m:
                Ls[-1].append(flat[at:at + x.numel()].view(x.shape))
                at += x.numel()
        s.update(plan=fmmgb.fmm_batch_create(trees, [q for _, q, _ in data], Ms, Ls), flat=flat)
    elif kind == "host":
        tree = fmmgb.fmm_build_lists(None, case["level"])
        s.update(tree=tree, hs=pipeline.HostStreamM2L(tree, 2, case["level"], p, prec=prec),
                 Mh=[d.cpu().pin_memory() for d in data],
                 Lh=[torch.empty(d.shape, dtype=d.dtype).pin_memory() for d in data])
    elif kind == "potential":
        xy, c, z = data
        tree = fmmgb.fmm_build_lists(None, case["level"])
        s.update(tree=tree, xy=xy, c=c, z=z)
        if not case["rebuild"]:
            s["potential"] = farfield.FmmPotential(tree, p, xy, c, z, prec)
    elif kind == "gradient":
        xy, c, z, w = data
        tree = fmmgb.fmm_build_lists(xy.cpu().numpy(), case["level"], leaf_cap=case["cap"])
        s.update(tree=tree, xy=xy.requires_grad_(True), c=c, z=torch.view_as_complex(z), w=w,
                 zleaf=farfield.leaf_boxes(tree, z))
    else:
        x, q, y = data
        g = _grid_log2(case["sigma"])
        nb, i32 = 4**g, dict(dtype=torch.int32, device=DEV)
        s.update(g=g, x=x, q=q, y=y, A=torch.empty((nb, p, p), device=DEV), G=torch.empty(y.shape[0], device=DEV),
                 sperm=torch.empty(x.shape[0], **i32), sstart=torch.empty(nb + 1, **i32),
                 tperm=torch.empty(y.shape[0], **i32), tstart=torch.empty(nb + 1, **i32), work=torch.empty(nb, **i32))
        if kind == "fgt_taylor":
            s.update(C=torch.empty_like(s["A"]), Y=torch.empty_like(s["A"]))
    return s


# ---------------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------------
def run(s):
    case = s["case"]
    kind, p, prec = case["kind"], case.get("p"), PRECS[case.get("prec", "fp32")]
    if kind == "m2l":
        fmmgb.fmm_m2l_levels(s["tree"], 2, p, s["Ms"], s["Ls"], prec=prec)
        return s["Ls"]
    if kind == "m2l_autograd":
        Ls = m2l_levels(s["tree"], p, s["Ms"])
        return {"L": [x.detach() for x in Ls], "G": list(torch.autograd.grad(Ls, s["Ms"], s["Ws"]))}
    if kind == "batched":
        s["plan"].run()
        return s["flat"]
    if kind == "host":
        s["hs"].run(s["Mh"], s["Lh"])
        s["hs"].sync()
        return s["Lh"]
    if kind == "potential":
        if case["rebuild"]:
            return farfield.FmmPotential(s["tree"], p, s["xy"], s["c"], s["z"], prec)()
        return s["potential"]()
    if kind == "gradient":
        J = farfield.far_field_objective(s["tree"], p, s["xy"], s["c"], None, s["z"], s["zleaf"], s["w"])
        return {"J": J.detach(), "grad": torch.autograd.grad(J, s["xy"])[0]}
    g, sigma = s["g"], case["sigma"]
    fmmgb.fgt_bin_points(g, s["x"], s["sperm"], s["sstart"], s["work"])
    fmmgb.fgt_p2h_binned(g, p, sigma, s["x"], s["q"], s["sperm"], s["A"])
    if kind == "fgt_taylor":
        fmmgb.fgt_h2t(g, NCUT, p, sigma, s["A"], s["C"], work=s["Y"], prec=prec)
        fmmgb.fgt_bin_points(g, s["y"], s["tperm"], s["tstart"], s["work"])
        fmmgb.fgt_t2p_binned(g, p, sigma, s["C"], s["y"], s["tperm"], s["tstart"], s["G"])
    else:
        fmmgb.fgt_bin_points(g, s["y"], s["tperm"], s["tstart"], s["work"])
        fmmgb.fgt_h2p(g, NCUT, p, sigma, s["A"], s["y"], s["tperm"], s["tstart"], s["G"], prec=prec)
    return s["G"]


# ---------------------------------------------------------------------------------------------------
# what a pass cannot do without: inputs read once, outputs written once; the products of the series as
# the method states them (one p x p complex product per translation, p^2 per target and source box)
# ---------------------------------------------------------------------------------------------------
def _translations(level, periodic=False):
    n = 2**level
    return 27 * n * n if periodic else (6 * n - 8) ** 2 - (3 * n - 2) ** 2


def _m2l_work(level, p, periodic=False):
    lv = range(2, level + 1)
    return 2 * 8 * p * sum(4**l for l in lv), 8 * p * p * sum(_translations(l, periodic) for l in lv)


def work(case):
    kind, p = case["kind"], case.get("p")
    if kind == "m2l":
        b, f = _m2l_work(case["level"], p, case["periodic"])
    elif kind == "m2l_autograd":
        # about one box of the deepest levels for every cap / 2 points, 20 list entries each
        boxes = min(2 * case["n"] / case["cap"], sum(4**l for l in range(2, case["level"] + 1)))
        b, f = 2 * 2 * 8 * p * boxes, 2 * 8 * p * p * 20 * boxes
    elif kind == "batched":
        each = [_m2l_work(L, q) for L, q in _batch_shapes(case, 0)]
        b, f = sum(x for x, _ in each), sum(x for _, x in each)
    elif kind == "host":
        b, f = (case["steps"] * v for v in _m2l_work(case["level"], p))
    elif kind == "potential":
        n, m = case["n"], case["m"] or case["n"]
        b = n * 24 + m * (16 + 8)
        f = _m2l_work(case["level"], p)[1] + 8.0 * m * 9 * n / 4 ** case["level"]
    elif kind == "gradient":
        boxes = min(2 * case["n"] / case["cap"], 4 ** case["level"])
        b, f = case["n"] * (24 + 16) + case["m"] * 40, 2 * (8 * p * p * 20 * boxes + case["n"] * 8 * p)
    else:
        n, m, nb = case["n"], case["m"], 4 ** _grid_log2(case["sigma"])
        b = n * 24 + m * (16 + 4)
        f = 2.0 * p * p * n + 2.0 * p * p * m
        taps = (2 * NCUT + 1)
        f += nb * 2 * taps * 2.0 * p**3 if kind == "fgt_taylor" else m * min(taps * taps, nb) * 2.0 * p * p
    return {"bytes": int(b), "flops": int(f)}


def tolerance(case):
    """About four times the error against ``exact`` over the listed and 30 drawn cases.  FP32 sums: 3.4e-7
    (M2L, largest difference 4e-5 of a value near the root mean square), 1.1e-6 (FGT), 3e-7 (gradient; its J is a
    sum of terms of both signs, 1.4e-6).  The potential: positions kept to 2^-24 of a box side, so the closest
    pairs set its 4e-5 to 1.6e-4 (largest 5e-3).  BF16 hi + lo operands: 5.3e-6 (M2L), 4.9e-6 (FGT); TF32 hi +
    lo: 1.6e-6."""
    kind, prec = case["kind"], case.get("prec", "fp32")
    if kind == "potential":
        return {"rel": 6e-4, "max": 2e-2}
    if kind == "gradient":
        return {"rel": 1e-5, "max": 4e-5}
    if kind.startswith("fgt"):
        return {"rel": 4.5e-6, "max": 2e-5} if prec == "fp32" else {"rel": 2e-5, "max": 1e-4}
    return {"fp32": {"rel": 1.5e-6, "max": 1.5e-4}, "bf16x3": {"rel": 2e-5, "max": 3e-4},
            "tf32x3": {"rel": 6e-6, "max": 7e-5}}[prec]


# ---------------------------------------------------------------------------------------------------
# the same results in 64 bits, in plain torch
# ---------------------------------------------------------------------------------------------------
def _m2l_matrix(dx, dy, p):
    """T[n][k] = (-1)^n C(n+k, k) D^-(n+k+1) for D = target centre - source centre = dx + i dy (box sides)."""
    D = complex(dx, dy)
    T = [[(-1) ** n * math.comb(n + k, k) * D ** -(n + k + 1) for k in range(p)] for n in range(p)]
    return torch.tensor(T, dtype=C64, device=DEV)


def _shifted(M, dx, dy, periodic):
    """M[side, side, p] (y, x) read at (y + dy, x + dx), zero outside or wrapped."""
    if periodic:
        return torch.roll(M, (-dy, -dx), (0, 1))
    side = M.shape[0]
    pad = torch.nn.functional.pad(torch.view_as_real(M).permute(2, 3, 0, 1), (3, 3, 3, 3))
    pad = torch.view_as_complex(pad.permute(2, 3, 0, 1).contiguous())
    return pad[3 + dy:3 + dy + side, 3 + dx:3 + dx + side]


def _m2l64(M, level, p, periodic=False, adjoint=False, exists=None):
    """The list sum of one level: M [4^level, p] complex128 -> [4^level, p]."""
    side = 2**level
    M = M.view(side, side, p)
    if exists is not None:
        M = M * exists.view(side, side, 1)
    out = torch.zeros_like(M)
    for dy in range(-3, 4):
        for dx in range(-3, 4):
            if max(abs(dx), abs(dy)) < 2:
                continue
            # the offset is in the list of the child classes for which it stays inside the parents' neighbours
            ok = torch.zeros((2, 2), dtype=torch.bool)
            for cy in (0, 1):
                for cx in (0, 1):
                    ok[cy, cx] = -1 <= (cx + dx) // 2 <= 1 and -1 <= (cy + dy) // 2 <= 1
            mask = ok.repeat(side // 2, side // 2).to(DEV)
            T = _m2l_matrix(dx, dy, p).conj() if adjoint else _m2l_matrix(-dx, -dy, p).T
            out = out + (_shifted(M, dx, dy, periodic) @ T) * mask[:, :, None]
    if exists is not None:
        out = out * exists.view(side, side, 1)
    return out.view(4**level, p)


def _exists(pts, level, cap):
    """Box existence per level of the adaptive tree: children with points of boxes with more than cap points."""
    out, parent_split = [torch.ones(1, dtype=torch.bool, device=DEV)], torch.tensor([pts.shape[0] > cap], device=DEV)
    for l in range(1, level + 1):
        side = 2**l
        b = _cells(pts, l)
        cnt = torch.bincount(b[:, 1] * side + b[:, 0], minlength=side * side)
        up = parent_split.view(side // 2, side // 2).repeat_interleave(2, 0).repeat_interleave(2, 1).reshape(-1)
        out.append(up & (cnt > 0))
        parent_split = out[-1] & (cnt > cap)
    return out


def _cells(pts, level):
    return torch.floor(pts.detach() * 2**level).clamp(0, 2**level - 1).to(torch.int64)


def _offsets(pts, cells, level):
    """(y - centre) / side of each point's box, complex."""
    d = pts * 2**level - (cells + 0.5)
    return torch.complex(d[:, 0], d[:, 1])


def _powers(d, p):
    out = [torch.ones_like(d)]
    for _ in range(p - 1):
        out.append(out[-1] * d)
    return torch.stack(out, 1)


def _p2m64(pts, c, level, p):
    cells = _cells(pts, level)
    box = cells[:, 1] * 2**level + cells[:, 0]
    M = torch.zeros((4**level, p), dtype=C64, device=DEV)
    return M.index_add(0, box, _powers(_offsets(pts, cells, level), p) * c[:, None])


def _m2m64(M, level, p):
    """Parent MEs (level - 1) from child MEs (level), radius-scaled."""
    half = 2 ** (level - 1)
    M = M.view(half, 2, half, 2, p)
    out = 0
    for cy in (0, 1):
        for cx in (0, 1):
            z = complex(cx - 0.5, cy - 0.5) / 2
            T = torch.tensor([[math.comb(j, k) * z ** (j - k) * 0.5**k if k <= j else 0 for k in range(p)]
                              for j in range(p)], dtype=C64, device=DEV)
            out = out + M[:, cy, :, cx] @ T.T
    return out.reshape(half * half, p)


def _l2l64(L, level, p):
    """Child LEs (level) from parent LEs (level - 1), radius-scaled."""
    half = 2 ** (level - 1)
    L = L.view(half, half, p)
    rows = []
    for cy in (0, 1):
        cols = []
        for cx in (0, 1):
            u = complex(cx - 0.5, cy - 0.5) / 2
            T = torch.tensor([[math.comb(n, j) * u ** (n - j) * 0.5 ** (j + 1) if n >= j else 0 for n in range(p)]
                              for j in range(p)], dtype=C64, device=DEV)
            cols.append(L @ T.T)
        rows.append(torch.stack(cols, 2))
    return torch.stack(rows, 1).reshape(4**level, p)


def _far64(xy, c, level, p, exists=None):
    """LEs of levels 2..level (list), after L2L: the far field of points xy of strength c."""
    Ms = {level: _p2m64(xy, c, level, p)}
    for l in range(level, 2, -1):
        Ms[l - 1] = _m2m64(Ms[l], l, p)
    Ls = {}
    for l in range(2, level + 1):
        Ls[l] = _m2l64(Ms[l], l, p, exists=None if exists is None else exists[l])
        if l > 2:
            Ls[l] = Ls[l] + _l2l64(Ls[l - 1], l, p)
    return Ls


def _l2p64(L, z, level, p):
    cells = _cells(z, level)
    box = cells[:, 1] * 2**level + cells[:, 0]
    return (L[box] * _powers(_offsets(z, cells, level), p)).sum(1) * 2**level


def _padded(pts, level):
    """Point indices by box, [4^level, most], -1 where a box has fewer."""
    cells = _cells(pts, level)
    box = cells[:, 1] * 2**level + cells[:, 0]
    order = torch.argsort(box, stable=True)
    cnt = torch.bincount(box, minlength=4**level)
    start = torch.cumsum(cnt, 0) - cnt
    tab = torch.full((4**level, int(cnt.max())), -1, dtype=torch.int64, device=DEV)
    b = box[order]
    tab[b, torch.arange(b.shape[0], device=DEV) - start[b]] = order
    return tab


def _near64(xy, c, z, level):
    side = 2**level
    st, tt = _padded(xy, level), _padded(z, level)
    phi = torch.zeros(z.shape[0], dtype=C64, device=DEV)
    step = max(1, 100_000_000 // (st.shape[1] * tt.shape[1]))
    for dy in (-1, 0, 1):
        for dx in (-1, 0, 1):
            for b0 in range(0, side * side, step):
                b = torch.arange(b0, min(b0 + step, side * side), device=DEV)
                sx, sy = b % side + dx, b // side + dy
                b = b[(sx >= 0) & (sx < side) & (sy >= 0) & (sy < side)]
                if not b.numel():
                    continue
                si, ti = st[b + dy * side + dx], tt[b]
                cs = torch.where(si >= 0, c[si.clamp(min=0)], 0.0)
                ps, pt = xy[si.clamp(min=0)], z[ti.clamp(min=0)]
                ex, ey = pt[:, :, None, 0] - ps[:, None, :, 0], pt[:, :, None, 1] - ps[:, None, :, 1]
                r2 = ex * ex + ey * ey
                w = torch.where(r2 > 0, cs[:, None, :] / r2, 0.0)
                v = torch.complex((w * ex).sum(2), -(w * ey).sum(2))
                ok = ti >= 0
                phi.index_add_(0, ti[ok], v[ok])
    return phi


def _hermite64(t, n):
    """h_0..h_{n-1}(t), h_k = exp(-t^2) H_k(t), on a new last axis."""
    h = [torch.exp(-t * t)]
    if n > 1:
        h.append(2 * t * h[0])
    for k in range(1, n - 1):
        h.append(2 * t * h[k] - 2 * k * h[k - 1])
    return torch.stack(h, -1)


def _taylor_powers(t, p, factorial):
    out = [torch.ones_like(t)]
    for a in range(1, p):
        out.append(out[-1] * t / (a if factorial else 1))
    return torch.stack(out, -1)


def _p2h64(x, q, g, p, sigma):
    cells = _cells(x, g)
    box = cells[:, 1] * 2**g + cells[:, 0]
    t = (x - (cells + 0.5) / 2**g) / (math.sqrt(2) * sigma)
    A = torch.zeros((4**g, p * p), dtype=F64, device=DEV)
    for i in range(0, x.shape[0], 1 << 18):
        s = slice(i, i + (1 << 18))
        w1, w2 = _taylor_powers(t[s, 0], p, True), _taylor_powers(t[s, 1], p, True)
        A.index_add_(0, box[s], (q[s, None, None] * w1[:, :, None] * w2[:, None, :]).reshape(-1, p * p))
    return A.view(4**g, p, p)


def _fgt_taylor64(x, q, y, g, p, sigma):
    side = 2**g
    A = _p2h64(x, q, g, p, sigma).view(side, side, p, p)  # [sy, sx, a1, a2]
    i = torch.arange(side, device=DEV)
    u = (i[None, :] - i[:, None]).to(F64) / side / (math.sqrt(2) * sigma)  # [source, target]
    h = _hermite64(u, 2 * p) * ((i[None, :] - i[:, None]).abs() <= NCUT)[..., None]
    a = torch.arange(p, device=DEV)
    f = torch.tensor([(-1) ** b / math.factorial(b) for b in range(p)], dtype=F64, device=DEV)
    H = h[:, :, a[:, None] + a[None, :]] * f  # [source, target, alpha, beta]
    Hm = H.permute(0, 2, 1, 3).reshape(side * p, side * p)  # (source, alpha), (target, beta)
    X = A.permute(0, 3, 1, 2).reshape(side * p, side * p) @ Hm  # (sy, a2), (tx, b1)
    C = (X.T @ Hm).view(side, p, side, p)  # (tx, b1), (ty, b2)
    C = C.permute(2, 0, 1, 3).reshape(side * side, p, p)
    cells = _cells(y, g)
    box = cells[:, 1] * side + cells[:, 0]
    t = (y - (cells + 0.5) / side) / (math.sqrt(2) * sigma)
    out = []
    for j in range(0, y.shape[0], 1 << 18):
        s = slice(j, j + (1 << 18))
        w1, w2 = _taylor_powers(t[s, 0], p, False), _taylor_powers(t[s, 1], p, False)
        out.append(torch.einsum("nab,na,nb->n", C[box[s]], w1, w2))
    return torch.cat(out)


def _fgt_hermite64(x, q, y, g, p, sigma):
    side = 2**g
    A = _p2h64(x, q, g, p, sigma).view(side, side, p, p)  # [sy, sx, a1, a2]
    scale = 1 / (math.sqrt(2) * sigma)
    centre = (torch.arange(side, device=DEV, dtype=F64) + 0.5) / side
    tab = _padded(y, g)
    cnt = (tab >= 0).sum(1).tolist()
    G = torch.zeros(y.shape[0], dtype=F64, device=DEV)
    for b in range(side * side):
        if not cnt[b]:
            continue
        tx, ty = b % side, b // side
        x0, x1, y0, y1 = max(tx - NCUT, 0), min(tx + NCUT, side - 1), max(ty - NCUT, 0), min(ty + NCUT, side - 1)
        j = tab[b, :cnt[b]]
        hx = _hermite64((y[j, 0, None] - centre[None, x0:x1 + 1]) * scale, p).reshape(cnt[b], -1)  # (sx, a1)
        hy = _hermite64((y[j, 1, None] - centre[None, y0:y1 + 1]) * scale, p).reshape(cnt[b], -1)  # (sy, a2)
        blk = A[y0:y1 + 1, x0:x1 + 1].permute(0, 3, 1, 2).reshape(hy.shape[1], hx.shape[1])
        G[j] = ((hy @ blk) * hx).sum(1)
    return G


def exact(case, seed):
    kind, p = case["kind"], case.get("p")
    data = _inputs(case, seed)
    if kind == "m2l":
        return [_m2l64(m.to(C64), l, p, case["periodic"]) for l, m in enumerate(data, 2)]
    if kind == "m2l_autograd":
        pts, Ms, Ws = data
        ex = _exists(pts, case["level"], case["cap"])
        return {"L": [_m2l64(m.to(C64), l, p, exists=ex[l]) for l, m in enumerate(Ms, 2)],
                "G": [_m2l64(w.to(C64), l, p, adjoint=True, exists=ex[l]) for l, w in enumerate(Ws, 2)]}
    if kind == "batched":
        return torch.cat([_m2l64(m.to(C64), l, q).reshape(-1) for _, q, Ms in data for l, m in enumerate(Ms, 2)])
    if kind == "host":
        out = []
        for d in data:
            at, parts = 0, []
            for l in range(2, case["level"] + 1):
                parts.append(_m2l64(d[at:at + 4**l * p].to(C64).view(-1, p), l, p).reshape(-1))
                at += 4**l * p
            out.append(torch.cat(parts))
        return out
    if kind == "potential":
        xy, c, z = data
        L = _far64(xy, c, case["level"], p)[case["level"]]
        return _l2p64(L, z, case["level"], p) + _near64(xy, c, z, case["level"])
    if kind == "gradient":
        xy, c, z, w = data
        xy = xy.requires_grad_(True)
        ex = _exists(xy, case["level"], case["cap"])
        Ls = _far64(xy, c, case["level"], p, exists=ex)
        leaf = torch.zeros(z.shape[0], dtype=torch.int64, device=DEV)
        for l in range(1, case["level"] + 1):
            cells = _cells(z, l)
            leaf[ex[l][cells[:, 1] * 2**l + cells[:, 0]]] = l
        J = 0
        for l in range(2, case["level"] + 1):
            at = leaf == l
            if bool(at.any()):
                J = J + (w[at] * _l2p64(Ls[l], z[at], l, p).real).sum()
        return {"J": J.detach(), "grad": torch.autograd.grad(J, xy)[0]}
    x, q, y = data
    f = _fgt_taylor64 if kind == "fgt_taylor" else _fgt_hermite64
    return f(x, q, y, _grid_log2(case["sigma"]), p, case["sigma"])
