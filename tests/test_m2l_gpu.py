"""GPU parity of the FP32 M2L path (fmm_m2l, fmm_m2l_adjoint, fmm_p2m, fmm_m2m)
against the FP64 oracle, through the C ABI.

Bar (spec tolerance for the FP32 path): relative L2 error of the
radius-scaled local coefficients of a level <= 1e-5, over all boxes and all n;
in addition every box's own relative error must stay below 1e-4 so that a
localised fault cannot hide in the level-wide norm.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

TOL_L2 = 1e-5
TOL_BOX = 1e-4


@pytest.fixture(scope="module")
def fmm():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1009_3457_gb300 import build, fmmgb

    build.build()
    fmmgb.load()
    return fmmgb


def _dev(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.complex64)).cuda()


def _host(t):
    return t.cpu().numpy().astype(np.complex128)


def _check(got, ref, tol_l2=TOL_L2, tol_box=TOL_BOX):
    err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
    assert err <= tol_l2, f"relative L2 {err:.3e} > {tol_l2:.1e}"
    box = np.linalg.norm(got - ref, axis=-1) / np.maximum(np.linalg.norm(ref, axis=-1), 1e-300)
    assert box.max() <= tol_box, f"worst box {box.max():.3e} at {int(box.argmax())}"
    return err


def _oracle_level(orc, level, p, M, periodic=False):
    return orc.scale_le(orc.m2l_uniform(level, p, M, periodic), level)


def test_m2l_small_workload(fmm, orc):
    """4096 points, uniform tree to level 4, p = 8: every level against the oracle."""
    cfg = workloads.CONFIGS["m2l_small"]
    p, L = cfg["p"], cfg["max_level"]
    xy, c = workloads.uniform_particles(cfg["n"], workloads.rng_for("m2l_small"))
    Ms = orc.upward_uniform(L, p, xy, c)
    tree = fmm.fmm_build_lists(None, L)
    for level in workloads.m2l_levels(L):
        Md = _dev(orc.scale_me(Ms[level], level))
        Ld = Md.new_empty(Md.shape)
        fmm.fmm_m2l(tree, level, p, Md, Ld)
        _check(_host(Ld), _oracle_level(orc, level, p, Ms[level]))
    fmm.fmm_sync_status()


@pytest.fixture(scope="module")
def medium_particles():
    return workloads.uniform_particles(6000, np.random.default_rng(123))


@pytest.mark.parametrize("p", [6, 8, 12, 16, 24])
def test_m2l_all_orders_levels_2_to_5(fmm, orc, medium_particles, p):
    """Levels 2, 3 (tile larger than the level: ragged), 4 (one full tile), 5 (2 x 2 tiles)."""
    xy, c = medium_particles
    Ms = orc.upward_uniform(5, p, xy, c)
    tree = fmm.fmm_build_lists(None, 5)
    for level in range(2, 6):
        Md = _dev(orc.scale_me(Ms[level], level))
        Ld = Md.new_empty(Md.shape)
        fmm.fmm_m2l(tree, level, p, Md, Ld)
        _check(_host(Ld), _oracle_level(orc, level, p, Ms[level]))


@pytest.mark.parametrize("level", [2, 3, 6])
def test_m2l_periodic_lists(fmm, orc, medium_particles, level):
    xy, c = medium_particles
    p = 12
    Ms = orc.upward_uniform(6, p, xy, c)
    tree = fmm.fmm_build_lists(None, 6, periodic=True)
    Md = _dev(orc.scale_me(Ms[level], level))
    Ld = Md.new_empty(Md.shape)
    fmm.fmm_m2l(tree, level, p, Md, Ld)
    _check(_host(Ld), _oracle_level(orc, level, p, Ms[level], periodic=True))


def test_m2l_accumulate_and_empty_levels(fmm, orc, medium_particles):
    import torch

    xy, c = medium_particles
    p = 8
    Ms = orc.upward_uniform(4, p, xy, c)
    tree = fmm.fmm_build_lists(None, 4)
    level = 4
    rng = np.random.default_rng(0)
    X = (rng.standard_normal((256, p)) + 1j * rng.standard_normal((256, p))).astype(np.complex64)
    Md = _dev(orc.scale_me(Ms[level], level))
    Ld = _dev(X)
    fmm.fmm_m2l(tree, level, p, Md, Ld, accumulate=True)
    _check(_host(Ld), X.astype(np.complex128) + _oracle_level(orc, level, p, Ms[level]))
    # levels 0 and 1 have empty interaction lists
    for lv in (0, 1):
        n = 4 ** lv
        Mz = _dev(np.ones((n, p)))
        Lz = _dev(np.full((n, p), 3.0))
        fmm.fmm_m2l(tree, lv, p, Mz, Lz, accumulate=True)
        assert np.all(_host(Lz) == 3.0)
        fmm.fmm_m2l(tree, lv, p, Mz, Lz)
        assert np.all(_host(Lz) == 0.0)
    torch.cuda.synchronize()


def test_m2l_is_deterministic(fmm, orc, medium_particles):
    xy, c = medium_particles
    p, level = 16, 5
    Ms = orc.upward_uniform(level, p, xy, c)
    tree = fmm.fmm_build_lists(None, level)
    Md = _dev(orc.scale_me(Ms[level], level))
    L1 = Md.new_empty(Md.shape)
    L2 = Md.new_empty(Md.shape)
    fmm.fmm_m2l(tree, level, p, Md, L1)
    fmm.fmm_m2l(tree, level, p, Md, L2)
    assert bool((L1 == L2).all())


@pytest.mark.parametrize("conj", [False, True])
@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("p,level", [(8, 3), (16, 5), (24, 4)])
def test_m2l_adjoint(fmm, orc, p, level, conj, periodic):
    """Scaled adjoint G~ = R_M A^T R_L W~  (R_M = diag r^k, R_L = diag r^(n+1)) against the
    oracle's explicit transpose; with FMM_CONJ the conjugate transpose."""
    rng = np.random.default_rng(level * 100 + p)
    n = 4 ** level
    W = rng.standard_normal((n, p)) + 1j * rng.standard_normal((n, p))
    tree = fmm.fmm_build_lists(None, level, periodic=periodic)
    Wd = _dev(W)
    Gd = Wd.new_empty(Wd.shape)
    fmm.fmm_m2l_adjoint(tree, level, p, Wd, Gd, conj=conj)
    Win = np.conj(W) if conj else W
    G = orc.unscale_me(orc.m2l_adjoint_uniform(level, p, orc.scale_le(Win, level), periodic), level)
    if conj:
        G = np.conj(G)
    _check(_host(Gd), G)


def test_upward_sweep_on_device(fmm, orc):
    """fmm_p2m + fmm_m2m (FP32 atomics) against the oracle's P2M/M2M, scaled units."""
    import torch

    xy, c = workloads.uniform_particles(50000, np.random.default_rng(99))
    p, L = 16, 6
    Ms = orc.upward_uniform(L, p, xy, c)
    xyd = torch.from_numpy(xy).cuda()
    cd = torch.from_numpy(c).cuda()
    Md = {L: torch.empty((4 ** L, p), dtype=torch.complex64, device="cuda")}
    fmm.fmm_p2m(L, p, xyd, cd, Md[L])
    for lv in range(L, 2, -1):
        Md[lv - 1] = torch.empty((4 ** (lv - 1), p), dtype=torch.complex64, device="cuda")
        fmm.fmm_m2m(lv, p, Md[lv], Md[lv - 1])
    for lv in range(2, L + 1):
        ref = orc.scale_me(Ms[lv], lv)
        got = _host(Md[lv])
        err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
        assert err < 2e-6, (lv, err)


def test_p2m_points_on_boundaries_and_outside(fmm, orc):
    """fmm_p2m with points on every cell boundary of the level, at 1.0 and just outside the
    unit square (clamped to the edge boxes): the offsets read off the coordinate bits and
    the FP64 fallback both agree with the oracle's P2M (Sec. 2.1 stage 2)."""
    import torch

    rng = np.random.default_rng(98)
    L, p, side = 4, 12, 16
    xy, c = workloads.uniform_particles(4000, rng)
    k = np.arange(side + 1) / side
    xy[:side + 1, 0] = k
    xy[side + 1:2 * side + 2, 1] = k
    xy[-4:] = [[1.0, 0.3], [1.01, 0.6], [-0.02, 0.2], [0.7, 1.03]]
    M = torch.zeros((4 ** L, p), dtype=torch.complex64, device="cuda")
    fmm.fmm_p2m(L, p, torch.from_numpy(xy).cuda(), torch.from_numpy(c).cuda(), M)
    fmm.fmm_sync_status()
    ref = orc.scale_me(orc.p2m_uniform(L, p, xy, c), L)
    err = np.linalg.norm(_host(M) - ref) / np.linalg.norm(ref)
    assert err < 2e-6, err


@pytest.mark.slow
def test_m2l_full_size_workload(fmm, orc):
    """2^22 points, uniform tree to level 8, p = 16, one launch per level (the benchmark's
    launch configuration): levels 2..7 compared in full, level 8 on sampled targets
    (all four corners, edge boxes and random interior boxes)."""
    cfg = workloads.CONFIGS["m2l_scale"]
    p, L = cfg["p"], cfg["max_level"]
    xy, c = workloads.uniform_particles(cfg["n"], workloads.rng_for("m2l_scale"))
    Ms = orc.upward_uniform(L, p, xy, c)
    tree = fmm.fmm_build_lists(None, L)
    outs = {}
    for level in workloads.m2l_levels(L):
        Md = _dev(orc.scale_me(Ms[level], level))
        Ld = Md.new_empty(Md.shape)
        fmm.fmm_m2l(tree, level, p, Md, Ld)
        outs[level] = Ld
    fmm.fmm_sync_status()
    for level in range(2, L):
        _check(_host(outs[level]), _oracle_level(orc, level, p, Ms[level]))
    n = 1 << L
    rng = np.random.default_rng(1)
    edge = [0, n - 1, n * (n - 1), n * n - 1, 1, n, 2 * n + 1, n * n - 2, (n // 2) * n]
    targets = np.unique(np.concatenate([edge, rng.integers(0, n * n, 3000)]))
    ref = orc.scale_le(orc.m2l_uniform_targets(L, p, Ms[L], targets), L)
    _check(_host(outs[L])[targets], ref)


@pytest.mark.parametrize("p", [8, 16, 24])
@pytest.mark.parametrize("periodic", [False, True])
def test_m2l_levels_single_launch(fmm, orc, medium_particles, p, periodic):
    """fmm_m2l_levels (levels 2..6 in one launch) equals the per-level oracle, and
    fmm_m2l_adjoint_levels equals the per-level adjoint."""
    xy, c = medium_particles
    Lmax = 6
    Ms = orc.upward_uniform(Lmax, p, xy, c)
    tree = fmm.fmm_build_lists(None, Lmax, periodic=periodic)
    levels = list(range(2, Lmax + 1))
    Md = [_dev(orc.scale_me(Ms[l], l)) for l in levels]
    Ld = [m.new_empty(m.shape) for m in Md]
    fmm.fmm_m2l_levels(tree, 2, p, Md, Ld)
    for l, out in zip(levels, Ld):
        _check(_host(out), _oracle_level(orc, l, p, Ms[l], periodic))
    Gd = [m.new_empty(m.shape) for m in Md]
    fmm.fmm_m2l_adjoint_levels(tree, 2, p, Ld, Gd, conj=True)
    for l, w, g in zip(levels, Ld, Gd):
        W = _host(w)
        G = np.conj(orc.unscale_me(orc.m2l_adjoint_uniform(l, p, orc.scale_le(np.conj(W), l), periodic), l))
        _check(_host(g), G)


def test_m2l_levels_including_empty_levels(fmm, orc, medium_particles):
    import torch

    xy, c = medium_particles
    p = 6
    Ms = orc.upward_uniform(3, p, xy, c)
    tree = fmm.fmm_build_lists(None, 3)
    Md = [_dev(np.ones((1, p))), _dev(np.ones((4, p))), _dev(orc.scale_me(Ms[2], 2)), _dev(orc.scale_me(Ms[3], 3))]
    Ld = [_dev(np.full(m.shape, 5.0)) for m in Md]
    fmm.fmm_m2l_levels(tree, 0, p, Md, Ld)
    torch.cuda.synchronize()
    assert np.all(_host(Ld[0]) == 0) and np.all(_host(Ld[1]) == 0)
    for l in (2, 3):
        _check(_host(Ld[l]), _oracle_level(orc, l, p, Ms[l]))


@pytest.mark.parametrize("prec_name", ["FMM_FP32", "FMM_TC_BF16X3", "FMM_TC_TF32X3"])
def test_levels_call_replays_from_a_cuda_graph(fmm, orc, prec_name):
    """fmm_m2l_levels recorded by a caller's stream capture (the persistent FP32 kernel with its
    work-counter reset; the tensor-core pre-pass and kernel) and replayed twice, accumulating:
    L = X + 3 M2L(M) after the warm call and two replays."""
    import torch

    prec = getattr(fmm, prec_name)
    p, L = 16, 7
    xy, c = workloads.uniform_particles(60000, np.random.default_rng(8))
    Ms = orc.upward_uniform(L, p, xy, c)
    tree = fmm.fmm_build_lists(None, L)
    levels = list(range(2, L + 1))
    rng = np.random.default_rng(9)
    X = {l: (rng.standard_normal((4 ** l, p)) + 1j * rng.standard_normal((4 ** l, p))) for l in levels}
    Md = [_dev(orc.scale_me(Ms[l], l)) for l in levels]
    Ld = [_dev(X[l]) for l in levels]
    fmm.fmm_m2l_levels(tree, 2, p, Md, Ld, prec=prec, accumulate=True)  # warm: tables, opt-ins, scratch
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="thread_local"):
        fmm.fmm_m2l_levels(tree, 2, p, Md, Ld, prec=prec, accumulate=True)
    g.replay()
    g.replay()
    torch.cuda.synchronize()
    fmm.fmm_sync_status()
    tol = 1e-4 if prec == fmm.FMM_TC_BF16X3 else TOL_L2  # TF32x3 is held to the FP32 bar
    for l, out in zip(levels, Ld):
        ref = orc.scale_le(orc.m2l_uniform(l, p, Ms[l]), l)
        got = (_host(out) - X[l].astype(np.complex64).astype(np.complex128)) / 3.0
        assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= tol, l


@pytest.mark.slow
@pytest.mark.parametrize("prec_name", ["FMM_FP32", "FMM_TC_BF16X3", "FMM_TC_TF32X3"])
def test_level_11_sampled_targets(fmm, orc, prec_name):
    """A level of 2048 x 2048 boxes (4M boxes, 65,536 FP32 tiles): seeded random scaled MEs,
    sampled targets on the corners, edges and interior against the oracle."""
    import torch

    prec = getattr(fmm, prec_name)
    p, level = 16, 11
    n = 1 << level
    rng = np.random.default_rng(1111)
    Ms = (rng.standard_normal((n * n, p)) + 1j * rng.standard_normal((n * n, p))).astype(np.complex64)
    tree = fmm.fmm_build_lists(None, level)
    Md = torch.from_numpy(Ms).cuda()
    Ld = torch.empty_like(Md)
    fmm.fmm_m2l(tree, level, p, Md, Ld, prec=prec)
    fmm.fmm_sync_status()
    edges = [0, 1, n - 2, n - 1]
    targets = [y * n + x for y in edges for x in edges] + list(rng.integers(0, n * n, 300))
    targets += [int(rng.integers(0, n)) for _ in range(20)]              # bottom row
    targets += [(n - 1) * n + int(rng.integers(0, n)) for _ in range(20)]  # top row
    targets = np.unique(np.array(targets, dtype=np.int64))
    M = orc.unscale_me(Ms.astype(np.complex128), level)
    ref = orc.scale_le(orc.m2l_uniform_targets(level, p, M, targets), level)
    got = _host(Ld)[targets]
    tol = 1e-4 if prec == fmm.FMM_TC_BF16X3 else TOL_L2  # TF32x3 is held to the FP32 bar
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= tol


def test_host_stream_pipeline_matches_direct_calls(fmm, orc):
    """pipeline.HostStreamM2L: five steps with different host ME sets (two device buffer
    sets, three streams) give exactly the LEs of fmm_m2l_levels on each set."""
    import torch
    from paper_1009_3457_gb300 import pipeline

    p, L = 8, 5
    tree = fmm.fmm_build_lists(None, L)
    levels = list(range(2, L + 1))
    rng = np.random.default_rng(17)
    host_in, host_out, refs = [], [], []
    for _ in range(5):
        Ms = [torch.from_numpy((rng.standard_normal((4 ** l, p)) + 1j * rng.standard_normal((4 ** l, p)))
                               .astype(np.complex64)).pin_memory() for l in levels]
        host_in.append(Ms)
        host_out.append([torch.empty_like(m).pin_memory() for m in Ms])
        Md = [m.cuda() for m in Ms]
        Ld = [torch.empty_like(m) for m in Md]
        fmm.fmm_m2l_levels(tree, 2, p, Md, Ld)
        refs.append([x.cpu() for x in Ld])
    pipe = pipeline.HostStreamM2L(tree, 2, L, p)
    pipe.run(host_in, host_out)
    # the flat form: all levels in one pinned buffer, one copy per direction
    flat_in = [torch.cat([m.reshape(-1) for m in ms]).pin_memory() for ms in host_in]
    flat_out = [torch.empty(pipe.flat_size(), dtype=torch.complex64).pin_memory() for _ in host_in]
    pipe.run(flat_in, flat_out)
    torch.cuda.synchronize()
    fmm.fmm_sync_status()
    for out, fo, ref in zip(host_out, flat_out, refs):
        for a, f, b in zip(out, pipe.level_views(fo), ref):
            assert torch.equal(a, b) and torch.equal(f, b)


@pytest.mark.parametrize("p", [6, 8, 12, 16, 24])
def test_m2l_single_sources_reach_their_lists_only(fmm, p):
    """One non-zero source box at a time (every child class, inside the domain, at a corner and
    at an edge, tiles with and without a neighbour), forward and conjugate adjoint: each target
    of its lists holds T(D) m to the FP32 rounding of a p-term sum, every other box exactly 0.
    The 27 offsets are folded by symmetry in the kernel, so each offset is checked apart."""
    import math
    import torch

    level, side = 4, 16
    tree = fmm.fmm_build_lists(None, level)
    lst, _ = tree.lists(level)
    rng = np.random.default_rng(p)
    nk = np.arange(p)
    binom = np.array([[math.comb(n + k, k) for k in range(p)] for n in range(p)], dtype=np.float64)
    for sx, sy in [(7, 6), (8, 9), (5, 8), (10, 11), (0, 0), (15, 3), (2, 15)]:
        m = (rng.standard_normal(p) + 1j * rng.standard_normal(p)).astype(np.complex64)
        src = sy * side + sx
        M = np.zeros((side * side, p), np.complex64)
        M[src] = m
        for adjoint in (False, True):
            Md, out = _dev(M), torch.full((side * side, p), float("nan"), dtype=torch.complex64, device="cuda")
            if adjoint:
                fmm.fmm_m2l_adjoint(tree, level, p, Md, out, conj=True)
            else:
                fmm.fmm_m2l(tree, level, p, Md, out)
            fmm.fmm_sync_status()
            got = _host(out)
            for t in range(side * side):
                if src not in lst[t]:
                    assert (got[t] == 0).all(), (sx, sy, t, adjoint)
                    continue
                d = complex(t % side - sx, t // side - sy)  # target - source (symmetric lists: adjoint of -d)
                D = -d if adjoint else d
                T = (-1.0) ** nk[:, None] * binom * D ** -(nk[:, None] + nk[None, :] + 1.0)
                T = T.conj().T if adjoint else T
                # p products and sums, two roundings of each scaling and of the operator's value, and the
                # folded combinations' few additions, on both parts: (2 p + 24) units of 2^-24
                bound = (2 * p + 24) * 2.0 ** -24 * (np.abs(T) @ np.abs(m))
                assert (np.abs(got[t] - T @ m) <= bound).all(), (sx, sy, t, adjoint)
