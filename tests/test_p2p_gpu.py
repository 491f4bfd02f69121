"""GPU parity of the near field (fmm_p2p, Sec. 2.1 stage 5, reading R15) and of the whole
FMM on the device (farfield.FmmPotential) against the FP64 oracle.

Bars.  The kernel keeps positions relative to the target box's centre in FP32, so a
pair's distance carries an absolute error of ~2^-24 x 1.5 box sides; a term's relative
error is that over the pair's distance, and the closest of m points in a box lies ~side/m
away.  Trees used as an FMM keep a few dozen points per finest box: there the bar is
relative L2 <= 1e-5 against the oracle's near field, every target within 1e-4 of
max |phi|.  The coarse cases below (4,000 points in one box at level 0, ~250 per box at
level 2) are checked at 2e-4 and 1e-4.  The whole FMM at p = 16 is held to 2e-5 of the
direct sum (the oracle's own FMM at p = 16 is within 3e-8 of it).
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fmm():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1009_3457_gb300 import build, fmmgb

    build.build()
    fmmgb.load()
    return fmmgb


def _bins(fmm, level, pts):
    import torch

    perm = torch.empty(pts.shape[0], dtype=torch.int32, device="cuda")
    start = torch.empty(4 ** level + 1, dtype=torch.int32, device="cuda")
    work = torch.empty(4 ** level, dtype=torch.int32, device="cuda")
    fmm.fmm_bin_points(level, pts, perm, start, work)
    return perm, start


def _p2p(fmm, level, xy, c, z, phi0=None):
    import torch

    xyd, cd = torch.from_numpy(xy).cuda(), torch.from_numpy(c).cuda()
    zd = torch.from_numpy(np.stack([z.real, z.imag], 1).copy()).cuda()
    sp, ss = _bins(fmm, level, xyd)
    tp, ts = _bins(fmm, level, zd)
    phi = torch.zeros(len(z), dtype=torch.complex64, device="cuda") if phi0 is None else \
        torch.from_numpy(phi0.astype(np.complex64)).cuda()
    fmm.fmm_p2p(level, xyd, cd, sp, ss, zd, tp, ts, phi, accumulate=phi0 is not None)
    fmm.fmm_sync_status()
    return phi.cpu().numpy().astype(np.complex128)


def _check(got, ref, l2=1e-5, worst=1e-4):
    err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
    w = np.abs(got - ref).max() / np.abs(ref).max()
    assert err <= l2 and w <= worst, f"relative L2 {err:.3e}, worst {w:.3e}"


@pytest.mark.parametrize("level,bar,nsrc", [(0, 2e-4, 4000), (2, 1e-4, 4000), (3, 1e-5, 4000), (5, 1e-5, 4000),
                                            (8, 1e-5, 262144), (10, 1e-5, 1048576)])
def test_p2p_matches_oracle(fmm, orc, level, bar, nsrc):
    """Levels 0 to 10, the finest (1M boxes) with ~1 source per box."""
    rng = np.random.default_rng(40 + level)
    xy, c = workloads.uniform_particles(nsrc, rng)
    z = rng.random(3000) + 1j * rng.random(3000)
    _check(_p2p(fmm, level, xy, c, z), orc.p2p_uniform(level, xy, c, z), l2=bar, worst=max(1e-4, 2 * bar))


@pytest.mark.parametrize("level,nsrc", [(3, 4000), (8, 262144)])
def test_p2p_shared_sm_grid_gives_the_same_result(fmm, orc, level, nsrc):
    """FMM_P2P_SHARE_SM only shrinks the persistent grid: on the same binning (the binning's
    order within a box is not fixed) every claim is summed the same way by whichever CTA
    takes it, so the result is bit-identical, and on the oracle's bar."""
    import torch

    rng = np.random.default_rng(60 + level)
    xy, c = workloads.uniform_particles(nsrc, rng)
    z = rng.random(3000) + 1j * rng.random(3000)
    xyd, cd = torch.from_numpy(xy).cuda(), torch.from_numpy(c).cuda()
    zd = torch.from_numpy(np.stack([z.real, z.imag], 1).copy()).cuda()
    sp, ss = _bins(fmm, level, xyd)
    tp, ts = _bins(fmm, level, zd)
    out = []
    for share in (False, True):
        phi = torch.zeros(len(z), dtype=torch.complex64, device="cuda")
        fmm.fmm_p2p(level, xyd, cd, sp, ss, zd, tp, ts, phi, share_sm=share)
        fmm.fmm_sync_status()
        out.append(phi.cpu())
    assert torch.equal(out[0], out[1])
    _check(out[1].numpy().astype(np.complex128), orc.p2p_uniform(level, xy, c, z))


def test_p2p_points_on_box_boundaries_and_outside(fmm, orc):
    """Sources on the level's box boundaries, targets one ulp either side of them, and
    points at 1.0 and just outside the unit square (clamped to the edge boxes)."""
    rng = np.random.default_rng(44)
    level, side = 3, 8
    xy, c = workloads.uniform_particles(3000, rng)
    k = np.arange(side + 1) / side
    xy[:side + 1, 0] = k
    xy[side + 1:2 * side + 2, 1] = k
    xy[-4:] = [[1.0, 0.3], [1.004, 0.6], [-0.003, 0.2], [0.7, 1.002]]
    zx = np.concatenate([np.nextafter(k, -1.0), np.nextafter(k, 2.0), rng.random(300), [1.0, 1.006, -0.002]])
    zy = rng.random(len(zx))
    _check(_p2p(fmm, level, xy, c, zx + 1j * zy), orc.p2p_uniform(level, xy, c, zx + 1j * zy))


def test_p2p_targets_on_sources_skip_themselves(fmm, orc):
    xy, c = workloads.uniform_particles(5000, np.random.default_rng(3))
    z = xy[:, 0] + 1j * xy[:, 1]
    _check(_p2p(fmm, 4, xy, c, z), orc.p2p_uniform(4, xy, c, z))


def test_p2p_clustered_sources_span_several_batches(fmm, orc):
    """Gaussian-mixture sources: boxes near the means hold thousands of points, so the
    3 x 3 neighbourhood is staged in several shared-memory batches (the coarse regime of
    the module's bars: 2e-4)."""
    xy, c = workloads.gmm_particles(30000, np.random.default_rng(8), ncomp=3)
    rng = np.random.default_rng(9)
    z = np.concatenate([rng.random(1500) + 1j * rng.random(1500), xy[:1500, 0] + 1j * xy[:1500, 1]])
    _check(_p2p(fmm, 4, xy, c, z), orc.p2p_uniform(4, xy, c, z), l2=2e-4, worst=4e-4)


def test_p2p_accumulate_and_ragged_counts(fmm, orc):
    rng = np.random.default_rng(12)
    xy, c = workloads.uniform_particles(3000, rng)
    for m in (1, 255, 257):
        z = rng.random(m) + 1j * rng.random(m)
        ref = orc.p2p_uniform(3, xy, c, z)
        base = 0.5 - 0.25j + np.zeros(m)
        _check(_p2p(fmm, 3, xy, c, z, phi0=base), ref + base)


@pytest.mark.parametrize("level,n", [(4, 8192), (5, 20000)])
def test_whole_fmm_on_device_matches_direct_sum(fmm, orc, level, n):
    """P2M, M2M, M2L, L2L, L2P and P2P, all library kernels, at the points themselves."""
    import torch
    from paper_1009_3457_gb300.farfield import FmmPotential

    xy, c = workloads.uniform_particles(n, np.random.default_rng(60 + level))
    tree = fmm.fmm_build_lists(xy, max_level=level)
    xyd = torch.from_numpy(xy).cuda()
    pot = FmmPotential(tree, 16, xyd, torch.from_numpy(c).cuda(), xyd)
    got = pot().cpu().numpy().astype(np.complex128)
    fmm.fmm_sync_status()
    pick = np.random.default_rng(1).choice(n, 400, replace=False)
    ref = orc.p2p_uniform(0, xy, c, xy[pick, 0] + 1j * xy[pick, 1])  # level 0: every other point
    assert np.linalg.norm(got[pick] - ref) / np.linalg.norm(ref) <= 2e-5
    # re-runnable: every buffer is rewritten (P2M sums with FP32 atomics, so runs agree to rounding)
    again = pot().cpu().numpy().astype(np.complex128)
    assert np.linalg.norm(again - got) / np.linalg.norm(got) <= 1e-6


def test_whole_fmm_full_size_sampled(fmm, orc):
    """2^22 uniform points, uniform tree to level 8, p = 16 (the M2L benchmark's tree): the
    potential at 120 sampled points against the direct sum over all other points."""
    import torch
    from paper_1009_3457_gb300.farfield import FmmPotential

    n = 1 << 22
    xy, c = workloads.uniform_particles(n, np.random.default_rng(77))
    tree = fmm.fmm_build_lists(xy, max_level=8)
    xyd = torch.from_numpy(xy).cuda()
    got = FmmPotential(tree, 16, xyd, torch.from_numpy(c).cuda(), xyd)().cpu().numpy().astype(np.complex128)
    fmm.fmm_sync_status()
    pick = np.random.default_rng(2).choice(n, 120, replace=False)
    ref = orc.p2p_uniform(0, xy, c, xy[pick, 0] + 1j * xy[pick, 1])  # level 0: every other point
    assert np.linalg.norm(got[pick] - ref) / np.linalg.norm(ref) <= 2e-5


@pytest.mark.parametrize("p", [8, 16, 24])
def test_p2m_binned_matches_oracle_and_repeats_exactly(fmm, orc, p):
    """fmm_p2m_binned (one block per box, no atomics) against the oracle's P2M in
    radius-scaled units, on uniform and clustered points; two runs are bit-identical."""
    import torch

    for xy, c, level in (workloads.uniform_particles(20000, np.random.default_rng(31)) + (5,),
                         workloads.gmm_particles(20000, np.random.default_rng(32), ncomp=3) + (6,)):
        xyd, cd = torch.from_numpy(xy).cuda(), torch.from_numpy(c).cuda()
        perm, start = _bins(fmm, level, xyd)
        M = torch.empty((4 ** level, p), dtype=torch.complex64, device="cuda")
        fmm.fmm_p2m_binned(level, p, xyd, cd, perm, start, M)
        fmm.fmm_sync_status()
        got = M.cpu().numpy().astype(np.complex128)
        ref = orc.scale_me(orc.p2m_uniform(level, p, xy, c), level)
        assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= 1e-5
        again = M.clone()
        fmm.fmm_p2m_binned(level, p, xyd, cd, perm, start, M)
        assert torch.equal(again, M)


@pytest.mark.parametrize("level,per_box", [(6, 8), (7, 0.5), (7, 8), (7, 31.9), (7, 32), (8, 8)])
def test_p2p_sparse_and_dense_claims(fmm, orc, level, per_box):
    """Both sides of the line between a CTA and a warp per claim (boxes, targets per box), with one
    box of thousands of targets and sources (several runs of targets, several pieces of sources),
    empty boxes, and accumulation; 900 targets against the oracle."""
    import torch

    nb = 4 ** level
    rng = np.random.default_rng(int(level * 100 + per_box))
    nz = int(per_box * nb)
    crowd = min(1500, nz // 4)
    z = np.concatenate([rng.random((nz - crowd, 2)), 0.37 + 0.9 * 0.5 ** level * rng.random((crowd, 2))])
    xy = np.concatenate([rng.random((30000, 2)), 0.37 + 0.9 * 0.5 ** level * rng.random((1000, 2))])
    c = rng.uniform(-1, 1, len(xy))
    pick = np.concatenate([rng.choice(nz, 600, replace=False), nz - crowd + rng.choice(crowd, 300, replace=False)])
    phi0 = rng.standard_normal(nz) + 1j * rng.standard_normal(nz)
    zz = z[:, 0] + 1j * z[:, 1]
    ref = orc.p2p_uniform(level, xy, c, zz[pick])
    # ~1000 sources in one box: the closest pair lies ~1e-3 box sides away (the bar of the coarse levels)
    got = _p2p(fmm, level, xy, c, zz, phi0=phi0)[pick] - phi0.astype(np.complex64)[pick]
    scale = np.abs(phi0[pick]) + np.abs(ref)
    assert np.linalg.norm(got - ref) <= 1e-4 * np.linalg.norm(ref)
    assert (np.abs(got - ref) <= 2e-4 * np.abs(ref).max() + 1e-6 * scale).all()


def test_chains_of_launches_replay_from_a_graph(fmm, orc):
    """Binning on a grid whose prefix is copied between two kernels, M2L of levels 0.. (memsets before
    the kernel) and the whole potential with its two streams, recorded in one CUDA graph and replayed,
    with other strengths too: equal to direct calls."""
    import torch

    from paper_1009_3457_gb300 import farfield

    level, p, n = 8, 8, 300_000
    rng = np.random.default_rng(12)
    sets = [(torch.from_numpy(rng.random((n, 2))).cuda(), torch.from_numpy(rng.uniform(-1, 1, n)).cuda())
            for _ in range(2)]
    tree = fmm.fmm_build_lists(None, level)
    xy, c = sets[0][0].clone(), sets[0][1].clone()
    Ms = [torch.view_as_complex(torch.randn((4 ** l, p, 2), device="cuda")) for l in range(level + 1)]
    Ls = [torch.full_like(m, float("nan")) for m in Ms]
    perm, start = _bins(fmm, level, xy)
    work = torch.empty(4 ** level, dtype=torch.int32, device="cuda")
    pot = farfield.FmmPotential(tree, p, xy, c, xy)
    fmm.fmm_m2l_levels(tree, 0, p, Ms, Ls)
    pot()
    torch.cuda.synchronize()
    want = [l.clone() for l in Ls]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        fmm.fmm_bin_points(level, xy, perm, start, work)
        fmm.fmm_m2l_levels(tree, 0, p, Ms, Ls)
        pot()
    for pts, q in sets:
        if pts is not sets[0][0]:
            c.copy_(q)  # the positions keep their bins
        for l in Ls:
            l.fill_(float("nan"))
        perm.zero_()
        start.zero_()
        graph.replay()
        fmm.fmm_sync_status()
        got = pot.phi.clone()
        pot()
        fmm.fmm_sync_status()
        assert torch.equal(torch.view_as_real(got), torch.view_as_real(pot.phi))
        for a, b in zip(Ls, want):
            assert torch.equal(torch.view_as_real(a), torch.view_as_real(b))
        ix = torch.clamp((xy * 2 ** level).floor().long(), 0, 2 ** level - 1)
        box = ix[:, 1] * 2 ** level + ix[:, 0]
        assert torch.equal(torch.diff(start).long(), torch.bincount(box, minlength=4 ** level))
        assert torch.equal(box[perm.long()], torch.sort(box).values)


@pytest.mark.parametrize("level,per_box", [(3, 100), (6, 8), (7, 0.3), (7, 20), (7, 40), (10, 0.6)])
def test_p2p_short_lived_blocks_equal_persistent_ones(fmm, level, per_box):
    """Both kernels, with blocks that end after a few claims (FMM_P2P_SHARE_SM; at level 10 more than
    two, the grid being bounded) and with persistent ones: the same bits, twice."""
    import torch

    g = torch.Generator(device="cuda").manual_seed(level)
    nz, n = int(per_box * 4 ** level), 20000
    z, xy = (torch.rand((k, 2), dtype=torch.float64, device="cuda", generator=g) for k in (nz, n))
    c = torch.rand(n, dtype=torch.float64, device="cuda", generator=g) - 0.5
    (sp, ss), (tp, ts) = _bins(fmm, level, xy), _bins(fmm, level, z)
    out = []
    for share in (False, True, False, True):
        phi = torch.full((nz,), float("nan"), dtype=torch.complex64, device="cuda")
        fmm.fmm_p2p(level, xy, c, sp, ss, z, tp, ts, phi, share_sm=share)
        fmm.fmm_sync_status()
        assert bool(torch.isfinite(torch.view_as_real(phi)).all())
        out.append(phi)
    for phi in out[1:]:
        assert torch.equal(torch.view_as_real(phi), torch.view_as_real(out[0]))


@pytest.mark.parametrize("level", [0, 3, 7])
@pytest.mark.parametrize("n", [1, 257, 32767, 32768, 4097 * 304, 1_300_001])
def test_binning_at_the_edges_of_its_blocks(fmm, level, n):
    """The three block shapes (256 threads x 4 points, 512 x 8, 1024 x 4), chunks shorter than a block's
    points and longer: the boxes' counts, and every point once in its own box."""
    import torch

    g = torch.Generator(device="cuda").manual_seed(n)
    pts = torch.rand((n, 2), dtype=torch.float64, device="cuda", generator=g) ** 2
    perm, start = _bins(fmm, level, pts)
    ix = (pts * 2 ** level).floor().long()
    box = ix[:, 1] * 2 ** level + ix[:, 0]
    assert torch.equal(torch.diff(start).long(), torch.bincount(box, minlength=4 ** level))
    assert torch.equal(box[perm.long()], torch.sort(box).values)
    assert torch.equal(torch.sort(perm).values.long(), torch.arange(n, device="cuda"))


@pytest.mark.parametrize("level", [7, 8])
def test_p2p_crowded_boxes_among_sparse_ones(fmm, orc, level):
    """A call whose sparse boxes go to the warp kernel and whose dense or crowded ones to the CTA kernel:
    boxes of 1, 31, 32, 33, 97, 320 and 500 targets (one run, and runs of several row counts), and few targets beside 1,023, 1,024 and 3,000 sources
    (in the box, and in its neighbours), at corners and inside, every such target against the oracle;
    the same bits with short-lived blocks."""
    import torch

    rng = np.random.default_rng(level)
    side = 2 ** level
    at = lambda bx, by, k: (np.array([bx, by]) + 0.02 + 0.96 * rng.random((k, 2))) / side
    z, xy = [rng.random((side * side // 8, 2))], [rng.random((2000, 2))]
    for i, m in enumerate((1, 31, 32, 33, 97, 320, 500)):
        z.append(at(4 * i, 0 if i % 2 else side - 1, m))
        xy.append(at(4 * i, 0 if i % 2 else side - 1, 7))
    for i, k in enumerate((1023, 1024, 3000)):
        z.append(at(10 * i + 3, side // 2, 5))
        xy.append(at(10 * i + 3 + i % 2, side // 2 + (i == 2), k))
    z, xy = np.concatenate(z), np.concatenate(xy)
    c = rng.uniform(-1, 1, len(xy))
    zz = z[:, 0] + 1j * z[:, 1]
    ref = orc.p2p_uniform(level, xy, c, zz)
    zd, xyd, cd = (torch.from_numpy(v).cuda() for v in (z, xy, c))
    (sp, ss), (tp, ts) = _bins(fmm, level, xyd), _bins(fmm, level, zd)
    out = []
    for share in (False, True):
        phi = torch.full((len(z),), float("nan"), dtype=torch.complex64, device="cuda")
        fmm.fmm_p2p(level, xyd, cd, sp, ss, zd, tp, ts, phi, share_sm=share)
        fmm.fmm_sync_status()
        out.append(phi)
    assert torch.equal(torch.view_as_real(out[0]), torch.view_as_real(out[1]))
    got = out[0].cpu().numpy().astype(np.complex128)
    # the bars of the coarse levels, as for the other crowded boxes above
    assert np.linalg.norm(got - ref) <= 1e-4 * np.linalg.norm(ref)
    assert np.abs(got - ref).max() <= 2e-4 * np.abs(ref).max()


def test_p2p_graph_keeps_its_buffer(fmm):
    """The per-device buffer grows inside a capture (more targets, then more sources, than any call
    before), and a graph captured before it grew replays what it did."""
    import torch

    level = 7
    g = torch.Generator(device="cuda").manual_seed(3)

    def problem(n, nz):
        xy, z = (torch.rand((k, 2), dtype=torch.float64, device="cuda", generator=g) for k in (n, nz))
        c = torch.rand(n, dtype=torch.float64, device="cuda", generator=g) - 0.5
        phi = torch.empty(nz, dtype=torch.complex64, device="cuda")
        (sp, ss), (tp, ts) = _bins(fmm, level, xy), _bins(fmm, level, z)
        return phi, lambda: fmm.fmm_p2p(level, xy, c, sp, ss, z, tp, ts, phi)

    torch.cuda.synchronize()
    grow = 6_000_000  # beyond every other call of these tests
    problems = [problem(1000, 2000), problem(1000, grow), problem(2 * grow, 2000), problem(8 * grow, 3000)]
    problems[0][1]()
    torch.cuda.synchronize()
    graphs = []
    for phi, call in problems:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, capture_error_mode="thread_local"):
            call()
        graphs.append(graph)
    for graph, (phi, call) in zip(graphs, problems):
        call()
        fmm.fmm_sync_status()
        want = phi.clone()
        phi.fill_(float("nan"))
        graph.replay()
        fmm.fmm_sync_status()
        assert torch.equal(torch.view_as_real(phi), torch.view_as_real(want))
