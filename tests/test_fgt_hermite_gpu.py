"""GPU parity of the FGT Hermite-series evaluation (fgt_h2p, Sec. 4.2, Eq. hermite),
the device binning of points by box (fgt_bin_points) and the binned P2H
(fgt_p2h_binned), against the FP64 oracle.

fgt_h2p has three forms: through Chebyshev coefficients of each target box (from 2 targets a box on
average, box sides of up to sqrt2 sigma / 2), and the direct sums on the CUDA cores and on the tensor
cores.  The grid of a sigma (workloads.fgt_grid_log2) has box sides of 0.25 to 0.5 sqrt2 sigma; the
tests of the direct kernels take the next coarser one, which the first form leaves to them.

Bars: binning is exact (the same box for every point, every point once);
G relative L2 over all targets <= 1e-5 (FP32) against the oracle evaluating
the same FP32 coefficients in FP64, and every target's error <= 1e-5 of
max |G|; the binned P2H relative L2 <= 1e-5 against the oracle's P2H.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

TOL_L2 = 1e-5
TOL_MAX = 1e-5


@pytest.fixture(scope="module")
def fmm():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1009_3457_gb300 import build, fmmgb

    build.build()
    fmmgb.load()
    return fmmgb


def _boxes(y, g):
    n = 1 << g
    ix = np.clip(np.floor(y[:, 0] * n), 0, n - 1).astype(np.int64)
    iy = np.clip(np.floor(y[:, 1] * n), 0, n - 1).astype(np.int64)
    return iy * n + ix


def _bin(fmm, g, y_dev):
    import torch

    n = y_dev.shape[0]
    perm = torch.empty(n, dtype=torch.int32, device="cuda")
    start = torch.empty(4 ** g + 1, dtype=torch.int32, device="cuda")
    work = torch.empty(4 ** g, dtype=torch.int32, device="cuda")
    fmm.fgt_bin_points(g, y_dev, perm, start, work)
    return perm, start


def _h2p(fmm, g, ncut, p, sigma, A32, y, G=None, accumulate=False):
    import torch

    yd = torch.from_numpy(np.ascontiguousarray(y, dtype=np.float64)).cuda()
    perm, start = _bin(fmm, g, yd)
    if G is None:
        G = torch.empty(len(y), dtype=torch.float32, device="cuda")
    fmm.fgt_h2p(g, ncut, p, sigma, torch.from_numpy(A32).cuda(), yd, perm, start, G, accumulate=accumulate)
    fmm.fmm_sync_status()
    return G.cpu().numpy().astype(np.float64)


def _check(got, ref):
    err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
    worst = np.abs(got - ref).max() / np.abs(ref).max()
    assert err <= TOL_L2 and worst <= TOL_MAX, f"relative L2 {err:.3e}, worst {worst:.3e}"
    return err


@pytest.fixture(scope="module")
def gmm_sources():
    return workloads.gmm_particles(20000, np.random.default_rng(91))


def test_bin_points_is_an_exact_counting_sort(fmm):
    import torch

    rng = np.random.default_rng(3)
    g = 5
    y = rng.random((50000, 2))
    y[:10] = [[0.0, 0.0], [1.0, 1.0], [-0.5, 0.3], [0.3, 1.5], [0.999999999, 0.5], [0.5, 0.03125],
              [0.03125, 0.0625], [1e-300, 0.9999999999999999], [2.0, -2.0], [0.5, 0.5]]
    y[10:5000] = [0.4, 0.6]  # one crowded box
    perm, start = _bin(fmm, g, torch.from_numpy(y).cuda())
    perm, start = perm.cpu().numpy(), start.cpu().numpy()
    box = _boxes(y, g)
    counts = np.bincount(box, minlength=4 ** g)
    assert start[0] == 0 and start[-1] == len(y)
    np.testing.assert_array_equal(np.diff(start), counts)
    assert np.array_equal(np.sort(perm), np.arange(len(y)))
    owner = np.repeat(np.arange(4 ** g), counts)
    np.testing.assert_array_equal(box[perm], owner)


def _edge_values(g):
    """Coordinates on and next to every cell boundary of the 2^g grid, the ends of [0, 1),
    subnormals, signed zeros, and values outside [0, 1) (clamped), infinities and NaN."""
    k = np.arange((1 << g) + 1) / (1 << g)
    v = np.concatenate([k, np.nextafter(k, -np.inf), np.nextafter(k, np.inf),
                        [0.0, -0.0, 5e-324, 1e-310, 1e-300, 1 - 2.0 ** -53, 1.0, 1.5, 2.0 ** 40, -1e-300, -3.0,
                         np.inf, -np.inf, np.nan, 0.5, 1.0 / 3.0]])
    return v


@pytest.mark.parametrize("g", [0, 1, 5, 10])
def test_bin_points_edge_coordinates(fmm, g):
    """The device places a coordinate by floor(v 2^g) exactly (read off the bits of the
    FP64 value), clamped to the grid, NaN to cell 0."""
    import torch

    v = _edge_values(g)
    rng = np.random.default_rng(17 + g)
    y = np.stack([np.concatenate([v, rng.permutation(v)]), np.concatenate([rng.permutation(v), v])], axis=1)
    side = 1 << g
    with np.errstate(invalid="ignore", over="ignore"):
        cell = np.floor(y * side)
    cell = np.clip(np.where(np.isnan(cell), 0.0, cell), 0, side - 1).astype(np.int64)
    box = cell[:, 1] * side + cell[:, 0]
    perm, start = _bin(fmm, g, torch.from_numpy(y).cuda())
    perm, start = perm.cpu().numpy(), start.cpu().numpy()
    counts = np.bincount(box, minlength=4 ** g)
    np.testing.assert_array_equal(np.diff(start), counts)
    np.testing.assert_array_equal(box[perm], np.repeat(np.arange(4 ** g), counts))


def test_bin_points_empty_and_single(fmm):
    import torch

    for n in (0, 1):
        y = torch.full((n, 2), 0.7, dtype=torch.float64, device="cuda")
        perm, start = _bin(fmm, 3, y)
        s = start.cpu().numpy()
        assert s[-1] == n and (np.diff(s) >= 0).all()
        if n:
            assert s[_boxes(np.full((1, 2), 0.7), 3)[0] + 1] == 1


@pytest.mark.parametrize("p", [4, 8, 12, 16])
def test_p2h_binned_matches_oracle(fmm, orc, gmm_sources, p):
    import torch

    x, q = gmm_sources
    for sigma in (0.2, 0.05):
        g = workloads.fgt_grid_log2(sigma)
        xd = torch.from_numpy(x).cuda()
        perm, _ = _bin(fmm, g, xd)
        A = torch.empty((4 ** g, p, p), dtype=torch.float32, device="cuda")
        fmm.fgt_p2h_binned(g, p, sigma, xd, torch.from_numpy(q).cuda(), perm, A)
        fmm.fmm_sync_status()
        ref = orc.fgt_p2h_grid(g, p, sigma, x, q)
        got = A.cpu().numpy().astype(np.float64)
        assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= 1e-5
        fmm.fgt_p2h_binned(g, p, sigma, xd, torch.from_numpy(q).cuda(), perm, A, accumulate=True)
        got2 = A.cpu().numpy().astype(np.float64)
        assert np.linalg.norm(got2 - 2 * ref) / np.linalg.norm(2 * ref) <= 1e-5


@pytest.mark.parametrize("coarser", [0, 1])
@pytest.mark.parametrize("p", [4, 8, 12, 16])
@pytest.mark.parametrize("sigma,ncut", [(0.2, 10), (0.1, 3), (0.05, 1), (0.1, 0)])
def test_h2p_matches_oracle(fmm, orc, gmm_sources, p, sigma, ncut, coarser):
    """Targets: uniform (many in boxes with no sources) plus a cluster of 700 in one
    box (coarser: several claims of one box by the direct kernel, a ragged last one)."""
    x, q = gmm_sources
    g = workloads.fgt_grid_log2(sigma) - coarser
    rng = np.random.default_rng(p * 100 + ncut)
    y = np.concatenate([rng.random((2500, 2)), 0.52 + 0.001 * rng.random((700, 2))])
    A32 = orc.fgt_p2h_grid(g, p, sigma, x, q).astype(np.float32)
    got = _h2p(fmm, g, ncut, p, sigma, A32, y)
    ref = orc.fgt_hermite_eval_grid(g, ncut, p, sigma, A32.astype(np.float64), y)
    _check(got, ref)


def test_h2p_accumulate_and_ragged_counts(fmm, orc, gmm_sources):
    import torch

    x, q = gmm_sources
    sigma, p, ncut = 0.1, 8, 4
    g = workloads.fgt_grid_log2(sigma)
    A32 = orc.fgt_p2h_grid(g, p, sigma, x, q).astype(np.float32)
    for n in (1, 31, 33, 511, 513):
        y = np.random.default_rng(n).random((n, 2))
        ref = orc.fgt_hermite_eval_grid(g, ncut, p, sigma, A32.astype(np.float64), y)
        _check(_h2p(fmm, g, ncut, p, sigma, A32, y), ref)
        G = torch.full((n,), 0.25, dtype=torch.float32, device="cuda")
        _check(_h2p(fmm, g, ncut, p, sigma, A32, y, G=G, accumulate=True), ref + 0.25)


@pytest.mark.parametrize("g", [0, 1, 6, 7])
def test_h2p_claim_order_grids(fmm, orc, g):
    """Claims are handed out heaviest neighbourhood first: one CTA builds that order for grids
    of up to 64 x 64 boxes, five launches (row prefix, keys, scan, scatter, claims) above.
    Grids of 1 x 1, 2 x 2 (the neighbourhood clipped to the grid), 64 x 64 and 128 x 128 boxes,
    a third of the source boxes empty, clustered targets (per box counts from 0 to thousands),
    G pre-filled with NaN: every target is evaluated once, against the oracle."""
    import math
    import torch

    rng = np.random.default_rng(300 + g)
    p, ncut = 8, 3
    n = 1 << g
    sigma = 2.0 ** -g / (math.sqrt(2.0) * 0.6)  # boxes that the direct kernel takes
    fact = np.array([math.factorial(a) for a in range(p)], float)
    A = rng.standard_normal((n * n, p, p)) * (0.3 ** (np.arange(p)[:, None] + np.arange(p)[None, :])) / np.outer(fact, fact)
    empty = rng.random(n * n) < 0.33
    empty[0] = False  # at least one source box holds coefficients
    A[empty] = 0.0
    A32 = A.astype(np.float32)
    c = rng.random((6, 2))
    y = np.concatenate([np.clip(c[i] + 0.03 * rng.standard_normal((3000, 2)), 0.0, 0.999999) for i in range(6)]
                       + [rng.random((2000, 2))])
    yd = torch.from_numpy(np.ascontiguousarray(y)).cuda()
    perm, start = _bin(fmm, g, yd)
    G = torch.full((len(y),), float("nan"), dtype=torch.float32, device="cuda")
    fmm.fgt_h2p(g, ncut, p, sigma, torch.from_numpy(A32).cuda(), yd, perm, start, G)
    fmm.fmm_sync_status()
    got = G.cpu().numpy().astype(np.float64)
    assert np.isfinite(got).all()
    ref = orc.fgt_hermite_eval_grid(g, ncut, p, sigma, A32.astype(np.float64), y)
    _check(got, ref)


def test_h2p_bad_permutation_sets_error_word(fmm):
    """A perm entry outside [0, n) is caught by the kernel's own bounds check: the
    target is skipped and fmm_sync_status reports FMM_EDEVICE; the context stays usable."""
    import torch

    g, p = 3, 4
    y = torch.from_numpy(np.random.default_rng(1).random((100, 2))).cuda()
    perm, start = _bin(fmm, g, y)
    perm[5] = 1000
    A = torch.zeros((4 ** g, p, p), dtype=torch.float32, device="cuda")
    A[:, 0, 0] = 1.0
    G = torch.zeros(100, dtype=torch.float32, device="cuda")
    fmm.fgt_h2p(g, 2, p, 0.2, A, y, perm, start, G)
    with pytest.raises(fmm.FmmError) as e:
        fmm.fmm_sync_status()
    assert e.value.code == fmm.FMM_EDEVICE
    fmm.fmm_sync_status()  # the word was cleared
    assert float(G.abs().sum()) > 0


@pytest.mark.parametrize("sigma,p", [(0.1, 8), (0.05, 12), (0.2, 16)])
def test_hermite_transform_on_device_matches_direct_sum(fmm, orc, sigma, p):
    """fgt_bin_points -> fgt_p2h_binned -> fgt_h2p: the whole transform through Hermite
    evaluation, against the direct Gauss sum (Eq. dgt), within truncation and cutoff."""
    import torch

    rng = np.random.default_rng(int(sigma * 1000) + p + 7)
    x, q = workloads.gmm_particles(20000, rng)
    y = rng.random((2000, 2))
    g = workloads.fgt_grid_log2(sigma)
    xd = torch.from_numpy(x).cuda()
    perm, _ = _bin(fmm, g, xd)
    A = torch.empty((4 ** g, p, p), dtype=torch.float32, device="cuda")
    fmm.fgt_p2h_binned(g, p, sigma, xd, torch.from_numpy(q).cuda(), perm, A)
    got = _h2p(fmm, g, workloads.FGT_NCUT, p, sigma, A.cpu().numpy(), y)
    direct = orc.fgt_direct(x, q, sigma, y)
    assert np.linalg.norm(got - direct) / np.linalg.norm(direct) <= 1e-5


@pytest.mark.parametrize("sigma,p,coarser", [(0.05, 16, 0), (0.2, 8, 0), (0.05, 16, 1), (0.2, 8, 1)])
def test_h2p_full_size_workload_sampled(fmm, orc, sigma, p, coarser):
    """2^20 Gaussian-mixture sources and 2^20 targets from the same mixture (n_cut = 10),
    the launch the benchmark times, and (coarser) one of the direct kernel; 1,500 sampled targets
    against the oracle."""
    import torch

    n = 1 << 20
    rng = np.random.default_rng(2024)
    x, q = workloads.gmm_particles(n, rng)
    y, _ = workloads.gmm_particles(n, np.random.default_rng(2025))
    g = workloads.fgt_grid_log2(sigma) - coarser
    xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    perm, _ = _bin(fmm, g, xd)
    A = torch.empty((4 ** g, p, p), dtype=torch.float32, device="cuda")
    fmm.fgt_p2h_binned(g, p, sigma, xd, torch.from_numpy(q).cuda(), perm, A)
    tperm, tstart = _bin(fmm, g, yd)
    G = torch.empty(n, dtype=torch.float32, device="cuda")
    fmm.fgt_h2p(g, workloads.FGT_NCUT, p, sigma, A, yd, tperm, tstart, G)
    fmm.fmm_sync_status()
    pick = np.random.default_rng(5).choice(n, 1500, replace=False)
    A64 = A.cpu().numpy().astype(np.float64)
    ref = orc.fgt_hermite_eval_grid(g, workloads.FGT_NCUT, p, sigma, A64, y[pick])
    _check(G.cpu().numpy().astype(np.float64)[pick], ref)


# ---------------------------------------------------------------------------
# tensor-core forms (p = 16): bar = the oracle's truncation error + 1e-4 in relative L2
# (split BF16, three products); the single-product form is checked at 1e-2.
# ---------------------------------------------------------------------------
TC_BAR = {"bf16x3": 1e-4, "bf16": 1e-2}


def _prec(fmm, name):
    return {"bf16x3": fmm.FMM_TC_BF16X3, "bf16": fmm.FMM_TC_BF16}[name]


def _h2p_tc(fmm, g, ncut, sigma, A32, y, prec, G=None, accumulate=False):
    import torch

    yd = torch.from_numpy(np.ascontiguousarray(y, dtype=np.float64)).cuda()
    perm, start = _bin(fmm, g, yd)
    if G is None:
        G = torch.empty(len(y), dtype=torch.float32, device="cuda")
    fmm.fgt_h2p(g, ncut, 16, sigma, torch.from_numpy(A32).cuda(), yd, perm, start, G, accumulate=accumulate,
                prec=prec)
    fmm.fmm_sync_status()
    return G.cpu().numpy().astype(np.float64)


def _rel(got, ref):
    return np.linalg.norm(got - ref) / np.linalg.norm(ref)


@pytest.mark.parametrize("coarser", [0, 1])
@pytest.mark.parametrize("name", ["bf16x3", "bf16"])
@pytest.mark.parametrize("sigma,ncut", [(0.2, 10), (0.1, 10), (0.05, 10), (0.1, 3), (0.05, 1), (0.1, 0), (0.05, 15)])
def test_h2p_tc_matches_oracle(fmm, orc, gmm_sources, name, sigma, ncut, coarser):
    """A tensor-core precision: served in FP32 through the coefficients, and (coarser) by the tensor-core
    kernel, the cluster in several claims of 128 targets; there it differs from the FP32 sums."""
    x, q = gmm_sources
    g = workloads.fgt_grid_log2(sigma) - coarser
    rng = np.random.default_rng(ncut + int(sigma * 100))
    y = np.concatenate([rng.random((2500, 2)), 0.52 + 0.001 * rng.random((700, 2))])
    A32 = orc.fgt_p2h_grid(g, 16, sigma, x, q).astype(np.float32)
    got = _h2p_tc(fmm, g, ncut, sigma, A32, y, _prec(fmm, name))
    ref = orc.fgt_hermite_eval_grid(g, ncut, 16, sigma, A32.astype(np.float64), y)
    trunc = _rel(orc.fgt_hermite_eval_grid(g, ncut, 16, sigma, orc.fgt_p2h_grid(g, 16, sigma, x, q), y),
                 orc.fgt_direct(x, q, sigma, y)) if ncut == 10 else 0.0
    err = _rel(got, ref)
    assert err <= trunc + TC_BAR[name], f"relative L2 {err:.3e}"
    assert np.abs(got - ref).max() <= 10 * TC_BAR[name] * np.abs(ref).max()
    fp32 = _h2p_tc(fmm, g, ncut, sigma, A32, y, fmm.FMM_FP32)
    assert np.array_equal(got, fp32) == (not coarser)
    if coarser and name == "bf16":  # one product of operands rounded to 8 bits: not the split form either
        assert err >= 1e-4


def test_h2p_tc_ragged_counts_and_accumulate(fmm, orc, gmm_sources):
    import torch

    x, q = gmm_sources
    sigma, ncut = 0.1, 4
    g = workloads.fgt_grid_log2(sigma)
    A32 = orc.fgt_p2h_grid(g, 16, sigma, x, q).astype(np.float32)
    for n in (1, 127, 128, 129, 300):
        y = np.random.default_rng(n + 5).random((n, 2))
        ref = orc.fgt_hermite_eval_grid(g, ncut, 16, sigma, A32.astype(np.float64), y)
        assert _rel(_h2p_tc(fmm, g, ncut, sigma, A32, y, fmm.FMM_TC_BF16X3), ref) <= 1e-4
        G = torch.full((n,), 0.5, dtype=torch.float32, device="cuda")
        got = _h2p_tc(fmm, g, ncut, sigma, A32, y, fmm.FMM_TC_BF16X3, G=G, accumulate=True)
        assert _rel(got, ref + 0.5) <= 1e-4


def test_h2p_tc_agrees_with_fp32_path_at_full_size(fmm, orc):
    """2^20 mixture targets, sigma 0.05, n_cut 10, on 16 x 16 boxes (wide ones, which the direct kernels
    take): the tensor-core result against the FP32 kernel's everywhere and the oracle on 1,500 sampled
    targets, accumulated too."""
    import torch

    n = 1 << 20
    x, q = workloads.gmm_particles(n, np.random.default_rng(2024))
    y, _ = workloads.gmm_particles(n, np.random.default_rng(2025))
    sigma, ncut = 0.05, workloads.FGT_NCUT
    g = workloads.fgt_grid_log2(sigma) - 1
    xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    perm, _ = _bin(fmm, g, xd)
    A = torch.empty((4 ** g, 16, 16), dtype=torch.float32, device="cuda")
    fmm.fgt_p2h_binned(g, 16, sigma, xd, torch.from_numpy(q).cuda(), perm, A)
    tperm, tstart = _bin(fmm, g, yd)
    G32 = torch.empty(n, dtype=torch.float32, device="cuda")
    Gtc = torch.empty(n, dtype=torch.float32, device="cuda")
    fmm.fgt_h2p(g, ncut, 16, sigma, A, yd, tperm, tstart, G32)
    fmm.fgt_h2p(g, ncut, 16, sigma, A, yd, tperm, tstart, Gtc, prec=fmm.FMM_TC_BF16X3)
    fmm.fmm_sync_status()
    g32, gtc = G32.cpu().numpy().astype(np.float64), Gtc.cpu().numpy().astype(np.float64)
    assert 0.0 < _rel(gtc, g32) <= 1e-4
    pick = np.random.default_rng(6).choice(n, 1500, replace=False)
    ref = orc.fgt_hermite_eval_grid(g, ncut, 16, sigma, A.cpu().numpy().astype(np.float64), y[pick])
    assert _rel(gtc[pick], ref) <= 1e-4
    fmm.fgt_h2p(g, ncut, 16, sigma, A, yd, tperm, tstart, Gtc, prec=fmm.FMM_TC_BF16X3, accumulate=True)
    fmm.fmm_sync_status()
    assert _rel(Gtc.cpu().numpy().astype(np.float64), 2 * gtc) <= 1e-6


# ---------------------------------------------------------------------------
# evaluation through per-box Chebyshev coefficients: taken at >= 2 targets per box on average, on
# grids up to 256 x 256, for box sides of up to 1/2 (in sqrt2 sigma)
# ---------------------------------------------------------------------------
def _decaying(rng, nbox, p):
    import math

    fact = np.array([math.factorial(a) for a in range(p)], float)
    A = rng.standard_normal((nbox, p, p)) * (0.35 ** (np.arange(p)[:, None] + np.arange(p)[None, :])) / np.outer(fact, fact)
    A[rng.random(nbox) < 0.25] = 0.0
    A[0, 0, 0] = 1.0
    return A.astype(np.float32)


@pytest.mark.parametrize("p,d", [(4, 0.5), (8, 0.4), (8, 0.95), (12, 0.79), (12, 0.82), (16, 0.26), (16, 0.72),
                                 (16, 0.73), (16, 1.29), (16, 1.31), (16, 0.5), (16, 0.501)])
def test_h2p_on_both_sides_of_the_chebyshev_rule(fmm, orc, p, d):
    """Box sides d (in sqrt2 sigma) on both sides of the line (1/2) between the coefficients and the
    direct sum, and target counts on both sides of two per box; targets on box edges,
    at 1.0 and outside the unit square (summed directly), and crowded into one box.  The bar is
    the FP32 bar of the direct kernel: the interpolation adds at most 4e-10 of a Hermite function's
    largest value, against sums rounded to ~1e-7."""
    import math

    g = 3
    nbox, n = 4 ** g, 1 << g
    sigma = 2.0 ** -g / (math.sqrt(2.0) * d)
    rng = np.random.default_rng(int(1000 * d) + p)
    A32 = _decaying(rng, nbox, p)
    k = np.arange(n + 1) / n
    edge = np.stack([np.concatenate([k, np.nextafter(k, -1), rng.random(3)]),
                     np.concatenate([rng.random(2 * n + 2), [1.0, 1.01, -0.02]])], 1)
    for ncut in (0, 2, 16):
        for m in (2 * nbox - 1, 2 * nbox, 2000):
            y = np.concatenate([edge, 0.3 + 0.05 * rng.random((max(0, m // 2 - len(edge)), 2))])
            y = np.concatenate([y, rng.random((m - len(y), 2))])
            ref = orc.fgt_hermite_eval_grid(g, ncut, p, sigma, A32.astype(np.float64), y)
            _check(_h2p(fmm, g, ncut, p, sigma, A32, y), ref)


@pytest.mark.parametrize("g", [0, 1, 2, 5, 8])
def test_h2p_chebyshev_grid_sizes(fmm, orc, g):
    """1 x 1 boxes to the largest grid taken (256 x 256), accumulating; at 256 x 256 the targets
    checked are 800 of them."""
    import math
    import torch

    p, ncut, nbox = 8, 3, 4 ** g
    sigma = 2.0 ** -g / (math.sqrt(2.0) * 0.45)
    rng = np.random.default_rng(g)
    A32 = _decaying(rng, nbox, p)
    y = rng.random((max(700, 2 * nbox + 77), 2))
    G = torch.full((len(y),), 0.25, dtype=torch.float32, device="cuda")
    got = _h2p(fmm, g, ncut, p, sigma, A32, y, G=G, accumulate=True)
    pick = rng.choice(len(y), min(800, len(y)), replace=False)
    _check(got[pick], orc.fgt_hermite_eval_grid(g, ncut, p, sigma, A32.astype(np.float64), y[pick]) + 0.25)


@pytest.mark.parametrize("p", [4, 8, 12, 16])
@pytest.mark.parametrize("g,k", [(1, 1), (1, 10), (1, 15), (1, 16), (1, 40), (3, 150), (5, 3)])
def test_h2p_targets_outside_the_unit_square(fmm, orc, p, g, k):
    """k targets outside the unit square (the nearest box's, summed directly) among those of the boxes:
    few of a warp's targets (the warp shares the source boxes of each) and many (a lane each), with
    neighbourhoods of one box and of the whole grid."""
    import math

    rng = np.random.default_rng(100 * g + k)
    sigma = 2.0 ** -g / (math.sqrt(2.0) * 0.45)
    A32 = _decaying(rng, 4 ** g, p)
    y = rng.random((max(32 - k, 4 * 4 ** g), 2))
    out = rng.choice(len(y), min(k, len(y)), replace=False)
    y[out, 0] = np.where(rng.random(len(out)) < 0.5, 1.0 + 0.05 * rng.random(len(out)), -0.05 * rng.random(len(out)))
    for ncut in (0, 16):
        _check(_h2p(fmm, g, ncut, p, sigma, A32, y),
               orc.fgt_hermite_eval_grid(g, ncut, p, sigma, A32.astype(np.float64), y))


@pytest.mark.parametrize("p", [4, 16])
@pytest.mark.parametrize("g,ncut,n", [(0, 0, 5), (0, 16, 5), (0, 16, 700), (1, 16, 9), (1, 2, 500), (2, 15, 800),
                                      (3, 7, 2 ** 17 - 1), (3, 10, 2 ** 17)])
def test_h2p_neighbourhoods_wider_than_the_grid(fmm, orc, p, g, ncut, n):
    """n_cut beyond the grid's side (as many offsets as the grid has), and both sides of the line between one
    and four targets a lane; 500 targets against the oracle."""
    import math

    rng = np.random.default_rng(10 * g + ncut)
    sigma = 2.0 ** -g / (math.sqrt(2.0) * 0.45)
    A32 = _decaying(rng, 4 ** g, p)
    y = rng.random((n, 2))
    pick = rng.choice(n, min(n, 500), replace=False)
    _check(_h2p(fmm, g, ncut, p, sigma, A32, y)[pick],
           orc.fgt_hermite_eval_grid(g, ncut, p, sigma, A32.astype(np.float64), y[pick]))


def _per_target_terms(g, sigma, A, box, y):
    """Sum over one source box of |A_a1a2 h_a1(t1) h_a2(t2)| at each target, and t1^2 + t2^2, in 64 bits."""
    p, n = A.shape[-1], 1 << g
    t = (y - (np.array([box % n, box // n]) + 0.5) / n) / (np.sqrt(2.0) * sigma)
    h = [np.exp(-t * t), 2 * t * np.exp(-t * t)]
    for m in range(1, p - 1):
        h.append(2 * t * h[m] - 2 * m * h[m - 1])
    h = np.abs(np.stack(h[:p]))
    return np.einsum("ab,an,bn->n", np.abs(A.astype(np.float64)), h[:, :, 0], h[:, :, 1]), (t * t).sum(1)


@pytest.mark.parametrize("p,d,g", [(16, 0.6, 3), (16, 1.0, 3), (16, 1.28, 3), (8, 0.95, 3), (12, 0.8, 3), (4, 1.9, 2),
                                   (16, 0.5, 4), (12, 0.5, 4), (8, 0.44, 4), (4, 0.5, 4), (16, 0.36, 5)])
def test_h2p_each_target_keeps_its_own_accuracy(fmm, orc, p, d, g):
    """Sources in one corner box alone, targets all over the grid, down to values of 1e-30: each
    target's error against the size of its own terms, not of the largest target's.  FP32: t1^2 + t2^2
    are the exponents, whose rounding (two roundings of the argument, one of its scaling to a power of
    2, each 2^-24 relative) is an absolute error of the logarithm; p-term recurrences and sums on both
    axes and the function's own error: (4 p + 32 + 4 (t1^2 + t2^2)) units of 2^-24 (a 32-bit emulation
    of the direct sum reaches 0.46 of that)."""
    import math

    n, rng = 1 << g, np.random.default_rng(int(100 * d) + p)
    sigma = 2.0 ** -g / (math.sqrt(2.0) * d)
    x = rng.random((60, 2)) / n
    A32 = orc.fgt_p2h_grid(g, p, sigma, x, rng.random(60)).astype(np.float32)
    y = rng.random((max(1500, 4 * n * n), 2))
    ref = orc.fgt_hermite_eval_grid(g, 16, p, sigma, A32.astype(np.float64), y)
    size, t2 = _per_target_terms(g, sigma, A32[0], 0, y)
    got = _h2p(fmm, g, 16, p, sigma, A32, y)
    ok = size > 1e-30
    over = (np.abs(got - ref) / ((4 * p + 32 + 4 * t2) * 2.0 ** -24 * size))[ok]
    assert over.max() <= 1.0, f"{over.max():.3g} of the bound, {int((over > 1).sum())} targets above it"


def test_h2p_nan_coefficients_reach_their_neighbourhood_only(fmm, orc):
    """A NaN coefficient makes every target within n_cut boxes NaN and leaves the others as they
    are; a NaN coordinate gives NaN at that target alone."""
    import math

    g, p, ncut = 4, 8, 2
    n = 1 << g
    sigma = 2.0 ** -g / (math.sqrt(2.0) * 0.45)
    rng = np.random.default_rng(8)
    A32 = _decaying(rng, n * n, p)
    y = rng.random((3000, 2))
    y[17] = [np.nan, 0.5]
    ref = orc.fgt_hermite_eval_grid(g, ncut, p, sigma, A32.astype(np.float64), np.nan_to_num(y, nan=0.5))
    bad = 5 * n + 9
    A32[bad, 3, 2] = np.nan
    got = _h2p(fmm, g, ncut, p, sigma, A32, y)
    b = _boxes(np.nan_to_num(y, nan=0.0), g)
    near = (np.abs(b % n - bad % n) <= ncut) & (np.abs(b // n - bad // n) <= ncut)
    near[17] = True
    assert np.isnan(got[near]).all() and np.isfinite(got[~near]).all()
    _check(got[~near], ref[~near])


def test_h2p_first_call_of_a_grid_size_inside_a_capture(fmm, orc):
    """The coefficients' workspace of a grid size is allocated on its first use, inside a stream capture
    too: the graph replays what direct calls give, beside them."""
    import math
    import torch

    g, p, ncut = 7, 4, 1
    nbox = 4 ** g
    sigma = 2.0 ** -g / (math.sqrt(2.0) * 0.45)
    rng = np.random.default_rng(70)
    A32 = _decaying(rng, nbox, p)
    y = rng.random((2 * nbox + 5, 2))
    yd, Ad = torch.from_numpy(y).cuda(), torch.from_numpy(A32).cuda()
    perm, start = _bin(fmm, g, yd)
    fmm.fmm_prepare(8)  # the scratch of the direct sum
    G = torch.zeros(len(y), dtype=torch.float32, device="cuda")
    warm = torch.zeros(100, dtype=torch.float32, device="cuda")
    yw = yd[:100].contiguous()
    wperm, wstart = _bin(fmm, g, yw)
    fmm.fgt_h2p(g, ncut, p, sigma, Ad, yw, wperm, wstart, warm)  # few targets: the direct sum, loaded and set up
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        fmm.fgt_h2p(g, ncut, p, sigma, Ad, yd, perm, start, G)
    graph.replay()
    fmm.fmm_sync_status()
    first = G.clone()
    G.zero_()
    fmm.fgt_h2p(g, ncut, p, sigma, Ad, yd, perm, start, G)
    fmm.fmm_sync_status()
    second = G.clone()
    G.zero_()
    graph.replay()
    fmm.fmm_sync_status()
    pick = rng.choice(len(y), 600, replace=False)
    ref = orc.fgt_hermite_eval_grid(g, ncut, p, sigma, A32.astype(np.float64), y[pick])
    for t in (first, second, G):
        _check(t.cpu().numpy().astype(np.float64)[pick], ref)
    assert torch.equal(first, second) and torch.equal(first, G)


@pytest.mark.parametrize("prec", ["fp32", "bf16x3", "bf16"])
def test_h2p_captures_after_a_call_of_the_other_form(prec):
    """A program whose only call was served through the Chebyshev coefficients captures one that takes the
    direct sums (their scratch, and the tensor cores' image and tile table, come inside the
    capture), and one of a grid not used before: in a process of its own, where nothing else
    has been allocated."""
    import os
    import subprocess
    import sys

    code = f"""
import math, torch
from paper_1009_3457_gb300 import fmmgb as fmm
prec = {{"fp32": fmm.FMM_FP32, "bf16x3": fmm.FMM_TC_BF16X3, "bf16": fmm.FMM_TC_BF16}}[{prec!r}]
torch.manual_seed(1)
def problem(g, n):
    y = torch.rand((n, 2), dtype=torch.float64, device="cuda")
    i = dict(dtype=torch.int32, device="cuda")
    perm, start, work = torch.empty(n, **i), torch.empty(4 ** g + 1, **i), torch.empty(4 ** g, **i)
    fmm.fgt_bin_points(g, y, perm, start, work)
    A, G = torch.rand((4 ** g, 16, 16), device="cuda"), torch.empty(n, device="cuda")
    A *= 0.1 ** torch.arange(16, device="cuda")[:, None] * 0.1 ** torch.arange(16, device="cuda")
    sigma = 2.0 ** -g / (math.sqrt(2.0) * 0.45)
    return G, lambda: fmm.fgt_h2p(g, 3, 16, sigma, A, y, perm, start, G, prec=prec)
problem(4, 2000)[1]()
todo = [problem(4, 300), problem(5, 700), problem(5, 4000)]
torch.cuda.synchronize()
graphs = []
for G, call in todo:
    graphs.append(torch.cuda.CUDAGraph())
    with torch.cuda.graph(graphs[-1], capture_error_mode="thread_local"):
        call()
for graph, (G, call) in zip(graphs, todo):
    graph.replay()
    fmm.fmm_sync_status()
    got = G.clone()
    G.fill_(float("nan"))
    call()
    fmm.fmm_sync_status()
    assert torch.equal(got, G) and bool(torch.isfinite(G).all())
print("captured")
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "captured" in r.stdout, r.stdout + r.stderr


@pytest.mark.parametrize("p", [4, 8, 12, 16])
def test_p2h_and_t2p_binned_runs_and_alignments(fmm, orc, p):
    """P2H over 256-point blocks of one box, of several and of many, the last one ragged, into
    coefficients 16-byte aligned and not; T2P at the same points from coefficients aligned and not
    (several targets of one box together, and a box per lane)."""
    import torch

    g, sigma = 3, 0.2
    rng = np.random.default_rng(p)
    x = np.concatenate([0.51 + 0.01 * rng.random((700, 2)), 0.13 + 0.3 * rng.random((300, 2)), rng.random((411, 2)),
                        [[1.0, 0.4], [1.02, 0.7], [-0.01, 0.3]]])
    q = rng.uniform(-1, 1, len(x))
    ref = orc.fgt_p2h_grid(g, p, sigma, x, q)
    xd, qd = torch.from_numpy(x).cuda(), torch.from_numpy(q).cuda()
    perm, start = _bin(fmm, g, xd)
    m = 4 ** g * p * p
    ev = orc.fgt_taylor_eval_grid(g, p, sigma, ref.astype(np.float32).astype(np.float64), x)
    for shift in (0, 1):
        A = torch.full((m + 1,), float("nan"), dtype=torch.float32, device="cuda")[shift:shift + m].view(4 ** g, p, p)
        fmm.fgt_p2h_binned(g, p, sigma, xd, qd, perm, A)
        fmm.fmm_sync_status()
        got = A.cpu().numpy().astype(np.float64)
        assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= 1e-5
        A.copy_(torch.from_numpy(ref.astype(np.float32)))
        G = torch.zeros(len(x), dtype=torch.float32, device="cuda")
        fmm.fgt_t2p_binned(g, p, sigma, A, xd, perm, start, G)
        fmm.fmm_sync_status()
        _check(G.cpu().numpy().astype(np.float64), ev)


@pytest.mark.parametrize("p", [4, 8, 12, 16])
@pytest.mark.parametrize("g,n", [(0, 1), (0, 33), (2, 31), (2, 129), (5, 1000), (4, 2 ** 14 - 1), (4, 2 ** 14),
                                 (5, 2 ** 18 - 1), (5, 2 ** 18), (8, 3000)])
def test_t2p_binned_one_and_four_targets_a_lane(fmm, orc, p, g, n):
    """T2P on both sides of the lines between four lanes a target, one, and four targets a lane, from coefficients 16-byte aligned and
    not, added and written: boxes of one target and of many, the last warp ragged."""
    import torch

    rng = np.random.default_rng(1000 * g + p)
    sigma = 2.0 ** -g / (np.sqrt(2.0) * 0.4)
    C = rng.standard_normal((4 ** g, p, p)).astype(np.float32)
    y = np.concatenate([rng.random((n - n // 3, 2)), 0.3 + 0.2 * rng.random((n // 3, 2))])
    pick = rng.choice(n, min(n, 500), replace=False)
    ref = orc.fgt_taylor_eval_grid(g, p, sigma, C.astype(np.float64), y[pick])
    yd = torch.from_numpy(y).cuda()
    perm, start = _bin(fmm, g, yd)
    for shift in (0, 1):
        Cd = torch.empty(C.size + 1, device="cuda")[shift:shift + C.size].view(C.shape)
        Cd.copy_(torch.from_numpy(C))
        for acc in (False, True):
            G = torch.full((n,), 0.5, dtype=torch.float32, device="cuda")
            fmm.fgt_t2p_binned(g, p, sigma, Cd, yd, perm, start, G, accumulate=acc)
            fmm.fmm_sync_status()
            _check(G.cpu().numpy().astype(np.float64)[pick], ref + (0.5 if acc else 0.0))


def test_t2p_and_h2p_report_a_bad_box_start(fmm):
    """A box start out of range, or a box that ends before it starts, sets the error word; the other
    boxes' targets are evaluated."""
    import torch

    g, p = 3, 4
    y = torch.from_numpy(np.random.default_rng(2).random((600, 2))).cuda()
    perm, start = _bin(fmm, g, y)
    C = torch.zeros((4 ** g, p, p), dtype=torch.float32, device="cuda")
    C[:, 0, 0] = 1.0
    for b, v in ((5, -3), (40, 601), (20, 0)):
        bad = start.clone()
        bad[b] = v
        for call in (lambda G: fmm.fgt_t2p_binned(g, p, 0.2, C, y, perm, bad, G),
                     lambda G: fmm.fgt_h2p(g, 2, p, 0.2, C, y, perm, bad, G)):
            G = torch.zeros(600, dtype=torch.float32, device="cuda")
            call(G)
            with pytest.raises(fmm.FmmError) as e:
                fmm.fmm_sync_status()
            assert e.value.code == fmm.FMM_EDEVICE
            fmm.fmm_sync_status()
            assert int((G > 0).sum()) > 500


@pytest.mark.parametrize("g", [6, 7, 8, 9])
def test_bin_points_scans_over_many_blocks(fmm, g):
    """Grids whose prefix is taken by one block (64 x 64) and by many, a few boxes crowded."""
    import torch

    rng = np.random.default_rng(g)
    y = np.concatenate([rng.random((20000, 2)), 0.7 + 1e-4 * rng.random((5000, 2)), np.full((777, 2), 0.999999)])
    perm, start = _bin(fmm, g, torch.from_numpy(y).cuda())
    box = _boxes(y, g)
    np.testing.assert_array_equal(np.diff(start.cpu().numpy()), np.bincount(box, minlength=4 ** g))
    assert int(start[0]) == 0
    pm = perm.cpu().numpy()
    np.testing.assert_array_equal(box[pm], np.sort(box))
    assert np.array_equal(np.sort(pm), np.arange(len(y)))
