"""GPU parity of the far-field stages around the M2L path (fmm_l2l, fmm_l2p and
their adjoints, fmm_p2m_adjoint) against references built from the FP64 oracle
only: the oracle's L2L and L2P routines, explicit conjugate transposes of the
maps the oracle applies to unit vectors, and central differences of the
oracle's P2M.  Scaled units at the library boundary."""
import numpy as np
import pytest

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


def _dev(a, dtype=np.complex64):
    import torch

    return torch.from_numpy(np.ascontiguousarray(a, dtype=dtype)).cuda()


def _host(t):
    return t.cpu().numpy().astype(np.complex128)


def _rel(got, ref):
    return np.linalg.norm(got - ref) / np.linalg.norm(ref)


def _oracle_l2l_scaled(orc, child_level, p, Lp):
    """Scaled L2L of a whole level from the oracle's physical-unit L2L."""
    n = 1 << child_level
    Lc = np.zeros((n * n, p), dtype=np.complex128)
    phys = orc.unscale_le(Lp, child_level - 1)
    for iy in range(n):
        for ix in range(n):
            shift = orc.box_centre(child_level, ix, iy) - orc.box_centre(child_level - 1, ix // 2, iy // 2)
            Lc[iy * n + ix] = orc.l2l(p, phys[(iy // 2) * (n // 2) + ix // 2], shift)
    return orc.scale_le(Lc, child_level)


@pytest.mark.parametrize("p", [8, 16])
def test_l2l_and_adjoint(fmm, orc, p):
    rng = np.random.default_rng(p)
    cl = 4
    nb_p, nb_c = 4 ** (cl - 1), 4 ** cl
    Lp = rng.standard_normal((nb_p, p)) + 1j * rng.standard_normal((nb_p, p))
    X = rng.standard_normal((nb_c, p)) + 1j * rng.standard_normal((nb_c, p))
    Lcd = _dev(X)
    fmm.fmm_l2l(cl, p, _dev(Lp), Lcd, accumulate=True)
    fmm.fmm_sync_status()
    ref = _oracle_l2l_scaled(orc, cl, p, Lp)
    assert _rel(_host(Lcd) - X.astype(np.complex64), ref) <= 1e-6
    # adjoint: conj transpose of the oracle's map (applied to unit parent vectors)
    W = rng.standard_normal((nb_c, p)) + 1j * rng.standard_normal((nb_c, p))
    Wp = _dev(np.zeros((nb_p, p)))
    fmm.fmm_l2l_adjoint(cl, p, _dev(W), Wp)
    fmm.fmm_sync_status()
    n = 1 << cl
    T = {}
    for c in range(4):  # T_c[j][n] from unit inputs, one child per class
        ix, iy = c & 1, c >> 1
        cols = []
        for k in range(p):
            e = np.zeros((nb_p, p), dtype=np.complex128)
            e[0, k] = 1.0
            cols.append(_oracle_l2l_scaled(orc, cl, p, e)[iy * n + ix])
        T[c] = np.stack(cols, axis=1)
    ref = np.zeros((nb_p, p), dtype=np.complex128)
    for iy in range(n):
        for ix in range(n):
            c = (ix & 1) + 2 * (iy & 1)
            ref[(iy // 2) * (n // 2) + ix // 2] += T[c].conj().T @ W[iy * n + ix]
    assert _rel(_host(Wp), ref) <= 1e-6


def _points(rng, n, level):
    import torch

    z = rng.random((n, 2))
    side = 1 << level
    ix = np.minimum((z[:, 0] * side).astype(np.int64), side - 1)
    iy = np.minimum((z[:, 1] * side).astype(np.int64), side - 1)
    box = iy * side + ix
    return z, box, torch.from_numpy(z).cuda(), torch.full((n,), level, dtype=torch.int32).cuda(), \
        torch.from_numpy(box).cuda()


@pytest.mark.parametrize("p", [8, 16])
def test_l2p_and_adjoint(fmm, orc, p):
    import torch

    rng = np.random.default_rng(10 + p)
    level, npts = 5, 300
    nb = 4 ** level
    Ls = rng.standard_normal((nb, p)) + 1j * rng.standard_normal((nb, p))
    z, box, zd, levd, boxd = _points(rng, npts, level)
    phi = torch.empty(npts, dtype=torch.complex64, device="cuda")
    fmm.fmm_l2p(p, zd, levd, boxd, {level: _dev(Ls)}, level, phi)
    fmm.fmm_sync_status()
    side = 1 << level
    phys = orc.unscale_le(Ls, level)
    ref = np.array([orc.l2p(p, phys[b], orc.box_centre(level, int(b % side), int(b // side)),
                            np.array([z[j, 0] + 1j * z[j, 1]]))[0] for j, b in enumerate(box)])
    assert _rel(_host(phi), ref) <= 1e-6
    # adjoint: G[b][n] = sum_j conj(A_jn) cot_j with A_jn = phi_j for the unit LE e_n of box b
    cot = rng.standard_normal(npts) + 1j * rng.standard_normal(npts)
    G = _dev(np.zeros((nb, p)))
    fmm.fmm_l2p_adjoint(p, zd, levd, boxd, _dev(cot), {level: G}, level)
    fmm.fmm_sync_status()
    ref = np.zeros((nb, p), dtype=np.complex128)
    for j, b in enumerate(box):
        centre = orc.box_centre(level, int(b % side), int(b // side))
        for k in range(p):
            e = np.zeros((1, p), dtype=np.complex128)
            e[0, k] = 1.0
            a = orc.l2p(p, orc.unscale_le(e, level)[0], centre, np.array([z[j, 0] + 1j * z[j, 1]]))[0]
            ref[b, k] += np.conj(a) * cot[j]
    assert _rel(_host(G), ref) <= 1e-5


@pytest.mark.parametrize("p", [8, 16])
def test_l2p_binned_matches_oracle_and_per_point_kernel(fmm, orc, p):
    """fmm_l2p_binned (one block per box over the binned points) against the oracle's
    L2P at each point's box and the per-point kernel: points in random order, on box
    boundaries, at 1.0 and just outside the unit square (clamped boxes)."""
    import torch

    rng = np.random.default_rng(40 + p)
    level, npts = 5, 3000
    side, nb = 1 << level, 4 ** level
    z = rng.random((npts, 2))
    k = np.arange(side + 1) / side
    z[:side + 1, 0] = k
    z[side + 1:2 * side + 2, 1] = np.nextafter(k, -1.0)
    z[-3:] = [[1.0, 0.5], [1.004, 0.2], [-0.002, 0.7]]
    Ls = rng.standard_normal((nb, p)) + 1j * rng.standard_normal((nb, p))
    zd = torch.from_numpy(z).cuda()
    perm = torch.empty(npts, dtype=torch.int32, device="cuda")
    start = torch.empty(nb + 1, dtype=torch.int32, device="cuda")
    fmm.fmm_bin_points(level, zd, perm, start, torch.empty(nb, dtype=torch.int32, device="cuda"))
    phi = torch.empty(npts, dtype=torch.complex64, device="cuda")
    fmm.fmm_l2p_binned(level, p, zd, perm, start, _dev(Ls), phi)
    fmm.fmm_sync_status()
    ix = np.clip(np.floor(z[:, 0] * side), 0, side - 1).astype(np.int64)
    iy = np.clip(np.floor(z[:, 1] * side), 0, side - 1).astype(np.int64)
    phys = orc.unscale_le(Ls, level)
    ref = np.array([orc.l2p(p, phys[iy[j] * side + ix[j]], orc.box_centre(level, int(ix[j]), int(iy[j])),
                            np.array([z[j, 0] + 1j * z[j, 1]]))[0] for j in range(npts)])
    got = _host(phi)
    assert _rel(got, ref) <= 1e-6
    # the per-point kernel on the same boxes
    phi2 = torch.empty_like(phi)
    lev = torch.full((npts,), level, dtype=torch.int32, device="cuda")
    fmm.fmm_l2p(p, zd, lev, torch.from_numpy(iy * side + ix).cuda(), {level: _dev(Ls)}, level, phi2)
    fmm.fmm_sync_status()
    assert _rel(got, _host(phi2)) <= 1e-6
    # accumulate
    fmm.fmm_l2p_binned(level, p, zd, perm, start, _dev(Ls), phi, accumulate=True)
    fmm.fmm_sync_status()
    assert _rel(_host(phi), 2 * ref) <= 1e-6


def test_l2p_binned_coarse_levels_and_bad_bins(fmm):
    """Levels 0 and 1 carry no LEs (phi = 0, L may be None); a box_start that does not bin
    the points sets the device error word."""
    import torch

    z = torch.rand((50, 2), dtype=torch.float64, device="cuda")
    perm = torch.arange(50, dtype=torch.int32, device="cuda")
    phi = torch.full((50,), 3.0 + 1.0j, dtype=torch.complex64, device="cuda")
    start = torch.tensor([0, 50], dtype=torch.int32, device="cuda")
    fmm.fmm_l2p_binned(0, 8, z, perm, start, None, phi)
    fmm.fmm_sync_status()
    assert float(phi.abs().max()) == 0.0
    bad = torch.tensor([0, 10, 5, 20, 50], dtype=torch.int32, device="cuda")  # a box with end < first
    L1 = torch.zeros((4, 8), dtype=torch.complex64, device="cuda")
    fmm.fmm_l2p_binned(1, 8, z, perm, bad, L1, phi)
    with pytest.raises(fmm.FmmError) as e:
        fmm.fmm_sync_status()
    assert e.value.code == fmm.FMM_EDEVICE


def test_l2p_reports_bad_leaves(fmm, orc):
    import torch

    z = torch.rand((4, 2), dtype=torch.float64, device="cuda")
    lev = torch.tensor([3, 3, 9, 3], dtype=torch.int32, device="cuda")  # level 9 has no array
    box = torch.tensor([0, 63, 0, 64], dtype=torch.int64, device="cuda")  # box 64 is outside level 3
    L3 = torch.zeros((64, 8), dtype=torch.complex64, device="cuda")
    phi = torch.empty(4, dtype=torch.complex64, device="cuda")
    fmm.fmm_l2p(8, z, lev, box, {3: L3}, 3, phi)
    with pytest.raises(fmm.FmmError) as e:
        fmm.fmm_sync_status()
    assert e.value.code == fmm.FMM_EDEVICE
    assert float(phi.abs().max()) == 0.0


def test_p2m_adjoint_matches_central_differences(fmm, orc):
    """grad of J = Re sum_b sum_k conj(G[b][k]) M~_b[k](y) in each point's position."""
    import torch

    rng = np.random.default_rng(3)
    p, level, n = 12, 4, 40
    xy = rng.random((n, 2))
    c = rng.uniform(-1, 1, n)
    nb = 4 ** level
    G = rng.standard_normal((nb, p)) + 1j * rng.standard_normal((nb, p))
    grad = torch.zeros((n, 2), dtype=torch.float64, device="cuda")
    fmm.fmm_p2m_adjoint(level, p, torch.from_numpy(xy).cuda(), torch.from_numpy(c).cuda(), _dev(G), grad)
    fmm.fmm_sync_status()
    side = 1 << level
    h = 1e-7

    def J(i, pos):
        ix, iy = min(int(xy[i, 0] * side), side - 1), min(int(xy[i, 1] * side), side - 1)
        b = iy * side + ix
        m = orc.scale_me(orc.p2m_box(pos[None, :], c[i:i + 1], orc.box_centre(level, ix, iy), p)[None, :], level)[0]
        return float(np.real(np.sum(np.conj(G[b]) * m)))

    ref = np.zeros((n, 2))
    for i in range(n):
        for a in range(2):
            pp, pm = xy[i].copy(), xy[i].copy()
            pp[a] += h
            pm[a] -= h
            ref[i, a] = (J(i, pp) - J(i, pm)) / (2 * h)
    got = grad.cpu().numpy()
    assert np.linalg.norm(got - ref) <= 1e-6 * np.linalg.norm(ref), np.linalg.norm(got - ref) / np.linalg.norm(ref)


def test_m2m_adjoint(fmm, orc):
    """Conjugate transpose of M2M against the oracle's M2M applied to unit child vectors."""
    rng = np.random.default_rng(21)
    p, cl = 12, 4
    nb_c, nb_p = 4 ** cl, 4 ** (cl - 1)
    W = rng.standard_normal((nb_p, p)) + 1j * rng.standard_normal((nb_p, p))
    Wc = _dev(np.zeros((nb_c, p)))
    fmm.fmm_m2m_adjoint(cl, p, _dev(W), Wc)
    fmm.fmm_sync_status()
    n = 1 << cl
    ref = np.zeros((nb_c, p), dtype=np.complex128)
    for c in range(4):  # scaled M2M matrix of child class c: parent[j] from child[k]
        ix, iy = c & 1, c >> 1
        cols = []
        for k in range(p):
            e = np.zeros((nb_c, p), dtype=np.complex128)
            e[iy * n + ix, k] = 1.0
            Mp = orc.scale_me(orc.m2m_uniform(cl, p, orc.unscale_me(e, cl)), cl - 1)
            cols.append(Mp[0])
        T = np.stack(cols, axis=1)
        for py in range(n // 2):
            for px in range(n // 2):
                ref[(2 * py + iy) * n + 2 * px + ix] = T.conj().T @ W[py * (n // 2) + px]
    assert _rel(_host(Wc), ref) <= 1e-6


@pytest.mark.parametrize("p", [6, 7, 8, 12, 16, 24])
@pytest.mark.parametrize("cl", [1, 2, 5])
def test_child_parent_translations_of_every_order(fmm, p, cl):
    """M2M, L2L and their conjugate transposes against their entries in FP64, written and
    accumulated: the orders with the four children folded (the last block ragged at p = 6, 12, 24)
    and one (7) that takes the general kernels.  FP32 sums of at most 4 p products: 1e-6."""
    import math

    rng = np.random.default_rng(100 * cl + p)
    half, nc = 1 << (cl - 1), 1 << cl
    n = np.arange(p)
    C = np.array([[math.comb(a, b) if b <= a else 0 for b in range(p)] for a in range(p)], float)
    par = rng.standard_normal((half, half, p)) + 1j * rng.standard_normal((half, half, p))
    chl = rng.standard_normal((nc, nc, p)) + 1j * rng.standard_normal((nc, nc, p))
    par, chl = par.astype(np.complex64), chl.astype(np.complex64)
    up, upa = np.zeros((2, half, half, p), complex)
    dn, dna = np.zeros((2, nc, nc, p), complex)
    for cy in (0, 1):
        for cx in (0, 1):
            z = complex(cx - 0.5, cy - 0.5) / 2
            Z = np.where(n[:, None] >= n[None, :], z ** np.maximum(n[:, None] - n[None, :], 0), 0)
            M2M = C * Z * 0.5 ** n[None, :]            # parent j from child k
            L2L = (C * Z * 0.5 ** (n[None, :] + 1)).T  # child j from parent n
            sub = np.s_[cy::2, cx::2]
            up += chl[sub] @ M2M.T
            upa += chl[sub] @ L2L.conj()
            dn[sub] = par @ L2L.T
            dna[sub] = par @ M2M.conj()
    for f, src, ref in ((fmm.fmm_m2m, chl, up), (fmm.fmm_l2l_adjoint, chl, upa), (fmm.fmm_l2l, par, dn),
                        (fmm.fmm_m2m_adjoint, par, dna)):
        src, ref = src.reshape(-1, p), ref.reshape(-1, p)
        out = _dev(np.full(ref.shape, np.nan))
        f(cl, p, _dev(src), out)
        fmm.fmm_sync_status()
        assert _rel(_host(out), ref) <= 1e-6
        x = (rng.standard_normal(ref.shape) + 1j * rng.standard_normal(ref.shape)).astype(np.complex64)
        out = _dev(x)
        f(cl, p, _dev(src), out, accumulate=True)
        fmm.fmm_sync_status()
        assert _rel(_host(out), ref + x) <= 1e-6


def test_p2m_orders_and_alignments(fmm, orc):
    """Per-point P2M with 16-byte atomics (even p, aligned rows) and 4-byte ones (odd p, rows only
    8-byte aligned) against each other's FP64 sums."""
    import torch

    rng = np.random.default_rng(77)
    level, side = 3, 8
    xy = np.concatenate([rng.random((3000, 2)), 0.4 + 0.01 * rng.random((500, 2)), [[1.0, 0.2], [-0.01, 0.5]]])
    c = rng.uniform(-1, 1, len(xy))
    cell = np.clip(np.floor(xy * side), 0, side - 1)
    d = (xy * side - cell - 0.5) @ np.array([1, 1j])
    box = (cell[:, 1] * side + cell[:, 0]).astype(int)
    for p, shift in ((16, 0), (16, 1), (7, 0), (2, 0), (1, 0)):
        ref = np.zeros((side * side, p), complex)
        np.add.at(ref, box, c[:, None] * d[:, None] ** np.arange(p))
        buf = torch.full((side * side * p + 1,), float("nan"), dtype=torch.complex64, device="cuda")
        M = buf[shift:shift + side * side * p].view(side * side, p)
        fmm.fmm_p2m(level, p, torch.from_numpy(xy).cuda(), torch.from_numpy(c).cuda(), M)
        fmm.fmm_sync_status()
        assert _rel(_host(M), ref) <= 1e-6, (p, shift)


@pytest.mark.parametrize("p", [6, 7, 8, 12, 16, 24])
@pytest.mark.parametrize("lmin,lmax", [(2, 3), (2, 4), (0, 2), (3, 7), (2, 8), (6, 8)])
def test_level_passes_equal_the_per_level_calls(fmm, p, lmin, lmax):
    """A pass over several levels (the coarse ones in one launch of a cluster, the finer ones and the
    general orders level by level) writes what the per-level calls write, bit for bit."""
    import torch

    g = torch.Generator(device="cuda").manual_seed(100 * lmax + p)
    lv = list(range(lmin, lmax + 1))

    def data():
        return [torch.view_as_complex(torch.randn((4 ** l, p, 2), device="cuda", generator=g)) for l in lv]

    def down(f, X):
        for i in range(1, len(lv)):
            f(lv[i], p, X[i - 1], X[i], accumulate=True)

    def up(f, X, **kw):
        for i in range(len(lv) - 1, 0, -1):
            f(lv[i], p, X[i], X[i - 1], **kw)

    for op, ref in ((fmm.SHIFT_M2M, lambda X: up(fmm.fmm_m2m, X)),
                    (fmm.SHIFT_L2L_ADJOINT, lambda X: up(fmm.fmm_l2l_adjoint, X, accumulate=True)),
                    (fmm.SHIFT_L2L, lambda X: down(fmm.fmm_l2l, X)),
                    (fmm.SHIFT_M2M_ADJOINT, lambda X: down(fmm.fmm_m2m_adjoint, X))):
        X = data()
        Y = [x.clone() for x in X]
        ref(X)
        fmm._shift_levels(op, p, lmin, Y, None)
        fmm.fmm_sync_status()
        for l, a, b in zip(lv, X, Y):
            assert torch.equal(torch.view_as_real(a), torch.view_as_real(b)), (op, l)
