"""Differentiable far-field objective on a quadtree, for gradients with respect to
source positions (the P2M -> M2L -> L2L -> L2P chain of Sec. 2.1 stages 2-4).

    J = sum_j w_j Re phi_far(z_j),

phi_far(z) the local expansion of z's leaf, after M2L over the lists of every
level 2..depth and L2L down the tree, evaluated at z.  Every stage runs in the
library's kernels, forward and backward:

    forward   fmm_p2m (finest level) -> fmm_m2m (upward) -> fmm_m2l_levels -> fmm_l2l (downward)
              -> fmm_l2p
    backward  fmm_l2p_adjoint -> fmm_l2l_adjoint (upward) -> fmm_m2l_adjoint_levels (conjugate)
              -> fmm_m2m_adjoint (downward) -> fmm_p2m_adjoint, giving dJ/dx, dJ/dy per point.

Every level's MEs come from the finest level's P2M by M2M, which equals the
P2M of all points in each box (exact for truncated series); on an adaptive tree
the M2L reads existing boxes only, so a point contributes down to its leaf and
no further, which is the frozen-leaf assignment.  Units at the library boundary
are radius-scaled: M~_k = m_k / r^k, L~_n = l_n r^(n+1).
"""
from __future__ import annotations

import torch

from . import fmmgb


def leaf_boxes(tree, xy: torch.Tensor):
    """(level, box) of the deepest existing box containing each point (library
    kernel ``fmm_leaf_boxes``).  xy: [N, 2] float64 on the device; returns
    (int32, int64) device tensors."""
    xy = xy.contiguous()
    lev = torch.empty(xy.shape[0], dtype=torch.int32, device=xy.device)
    box = torch.empty(xy.shape[0], dtype=torch.int64, device=xy.device)
    fmmgb.fmm_leaf_boxes(tree, xy, lev, box)
    return lev, box


def _level_block(levels, p: int, device, zero: bool):
    """One complex64 allocation for the [4^l, p] arrays of `levels`, and each level's address (a tensor
    and an allocation per level cost the host more than the kernels they served)."""
    sizes = [4 ** l * p for l in levels]
    flat = (torch.zeros if zero else torch.empty)(sum(sizes), dtype=torch.complex64, device=device)
    at, out = flat.data_ptr(), []
    for n in sizes:
        out.append(at)
        at += 8 * n
    return flat, out


class FarFieldObjective(torch.autograd.Function):
    """J(xy) for fixed strengths, evaluation points and weights (see the module docstring)."""

    @staticmethod
    def forward(ctx, xy, tree, p, c, zxy, zlev, zbox, w):
        L = tree.max_level
        dev = xy.device
        st = fmmgb._stream(None)  # looked up once
        levels = list(range(2, L + 1))
        mem_m, Ms = _level_block(levels, p, dev, zero=False)
        fmmgb.fmm_p2m(L, p, xy, c, Ms[-1], stream=st)  # finest level, then M2M upward (exact for truncated series)
        fmmgb._shift_levels(fmmgb.SHIFT_M2M, p, 2, Ms, st)
        mem_l, Ls = _level_block(levels, p, dev, zero=tree.adaptive)  # M2L leaves absent boxes as they are
        fmmgb.fmm_m2l_levels(tree, 2, p, Ms, Ls, stream=st)
        fmmgb._shift_levels(fmmgb.SHIFT_L2L, p, 2, Ls, st)
        phi = torch.empty(zxy.shape[0], dtype=torch.complex64, device=dev)
        fmmgb.fmm_l2p(p, zxy, zlev, zbox, dict(zip(levels, Ls)), L, phi, stream=st)
        del mem_m, mem_l  # in use on the stream until here
        ctx.save_for_backward(xy, c, zxy, zlev, zbox, w)
        ctx.tree, ctx.p = tree, p
        return torch.sum(w * phi.real.to(torch.float64))

    @staticmethod
    def backward(ctx, gJ):
        xy, c, zxy, zlev, zbox, w = ctx.saved_tensors
        tree, p = ctx.tree, ctx.p
        L = tree.max_level
        levels = list(range(2, L + 1))
        dev = xy.device
        cot = (gJ * w).to(torch.complex64)  # dJ/dphi (real weights)
        st = fmmgb._stream(None)  # looked up once
        mem_g, Gs = _level_block(levels, p, dev, zero=True)
        fmmgb.fmm_l2p_adjoint(p, zxy, zlev, zbox, cot, dict(zip(levels, Gs)), L, stream=st)
        fmmgb._shift_levels(fmmgb.SHIFT_L2L_ADJOINT, p, 2, Gs, st)
        mem_w, Ws = _level_block(levels, p, dev, zero=tree.adaptive)
        fmmgb.fmm_m2l_adjoint_levels(tree, 2, p, Gs, Ws, conj=True, stream=st)
        fmmgb._shift_levels(fmmgb.SHIFT_M2M_ADJOINT, p, 2, Ws, st)  # M_l = M2M(M_{l+1}): coarse to fine
        grad = torch.empty_like(xy)  # every point is written
        fmmgb.fmm_p2m_adjoint(L, p, xy, c, Ws[-1], grad, stream=st)
        del mem_g, mem_w
        return grad, None, None, None, None, None, None, None


def far_field_objective(tree, p: int, xy: torch.Tensor, c: torch.Tensor, leaf, z: torch.Tensor, z_leaf,
                        w: torch.Tensor) -> torch.Tensor:
    """J (a 0-d float64 tensor), differentiable in xy ([N, 2] float64, CUDA).

    c: [N] float64 strengths; z: [Z] complex128 evaluation points; z_leaf: their
    (levels, boxes) from ``leaf_boxes``; w: [Z] float64 weights.  `leaf`, the
    sources' leaves, is implied by their positions (each point is binned at
    every level and absent boxes are skipped) and is accepted for symmetry."""
    del leaf
    zxy = torch.view_as_real(z.to(torch.complex128)).contiguous()
    zlev, zbox = z_leaf
    return FarFieldObjective.apply(xy.contiguous(), tree, p, c.contiguous(), zxy, zlev.to(torch.int32).contiguous(),
                                   zbox.to(torch.int64).contiguous(), w.contiguous())


class FmmPotential:
    """The whole FMM on a uniform tree to level L (Sec. 2.1 stages 2-5), every stage a
    library kernel: P2M at level L (on the binned points), M2M up, M2L over the interaction lists of levels 2..L,
    L2L down, L2P at each target's level-L box (on the binned targets), plus the near
    field (own and adjacent boxes) by ``fmm_p2p``.

        phi(z) = sum_i c_i / (z - y_i)   (sources at exactly z skipped)

    The near field and the far field up to L2L are independent: the near field runs on the
    current stream (writing phi, with FMM_P2P_SHARE_SM so that its blocks end after a few
    boxes), the far field on a second stream of higher priority, whose kernels take the places
    that free up, and L2P adds into phi once both are done.  Buffers are allocated once;
    ``__call__`` enqueues the whole evaluation, ending on the current stream (capturable as a
    CUDA graph after a first call)."""

    def __init__(self, tree, p: int, xy: torch.Tensor, c: torch.Tensor, z: torch.Tensor, prec: int = 0):
        if tree.adaptive or tree.periodic or tree.max_level < 2:
            raise ValueError("FmmPotential takes a uniform, non-periodic tree of depth >= 2")
        self.tree, self.p, self.prec = tree, p, prec
        self.L = L = tree.max_level
        dev = xy.device
        self.xy, self.c, self.z = xy.contiguous(), c.contiguous(), z.contiguous()
        self.levels = list(range(2, L + 1))
        # one allocation for the MEs and LEs, one for the binnings: a small problem's buffers cost the
        # host more than its kernels
        sizes = [4 ** l * p for l in self.levels]
        flat = torch.empty(2 * sum(sizes), dtype=torch.complex64, device=dev).split(sizes + sizes)
        arrays = [t.view(-1, p) for t in flat]
        self.Ms, self.Ls = arrays[:len(sizes)], arrays[len(sizes):]
        nb, n, nz = 4 ** L, self.xy.shape[0], self.z.shape[0]
        self.sperm, self.sstart, self.tperm, self.tstart, work = torch.empty(
            n + nz + 3 * nb + 2, dtype=torch.int32, device=dev).split([n, nb + 1, nz, nb + 1, nb])
        st = fmmgb._stream(None)
        fmmgb.fmm_bin_points(L, self.xy, self.sperm, self.sstart, work, stream=st)
        fmmgb.fmm_bin_points(L, self.z, self.tperm, self.tstart, work, stream=st)
        self.phi = torch.empty(nz, dtype=torch.complex64, device=dev)
        self.side = torch.cuda.Stream(device=dev, priority=-1)

    def __call__(self) -> torch.Tensor:
        p, L = self.p, self.L
        cur = torch.cuda.current_stream(self.phi.device)
        st, far = fmmgb._stream(None), self.side.cuda_stream
        self.side.wait_stream(cur)  # the inputs and the expansions are the current stream's until here
        fmmgb.fmm_p2p(L, self.xy, self.c, self.sperm, self.sstart, self.z, self.tperm, self.tstart, self.phi,
                      stream=st, share_sm=True)
        fmmgb.fmm_p2m_binned(L, p, self.xy, self.c, self.sperm, self.sstart, self.Ms[-1], stream=far)
        fmmgb._shift_levels(fmmgb.SHIFT_M2M, p, 2, self.Ms, far)
        fmmgb.fmm_m2l_levels(self.tree, 2, p, self.Ms, self.Ls, prec=self.prec, stream=far)
        fmmgb._shift_levels(fmmgb.SHIFT_L2L, p, 2, self.Ls, far)
        cur.wait_stream(self.side)
        fmmgb.fmm_l2p_binned(L, p, self.z, self.tperm, self.tstart, self.Ls[-1], self.phi, accumulate=True, stream=st)
        return self.phi
