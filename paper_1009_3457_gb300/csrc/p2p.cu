// p2p.cu -- the near field of a uniform quadtree at its finest level
// (Sec. 2.1 stage 5: Eq. n_body restricted to each target's own and adjacent
// boxes, the complement of the interaction lists of every level):
//
//   phi(z) (+)= sum_{i : box(y_i) adjacent to or equal box(z), y_i != z} c_i / (z - y_i).
//
// Targets and sources are binned by box (fmm_bin_points); a pre-pass copies the
// sources into box order, each as its position relative to its own box's
// centre in box sides (read off the bits of the FP64 position, kept in FP32)
// and strength, so a box's sources are one contiguous range and staging adds
// only the exact offset between box centres (-1, 0 or 1) -- no FP64
// arithmetic per staged source or per claim.  Runs of targets of one box are
// claimed from a table; two kernels take them:
//   - fmm_p2p_kernel, dense or crowded boxes, or few boxes: a CTA of 128 threads a claim of
//     up to 96 targets.  It gathers the sources of the 3 x 3 neighbourhood
//     into shared memory in batches, and each warp sums the run's targets (one to
//     three rows of 32, as many as the run fills, one target per lane and row)
//     against a quarter of every batch; the four partial sums of a target meet in
//     shared memory;
//   - fmm_p2p_warp_kernel, the sparse boxes where they are many: a warp a claim of up to 64 targets, eight
//     lanes for the targets and four for the sources, so that a run of 16 targets
//     fills the warp (a row of 32 lanes was half empty), and no barrier.
// In FP32:
//   1/(dx + i dy) = (dx - i dy) / r2 with one approximate reciprocal per pair,
// dx, dy in box sides, and the sums scaled by 2^level (exact) at the end.
// Positions relative to the target box keep |dx|, |dy| <= 1.5 box sides, so
// FP32 carries the difference of two nearby points to ~2^-24 of a box side.
// A source at the target's position (the point itself, when targets are the
// sources) contributes nothing: r^2 carries a 1e-30 offset and dx = dy = 0.
#include <algorithm>

#include "fgt_hermite.cuh"

namespace fmmgb {

constexpr int kP2pThreads = 128;
constexpr int kP2pWarps = kP2pThreads / 32;     // each takes a quarter of the sources
constexpr int kP2pR = 3;                        // targets per lane (rows of 32 targets per claim)
constexpr int kP2pRun = 32 * kP2pR;             // targets per claim
constexpr int kP2pBatch = 1024;                 // sources per shared-memory batch
// The CTA kernel's CTAs, and with FMM_P2P_SHARE_SM the warp kernel's, take one claim or a few each and
// end: kernels of a stream of higher priority take their places, and no claim waits behind a heavy one
// that a persistent CTA holds.  The potential of 2^22 points with the far field beside it: 1,240 us with
// persistent CTAs (8 per SM), 1,167 / 1,157 / 1,163 / 1,169 with 1 / 2 / 3 / 4 claims; the near field alone, persistent
// and so: 2^22 uniform points at level 8 939 and 915, 2^19 clustered at level 7 696 and 530, 2^17 at level 6 218 and
// 181.  Where few, a CTA each: two a CTA left SMs idle (2^15 clustered points at level 5 80 us and 57).
// A warp a claim loses alone (2^22 points at level 9 689 -> 731), so that without the flag the warp kernel
// persists.
constexpr int kP2pShareOne = 1 << 14;           // claims: a CTA (warp) each up to here, beyond it two
constexpr int kP2pShareGrid = 1 << 16;          // more claims a CTA rather than more CTAs (most find none)
// CTAs per SM of the CTA kernel beside the warp kernel (four times the resident ones): 16 / 32 / 64 for 2^20 clustered points at level 8 642 / 601 /
// 566 us, for 2^18 uniform ones at level 7, which leave it nothing, 66 / 68 / 73 (64 before it).
constexpr int kP2pSplitGrid = 36;
// With the flag a call of few claims, or beside the warp kernel, leaves room on each SM: shared memory for 7
// CTAs of the CTA kernel where registers allow 9, since among crowded boxes a claim lasts tens of
// microseconds and the other stream's kernels wait for it (the whole potential of 2^17 clustered points at
// level 6 263 -> 224 us, uniform 61 both; 2^22 uniform points lose, 1,106 -> 1,183).
constexpr int kP2pRoomSmem = 12 << 10;
// The warp kernel takes calls of fewer than kP2pDense targets a box on average, on kP2wBoxes boxes or
// more (fewer claims than warps otherwise).  us, CTA / warp: 16 a box at level 5 26 / 35, level 6 31 / 35,
// level 7 68 / 62, level 8 216 / 170, level 9 914 / 676; 32 a box at level 6 41 / 55, level 7 105 / 110,
// level 8 374 / 344; 64 a box at level 8 931 / 1,038.
constexpr int kP2pDense = 32, kP2wBoxes = 1 << 14;
// And of such a call only the boxes with fewer than kP2wBoxTargets targets and kP2wSources sources around
// them; the others go to the CTA kernel, beside it.  (All boxes to the warp kernel left its warps waiting
// for the crowded ones; us, before the warp kernel / that / so, Gaussian mixtures: 2^18 points at level 7 250 / 450 / 200,
// at level 8 153 / 213 / 87, 2^20 at level 8 709 / 1,004 / 550, at level 9 501 / 430 / 255.  32 / 48 / 64 targets
// with ordinary launches: 264 / 275 / 302, 133 / 143 / 172, 682 / 706 / 743, 319 / 341 / 418; 512 to 2,048 sources
// measured alike.)
constexpr int kP2wBoxTargets = 32, kP2wSources = 1024;
// the warp kernel
constexpr int kP2wLanes = 8;                    // target lanes; the other factor 4 splits the sources
constexpr int kP2wSplit = 32 / kP2wLanes;
constexpr int kP2wPairs = 4;                    // packed target pairs per lane, at most
constexpr int kP2wRun = 2 * kP2wLanes * kP2wPairs;  // targets per claim
constexpr int kP2wChunk = 96;                   // sources per staging buffer of a warp
constexpr int kP2wCtas = 7;                     // resident CTAs per SM (72 registers)
// added to every r^2 (in box sides squared): a source at the target's position
// (dx = dy = 0) then contributes exactly 0 -- c / 1e-30 is finite for |c| < 3e8 -- and
// any other pair changes by a relative 1e-30 / r^2 (below FP32 rounding for distances
// above 1e-11 box sides; positions resolve 2^-31 of a side, 4.7e-10)
constexpr float kP2pTiny = 1e-30f;

struct P2pArgs {
    int level, n, nz, accumulate;
    const float4* src;  // sources in box order: x, y relative to their own box's centre, c (p2p_sort_kernel)
    const int* sstart;
    const double* z;
    const int* tperm;
    const int* nclaim;  // claims in the table
    const int4* tab;    // claim table (p2p_claim_table_kernel), room for ntab entries
    int ntab;
    float2* phi;
    int* cursor;  // of the warp kernel: [0] next claim index, [1] warps finished; NULL: a warp takes every
                  // (number of warps)-th place of the table and ends
    int go;       // the other kernel may start beside this one
    int* err;
};

// sources in box order, so that a box's sources are one contiguous range; positions relative to
// the centre of their own box in box sides, read off the bits of the FP64 coordinates and kept
// in FP32 (|x - c| <= 1/2)
__global__ void p2p_sort_kernel(int level, const double* __restrict__ xy, const double* __restrict__ c,
                                const int* __restrict__ perm, int n, float4* __restrict__ out, int* err)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int i = __ldg(perm + k);
    if ((unsigned)i >= (unsigned)n) {
        atomicOr(err, DEV_ERR_CHECK);
        out[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    const double x = __ldg(xy + 2 * (size_t)i), y = __ldg(xy + 2 * (size_t)i + 1);
    const float cf = (float)__ldg(c + i);
    long long X, Y;
    if (grid_fixed31(x, level, X) && grid_fixed31(y, level, Y)) {
        out[k] = make_float4(cell_offset31(X), cell_offset31(Y), cf, 0.f);  // offset in box sides
        return;
    }
    // outside the unit square: the clamped box, offset in FP64 (x 2^level is exact)
    const int side = 1 << level;
    const double px = x * side, py = y * side;
    const int ix = !(px >= 0.0) ? 0 : (px >= side ? side - 1 : (int)px);
    const int iy = !(py >= 0.0) ? 0 : (py >= side ? side - 1 : (int)py);
    out[k] = make_float4((float)(px - (ix + 0.5)), (float)(py - (iy + 0.5)), cf, 0.f);
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Packed two-lane FP32 (PTX f32x2): two targets of a lane in one 64-bit register pair.
__device__ __forceinline__ unsigned long long p2_pk(float a, float b)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 p2_upk(unsigned long long v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ unsigned long long p2_sub(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long p2_add(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long p2_mul(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long p2_fma(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// One warp's share of a staged batch (sources warp, warp + 4, ...) against the
// claim's NR occupied rows of 32 targets (NR warp-uniform: empty rows cost nothing).
// Rows 0 and 1 run as one packed pair (dx, dy, r^2, the weight and both sums in
// f32x2 operations; the two reciprocals stay scalar), row 2 alone.
template <int NR>
__device__ __forceinline__ void p2p_batch(const float4* __restrict__ s_src, int cnt, int warp, const float* zx,
                                          const float* zy, float* re, float* im)
{
    if constexpr (NR >= 2) {
        const unsigned long long zx01 = p2_pk(zx[0], zx[1]), zy01 = p2_pk(zy[0], zy[1]);
        const unsigned long long tiny = p2_pk(kP2pTiny, kP2pTiny);
        unsigned long long re01 = p2_pk(re[0], re[1]), im01 = p2_pk(-im[0], -im[1]);  // im01 sums +w dy
        float re2 = NR > 2 ? re[2] : 0.f, im2 = NR > 2 ? im[2] : 0.f;
#pragma unroll 8
        for (int i = warp; i < cnt; i += kP2pWarps) {
            const float4 v = s_src[i];
            const unsigned long long dx = p2_sub(zx01, p2_pk(v.x, v.x)), dy = p2_sub(zy01, p2_pk(v.y, v.y));
            const float2 r2 = p2_upk(p2_fma(dx, dx, p2_fma(dy, dy, tiny)));
            const unsigned long long w = p2_mul(p2_pk(v.z, v.z), p2_pk(rcp_approx(r2.x), rcp_approx(r2.y)));
            re01 = p2_fma(w, dx, re01);
            im01 = p2_fma(w, dy, im01);
            if constexpr (NR > 2) {
                const float ex = zx[2] - v.x, ey = zy[2] - v.y;
                const float q2 = fmaf(ex, ex, fmaf(ey, ey, kP2pTiny));
                const float u = v.z * rcp_approx(q2);
                re2 = fmaf(u, ex, re2);
                im2 = fmaf(-u, ey, im2);
            }
        }
        const float2 a = p2_upk(re01), b = p2_upk(im01);
        re[0] = a.x;
        re[1] = a.y;
        im[0] = -b.x;
        im[1] = -b.y;
        if constexpr (NR > 2) {
            re[2] = re2;
            im[2] = im2;
        }
    } else {
#pragma unroll 4
        for (int i = warp; i < cnt; i += kP2pWarps) {
            const float4 v = s_src[i];
            const float dx = zx[0] - v.x, dy = zy[0] - v.y;
            const float r2 = fmaf(dx, dx, fmaf(dy, dy, kP2pTiny));
            const float w = v.z * rcp_approx(r2);
            re[0] = fmaf(w, dx, re[0]);
            im[0] = fmaf(-w, dy, im[0]);
        }
    }
}

// Claim table: one entry (first, end, box) per run of targets of one box, a box's targets cut
// into runs of at most `most`, alike in whole rows of `row` targets (runs alike in targets leave every
// run's last row half empty: 320 targets in 12 rows of 32 instead of 10; 2^22 points in a band of 1/20 of the square at
// level 9 3,834 -> 3,437 us).  The runs of a warp's 32 boxes take consecutive places
// from one addition to *nclaim (zero before); the order of the table only sets the order in
// which claims are taken.  Places past `cap`, or a box_start that does not bin [0, nz), set the
// error word (and those runs are skipped).  (A scan of the boxes' counts by one block, to give every
// run a place of its own, took 73 us at 256 x 256 boxes and 290 us at 512 x 512.)
struct P2pTable {
    int row, most, cap;
    int* nclaim;
    int4* tab;
};

// The whole warp: the runs of its boxes (n of [f, e) each) into the table.
__device__ __forceinline__ void p2p_append(const P2pTable& t, int n, int f, int e, int b, int* err)
{
    const int lane = threadIdx.x & 31;
    int x = n;  // inclusive scan over the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += v;
    }
    int at = 0;
    if (lane == 31 && x > 0) at = atomicAdd(t.nclaim, x);
    at = __shfl_sync(0xffffffffu, at, 31) + x - n;
    if (n <= 0) return;
    const int64_t rows = (e - f + t.row - 1) / t.row;
    for (int k = 0; k < n; ++k) {
        if ((unsigned)(at + k) >= (unsigned)t.cap) {
            atomicOr(err, DEV_ERR_CHECK);
            return;
        }
        t.tab[at + k] = make_int4(f + t.row * (int)(k * rows / n), min(f + t.row * (int)((k + 1) * rows / n), e), b, 0);
    }
}

// cta: the runs of the CTA kernel; warp: of the warp kernel (cap 0: every box to the CTA kernel).
__global__ void p2p_claim_table_kernel(int level, const int* __restrict__ tstart, int nz, const int* __restrict__ sstart,
                                       P2pTable cta, P2pTable warp, int* err)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x, side = 1 << level, nbox = side * side;
    int f = 0, e = 0;
    if (b < nbox) {
        f = tstart[b];
        e = tstart[b + 1];
        if (f < 0 || e > nz || f > e) {
            atomicOr(err, DEV_ERR_CHECK);
            e = min(e, nz);
            if (f < 0 || f > e) f = e = 0;
        }
    }
    const int m = e - f;
    bool sparse = false;
    if (warp.cap) {
        sparse = m < kP2wBoxTargets;
        if (sparse && m > 0) {  // the sources of the 3 x 3 neighbourhood: a run of boxes a row
            const int tx = b & (side - 1), ty = b >> level;
            int64_t src = 0;
            for (int y = max(ty - 1, 0); y <= min(ty + 1, side - 1); ++y)
                src += (int64_t)sstart[y * side + min(tx + 1, side - 1) + 1] - sstart[y * side + max(tx - 1, 0)];
            sparse = src < kP2wSources;
        }
        p2p_append(warp, sparse ? (m + warp.most - 1) / warp.most : 0, f, e, b, err);
    }
    p2p_append(cta, sparse ? 0 : (m + cta.most - 1) / cta.most, f, e, b, err);
}

// (The arguments as a grid constant: 2^22 points at level 8 947 -> 911 us.)
__global__ void __launch_bounds__(kP2pThreads) fmm_p2p_kernel(const __grid_constant__ P2pArgs a)
{
    __shared__ float4 s_src[kP2pBatch];  // position relative to the target box's centre (box sides), c
    __shared__ int4 s_claim;
    __shared__ int s_box[9], s_cnt[9];  // first sorted source and source count of each neighbour box
    __shared__ float s_ox[9], s_oy[9];  // centre of each neighbour box minus the target box's (box sides)
    __shared__ float2 s_part[kP2pWarps - 1][kP2pRun];  // partial sums of warps 1..3

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int side = 1 << a.level;
    if (a.go) after_go();
    const int total = min(__ldg(a.nclaim), a.ntab);
    if (total <= 0) return;  // the same for every CTA
    for (int k = blockIdx.x;; k += gridDim.x) {
        if (tid == 0) s_claim = k < total ? __ldg(a.tab + k) : make_int4(-1, -1, 0, 0);
        __syncthreads();
        const int4 cl = s_claim;
        const int first = cl.x, end = cl.y, box = cl.z;
        if (first < 0) break;
        const int nrow = (end - first + 31) >> 5;  // occupied rows of 32 targets (0..kP2pR)
        const int tx = box & (side - 1), ty = box >> a.level;
        if (tid < 9) {  // the 3 x 3 neighbourhood, one box per thread
            const int sx = tx + tid % 3 - 1, sy = ty + tid / 3 - 1;
            s_ox[tid] = (float)(tid % 3 - 1);
            s_oy[tid] = (float)(tid / 3 - 1);
            int b0 = -1, m = 0;
            if (sx >= 0 && sy >= 0 && sx < side && sy < side) {
                const int b = sy * side + sx;
                b0 = __ldg(a.sstart + b);
                m = __ldg(a.sstart + b + 1) - b0;
                if (m <= 0 || b0 < 0 || b0 + m > a.n) {
                    b0 = -1;
                    m = 0;
                }
            }
            s_box[tid] = b0;
            s_cnt[tid] = m;
        }

        int tj[kP2pR];
        float zx[kP2pR], zy[kP2pR], re[kP2pR], im[kP2pR];
#pragma unroll
        for (int r = 0; r < kP2pR; ++r) {
            const int pos = first + r * 32 + lane;
            tj[r] = -1;
            zx[r] = zy[r] = re[r] = im[r] = 0.f;
            if (pos < end) {
                const int j = __ldg(a.tperm + pos);
                if ((unsigned)j < (unsigned)a.nz) {
                    tj[r] = j;
                    const double x = __ldg(a.z + 2 * (size_t)j), y = __ldg(a.z + 2 * (size_t)j + 1);
                    long long X, Y;
                    if (grid_fixed31(x, a.level, X) && grid_fixed31(y, a.level, Y) && (int)(X >> 31) == tx &&
                        (int)(Y >> 31) == ty) {
                        zx[r] = cell_offset31(X);  // in the claimed box: no FP64 arithmetic
                        zy[r] = cell_offset31(Y);
                    } else {  // outside it (coordinates outside the unit square): FP64, x 2^level exact
                        zx[r] = (float)(x * side - (tx + 0.5));
                        zy[r] = (float)(y * side - (ty + 0.5));
                    }
                } else if (warp == 0) {
                    atomicOr(a.err, DEV_ERR_CHECK);
                }
            }
        }
        __syncthreads();
        int pre[10];  // prefix of the neighbour boxes' source counts
        pre[0] = 0;
#pragma unroll
        for (int q = 0; q < 9; ++q) pre[q + 1] = pre[q] + s_cnt[q];
        const int S = pre[9];

        for (int base = 0; base < S; base += kP2pBatch) {
            const int cnt = min(kP2pBatch, S - base);
            for (int i = tid; i < cnt; i += kP2pThreads) {
                const int g = base + i;
                int q = 0;
#pragma unroll
                for (int t = 1; t < 9; ++t) q += pre[t] <= g;  // the neighbour box holding source g
                const int b0 = s_box[q];
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (b0 >= 0) {
                    int off = 0;  // pre[q], with registers indexed by constants only
#pragma unroll
                    for (int t = 1; t < 9; ++t) off = t == q ? pre[t] : off;
                    const float4 u = a.src[b0 + (g - off)];
                    v.x = u.x + s_ox[q];
                    v.y = u.y + s_oy[q];
                    v.z = u.z;
                }
                s_src[i] = v;
            }
            __syncthreads();
            switch (nrow) {
                case 0: break;  // a run the claim table flagged (error word set)
                case 1: p2p_batch<1>(s_src, cnt, warp, zx, zy, re, im); break;
                case 2: p2p_batch<2>(s_src, cnt, warp, zx, zy, re, im); break;
                default: p2p_batch<3>(s_src, cnt, warp, zx, zy, re, im); break;
            }
            __syncthreads();  // the batch buffer is refilled next
        }
        if (warp > 0) {
#pragma unroll
            for (int r = 0; r < kP2pR; ++r)
                if (r < nrow) s_part[warp - 1][r * 32 + lane] = make_float2(re[r], im[r]);
        }
        __syncthreads();
        if (warp > 0) continue;  // warp 0 writes; every warp is back at the claim's barrier next
#pragma unroll
        for (int r = 0; r < kP2pR; ++r) {
            if (tj[r] < 0) continue;
            float2 o = make_float2(re[r], im[r]);
#pragma unroll
            for (int q = 0; q < kP2pWarps - 1; ++q) {
                o.x += s_part[q][r * 32 + lane].x;
                o.y += s_part[q][r * 32 + lane].y;
            }
            o.x *= (float)side;  // 1/(z - y) = 2^level / ((z - y) in box sides): exact scaling
            o.y *= (float)side;
            if (a.accumulate) {
                const float2 old = a.phi[tj[r]];
                o.x += old.x;
                o.y += old.y;
            }
            a.phi[tj[r]] = o;
        }
    }
}

__device__ __forceinline__ void p2p_copy16(void* smem, const void* gmem)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}

// A warp's claim: m <= 16 NP targets of box (tx, ty) from place `first` on, against the 3 x 3
// neighbourhood, lane q < 9 holding box q's first sorted source b0 and count n.  A lane keeps 2 NP
// targets as packed pairs (dx, dy, r^2, the weight and both sums in f32x2 operations, the two
// reciprocals scalar) and takes every fourth source.  A box's sources are one run of the sorted
// array; the warp copies them into one of its two buffers asynchronously while it sums the other.
// im sums +w dy.
template <int NP>
__device__ __forceinline__ void p2p_claim(const P2pArgs& a, int first, int m, int tx, int ty, int b0, int n,
                                          float4* buf)
{
    const int lane = threadIdx.x & 31, tl = lane & (kP2wLanes - 1), sl = lane / kP2wLanes;
    const int side = 1 << a.level;
    unsigned long long zx[NP], zy[NP], re[NP], im[NP];
    auto target = [&](int k) {  // index of the lane's target k (-1: none)
        const int t = kP2wLanes * k + tl;
        const int j = t < m ? a.tperm[first + t] : -1;
        return (unsigned)j < (unsigned)a.nz ? j : -1;
    };
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        float2 z[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = target(2 * p + h);
            z[h] = make_float2(0.f, 0.f);
            if (j < 0) {
                if (kP2wLanes * (2 * p + h) + tl < m) atomicOr(a.err, DEV_ERR_CHECK);
                continue;
            }
            const double x = a.z[2 * (size_t)j], y = a.z[2 * (size_t)j + 1];
            long long X, Y;
            if (grid_fixed31(x, a.level, X) && grid_fixed31(y, a.level, Y) && (int)(X >> 31) == tx &&
                (int)(Y >> 31) == ty) {
                z[h] = make_float2(cell_offset31(X), cell_offset31(Y));  // in the claimed box: no FP64 arithmetic
            } else {  // outside it (coordinates outside the unit square): FP64, x 2^level exact
                z[h] = make_float2((float)(x * side - (tx + 0.5)), (float)(y * side - (ty + 0.5)));
            }
        }
        zx[p] = p2_pk(z[0].x, z[1].x);
        zy[p] = p2_pk(z[0].y, z[1].y);
        re[p] = im[p] = 0ull;
    }
    const unsigned long long tiny = p2_pk(kP2pTiny, kP2pTiny);
    // the neighbourhood's sources, box by box in pieces of up to kP2wChunk: piece [at, at + cnt) of box q
    int q = -1, at = 0, s1 = 0, cnt = 0;
    float ox = 0.f, oy = 0.f;
    auto next = [&](float4* buf) {  // the next piece, its copies issued (one group, empty past the end)
        at += cnt;
        while (at >= s1 && q < 8) {
            ++q;
            at = __shfl_sync(0xffffffffu, b0, q);
            s1 = at + __shfl_sync(0xffffffffu, n, q);
        }
        cnt = min(kP2wChunk, s1 - at);
        ox = (float)(q % 3 - 1);  // the box's centre from the target box's
        oy = (float)(q / 3 - 1);
        for (int i = lane; i < cnt; i += 32) p2p_copy16(buf + i, a.src + at + i);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    next(buf);
    for (int k = 0; cnt > 0; k ^= 1) {
        const float4* cur = buf + k * kP2wChunk;
        const int m0 = cnt;
        const float cx = -ox, cy = -oy;
        next(buf + (k ^ 1) * kP2wChunk);
        asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        __syncwarp();
#pragma unroll 2
        for (int i = sl; i < m0; i += kP2wSplit) {
            const float4 u = cur[i];
            const float x = cx - u.x, y = cy - u.y;
            const unsigned long long vx = p2_pk(x, x), vy = p2_pk(y, y), c = p2_pk(u.z, u.z);
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const unsigned long long dx = p2_add(zx[p], vx), dy = p2_add(zy[p], vy);
                const float2 r2 = p2_upk(p2_fma(dx, dx, p2_fma(dy, dy, tiny)));
                const unsigned long long w = p2_mul(c, p2_pk(rcp_approx(r2.x), rcp_approx(r2.y)));
                re[p] = p2_fma(w, dx, re[p]);
                im[p] = p2_fma(w, dy, im[p]);
            }
        }
        __syncwarp();  // the buffer has been read
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        const float2 r = p2_upk(re[p]), i = p2_upk(im[p]);
        float v[4] = {r.x, i.x, r.y, i.y};
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int o = kP2wLanes; o < 32; o <<= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (sl != (2 * p + h) % kP2wSplit) continue;  // the source lanes share the stores
            const int j = target(2 * p + h);
            if (j < 0) continue;
            // 1/(z - y) = 2^level / ((z - y) in box sides): exact scaling
            float2 o = make_float2(v[2 * h] * (float)side, -v[2 * h + 1] * (float)side);
            if (a.accumulate) {
                const float2 old = a.phi[j];
                o.x += old.x;
                o.y += old.y;
            }
            a.phi[j] = o;
        }
    }
}

// Runs beside the CTA kernel of the same call, in the room that one leaves (nothing it reads is
// written by that kernel).
__global__ void __launch_bounds__(kP2pThreads, kP2wCtas) fmm_p2p_warp_kernel(const __grid_constant__ P2pArgs a)
{
    __shared__ float4 s_src[kP2pThreads / 32][2 * kP2wChunk];  // two staging buffers a warp
    const int lane = threadIdx.x & 31;
    float4* buf = s_src[threadIdx.x >> 5];
    const int side = 1 << a.level;
    const int total = min(*a.nclaim, a.ntab);
    // lane 0 fetches the index of the warp's next claim one claim ahead
    const int warp = (int)blockIdx.x * (kP2pThreads / 32) + (threadIdx.x >> 5), nwarp = (int)gridDim.x * (kP2pThreads / 32);
    int knext = !a.cursor ? warp : lane == 0 ? atomicAdd(a.cursor, 1) : 0;
    for (;;) {
        const int k = __shfl_sync(0xffffffffu, knext, 0);
        if (k >= total) break;
        if (lane == 0) knext = !a.cursor ? k + nwarp : atomicAdd(a.cursor, 1);
        const int4 cl = a.tab[k];
        const int first = cl.x, m = cl.y - cl.x, box = cl.z;
        const int tx = box & (side - 1), ty = box >> a.level;
        int b0 = 0, n = 0;
        if (lane < 9) {  // the 3 x 3 neighbourhood, one box per lane
            const int sx = tx + lane % 3 - 1, sy = ty + lane / 3 - 1;
            if (sx >= 0 && sy >= 0 && sx < side && sy < side) {
                const int b = sy * side + sx;
                b0 = a.sstart[b];
                n = a.sstart[b + 1] - b0;
                if (n < 0 || b0 < 0 || b0 + n > a.n) {
                    atomicOr(a.err, DEV_ERR_CHECK);
                    b0 = n = 0;
                }
            }
        }
        switch ((m + 2 * kP2wLanes - 1) / (2 * kP2wLanes)) {
            case 1: p2p_claim<1>(a, first, m, tx, ty, b0, n, buf); break;
            case 2: p2p_claim<2>(a, first, m, tx, ty, b0, n, buf); break;
            case 3: p2p_claim<3>(a, first, m, tx, ty, b0, n, buf); break;
            default: p2p_claim<4>(a, first, m, tx, ty, b0, n, buf); break;
        }
    }
    // the last warp to finish returns the cursor slot to zero for its next use
    if (lane == 0 && a.cursor) {
        __threadfence();
        if (atomicAdd(a.cursor + 1, 1) == (int)gridDim.x * (kP2pThreads / 32) - 1) {
            atomicExch(a.cursor, 0);
            atomicExch(a.cursor + 1, 0);
        }
    }
    after_wait();  // what follows in the stream waits for the CTA kernel too
}

// The sources in box order and the claim table of a call.
static KeptBuffer g_p2p_buffer;

// The claims of table t, by the warp kernel or by the CTA kernel, alone or (split) before the warp kernel.
static int p2p_launch(bool warp, bool split, P2pArgs& a, const P2pTable& t, bool share, cudaStream_t st)
{
    auto kern = warp ? fmm_p2p_warp_kernel : fmm_p2p_kernel;
    const int64_t ctas = warp ? ((int64_t)t.cap + kP2pThreads / 32 - 1) / (kP2pThreads / 32) : t.cap;
    int sms = 0;
    if (int rc = device_sm_count(&sms)) return rc;
    a.go = split;
    a.nclaim = t.nclaim;
    a.tab = t.tab;
    a.ntab = t.cap;
    a.cursor = nullptr;
    int64_t grid = 0;
    if (warp && !share) {
        if (int rc = tile_counter(&a.cursor, st)) return rc;
        static int occ_cache;
        int occ = __atomic_load_n(&occ_cache, __ATOMIC_ACQUIRE);
        if (!occ) {
            FMM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kP2pThreads, 0));
            occ = std::max(occ, 1);
            __atomic_store_n(&occ_cache, occ, __ATOMIC_RELEASE);
        }
        grid = std::min<int64_t>((int64_t)occ * sms, ctas);
    } else {
        grid = split ? std::min<int64_t>(ctas, kP2pSplitGrid * sms)
                     : (ctas <= kP2pShareOne ? ctas : std::min<int64_t>((ctas + 1) / 2, kP2pShareGrid));
    }
    if (warp) {
        FMM_CUDA_TRY(launch_after(kern, (unsigned)grid, kP2pThreads, 0, st, a));
    } else {
        kern<<<(unsigned)grid, kP2pThreads, share && (split || ctas <= kP2pShareOne) ? kP2pRoomSmem : 0, st>>>(a);
        FMM_CUDA_TRY(cudaGetLastError());
    }
    return FMM_OK;
}

}  // namespace fmmgb

using namespace fmmgb;

extern "C" int fmm_p2p(int32_t level, const double* xy, const double* c, int64_t n, const int32_t* src_perm,
                       const int32_t* src_start, const double* z, int64_t nz, const int32_t* tgt_perm,
                       const int32_t* tgt_start, void* phi, int32_t flags, void* stream)
{
    clear_error();
    if (level < 0 || level > 10) return fail(FMM_EINVAL, "fmm_p2p: level %d outside 0..10", level);
    if (n < 0 || n > INT32_MAX || nz < 0 || nz > INT32_MAX)
        return fail(FMM_EINVAL, "fmm_p2p: point counts must lie in 0..2^31-1");
    if (!src_start || !tgt_start || (n > 0 && (!xy || !c || !src_perm)) || (nz > 0 && (!z || !tgt_perm || !phi)))
        return fail(FMM_EINVAL, "fmm_p2p: NULL pointer");
    if (((uintptr_t)xy & 7) || ((uintptr_t)c & 7) || ((uintptr_t)z & 7) || ((uintptr_t)phi & 7) ||
        ((uintptr_t)src_perm & 3) || ((uintptr_t)src_start & 3) || ((uintptr_t)tgt_perm & 3) ||
        ((uintptr_t)tgt_start & 3))
        return fail(FMM_EINVAL, "fmm_p2p: misaligned pointer (xy, c, z, phi 8 bytes; int32 arrays 4)");
    if (flags & ~(FMM_ACCUMULATE | FMM_P2P_SHARE_SM)) return fail(FMM_EINVAL, "fmm_p2p: unknown flags 0x%x", flags);
    if (nz == 0) return FMM_OK;
    cudaStream_t st = (cudaStream_t)stream;
    P2pArgs args;
    args.level = level;
    args.n = (int)n;
    args.nz = (int)nz;
    args.accumulate = (flags & FMM_ACCUMULATE) ? 1 : 0;
    args.sstart = src_start;
    args.z = z;
    args.tperm = tgt_perm;
    args.phi = reinterpret_cast<float2*>(phi);
    if (int rc = device_error_word(&args.err)) return rc;
    const int nbox = 1 << (2 * level);
    // every box to the CTA kernel, or the sparse ones to the warp kernel (the lines: above)
    const bool dense = nz >= (int64_t)kP2pDense * nbox || nbox < kP2wBoxes;
    // one buffer: the sources in box order, the claim tables, the numbers of claims
    const int64_t boxes = std::min<int64_t>(nbox, nz);
    // claims can be no more than the rooms of the tables
    P2pTable cta{32, kP2pRun, (int)(nz / kP2pRun + boxes)}, warp{2 * kP2wLanes, kP2wRun, dense ? 0 : (int)(nz / kP2wRun + boxes)};
    float4* src = nullptr;
    if (int rc = kept_buffer(g_p2p_buffer, (size_t)(n + cta.cap + warp.cap + 1) * sizeof(float4), (void**)&src)) return rc;
    cta.tab = reinterpret_cast<int4*>(src + n);
    warp.tab = cta.tab + cta.cap;
    cta.nclaim = reinterpret_cast<int*>(warp.tab + warp.cap);
    warp.nclaim = cta.nclaim + 1;
    FMM_CUDA_TRY(cudaMemsetAsync(cta.nclaim, 0, 2 * sizeof(int), st));
    p2p_claim_table_kernel<<<(unsigned)((nbox + 255) / 256), 256, 0, st>>>(level, tgt_start, (int)nz, src_start, cta, warp,
                                                                          args.err);
    FMM_CUDA_TRY(cudaGetLastError());
    if (n > 0) {
        p2p_sort_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(level, xy, c, src_perm, (int)n, src, args.err);
        FMM_CUDA_TRY(cudaGetLastError());
    }
    args.src = src;
    const bool share = (flags & FMM_P2P_SHARE_SM) != 0;
    if (int rc = p2p_launch(false, !dense, args, cta, share, st)) return rc;
    return dense ? FMM_OK : p2p_launch(true, false, args, warp, share, st);
}
