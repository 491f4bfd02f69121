// fgt_cheb.cu -- the FGT's Hermite evaluation (Sec. 4.2, Eq. hermite) with the sums over
// source boxes taken once per target box instead of once per target.
//
// At the targets of one box the transform is a smooth function of the offset u = (y - t_C)/(sqrt2 sigma),
//   F(u1, u2) = sum_{k1,k2} sum_{a1,a2} A_B[a1][a2] h_a1(u1 + k1 d) h_a2(u2 + k2 d),
// (k1, k2) the box offset target - source, d = box side / (sqrt2 sigma), |u| <= d/2.  Each
// h_a(u + k d) is replaced by its Chebyshev interpolant of Q nodes on |u| <= d/2, whose
// coefficients W_k[a][m] (formed in FP64, the same for every box) turn the sums into two
// one-dimensional contractions over the grid,
//   X[sy][tx][a2][m] = sum_{k1,a1} A[sy][tx - k1][a1][a2] W_k1[a1][m]
//   C[ty][tx][m][l]  = sum_{k2,a2} X[ty - k2][tx][a2][m] W_k2[a2][l],
// and a target's value is sum_{m,l} C[m][l] T_m(x1) T_l(x2), x = 2u/d: Q^2 multiply-adds a
// target instead of p^2 a target and source box (441 boxes at n_cut = 10).
//
// Error.  The interpolant of h_a differs from it by at most
//   2 (d/4)^Q / Q! max |h_a^(Q)|,  |h_a^(Q)| = |h_(a+Q)| <= 1.09 sqrt(2^(a+Q) (a+Q)!)
// (Cramer's inequality), so relative to h_a's own largest value, 1.09 sqrt(2^a a!), by
//   2 (d/4)^Q sqrt(2^Q (a+Q)!/a!) / Q!,
// 4e-10 for Q = 12, a = 15 and d = 1/2, the widest box that is taken.  That bound, and the FP32
// rounding of a box's sums, are relative to the largest values in the box; a target's own value can be
// smaller: over a box k boxes away h(u + k d) falls by about exp(2 k d^2) in each dimension.  So
// wider boxes keep the direct sum, which is accurate target by target (one source box (4, 4) boxes
// away, d = 0.95, 99 of 100 targets: 4e-6 of their values direct, 3e-3 through 16 nodes), and so do the
// boxes that the sources reach from afar only (d = 1/2, (10, 10) boxes away: 6e-6 direct, 2e-4).
// The contractions carry two limits of ln |field| over each target box besides, with m_B the largest
// coefficient of a source box: max_B (ln m_B - r^2) for the distance r to B's centre of the
// box's nearest point and of its farthest, per axis (|k| -+ 1/2) d.  Boxes where they lie more than
// kChebLoss apart are listed and summed directly.  In 32-bit emulation of random
// source boxes (1 to 6 of them up to 10 away, strengths over 8 decades) the rms error relative to a target's
// own terms is at most the direct sum's up to 5 (at 4 to 5: 3.2e-7 against 6.7e-7, d = 0.44; at 6 to 8 2.9e-6
// against 1.3e-6).
// The sums are FP32, as in the direct kernel.
//
// Measured at p = 16, n_cut = 10: 2^20 clustered targets, 32 x 32 boxes (263.6M target-box pairs)
// 2,350 us direct -> 46 us (table 6, contractions 7 and 6, evaluation 26, which is bound by the
// gathers of the targets and the scattered results); 3*10^5 targets, 16 x 16 boxes, against the
// tensor-core form 128 -> 26 us.  Error against 64 bits on the same coefficients, mean of 20 draws:
// 2.7e-7 -> 1.6e-7 (3.4e-6 where BF16x3 is asked for): a target's value sums 144 terms instead of
// 10^5.  A tap's P terms are summed apart before they join the sum over the taps: 1.9e-7 -> 1.6e-7, and
// 173 -> 169 us for the whole transform.
//
// The rule's other lines: at least 2 targets per box on average (uniform targets and sources, p = 16,
// n_cut = 10, just below the line, direct, and on it: 8 x 8 boxes 87 and 25 us, 32 x 32 1,350 and 44, 256 x 256
// 59,800 and 605; sources in one box in a hundred there 1,164 and 643, in one box alone 519 and 606) and
// grids of up to 256 x 256 boxes (90 MB of workspace; one allocation per grid size and device, kept).  A target outside its box
// (coordinates outside the unit square, or a binning that assigns it elsewhere) is summed
// directly too.
#include <algorithm>
#include <mutex>

#include "fgt_hermite.cuh"

namespace fmmgb {

constexpr int kChebMaxLog2 = 8;
constexpr int kChebMaxCut = 16;
constexpr int kChebQ = 12;           // nodes per dimension
constexpr double kChebMaxSide = 0.5;  // widest box, in sqrt2 sigma
constexpr float kChebLoss = 5.f;      // largest fall of ln |field| over a box (see above)
constexpr size_t kChebTableFloats = (size_t)(2 * kChebMaxCut + 1) * 16 * kChebQ;

// What the contractions and the listed boxes read (see above).
struct ChebLimits {
    float2* box;           // [sy][sx]: ln of the largest |coefficient| of the source box, twice
    float2* line;          // [tx][sy]: the limits contracted along x, (nearest, farthest)
    unsigned char* nz;     // [box] any non-zero coefficient
    unsigned char* apart;  // [box] summed directly
    H2pList list;
};

// The first 2 ncut + 1 CTAs: W[k][a][m] for the offset (k - ncut) d, one CTA each, FP64.  The others:
// the source boxes' l.box and l.nz, a warp each.
template <int P, int Q>
__global__ void __launch_bounds__(256) cheb_table_kernel(int ncut, double d, int nbox, const float* A, float* __restrict__ W,
                                                         ChebLimits l)
{
    __shared__ double s_h[P][Q], s_cos[4 * Q];
    const int tid = threadIdx.x, k = blockIdx.x;
    after_go();
    if (k > 2 * ncut) {
        after_wait();
        const int b = (k - 2 * ncut - 1) * 8 + tid / 32, lane = tid % 32;
        if (b >= nbox) return;
        unsigned m = 0;
        for (int i = lane; i < P * P / 4; i += 32) {
            const float4 v = reinterpret_cast<const float4*>(A + (size_t)b * P * P)[i];
            m = max(m, max(max(__float_as_uint(v.x) & 0x7FFFFFFFu, __float_as_uint(v.y) & 0x7FFFFFFFu),
                           max(__float_as_uint(v.z) & 0x7FFFFFFFu, __float_as_uint(v.w) & 0x7FFFFFFFu)));
        }
        m = __reduce_max_sync(0xffffffffu, m);
        if (lane) return;
        const float ln = m < 0x7F800000u ? logf(__uint_as_float(m)) : INFINITY;  // infinite: not finite
        l.box[b] = make_float2(ln, ln);
        l.nz[b] = m != 0;
        return;
    }
    if (tid < 4 * Q) s_cos[tid] = cospi((double)tid / (2.0 * Q));
    __syncthreads();
    if (tid < Q) {
        const double t = 0.5 * d * s_cos[2 * tid + 1] + (double)(k - ncut) * d;
        double h0 = exp(-t * t), h1 = 2.0 * t * h0;
        s_h[0][tid] = h0;
#pragma unroll
        for (int a = 1; a < P; ++a) {
            s_h[a][tid] = h1;
            const double h2 = 2.0 * t * h1 - 2.0 * a * h0;
            h0 = h1;
            h1 = h2;
        }
    }
    __syncthreads();
    after_wait();  // an earlier call may still read the table and the list
    if (k == 0 && tid == 0) *l.list.count = 0;
    for (int e = tid; e < P * Q; e += 256) {
        const int a = e / Q, m = e % Q;
        double s = 0.0;
#pragma unroll
        for (int i = 0; i < Q; ++i) s += s_h[a][i] * s_cos[(2 * i + 1) * m % (4 * Q)];
        W[(size_t)k * P * Q + e] = (float)(s * (m ? 2.0 : 1.0) / Q);
    }
}

// One contraction along a line of boxes.  in: [line][s][c < P][r < R]; out: [t][line][r][m < Q]
// (so the second contraction, along the other axis, finds its line contiguous and contracts
// the other index).  A CTA takes kSeg target boxes of a line and stages their window of
// kSeg + 2 n_cut source boxes and the table; a thread owns (box, r) and all Q outputs, over
// every kTaps-th tap, so a step is one scalar and Q/4 broadcast 16-byte shared loads for Q
// multiply-adds; the taps' sums are added in registers and the groups' meet in shared memory.
// The limits of ln |field| (see above) are contracted beside them, max for sum: along x from l.box into
// l.line, along y (LAST) into the list of the boxes summed directly, whose first coefficient becomes NaN.
constexpr int kSeg = 4;
constexpr int kTaps = 4;
constexpr int kEvalThreads = 128;  // of the evaluation's CTAs, and targets of a listed box per claim

template <int P, int R, int Q>
struct ChebPass {
    static constexpr int THREADS = kSeg * kTaps * R;
    static constexpr int BOX = P * R + (R + 32 - P * R % 32) % 32;  // floats per staged box (bank skew R)
    static constexpr int OUT = kSeg * R * Q;
    static size_t smem(int ncut)
    {
        const size_t win = (size_t)(kSeg + 2 * ncut) * BOX, red = (size_t)kTaps * OUT;
        return ((win > red ? win : red) + (size_t)(2 * ncut + 1) * P * Q) * sizeof(float);
    }
};

// The order of floats as that of integers (NaN aside), and back.
__device__ __forceinline__ int float_key(float x)
{
    const int i = __float_as_int(x);
    return i ^ (i >> 31 & 0x7FFFFFFF);
}

template <int P, int R, int Q, bool LAST>
__global__ void __launch_bounds__(kSeg* kTaps* R)
    cheb_pass_kernel(int side, int ncut, const float* in, const float* W, float* __restrict__ out, float d, ChebLimits l,
                     const int* box_start)
{
    __shared__ float2 s_lim[kSeg + 2 * kChebMaxCut];  // of the window's boxes
    __shared__ bool s_apart[kSeg];
    using C = ChebPass<P, R, Q>;
    extern __shared__ float4 cheb_smem[];
    const int taps = 2 * ncut + 1;
    float* s_tab = reinterpret_cast<float*>(cheb_smem);  // [taps][P][Q]
    float* s_win = s_tab + taps * P * Q;                 // [kSeg + 2 ncut][BOX], then the groups' sums
    const int tid = threadIdx.x, line = blockIdx.y, t0 = blockIdx.x * kSeg;
    after_go();
    after_wait();
    const int nwin = kSeg + 2 * ncut;
    static_assert(C::THREADS >= kSeg + 2 * kChebMaxCut);
    for (int i = tid; i < taps * P * Q / 4; i += C::THREADS)
        reinterpret_cast<float4*>(s_tab)[i] = reinterpret_cast<const float4*>(W)[i];
    float2 lim = make_float2(-INFINITY, -INFINITY);
    if (const int s = t0 - ncut + tid; tid < nwin && s >= 0 && s < side) lim = (LAST ? l.line : l.box)[line * side + s];
    constexpr int B4 = P * R / 4;
    for (int i = tid; i < nwin * B4; i += C::THREADS) {
        const int b = i / B4, s = t0 - ncut + b;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (s >= 0 && s < side) v = reinterpret_cast<const float4*>(in + ((size_t)line * side + s) * P * R)[i % B4];
        *reinterpret_cast<float4*>(s_win + b * C::BOX + 4 * (i % B4)) = v;
    }
    if (tid < nwin) s_lim[tid] = lim;
    __syncthreads();
    const int group = tid / (kSeg * R), e = tid % (kSeg * R), seg = e / R, r = e % R;
    float sum[Q];
#pragma unroll
    for (int m = 0; m < Q; ++m) sum[m] = 0.f;
    for (int j = group; j < taps; j += kTaps) {  // source box t + j - ncut: offset ncut - j
        const float* v = s_win + (seg + j) * C::BOX + r;
        const float4* w = reinterpret_cast<const float4*>(s_tab + (2 * ncut - j) * P * Q);
        float acc[Q];
#pragma unroll
        for (int m = 0; m < Q; ++m) acc[m] = 0.f;
#pragma unroll 4
        for (int c = 0; c < P; ++c) {
            const float x = v[c * R];
#pragma unroll
            for (int q = 0; q < Q / 4; ++q) {
                const float4 h = w[c * (Q / 4) + q];
                acc[4 * q] = fmaf(x, h.x, acc[4 * q]);
                acc[4 * q + 1] = fmaf(x, h.y, acc[4 * q + 1]);
                acc[4 * q + 2] = fmaf(x, h.z, acc[4 * q + 2]);
                acc[4 * q + 3] = fmaf(x, h.w, acc[4 * q + 3]);
            }
        }
#pragma unroll
        for (int m = 0; m < Q; ++m) sum[m] += acc[m];
    }
    // the limits, after the sums (before them the first pass took 2 us more); the last warps have fewer taps
    for (int t = C::THREADS / 32 - 1 - tid / 32; t < kSeg; t += C::THREADS / 32) {
        const int lane = tid & 31;
        int hi = float_key(-INFINITY), lo = hi;
        for (int j = lane; j < taps; j += 32) {
            const float2 m = s_lim[t + j];
            const float k = (float)abs(j - ncut), near = fmaxf(k - 0.5f, 0.f) * d, far = (k + 0.5f) * d;
            hi = max(hi, float_key(m.x - near * near));
            lo = max(lo, float_key(m.y - far * far));
        }
        hi = __reduce_max_sync(0xffffffffu, hi);
        lo = __reduce_max_sync(0xffffffffu, lo);
        const int b = (t0 + t) * side + line;
        if (lane || t0 + t >= side) continue;
        const float2 m = make_float2(__int_as_float(hi ^ (hi >> 31 & 0x7FFFFFFF)), __int_as_float(lo ^ (lo >> 31 & 0x7FFFFFFF)));
        if constexpr (!LAST) {
            l.line[b] = m;
        } else {
            // m.x = -inf: no source box holds anything; inf - inf: a coefficient is not finite
            const bool apart = m.x > -INFINITY && !(m.x - m.y <= kChebLoss);
            l.apart[b] = s_apart[t] = apart;
            const int n = apart ? box_start[b + 1] - box_start[b] : 0;
            if (n > 0) {
                const unsigned long long old =
                    atomicAdd(l.list.count, (1ull << 32) | (unsigned)((n + kEvalThreads - 1) / kEvalThreads));
                l.list.box[old >> 32] = b;
                l.list.claim[old >> 32] = (int)old;
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < Q / 4; ++q)
        *reinterpret_cast<float4*>(s_win + group * C::OUT + e * Q + 4 * q) =
            make_float4(sum[4 * q], sum[4 * q + 1], sum[4 * q + 2], sum[4 * q + 3]);
    __syncthreads();
    for (int i = tid; i < C::OUT; i += C::THREADS) {
        const int t = t0 + i / (R * Q);
        if (t >= side) break;
        float v = 0.f;
#pragma unroll
        for (int k = 0; k < kTaps; ++k) v += s_win[k * C::OUT + i];
        if (LAST && i % (R * Q) == 0 && s_apart[i / (R * Q)]) v = NAN;
        out[((size_t)t * side + line) * (R * Q) + i % (R * Q)] = v;
    }
}

struct ChebEval : H2pSums {
    const float* C;
    const unsigned char* apart;  // of ChebLimits
    H2pList list;
};

// The direct sum for one target assigned to `box`, as the direct kernel takes it (source boxes without
// a non-zero coefficient are skipped): source boxes first, first + step, ... of the neighbourhood.
template <int P>
__device__ __noinline__ float cheb_direct(const ChebEval& a, int box, double y0, double y1, int first, int step)
{
    const int side = 1 << a.g, tx = box & (side - 1), ty = box >> a.g;
    const int sx0 = max(tx - a.ncut, 0), w = min(tx + a.ncut, side - 1) - sx0 + 1;
    const int sy0 = max(ty - a.ncut, 0), nb = w * (min(ty + a.ncut, side - 1) - sy0 + 1);
    const float u1 = (float)((y0 * side - (tx + 0.5)) * a.d), u2 = (float)((y1 * side - (ty + 0.5)) * a.d);
    float acc = 0.f, h2[P];
    int row = -1;
#pragma unroll 1
    for (int i = first; i < nb; i += step) {
        const int sx = sx0 + i % w, sy = sy0 + i / w;
        if (!a.nz[sy * side + sx]) continue;
        if (sy != row) {
            row = sy;
            hermite_functions<P>(u2 + (float)((double)(ty - sy) * a.d), h2);
        }
        // Clenshaw's backward recurrence over a1 for h_(a+1) = 2t h_a - 2a h_(a-1)
        const float t1 = u1 + (float)((double)(tx - sx) * a.d), tt = t1 + t1;
        const float4* Ab = reinterpret_cast<const float4*>(a.A + ((size_t)sy * side + sx) * P * P);
        float c1 = 0.f, c2 = 0.f;
#pragma unroll
        for (int a1 = P - 1; a1 >= 0; --a1) {
            float t = fmaf(tt, c1, -(float)(2 * (a1 + 1)) * c2);
#pragma unroll
            for (int q = 0; q < P / 4; ++q) {
                const float4 v = Ab[a1 * (P / 4) + q];
                t = fmaf(v.x, h2[4 * q], t);
                t = fmaf(v.y, h2[4 * q + 1], t);
                t = fmaf(v.z, h2[4 * q + 2], t);
                t = fmaf(v.w, h2[4 * q + 3], t);
            }
            c2 = c1;
            c1 = t;
        }
        acc = fmaf(__expf(-t1 * t1), c1, acc);
    }
    return acc;
}

// The direct sums of a warp's targets (box < 0: none).  A few take the whole warp one after another, a
// share of the source boxes a lane; many take a lane each.  2^20 targets on 32 x 32 boxes, n_cut = 10,
// 61 us with none outside the unit square: with one 1,842 us a lane each always, 86 us so; with one in a
// hundred (crowded into the edge boxes) 7.4 ms and 2.7 ms, where the direct kernel takes 4.4 ms for all.
constexpr int kApartShared = 15;
template <int P>
__device__ __noinline__ float cheb_apart(const ChebEval& a, int box, double y0, double y1)
{
    unsigned todo = __ballot_sync(0xffffffffu, box >= 0);
    float out = 0.f;
    if (__popc(todo) > kApartShared) {
        if (box >= 0) out = cheb_direct<P>(a, box, y0, y1, 0, 1);
        return out;
    }
    const int lane = threadIdx.x & 31;
    for (; todo; todo &= todo - 1) {
        const int l = __ffs(todo) - 1;
        float s = cheb_direct<P>(a, __shfl_sync(0xffffffffu, box, l), __shfl_sync(0xffffffffu, y0, l),
                                 __shfl_sync(0xffffffffu, y1, l), lane, 32);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == l) out = s;
    }
    return out;
}

// sum_{m,l} c[m][l] T_m(x1) T_l(x2) for NR targets of one box (or, with NR = 1, of a box per lane).
template <int Q, int NR>
__device__ __forceinline__ void cheb_sum(const float* c, const float* x1, const float* x2, float* out)
{
    float T[NR][Q], b1[NR], b2[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        T[r][0] = 1.f;
        T[r][1] = x2[r];
#pragma unroll
        for (int l = 2; l < Q; ++l) T[r][l] = fmaf(x2[r] + x2[r], T[r][l - 1], -T[r][l - 2]);
        b1[r] = b2[r] = 0.f;
    }
    const float4* c4 = reinterpret_cast<const float4*>(c);
#pragma unroll
    for (int m = Q - 1; m >= 0; --m) {  // Clenshaw over m: b_m = row_m + 2 x1 b_(m+1) - b_(m+2)
        float row[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) row[r] = fmaf(m ? x1[r] + x1[r] : x1[r], b1[r], -b2[r]);
#pragma unroll
        for (int q = 0; q < Q / 4; ++q) {
            const float4 v = c4[m * (Q / 4) + q];
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                row[r] = fmaf(v.x, T[r][4 * q], row[r]);
                row[r] = fmaf(v.y, T[r][4 * q + 1], row[r]);
                row[r] = fmaf(v.z, T[r][4 * q + 2], row[r]);
                row[r] = fmaf(v.w, T[r][4 * q + 3], row[r]);
            }
        }
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            b2[r] = b1[r];
            b1[r] = row[r];
        }
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) out[r] = b1[r];
}

// Places base + 32 r + lane, r < NR, of the binned targets: tj[r] the target's index (-1: past the
// end, or a perm entry out of range, which sets the error word), tb[r] the box of its coordinates
// where that box holds the place, else -1, (o0, o1) its offset from that box's centre in box sides.
// The loads of all rows are in flight together: index, coordinates and box range are three round
// trips a warp instead of three a row (2^20 targets: 30 -> 26 us; fewer rows a lane, for more warps on an
// SM, measured the same).
template <int NR>
__device__ __forceinline__ void binned_targets(const double* y, const int* perm, const int* box_start, int g, int n,
                                               int64_t base, int* err, int* tj, int* tb, float* o0, float* o1)
{
    double y0[NR], y1[NR];
    int f[NR], e[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) tj[r] = base + 32 * r < n ? perm[base + 32 * r] : -1;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const size_t j = (unsigned)tj[r] < (unsigned)n ? tj[r] : 0;
        y0[r] = y[2 * j];
        y1[r] = y[2 * j + 1];
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        long long X0, X1;
        tb[r] = -1;
        o0[r] = o1[r] = 0.f;
        if (grid_fixed31(y0[r], g, X0) && grid_fixed31(y1[r], g, X1)) {
            tb[r] = ((int)(X1 >> 31) << g) + (int)(X0 >> 31);
            o0[r] = cell_offset31(X0);
            o1[r] = cell_offset31(X1);
        }
        f[r] = box_start[max(tb[r], 0)];
        e[r] = box_start[max(tb[r], 0) + 1];
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int64_t pos = base + 32 * r;
        if ((unsigned)tj[r] >= (unsigned)n) {
            if (pos < n) atomicOr(err, DEV_ERR_CHECK);
            tj[r] = tb[r] = -1;
        } else if (tb[r] >= 0 && !(bin_range_ok(f[r], e[r], n) && f[r] <= pos && pos < e[r])) {
            tb[r] = -1;
        }
    }
}
// A warp takes 32 ROWS consecutive binned targets: together where they share a box (uniform
// 16-byte loads of its coefficients, each feeding 4 ROWS multiply-adds a lane), else a row of
// 32 at a time with a box per lane.  ROWS is 4, or 1 for fewer than kEvalWide targets, which leave the SMs
// warps to spare (whole calls on 1 to 4^7 boxes, p = 8 and 16, n_cut = 0 to 10, one row against four: 0.73 of the
// time for 2,000 targets, 0.85 for 10^5, 1.00 for 2*10^5, 1.13 for 3*10^5).
constexpr int64_t kEvalWide = 1 << 17;

template <int P, int Q, int ROWS>
__device__ __forceinline__ void cheb_eval_warp(const ChebEval& a, int64_t base)
{
    const int lane = threadIdx.x & 31, side = 1 << a.g, nbox = side * side;
    int tj[ROWS], tb[ROWS];  // target, its box (-1: evaluated apart)
    float x1[ROWS], x2[ROWS], out[ROWS];
    binned_targets<ROWS>(a.y, a.perm, a.box_start, a.g, a.n, base + lane, a.err, tj, tb, x1, x2);
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        x1[r] *= 2.f;
        x2[r] *= 2.f;
        out[r] = 0.f;
    }
    const int b0 = __shfl_sync(0xffffffffu, tb[0], 0);
    bool same = b0 >= 0;
#pragma unroll
    for (int r = 0; r < ROWS; ++r) same &= tb[r] == b0 || base + 32 * r + lane >= a.n;
    if (__all_sync(0xffffffffu, same)) {
        cheb_sum<Q, ROWS>(a.C + (size_t)b0 * Q * Q, x1, x2, out);
    } else {
#pragma unroll 1
        for (int r = 0; r < ROWS; ++r) {
            // registers indexed by constants only
            float u1 = 0.f, u2 = 0.f, v = 0.f;
            int b = -1, j = -1;
#pragma unroll
            for (int k = 0; k < ROWS; ++k)
                if (k == r) {
                    u1 = x1[k];
                    u2 = x2[k];
                    b = tb[k];
                    j = tj[k];
                }
            if (b >= 0) cheb_sum<Q, 1>(a.C + (size_t)b * Q * Q, &u1, &u2, &v);
            if (__any_sync(0xffffffffu, b < 0 && j >= 0)) {
                int lo = -1;  // the assigned box
                double y0 = 0.0, y1 = 0.0;
                if (b < 0 && j >= 0) {
                    lo = bin_find(a.box_start, nbox, (int)(base + 32 * r + lane), a.n);
                    if (lo >= 0 && a.apart[lo]) {
                        lo = j = -1;
                    } else if (lo >= 0) {
                        y0 = a.y[2 * (size_t)j];
                        y1 = a.y[2 * (size_t)j + 1];
                    } else {  // box_start does not bin [0, n)
                        atomicOr(a.err, DEV_ERR_CHECK);
                        j = -1;
                    }
                }
                const float w = cheb_apart<P>(a, lo, y0, y1);
                if (lo >= 0) v = w;
            }
#pragma unroll
            for (int k = 0; k < ROWS; ++k)
                if (k == r) {
                    out[k] = v;
                    tj[k] = j;
                }
        }
    }
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
        // NaN of a box that is summed directly: left to that sum
        if (tj[r] >= 0 && !(isnan(out[r]) && tb[r] >= 0 && a.apart[tb[r]])) a.G[tj[r]] = a.accumulate ? a.G[tj[r]] + out[r] : out[r];
}

// A CTA that has evaluated its own targets takes its share of the claims on the listed boxes, 128
// targets each, one a thread.  (A launch of the direct kernel after this one cost 7 us more for an empty list,
// and so did CTAs of their own before the others.)
template <int P, int Q, int ROWS>
__global__ void __launch_bounds__(kEvalThreads) cheb_eval_kernel(ChebEval a)
{
    __shared__ H2pShared<kEvalThreads> sh;
    __shared__ int s_claim[3];
    extern __shared__ float4 cheb_smem[];
    const int nbox = 1 << (2 * a.g);
    after_go();
    after_wait();
    const int64_t base = ((int64_t)blockIdx.x * (kEvalThreads / 32) + (threadIdx.x >> 5)) * (32 * ROWS);
    bin_check(a.box_start, nbox, a.n, a.err);
    const unsigned long long count = *a.list.count;
    if (base < a.n) cheb_eval_warp<P, Q, ROWS>(a, base);
    if (blockIdx.x >= (unsigned)count) return;
    h2p_offsets(sh, a);
    for (unsigned k = blockIdx.x; k < (unsigned)count; k += gridDim.x) {
        if (threadIdx.x == 0)
            h2p_claim_range_ordered(a.list.claim, a.list.box, a.box_start, nbox, (int)(count >> 32), a.n, kEvalThreads, k,
                                    s_claim, s_claim + 1, s_claim + 2);
        __syncthreads();
        const int first = s_claim[0], end = s_claim[1], box = s_claim[2];
        if (first < end) h2p_run<P, 1, kEvalThreads>(a, sh, reinterpret_cast<float*>(cheb_smem), first, end, box);
        __syncthreads();  // the claim has been read
    }
}

// Per device and grid size: table | X [4^g][16][12] | C [4^g][12][12] | the list's count | l.box, l.line
// [4^g] | the list's boxes and claims [4^g] | nz, apart [4^g] (bytes), allocated on first use and
// kept (captured graphs hold its address).  NULL, without an error, when there is no room for it.
static int cheb_workspace(int g, float** out)
{
    static std::mutex mu;
    static float* buf[64][kChebMaxLog2 + 1];
    int dev = 0;
    FMM_CUDA_TRY(cudaGetDevice(&dev));
    *out = nullptr;
    if (dev < 0 || dev >= 64) return FMM_OK;  // the direct sum serves it
    std::lock_guard<std::mutex> lk(mu);
    if (!buf[dev][g]) {
        const size_t bytes = (kChebTableFloats + 2 + ((size_t)((16 + kChebQ) * kChebQ + 7) << (2 * g))) * sizeof(float);
        if (capture_safe_malloc((void**)&buf[dev][g], bytes) != cudaSuccess) return FMM_OK;
    }
    *out = buf[dev][g];
    return FMM_OK;
}

template <int P, int Q = kChebQ>
static int cheb_launch(const H2pSums& e, float* ws, cudaStream_t st)
{
    using C1 = ChebPass<P, P, Q>;
    using C2 = ChebPass<P, Q, Q>;
    const int side = 1 << e.g;
    float *W = ws, *X = W + kChebTableFloats, *C = X + ((size_t)16 * kChebQ << (2 * e.g));
    static unsigned long long opted[2];
    if (int rc = smem_opt_in((const void*)cheb_pass_kernel<P, P, Q, false>, (int)C1::smem(kChebMaxCut), &opted[0])) return rc;
    if (int rc = smem_opt_in((const void*)cheb_pass_kernel<P, Q, Q, true>, (int)C2::smem(kChebMaxCut), &opted[1])) return rc;
    const size_t nbox = (size_t)1 << (2 * e.g);
    ChebLimits l;
    l.list.count = reinterpret_cast<unsigned long long*>(C + kChebQ * kChebQ * nbox);
    l.box = reinterpret_cast<float2*>(l.list.count + 1);
    l.line = l.box + nbox;
    l.list.box = reinterpret_cast<int*>(l.line + nbox);
    l.list.claim = l.list.box + nbox;
    l.nz = reinterpret_cast<unsigned char*>(l.list.claim + nbox);
    l.apart = l.nz + nbox;
    FMM_CUDA_TRY(launch_after(cheb_table_kernel<P, Q>, 2 * e.ncut + 1 + (unsigned)(nbox + 7) / 8, 256, 0, st, e.ncut, e.d, (int)nbox, e.A, W, l));
    const dim3 grid((side + kSeg - 1) / kSeg, side);
    FMM_CUDA_TRY(launch_after(cheb_pass_kernel<P, P, Q, false>, grid, C1::THREADS, C1::smem(e.ncut), st, side, e.ncut, e.A, W, X,
                              (float)e.d, l, e.box_start));
    FMM_CUDA_TRY(launch_after(cheb_pass_kernel<P, Q, Q, true>, grid, C2::THREADS, C2::smem(e.ncut), st, side, e.ncut, X, W, C,
                              (float)e.d, l, e.box_start));
    ChebEval a;
    static_cast<H2pSums&>(a) = e;
    a.nz = l.nz;
    a.C = C;
    a.apart = l.apart;
    a.list = l.list;
    int sms = 0;
    if (int rc = device_sm_count(&sms)) return rc;
    const bool wide = a.n >= kEvalWide;
    // with few targets, CTAs enough for the listed boxes (2^14 uniform targets
    // on 32 x 32 boxes, all sources in a spot of 2 % of the side, d = 0.44: 150 -> 63 us)
    const unsigned blocks = std::max(bin_blocks(a.n, kEvalThreads * (wide ? 4 : 1), (int64_t)nbox, kEvalThreads),
                                     (unsigned)std::min<size_t>(nbox, 2 * (size_t)sms));
    auto eval = wide ? cheb_eval_kernel<P, Q, 4> : cheb_eval_kernel<P, Q, 1>;
    FMM_CUDA_TRY(launch_after(eval, blocks, kEvalThreads, H2pSmem<P>::bytes, st, a));
    return FMM_OK;
}

int launch_fgt_h2p_cheb(int g, int ncut, int p, double d, const float* A, const double* y, int n, const int* perm,
                        const int* box_start, float* G, bool accumulate, int* err, cudaStream_t st, bool* done)
{
    *done = false;
    if (d > kChebMaxSide || g > kChebMaxLog2 || n < (2 << (2 * g))) return FMM_OK;
    float* ws = nullptr;
    if (int rc = cheb_workspace(g, &ws)) return rc;
    if (!ws) return FMM_OK;
    *done = true;
    ncut = std::min(ncut, (1 << g) - 1);  // no more offsets than the grid has (1 box, n_cut = 10: 16.7 -> 11 us)
    const H2pSums e{g, ncut, n, d, A, y, perm, box_start, nullptr, G, accumulate ? 1 : 0, err};
    switch (p) {
        case 4: return cheb_launch<4>(e, ws, st);
        case 8: return cheb_launch<8>(e, ws, st);
        case 12: return cheb_launch<12>(e, ws, st);
        default: return cheb_launch<16>(e, ws, st);
    }
}

}  // namespace fmmgb
