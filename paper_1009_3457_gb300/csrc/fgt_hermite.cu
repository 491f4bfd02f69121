// fgt_hermite.cu -- the fast Gauss transform evaluated directly from Hermite
// series at target points (Sec. 4.2, Eq. hermite), over the n_cut
// neighbourhood of each target's box on the uniform 2^g x 2^g grid:
//
//   G(y) (+)= sum_{B : max(|sx-tx|,|sy-ty|) <= n_cut}
//               sum_{a1,a2 < p} A_B[a1][a2] h_a1((y1 - sB1)/(sqrt2 sigma)) h_a2((y2 - sB2)/(sqrt2 sigma)),
//
// h_n(t) = exp(-t^2) H_n(t).  Targets are first binned by box (a counting
// sort on the device), so that one CTA serves a run of targets of one box and
// stages each source box's p x p coefficients in shared memory once for all
// of them -- the paper's design point of keeping the series coefficients in
// shared memory for a block of targets, without its per-call size limits.
// The same binning gives a P2H (Eq. A_alpha) without contended atomics.
//
// Evaluation kernel (FP32, CUDA cores; no dense contraction here that tensor
// cores could take without forming an m x p^2 operand per box):
//   - persistent CTAs of 128 threads claim runs of up to 128 R targets of one
//     box by an atomic claim index and a per-box claim table built just
//     before (a scan of ceil(targets / run) over the boxes);
//   - the neighbourhood is walked one source row at a time: the row's boxes
//     are contiguous in A and are copied to shared memory with cp.async,
//     double-buffered, while the previous row is evaluated;
//   - per thread R targets; per row h_b(t2) is formed once by the three-term
//     recurrence h_{n+1} = 2t h_n - 2n h_{n-1}; per box
//     acc += sum_a h_a(t1) sum_b A[a][b] h_b(t2), the outer sum by Clenshaw's
//     backward recurrence (p^2 + 2p multiply-adds, the A rows read as broadcast
//     float4 from shared memory);
//   - t = u + k d with u = (y - t_C)/(sqrt2 sigma) formed once per target in
//     FP64 and k d (k = tx - sx, d = side/(sqrt2 sigma)) from a small table,
//     so no FP64 arithmetic runs per box;
//   - boxes whose coefficients are all zero (no sources) are skipped.
#include <mutex>

#include "fgt_hermite.cuh"

namespace fmmgb {

// ---------------------------------------------------------------------------
// binning of points by grid box
// ---------------------------------------------------------------------------
constexpr int kBinThreads = 256;
constexpr int kScanThreads = 1024;

__device__ __forceinline__ int fgt_grid_box(double x, double y, int g)
{
    // floor(v 2^g) per coordinate, clamped to the grid; NaN and negatives to cell 0
    return grid_cell(y, g) * (1 << g) + grid_cell(x, g);
}

// Warp-aggregated counting: the lanes of a warp whose points share a box make
// one atomic between them (clustered inputs put many points of a warp in one
// box), and each lane learns its rank among them.  Every lane of the warp calls
// it (key < 0: no point); returns the box's count before the warp's additions
// plus the lane's rank, or -1 without a point.
__device__ __forceinline__ int warp_box_claim(int* __restrict__ counter, int key)
{
    const unsigned peers = __match_any_sync(0xffffffffu, key);
    const int lane = threadIdx.x & 31, leader = __ffs(peers) - 1;
    int base = 0;
    if (key >= 0 && lane == leader) base = atomicAdd(&counter[key], __popc(peers));
    base = __shfl_sync(0xffffffffu, base, leader);
    return key >= 0 ? base + __popc(peers & ((1u << lane) - 1u)) : -1;
}

// grid-stride over warps: all 32 lanes of a warp take part in every round
__global__ void bin_count_kernel(int g, const double* __restrict__ y, int64_t n, int* __restrict__ counts)
{
    after_go();
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w = w0; 32 * w < n; w += nw) {
        const int64_t i = 32 * w + lane;
        const int key = i < n ? fgt_grid_box(__ldg(y + 2 * i), __ldg(y + 2 * i + 1), g) : -1;
        warp_box_claim(counts, key);
    }
}

// One CTA: exclusive scan of v(0..nbox-1) into out[0..nbox] (out[nbox] = total); put(i, prefix)
// also receives each prefix.
template <class Load, class Put>
__device__ void block_exclusive_scan(int nbox, Load v, Put put, int* out)
{
    __shared__ int s_warp[kScanThreads / 32];
    __shared__ int s_carry;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) s_carry = 0;
    __syncthreads();
    for (int base = 0; base < nbox; base += kScanThreads) {
        const int i = base + tid;
        const int c = i < nbox ? v(i) : 0;
        int x = c;  // inclusive warp scan
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += t;
        }
        if (lane == 31) s_warp[warp] = x;
        __syncthreads();
        if (warp == 0) {
            int w = s_warp[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += t;
            }
            s_warp[lane] = w;
        }
        __syncthreads();
        const int excl = s_carry + (warp ? s_warp[warp - 1] : 0) + x - c;
        if (i < nbox) {
            out[i] = excl;
            put(i, excl);
        }
        __syncthreads();
        if (tid == kScanThreads - 1) s_carry = excl + c;
        __syncthreads();
    }
    if (tid == 0) out[nbox] = s_carry;
}

// box_start[0..nbox] = exclusive scan of counts; counts becomes the scatter cursor (the same prefix)
__global__ void __launch_bounds__(kScanThreads) bin_scan_kernel(int nbox, int* counts, int* __restrict__ box_start)
{
    after_go();
    after_wait();
    block_exclusive_scan(
        nbox, [&](int i) { return counts[i]; }, [&](int i, int e) { counts[i] = e; }, box_start);
}

// The same for larger grids, a block per kScanTile boxes: a block adds up every count before its
// own tile (read from L2: at most the whole array, 4 MB at 1024 x 1024 boxes, a block) and scans
// its tile, so the blocks need not meet.  The counts stay as they are; the cursors are a copy.
// One block's rounds of barriers one after another took 1.1 us per 1,024 boxes: binning 2^22 points
// on 256 x 256 and 512 x 512 boxes 147 -> 114 and 263 -> 119 us, 2^18 points on 1024 x 1024
// 735 -> 95 us.
constexpr int kScanTile = 4096;

__global__ void __launch_bounds__(kScanThreads) bin_scan_tiles_kernel(int nbox, const int* counts,
                                                                      int* __restrict__ box_start)
{
    __shared__ int s_warp[kScanThreads / 32], s_before;
    after_go();
    after_wait();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, first = blockIdx.x * kScanTile;
    int before = 0;
#pragma unroll 4
    for (int i = tid; i < first; i += kScanThreads) before += counts[i];
    before = __reduce_add_sync(0xffffffffu, before);
    if (lane == 0) s_warp[warp] = before;
    __syncthreads();
    if (warp == 0) {
        const int v = __reduce_add_sync(0xffffffffu, s_warp[lane]);
        if (lane == 0) s_before = v;
    }
    // four consecutive boxes a thread
    int c[4], sum = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int i = first + 4 * tid + k;
        c[k] = i < nbox ? counts[i] : 0;
        sum += c[k];
    }
    int x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += t;
    }
    __syncthreads();  // s_warp has been read, s_before written
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = s_warp[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += t;
        }
        s_warp[lane] = w;
    }
    __syncthreads();
    int at = s_before + (warp ? s_warp[warp - 1] : 0) + x - sum;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int i = first + 4 * tid + k;
        if (i < nbox) box_start[i] = at;
        at += c[k];
        if (i == nbox - 1) box_start[nbox] = at;
    }
}

__global__ void bin_scatter_kernel(int g, const double* y, int64_t n, int* __restrict__ cursor,
                                   int* __restrict__ perm)
{
    after_go();
    after_wait();
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w = w0; 32 * w < n; w += nw) {
        const int64_t i = 32 * w + lane;
        const int key = i < n ? fgt_grid_box(y[2 * i], y[2 * i + 1], g) : -1;
        const int slot = warp_box_claim(cursor, key);
        if (slot >= 0) perm[slot] = (int)i;
    }
}

// Small grids (up to 4^7 boxes): a block counts its contiguous chunk of points in a
// shared-memory histogram, so contended boxes (clustered points) cost shared-memory
// atomics, and the global counters see one addition per box a block touches.
constexpr int kBinSmemMaxLog2 = 7;

// A block of T threads, LOADS points a thread in flight at a time (a load and a shared atomic in
// turn left a thread waiting for each point's load).  fgt_bin_points takes
//   - 1024 x 4 on grids of 4^6 boxes or more and 2^15 points or more: a histogram of 16 to 64 KB
//     leaves room for few blocks, which then need their threads (2^20 points on 4^7 boxes 49 -> 33 us, 37
//     with 512 threads; 2^18 on 4^6 20.5 -> 16.4).  A block scatters 4,096 points at most and walks its counters
//     for them; two passes over the block's whole share of the points are still slower (2^22 / 2^24 / 2^26 points on
//     4^7 boxes 93 -> 73, 490 -> 248, 3,258 -> 909 us, on 4^6 66 -> 57, 464 -> 198, 2,668 -> 737);
//   - 512 x 8 on smaller grids and 2^19 points or more (on 4^5 boxes 2^18.5 / 2^19 / 2^19.5 points 20.9 / 23.0 / 26.8
//     -> 19.4 / 19.0 / 20.5 us, the first by 256 x 4; 2^20 27 -> 22.5; 1024 threads 21, but
//     they fill the SMs, and the next kernel's early part, the table of the Hermite evaluation, then waits:
//     163 against 153 us for that transform);
//   - 256 x 4 else: few blocks start and meet sooner (2^12 points 8.4 us against 9.6 with 1024
//     threads; the Hermite transform of 3e5 points 79 us against 84 with 512).
// Coordinates of the points first, first + T, ... (LOADS of them, below i1).
template <int T, int LOADS>
__device__ __forceinline__ void load_points(const double* y, int64_t first, int64_t i1,
                                            double (&a)[LOADS], double (&b)[LOADS])
{
#pragma unroll
    for (int u = 0; u < LOADS; ++u) {
        const int64_t k = first + u * T;
        a[u] = k < i1 ? y[2 * k] : 0.0;
        b[u] = k < i1 ? y[2 * k + 1] : 0.0;
    }
}

template <int T, int LOADS>
__global__ void __launch_bounds__(T) bin_count_smem_kernel(int g, const double* __restrict__ y, int64_t n, int64_t chunk,
                                                           int* __restrict__ counts)
{
    after_go();
    extern __shared__ int s_cnt[];
    const int nbox = 1 << (2 * g);
    for (int b = threadIdx.x; b < nbox; b += T) s_cnt[b] = 0;
    __syncthreads();
    const int64_t i0 = (int64_t)blockIdx.x * chunk, i1 = i0 + chunk < n ? i0 + chunk : n;
    for (int64_t i = i0 + threadIdx.x; i < i1; i += LOADS * T) {
        double a[LOADS], b[LOADS];
        load_points<T, LOADS>(y, i, i1, a, b);
#pragma unroll
        for (int u = 0; u < LOADS; ++u)
            if (i + u * T < i1) atomicAdd(&s_cnt[fgt_grid_box(a[u], b[u], g)], 1);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < nbox; b += T)
        if (s_cnt[b]) atomicAdd(&counts[b], s_cnt[b]);
}

// The scatter over chunks of up to LOADS points a thread: the counting addition gives a point
// its rank among the block's points of its box, which the thread keeps; the block reserves each
// touched box's range with one global atomic, and a point goes to that range's start + rank.  The
// coordinates are read once, with one shared atomic a point (a second pass over both before).
template <int T, int LOADS>
__global__ void __launch_bounds__(T) bin_scatter_smem_kernel(int g, const double* y, int64_t n, int64_t chunk,
                                                             int* __restrict__ cursor, int* __restrict__ perm)
{
    after_go();
    extern __shared__ int s_cnt[];
    const int nbox = 1 << (2 * g);
    for (int b = threadIdx.x; b < nbox; b += T) s_cnt[b] = 0;
    after_wait();
    __syncthreads();
    const int64_t i0 = (int64_t)blockIdx.x * chunk, i1 = i0 + chunk < n ? i0 + chunk : n, i = i0 + threadIdx.x;
    double a[LOADS], b[LOADS];
    load_points<T, LOADS>(y, i, i1, a, b);
    int box[LOADS], rank[LOADS];
#pragma unroll
    for (int u = 0; u < LOADS; ++u) {
        box[u] = fgt_grid_box(a[u], b[u], g);
        if (i + u * T < i1) rank[u] = atomicAdd(&s_cnt[box[u]], 1);
    }
    __syncthreads();
    for (int c = threadIdx.x; c < nbox; c += T)
        if (s_cnt[c]) s_cnt[c] = atomicAdd(&cursor[c], s_cnt[c]);  // this block's first slot in box c
    __syncthreads();
#pragma unroll
    for (int u = 0; u < LOADS; ++u)
        if (i + u * T < i1) perm[s_cnt[box[u]] + rank[u]] = (int)(i + u * T);
}

static int bin_grid(int64_t n)
{
    int sms = 0;
    if (device_sm_count(&sms) || sms <= 0) sms = 148;
    const int64_t want = (n + kBinThreads - 1) / kBinThreads;
    return (int)(want < 8LL * sms ? (want > 0 ? want : 1) : 8LL * sms);
}

// ---------------------------------------------------------------------------
// P2H from binned sources (Eq. A_alpha): a CTA takes 256 consecutive binned
// points, forms q t1^a1 / a1! and t2^a2 / a2! for each in shared memory, and a
// thread sums a 4 x 4 block of their products over one of 16 groups of 16
// consecutive points: two 16-byte shared loads feed 16 multiply-adds (a thread
// per coefficient read two words for each).  Where the CTA's points lie in one
// box the groups' sums meet in shared memory and A gets one addition per
// coefficient; otherwise each group adds its runs of one box to A itself, four
// coefficients an atomic where A is 16-byte aligned (VEC).
// 2^20 clustered sources on 32 x 32 boxes, p = 16: 87 -> 40 us, of which the points' gathers are
// about half.
// ---------------------------------------------------------------------------
constexpr int kP2hPoints = 256;
constexpr int kP2hGroups = 16;
constexpr int kP2hPer = kP2hPoints / kP2hGroups;

template <int P, bool VEC>
__global__ void __launch_bounds__(kP2hPoints) fgt_p2h_binned_kernel(int g, double inv_c, float dcell,
                                                                    const double* __restrict__ x,
                                                                    const double* __restrict__ q, int n,
                                                                    const int* __restrict__ perm,
                                                                    float* __restrict__ A, int* err)
{
    // row strides of whole 16-byte words whose multiples spread over the banks
    constexpr int S = P == 12 ? 20 : P + 4, T = P / 4;
    __shared__ __align__(16) float s_w1[kP2hPoints * S];
    __shared__ __align__(16) float s_w2[kP2hPoints * S];
    __shared__ int s_box[kP2hPoints];
    const int tid = threadIdx.x;
    const int base = blockIdx.x * kP2hPoints;
    const int cnt = min(kP2hPoints, n - base);
    if (tid < cnt) {
        const int j = perm[base + tid];
        if ((unsigned)j < (unsigned)n) {
            const double x0 = x[2 * (size_t)j], x1 = x[2 * (size_t)j + 1];
            const int side = 1 << g;
            int b;
            float t1, t2;
            long long X0, X1;
            if (grid_fixed31(x0, g, X0) && grid_fixed31(x1, g, X1)) {
                // offsets from the box centre in box sides, times side / (sqrt2 sigma)
                b = (int)(X1 >> 31) * side + (int)(X0 >> 31);
                t1 = cell_offset31(X0) * dcell;
                t2 = cell_offset31(X1) * dcell;
            } else {  // outside the unit square: clamped box, offset in FP64
                b = fgt_grid_box(x0, x1, g);
                t1 = (float)((x0 * side - ((b & (side - 1)) + 0.5)) / side * inv_c);
                t2 = (float)((x1 * side - ((b >> g) + 0.5)) / side * inv_c);
            }
            float w1[P], w2[P];
            w1[0] = (float)q[j];
            w2[0] = 1.f;
#pragma unroll
            for (int a = 1; a < P; ++a) {
                w1[a] = w1[a - 1] * t1 * (1.f / (float)a);
                w2[a] = w2[a - 1] * t2 * (1.f / (float)a);
            }
#pragma unroll
            for (int a = 0; a < P; a += 4) {
                *reinterpret_cast<float4*>(s_w1 + tid * S + a) = make_float4(w1[a], w1[a + 1], w1[a + 2], w1[a + 3]);
                *reinterpret_cast<float4*>(s_w2 + tid * S + a) = make_float4(w2[a], w2[a + 1], w2[a + 2], w2[a + 3]);
            }
            s_box[tid] = b;
        } else {
            atomicOr(err, DEV_ERR_CHECK);
            s_box[tid] = -1;
        }
    }
    bool one = true;  // every point of the CTA in the first one's box
    __syncthreads();
    if (tid < cnt) one = s_box[tid] == s_box[0];
    one = __syncthreads_and(one) && s_box[0] >= 0;

    const int group = tid / (T * T), tile = tid % (T * T), a1 = 4 * (tile / T), a2 = 4 * (tile % T);
    const bool work = group < kP2hGroups;
    float acc[4][4];
    auto clear = [&] {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    };
    auto flush = [&](int b) {
        float* dst = A + (size_t)b * P * P + a1 * P + a2;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if constexpr (VEC) {
                atomicAdd(reinterpret_cast<float4*>(dst + i * P), make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]));
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) atomicAdd(dst + i * P + j, acc[i][j]);
            }
        }
    };
    clear();
    if (work) {
        int cur = -1;
        for (int k = group * kP2hPer; k < min((group + 1) * kP2hPer, cnt); ++k) {
            if (!one) {
                const int b = s_box[k];
                if (b != cur) {
                    if (cur >= 0) flush(cur);
                    clear();
                    cur = b;
                }
                if (b < 0) continue;
            }
            const float4 u = *reinterpret_cast<const float4*>(s_w1 + k * S + a1);
            const float4 v = *reinterpret_cast<const float4*>(s_w2 + k * S + a2);
            const float uu[4] = {u.x, u.y, u.z, u.w}, vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(uu[i], vv[j], acc[i][j]);
        }
        if (!one && cur >= 0) flush(cur);
    }
    if (!one) return;  // the same for the whole block
    __syncthreads();   // the points' factors have been read: their room takes the groups' sums
    float* s_sum = s_w1;
    if (work)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) s_sum[group * P * P + (a1 + i) * P + a2 + j] = acc[i][j];
    __syncthreads();
    if (tid < P * P) {
        float v = 0.f;
#pragma unroll
        for (int k = 0; k < kP2hGroups; ++k) v += s_sum[k * P * P + tid];
        atomicAdd(&A[(size_t)s_box[0] * P * P + tid], v);
    }
}

// ---------------------------------------------------------------------------
// Hermite evaluation at binned targets
// ---------------------------------------------------------------------------
template <int P>
struct H2pCfg {
    // 4 targets per thread: each broadcast 16-byte load of A feeds 16 FMAs; 64-thread CTAs at
    // p >= 12 keep a claim at 256 targets (a box's last claim is partly idle)
    static constexpr int R = 4;                        // targets per thread
    static constexpr int THREADS = P >= 12 ? 64 : 128;
    static constexpr int CH = THREADS * R;             // targets per claim
    static constexpr int PP = P * P;
    static constexpr size_t smem = H2pSmem<P>::bytes;
};

struct H2pArgs : H2pSums {
    const int* claims;        // [nbox + 1] claim-index prefix over the boxes in `order`
    const int* order;         // [nbox] the boxes, heaviest neighbourhood first (h2p_order_*)
    int* cursor;  // [0] next claim index, [1] CTAs finished
};

// flag[b] = any coefficient of box b is non-zero (one warp per box)
__global__ void fgt_box_flags_kernel(const float* __restrict__ A, int nbox, int pp, unsigned char* __restrict__ flag)
{
    const int b = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (b >= nbox) return;
    bool nz = false;
    for (int i = lane; i < pp; i += 32) nz |= A[(size_t)b * pp + i] != 0.f;
    nz = __any_sync(0xffffffffu, nz);
    if (lane == 0) flag[b] = nz ? 1 : 0;
}

// claims[0..nbox]: exclusive scan of ceil(targets of box b / ch), the table that maps a claim
// index to its box; a box_start that decreases counts as empty and is reported.
__global__ void __launch_bounds__(kScanThreads) h2p_claims_kernel(int nbox, const int* __restrict__ box_start, int ch,
                                                                  int* __restrict__ claims, int* err)
{
    block_exclusive_scan(
        nbox,
        [&](int i) {
            const int m = box_start[i + 1] - box_start[i];
            if (m < 0) atomicOr(err, DEV_ERR_CHECK);
            return m > 0 ? (m + ch - 1) / ch : 0;
        },
        [](int, int) {}, claims);
}

// ---------------------------------------------------------------------------
// Claim order.  A claim's work is its targets times the non-empty source boxes of
// its box's n_cut neighbourhood, and a claim is large (a few hundred microseconds
// of one CTA), so claims handed out in box order leave SMs idle at the end of the
// launch.  The boxes are counting-sorted by that count, heaviest first (longest
// processing time first), and the claim table runs over that order.  Only the order
// in which claims are taken changes: every target is still evaluated by one thread
// with the same arithmetic.
// ---------------------------------------------------------------------------
constexpr int kH2pKeys = kH2pMaxBoxes + 2;  // neighbourhood counts 0..kH2pMaxBoxes, and "no targets"

// rp[y][x] = nz[y][0] + ... + nz[y][x]: one warp per grid row, 32 columns per step
__global__ void h2p_row_prefix_kernel(const unsigned char* __restrict__ nz, int g, int* __restrict__ rp)
{
    const int side = 1 << g, lane = threadIdx.x & 31;
    const int y = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5);
    if (y >= side) return;
    int carry = 0;
    for (int x0 = 0; x0 < side; x0 += 32) {
        const int x = x0 + lane;
        int v = x < side ? (int)(nz[(size_t)y * side + x] != 0) : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += t;
        }
        if (x < side) rp[(size_t)y * side + x] = carry + v;
        carry += __shfl_sync(0xffffffffu, v, 31);
    }
}

// key[b] = kH2pMaxBoxes - (non-empty source boxes within n_cut of b), or kH2pKeys - 1 for a box
// without targets; hist[key] counts the boxes of each key
__global__ void h2p_order_keys_kernel(const int* __restrict__ rp, const int* __restrict__ box_start, int g, int ncut,
                                      int* __restrict__ key, int* __restrict__ hist)
{
    const int side = 1 << g, nbox = side * side;
    const int b = (int)(blockIdx.x * (size_t)blockDim.x + threadIdx.x);
    if (b >= nbox) return;
    int k = kH2pKeys - 1;
    if (box_start[b + 1] > box_start[b]) {
        const int tx = b & (side - 1), ty = b >> g;
        const int x0 = max(tx - ncut, 0), x1 = min(tx + ncut, side - 1);
        const int y0 = max(ty - ncut, 0), y1 = min(ty + ncut, side - 1);
        int w = 0;
        for (int yy = y0; yy <= y1; ++yy) {
            const int* r = rp + (size_t)yy * side;
            w += r[x1] - (x0 > 0 ? r[x0 - 1] : 0);
        }
        k = kH2pMaxBoxes - w;
    }
    key[b] = k;
    atomicAdd(hist + k, 1);
}

// the boxes in key order (within a key in no particular order): a counting sort's scatter
__global__ void h2p_order_scatter_kernel(const int* __restrict__ key, int nbox, int* __restrict__ cursor,
                                         int* __restrict__ order)
{
    const int b = (int)(blockIdx.x * (size_t)blockDim.x + threadIdx.x);
    if (b >= nbox) return;
    order[atomicAdd(cursor + key[b], 1)] = b;
}

// cursor[0..kH2pKeys]: exclusive scan of the key histogram, the scatter cursors (one CTA)
__global__ void __launch_bounds__(kScanThreads) h2p_order_scan_kernel(const int* __restrict__ hist,
                                                                      int* __restrict__ cursor)
{
    block_exclusive_scan(
        kH2pKeys, [&](int i) { return hist[i]; }, [](int, int) {}, cursor);
}

// claims[0..nbox]: exclusive scan over the boxes in `order` of ceil(targets / ch)
__global__ void __launch_bounds__(kScanThreads) h2p_claims_ordered_kernel(int nbox, const int* __restrict__ box_start,
                                                                          const int* __restrict__ order, int ch,
                                                                          int* __restrict__ claims, int* err)
{
    block_exclusive_scan(
        nbox,
        [&](int i) {
            const int b = order[i];
            const int m = box_start[b + 1] - box_start[b];
            if (m < 0) atomicOr(err, DEV_ERR_CHECK);
            return m > 0 ? (m + ch - 1) / ch : 0;
        },
        [](int, int) {}, claims);
}

// The same for grids of up to kH2pOrderSmall boxes in one CTA (one launch instead of five):
// row prefix and key histogram in shared memory, then order and claims.
constexpr int kH2pOrderSmall = 4096;
constexpr int kH2pOrderPer = kH2pOrderSmall / kScanThreads;  // boxes per thread
__global__ void __launch_bounds__(kScanThreads) h2p_order_small_kernel(const unsigned char* __restrict__ nz,
                                                                       const int* __restrict__ box_start, int g,
                                                                       int ncut, int ch, int* __restrict__ order,
                                                                       int* __restrict__ claims, int* err)
{
    __shared__ int s_rp[kH2pOrderSmall];
    __shared__ int s_hist[kH2pKeys];
    __shared__ int s_cur[kH2pKeys + 1];
    const int tid = threadIdx.x, side = 1 << g, nbox = side * side;
    for (int b = tid; b < nbox; b += kScanThreads) s_rp[b] = nz[b] != 0;
    for (int k = tid; k < kH2pKeys; k += kScanThreads) s_hist[k] = 0;
    __syncthreads();
    if (tid < side) {
        int c = 0;
        for (int x = 0; x < side; ++x) s_rp[tid * side + x] = (c += s_rp[tid * side + x]);
    }
    __syncthreads();
    int key[kH2pOrderPer];
#pragma unroll
    for (int j = 0; j < kH2pOrderPer; ++j) {
        const int b = tid + j * kScanThreads;
        key[j] = -1;
        if (b >= nbox) continue;
        int k = kH2pKeys - 1;
        if (box_start[b + 1] > box_start[b]) {
            const int tx = b & (side - 1), ty = b >> g;
            const int x0 = max(tx - ncut, 0), x1 = min(tx + ncut, side - 1);
            const int y0 = max(ty - ncut, 0), y1 = min(ty + ncut, side - 1);
            int w = 0;
            for (int yy = y0; yy <= y1; ++yy) w += s_rp[yy * side + x1] - (x0 > 0 ? s_rp[yy * side + x0 - 1] : 0);
            k = kH2pMaxBoxes - w;
        }
        key[j] = k;
        atomicAdd(s_hist + k, 1);
    }
    __syncthreads();
    block_exclusive_scan(
        kH2pKeys, [&](int i) { return s_hist[i]; }, [](int, int) {}, s_cur);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kH2pOrderPer; ++j)
        if (key[j] >= 0) order[atomicAdd(s_cur + key[j], 1)] = tid + j * kScanThreads;
    __syncthreads();  // the order, written by this block, is visible to it
    block_exclusive_scan(
        nbox,
        [&](int i) {
            const int b = order[i];
            const int m = box_start[b + 1] - box_start[b];
            if (m < 0) atomicOr(err, DEV_ERR_CHECK);
            return m > 0 ? (m + ch - 1) / ch : 0;
        },
        [](int, int) {}, claims);
}

// Claim k = the next unclaimed index: run [first, end) of at most ch binned targets of one box
// (the claim table runs over the boxes in a.order).  Returns false when no claim is left.
__device__ bool h2p_claim(const H2pArgs& a, int nbox, int ch, int* first, int* end, int* box)
{
    const int total = __ldg(a.claims + nbox);
    const int k = atomicAdd(a.cursor, 1);
    if (k >= total) return false;
    h2p_claim_range_ordered(a.claims, a.order, a.box_start, nbox, nbox, a.n, ch, k, first, end, box);
    if (*first >= *end) atomicOr(a.err, DEV_ERR_CHECK);  // box_start does not bin [0, n)
    return true;
}

template <int P>
__global__ void __launch_bounds__(H2pCfg<P>::THREADS) fgt_h2p_kernel(H2pArgs a)
{
    using C = H2pCfg<P>;
    extern __shared__ float4 h2p_smem[];
    __shared__ H2pShared<C::THREADS> sh;
    __shared__ int s_claim[4];
    const int tid = threadIdx.x, side = 1 << a.g, nbox = side * side;
    h2p_offsets(sh, a);

    for (;;) {
        if (tid == 0) {
            int f = 0, e = 0, b = 0;
            if (!h2p_claim(a, nbox, C::CH, &f, &e, &b)) f = e = -1;
            s_claim[0] = f;
            s_claim[1] = e;
            s_claim[2] = b;
        }
        __syncthreads();
        const int first = s_claim[0], end = s_claim[1], box = s_claim[2];
        if (first < 0) break;
        if (first >= end) {  // an inconsistent claim (reported); keep s_claim stable until all have read it
            __syncthreads();
            continue;
        }
        h2p_run<P, C::R, C::THREADS>(a, sh, reinterpret_cast<float*>(h2p_smem), first, end, box);
    }
    // the last CTA to finish returns the cursor slot to zero for its next use
    if (tid == 0) {
        __threadfence();
        if (atomicAdd(a.cursor + 1, 1) == (int)gridDim.x - 1) {
            atomicExch(a.cursor, 0);
            atomicExch(a.cursor + 1, 0);
        }
    }
}

int launch_h2p_claims(int nbox, const int* box_start, int ch, int* claims, int* err, cudaStream_t st)
{
    h2p_claims_kernel<<<1, kScanThreads, 0, st>>>(nbox, box_start, ch, claims, err);
    FMM_CUDA_TRY(cudaGetLastError());
    return FMM_OK;
}

// The claim order and the claim table over it, runs of ch targets: one CTA for grids of up to
// kH2pOrderSmall boxes, else row prefix, keys, histogram scan, scatter and claims as five
// launches.  nz: the source boxes' non-empty flags (already set); order points at the scratch
// words after the claims array.
static int h2p_order_claims(const unsigned char* nz, const int* box_start, int g, int ncut, int ch, int* order, int* claims,
                     int* err, cudaStream_t st)
{
    const int nbox = 1 << (2 * g), side = 1 << g;
    if (nbox <= kH2pOrderSmall) {
        h2p_order_small_kernel<<<1, kScanThreads, 0, st>>>(nz, box_start, g, ncut, ch, order, claims, err);
        FMM_CUDA_TRY(cudaGetLastError());
        return FMM_OK;
    }
    int* rp = order + nbox;               // [nbox] row prefix of the flags
    int* hist = rp + nbox;                // [kH2pKeys] key histogram
    int* cursor = hist + kH2pKeys;        // [kH2pKeys + 1] scatter cursors (their scan, total last)
    int* key = cursor + kH2pKeys + 1;     // [nbox]
    FMM_CUDA_TRY(cudaMemsetAsync(hist, 0, sizeof(int) * kH2pKeys, st));
    h2p_row_prefix_kernel<<<(side * 32 + 255) / 256, 256, 0, st>>>(nz, g, rp);
    FMM_CUDA_TRY(cudaGetLastError());
    h2p_order_keys_kernel<<<(nbox + 255) / 256, 256, 0, st>>>(rp, box_start, g, ncut, key, hist);
    FMM_CUDA_TRY(cudaGetLastError());
    h2p_order_scan_kernel<<<1, kScanThreads, 0, st>>>(hist, cursor);
    FMM_CUDA_TRY(cudaGetLastError());
    h2p_order_scatter_kernel<<<(nbox + 255) / 256, 256, 0, st>>>(key, nbox, cursor, order);
    FMM_CUDA_TRY(cudaGetLastError());
    h2p_claims_ordered_kernel<<<1, kScanThreads, 0, st>>>(nbox, box_start, order, ch, claims, err);
    FMM_CUDA_TRY(cudaGetLastError());
    return FMM_OK;
}

template <int P>
static void p2h_binned_launch(int g, double inv_c, float dcell, const double* x, const double* q, int n,
                              const int* perm, float* A, int* err, unsigned grid, cudaStream_t st)
{
    if (((uintptr_t)A & 15) == 0)
        fgt_p2h_binned_kernel<P, true><<<grid, kP2hPoints, 0, st>>>(g, inv_c, dcell, x, q, n, perm, A, err);
    else
        fgt_p2h_binned_kernel<P, false><<<grid, kP2hPoints, 0, st>>>(g, inv_c, dcell, x, q, n, perm, A, err);
}

template <int P>
static int h2p_launch(const H2pArgs& args, cudaStream_t st)
{
    using C = H2pCfg<P>;
    static unsigned long long opted;
    static int occ;
    static std::mutex mu;
    if (int rc = smem_opt_in((const void*)fgt_h2p_kernel<P>, (int)C::smem, &opted)) return rc;
    {
        std::lock_guard<std::mutex> lk(mu);
        if (!occ) {
            FMM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fgt_h2p_kernel<P>, C::THREADS, C::smem));
            if (occ < 1) occ = 1;
        }
    }
    int sms = 0;
    if (int rc = device_sm_count(&sms)) return rc;
    const int nbox = 1 << (2 * args.g);
    fgt_box_flags_kernel<<<(nbox + 7) / 8, 256, 0, st>>>(args.A, nbox, C::PP, const_cast<unsigned char*>(args.nz));
    FMM_CUDA_TRY(cudaGetLastError());
    // the claim order (heaviest neighbourhood first), then the claim table over it
    if (int rc = h2p_order_claims(args.nz, args.box_start, args.g, args.ncut, C::CH, const_cast<int*>(args.order),
                                  const_cast<int*>(args.claims), args.err, st))
        return rc;
    const int64_t most = (int64_t)args.n / C::CH + nbox;  // claims can be no more
    const int grid = (int)std::min<int64_t>((int64_t)occ * sms, most > 0 ? most : 1);
    fgt_h2p_kernel<P><<<grid, C::THREADS, C::smem, st>>>(args);
    FMM_CUDA_TRY(cudaGetLastError());
    return FMM_OK;
}

}  // namespace fmmgb

using namespace fmmgb;

extern "C" int fgt_bin_points(int32_t grid_log2, const double* y, int64_t n, int32_t* perm, int32_t* box_start,
                              int32_t* work, void* stream)
{
    clear_error();
    if (grid_log2 < 0 || grid_log2 > 10) return fail(FMM_EINVAL, "fgt_bin_points: grid_log2 %d outside 0..10", grid_log2);
    if (n < 0 || n > INT32_MAX) return fail(FMM_EINVAL, "fgt_bin_points: n = %lld outside 0..2^31-1", (long long)n);
    if (!box_start || !work || (n > 0 && (!y || !perm))) return fail(FMM_EINVAL, "fgt_bin_points: NULL pointer");
    if (((uintptr_t)y & 7) || ((uintptr_t)perm & 3) || ((uintptr_t)box_start & 3) || ((uintptr_t)work & 3))
        return fail(FMM_EINVAL, "fgt_bin_points: misaligned pointer (y 8 bytes, int32 arrays 4)");
    const int nbox = 1 << (2 * grid_log2);
    if ((const void*)work < (const void*)(box_start + nbox + 1) && (const void*)box_start < (const void*)(work + nbox))
        return fail(FMM_EINVAL, "fgt_bin_points: work overlaps box_start");
    cudaStream_t st = (cudaStream_t)stream;
    FMM_CUDA_TRY(cudaMemsetAsync(work, 0, sizeof(int) * (size_t)nbox, st));
    const bool smem = grid_log2 <= kBinSmemMaxLog2;
    const int smem_bytes = smem ? (int)sizeof(int) * nbox : 0;
    // 0: 256 threads x 4 points, 1: 512 x 8, 2: 1024 x 4 (the lines: above the kernels)
    const int form = grid_log2 >= 6 && n >= 1 << 15 ? 2 : grid_log2 < 6 && n >= 1 << 19 ? 1 : 0;
    const int threads = 256 << form, most = form ? 4096 : 1024;
    using Count = void (*)(int, const double*, int64_t, int64_t, int*);
    using Scatter = void (*)(int, const double*, int64_t, int64_t, int*, int*);
    static constexpr Count counts[] = {bin_count_smem_kernel<256, 4>, bin_count_smem_kernel<512, 8>,
                                        bin_count_smem_kernel<1024, 4>};
    static constexpr Scatter scatters[] = {bin_scatter_smem_kernel<256, 4>, bin_scatter_smem_kernel<512, 8>,
                                           bin_scatter_smem_kernel<1024, 4>};
    int grid = bin_grid(n);
    int64_t chunk = 0;
    if (smem && n > 0) {
        // every form opted in by the first call on a device, for the largest such grid: no later call,
        // in a capture or not, is a form's first
        static unsigned long long all, opted[3][2];
        int dev = 0;
        FMM_CUDA_TRY(cudaGetDevice(&dev));
        if (dev < 0 || dev >= 64 || !(__atomic_load_n(&all, __ATOMIC_ACQUIRE) >> dev & 1)) {
            constexpr int kMaxBytes = (int)sizeof(int) << (2 * kBinSmemMaxLog2);
            for (int f = 0; f < 3; ++f) {
                if (int rc = smem_opt_in((const void*)counts[f], kMaxBytes, &opted[f][0])) return rc;
                if (int rc = smem_opt_in((const void*)scatters[f], kMaxBytes, &opted[f][1])) return rc;
            }
            __atomic_fetch_or(&all, 1ull << dev, __ATOMIC_RELEASE);
        }
        int sms = 0;
        if (device_sm_count(&sms) || sms <= 0) sms = 148;
        grid = (int)std::min<int64_t>(2LL * sms, (n + threads - 1) / threads);
        chunk = (n + grid - 1) / grid;
    }
    if (n > 0) {
        if (smem)
            counts[form]<<<grid, threads, smem_bytes, st>>>(grid_log2, y, n, chunk, work);
        else
            bin_count_kernel<<<grid, kBinThreads, 0, st>>>(grid_log2, y, n, work);
        FMM_CUDA_TRY(cudaGetLastError());
    }
    if (nbox <= kScanTile) {
        FMM_CUDA_TRY(launch_after(bin_scan_kernel, 1, kScanThreads, 0, st, nbox, work, box_start));
    } else {
        FMM_CUDA_TRY(launch_after(bin_scan_tiles_kernel, nbox / kScanTile, kScanThreads, 0, st, nbox, work, box_start));
        FMM_CUDA_TRY(cudaMemcpyAsync(work, box_start, sizeof(int) * (size_t)nbox, cudaMemcpyDeviceToDevice, st));
    }
    if (n > 0) {
        if (smem) {
            chunk = std::min<int64_t>(chunk, most);  // points of a scatter block
            FMM_CUDA_TRY(launch_after(scatters[form], (unsigned)((n + chunk - 1) / chunk), threads, smem_bytes, st, grid_log2, y, n,
                                      chunk, work, perm));
        } else {
            FMM_CUDA_TRY(launch_after(bin_scatter_kernel, grid, kBinThreads, 0, st, grid_log2, y, n, work, perm));
        }
    }
    return FMM_OK;
}

extern "C" int fmm_bin_points(int32_t level, const double* y, int64_t n, int32_t* perm, int32_t* box_start,
                              int32_t* work, void* stream)
{
    // the boxes of quadtree level l are the cells of the 2^l x 2^l grid (reading R5)
    return fgt_bin_points(level, y, n, perm, box_start, work, stream);
}

extern "C" int fgt_p2h_binned(int32_t grid_log2, int32_t p, double sigma, const double* x, const double* q, int64_t n,
                              const int32_t* perm, float* A, int32_t flags, void* stream)
{
    clear_error();
    if (grid_log2 < 0 || grid_log2 > 10) return fail(FMM_EINVAL, "fgt_p2h_binned: grid_log2 %d outside 0..10", grid_log2);
    if (!fgt_supported(p)) return fail(FMM_EINVAL, "fgt_p2h_binned: unsupported p = %d (4, 8, 12, 16)", p);
    if (!(sigma > 0.0) || !(sigma < 1e300)) return fail(FMM_EINVAL, "fgt_p2h_binned: sigma must be positive and finite");
    if (n < 0 || n > INT32_MAX) return fail(FMM_EINVAL, "fgt_p2h_binned: n = %lld outside 0..2^31-1", (long long)n);
    if (!A || (n > 0 && (!x || !q || !perm))) return fail(FMM_EINVAL, "fgt_p2h_binned: NULL pointer");
    if (((uintptr_t)x & 7) || ((uintptr_t)q & 7) || ((uintptr_t)perm & 3) || ((uintptr_t)A & 3))
        return fail(FMM_EINVAL, "fgt_p2h_binned: misaligned pointer");
    if (flags & ~FMM_ACCUMULATE) return fail(FMM_EINVAL, "fgt_p2h_binned: unknown flags 0x%x", flags);
    cudaStream_t st = (cudaStream_t)stream;
    const size_t bytes = ((size_t)1 << (2 * grid_log2)) * (size_t)p * p * sizeof(float);
    if (!(flags & FMM_ACCUMULATE)) FMM_CUDA_TRY(cudaMemsetAsync(A, 0, bytes, st));
    if (n == 0) return FMM_OK;
    int* err = nullptr;
    if (int rc = device_error_word(&err)) return rc;
    const unsigned grid = (unsigned)((n + kP2hPoints - 1) / kP2hPoints);
    const double inv_c = 1.0 / (sqrt(2.0) * sigma);
    const float dcell = (float)(ldexp(1.0, -grid_log2) * inv_c);  // box side / (sqrt2 sigma)
    const int nn = (int)n;
    switch (p) {
        case 4: p2h_binned_launch<4>(grid_log2, inv_c, dcell, x, q, nn, perm, A, err, grid, st); break;
        case 8: p2h_binned_launch<8>(grid_log2, inv_c, dcell, x, q, nn, perm, A, err, grid, st); break;
        case 12: p2h_binned_launch<12>(grid_log2, inv_c, dcell, x, q, nn, perm, A, err, grid, st); break;
        default: p2h_binned_launch<16>(grid_log2, inv_c, dcell, x, q, nn, perm, A, err, grid, st); break;
    }
    FMM_CUDA_TRY(cudaGetLastError());
    return FMM_OK;
}

extern "C" int fgt_h2p(int32_t grid_log2, int32_t n_cut, int32_t p, int32_t prec, double sigma, const float* A,
                       const double* y, int64_t n, const int32_t* perm, const int32_t* box_start, float* G,
                       int32_t flags, void* stream)
{
    clear_error();
    if (prec == FMM_TC_TF32X3) return fail(FMM_EUNSUPPORTED, "fgt_h2p: FMM_TC_TF32X3 is an M2L precision");
    if (prec != FMM_FP32 && prec != FMM_TC_BF16X3 && prec != FMM_TC_BF16)
        return fail(FMM_EINVAL, "fgt_h2p: unknown precision %d", prec);
    if (prec != FMM_FP32 && p != 16)
        return fail(FMM_EUNSUPPORTED, "fgt_h2p: the tensor-core forms take p = 16 (got %d)", p);
    if (prec != FMM_FP32 && n_cut > 15)
        return fail(FMM_EUNSUPPORTED, "fgt_h2p: the tensor-core forms take n_cut <= 15 (got %d)", n_cut);
    if (grid_log2 < 0 || grid_log2 > 10) return fail(FMM_EINVAL, "fgt_h2p: grid_log2 %d outside 0..10", grid_log2);
    if (n_cut < 0 || n_cut > kH2pMaxCut) return fail(FMM_EINVAL, "fgt_h2p: n_cut %d outside 0..%d", n_cut, kH2pMaxCut);
    if (!fgt_supported(p)) return fail(FMM_EINVAL, "fgt_h2p: unsupported p = %d (4, 8, 12, 16)", p);
    if (!(sigma > 0.0) || !(sigma < 1e300)) return fail(FMM_EINVAL, "fgt_h2p: sigma must be positive and finite");
    if (n < 0 || n > INT32_MAX) return fail(FMM_EINVAL, "fgt_h2p: n = %lld outside 0..2^31-1", (long long)n);
    if (!A || !box_start || (n > 0 && (!y || !perm || !G))) return fail(FMM_EINVAL, "fgt_h2p: NULL pointer");
    if (((uintptr_t)A & 15) || ((uintptr_t)y & 7) || ((uintptr_t)perm & 3) || ((uintptr_t)box_start & 3) ||
        ((uintptr_t)G & 3))
        return fail(FMM_EINVAL, "fgt_h2p: misaligned pointer (A 16 bytes, y 8, the rest 4)");
    if (flags & ~FMM_ACCUMULATE) return fail(FMM_EINVAL, "fgt_h2p: unknown flags 0x%x", flags);
    if (n == 0) return FMM_OK;
    H2pArgs args;
    args.g = grid_log2;
    args.ncut = n_cut;
    args.n = (int)n;
    args.d = ldexp(1.0, -grid_log2) / (sqrt(2.0) * sigma);
    args.A = A;
    args.y = y;
    args.perm = perm;
    args.box_start = box_start;
    args.G = G;
    args.accumulate = (flags & FMM_ACCUMULATE) ? 1 : 0;
    cudaStream_t st = (cudaStream_t)stream;
    if (int rc = device_error_word(&args.err)) return rc;
    if (int rc = tile_counter(&args.cursor, st)) return rc;  // whichever form serves a first call, a captured one may take the other
    // every precision: the Chebyshev form is FP32 throughout and faster than either direct form
    bool done = false;
    if (int rc = launch_fgt_h2p_cheb(grid_log2, n_cut, p, args.d, A, y, args.n, perm, box_start, G,
                                     args.accumulate != 0, args.err, st, &done))
        return rc;
    if (done) return FMM_OK;
    unsigned char* nzbuf = nullptr;
    if (int rc = fgt_flag_buffer(&nzbuf)) return rc;
    args.nz = nzbuf;
    args.claims = reinterpret_cast<const int*>(nzbuf + kFgtFlagBytes);
    args.order = args.claims + ((size_t)1 << 20) + 1;
    if (prec != FMM_FP32) {
        const int nbox = 1 << (2 * grid_log2);
        if (int rc = launch_h2p_claims(nbox, box_start, 128, const_cast<int*>(args.claims), args.err, st)) return rc;
        return launch_fgt_h2p_tc(grid_log2, n_cut, args.d, prec == FMM_TC_BF16X3, A, y, args.n, perm, box_start,
                                 args.claims, G, args.accumulate != 0, args.err, st);
    }
    switch (p) {
        case 4: return h2p_launch<4>(args, st);
        case 8: return h2p_launch<8>(args, st);
        case 12: return h2p_launch<12>(args, st);
        default: return h2p_launch<16>(args, st);
    }
}
