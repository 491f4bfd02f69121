// fgt_eval.cu -- Taylor-series evaluation of the fast Gauss transform at
// target points (Sec. 2.2, Eq. taylor): each target takes the Taylor
// coefficients C of its own box of the uniform grid,
//   G(y) (+)= sum_{b1,b2 < p} C[box][b1][b2] t1^b1 t2^b2,  t = (y - t_C) / (sqrt(2) sigma).
// With P2H and H2T this completes the transform on the device.  Horner in
// FP32 on t formed in FP64 (|t| <= 0.36 on the workload grids).
#include "fgt_hermite.cuh"

namespace fmmgb {

template <int P>
__global__ void fgt_t2p_kernel(int g, double inv_scale, const float* __restrict__ C, int64_t n,
                               const double* __restrict__ y, float* __restrict__ G, int accumulate)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int side = 1 << g;
    const double px = y[2 * i] * side, py = y[2 * i + 1] * side;
    int ix = (int)floor(px), iy = (int)floor(py);
    ix = ix < 0 ? 0 : (ix > side - 1 ? side - 1 : ix);
    iy = iy < 0 ? 0 : (iy > side - 1 ? side - 1 : iy);
    const float t1 = (float)((px - (ix + 0.5)) / side * inv_scale);
    const float t2 = (float)((py - (iy + 0.5)) / side * inv_scale);
    const float4* cb = reinterpret_cast<const float4*>(C + ((size_t)iy * side + ix) * P * P);
    float outer = 0.f;
#pragma unroll 1
    for (int b1 = P - 1; b1 >= 0; --b1) {
        float row[P];
#pragma unroll
        for (int q = 0; q < P / 4; ++q) {
            const float4 v = __ldg(cb + b1 * (P / 4) + q);
            row[4 * q] = v.x;
            row[4 * q + 1] = v.y;
            row[4 * q + 2] = v.z;
            row[4 * q + 3] = v.w;
        }
        float inner = 0.f;
#pragma unroll
        for (int b2 = P - 1; b2 >= 0; --b2) inner = fmaf(inner, t2, row[b2]);
        outer = fmaf(outer, t1, inner);
    }
    G[i] = accumulate ? G[i] + outer : outer;
}

template <int P>
static int t2p_p(int g, double sigma, const float* C, int64_t n, const double* y, float* G, bool acc, cudaStream_t st)
{
    fgt_t2p_kernel<P><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(g, 1.0 / (sqrt(2.0) * sigma), C, n, y, G,
                                                                   acc ? 1 : 0);
    FMM_CUDA_TRY(cudaGetLastError());
    return FMM_OK;
}

// T2P at targets binned by box (fgt_bin_points).  A warp takes 128 consecutive binned targets,
// four per lane: where they share a box, each uniform 16-byte load of its coefficients (served
// by the L1) feeds 16 multiply-adds a lane; else a row of 32 targets at a time, each lane from
// its own box.  A warp's work does not depend on how the targets are spread over the boxes (a
// block per box left the SMs waiting for the crowded boxes), and a scalar shared load per
// multiply-add is gone.  Target offsets are read off the bits of the FP64 coordinates.
// 2^20 uniform targets on 32 x 32 boxes, p = 16: 40 -> 26 us, bound by the gathers and the
// scattered results.
// Fewer than kT2pWide targets leave the SMs warps to spare: one target a lane, since four rows
// one after the other are four times the latency (p = 16, 32 x 32 boxes, us, one / four: 300 targets 7.0 / 16.7,
// 10^4 4.7 / 12.3, 2*10^5 9.5 / 11.3, 3*10^5 14.1 / 12.0, 2^20 38 / 26).  Fewer than kT2pSplit: four lanes a
// target, a quarter of its coefficients' rows each (1 to 4^10 boxes, all p, four lanes against one: 0.8 of the time for 30 to
// 3,000 targets, 0.90 for 10^4, 0.97 for 2*10^4, 1.06 for 3*10^4).
constexpr int kT2pThreads = 128;
constexpr int64_t kT2pWide = 1 << 18, kT2pSplit = 1 << 14;

template <bool VEC>
__device__ __forceinline__ float4 t2p_load4(const float* c)
{
    if constexpr (VEC) return *reinterpret_cast<const float4*>(c);
    return make_float4(c[0], c[1], c[2], c[3]);
}

// sum_{b1 < B, b2 < P} c[b1][b2] t1^b1 t2^b2 by Horner's rule, NR targets of one box (NR = 1: a box per lane)
template <int P, int B, int NR, bool VEC>
__device__ __forceinline__ void t2p_sum(const float* c, const float* t1, const float* t2, float* out)
{
#pragma unroll
    for (int r = 0; r < NR; ++r) out[r] = 0.f;
#pragma unroll (NR == 1 ? B : 4)
    for (int b1 = B - 1; b1 >= 0; --b1) {
        float inner[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) inner[r] = 0.f;
#pragma unroll
        for (int q = P / 4 - 1; q >= 0; --q) {
            const float4 v = t2p_load4<VEC>(c + b1 * P + 4 * q);
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                inner[r] = fmaf(inner[r], t2[r], v.w);
                inner[r] = fmaf(inner[r], t2[r], v.z);
                inner[r] = fmaf(inner[r], t2[r], v.y);
                inner[r] = fmaf(inner[r], t2[r], v.x);
            }
        }
#pragma unroll
        for (int r = 0; r < NR; ++r) out[r] = fmaf(out[r], t1[r], inner[r]);
    }
}

template <int P, bool VEC, int ROWS, int SPLIT>
__global__ void __launch_bounds__(kT2pThreads) fgt_t2p_binned_kernel(int g, double inv_scale, float dcell,
                                                                     const float* C, int n, const double* y,
                                                                     const int* perm, const int* box_start,
                                                                     float* __restrict__ G, int accumulate, int* err)
{
    const int lane = threadIdx.x & 31, side = 1 << g, nbox = side * side, part = lane % SPLIT;
    after_wait();
    const int64_t base = ((int64_t)blockIdx.x * (kT2pThreads / 32) + (threadIdx.x >> 5)) * (32 * ROWS / SPLIT);
    bin_check(box_start, nbox, n, err);
    if (base >= n) return;
    int tj[ROWS], tb[ROWS];
    float t1[ROWS], t2[ROWS], out[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        const int64_t pos = base + 32 * r + lane / SPLIT;
        tj[r] = tb[r] = -1;
        t1[r] = t2[r] = out[r] = 0.f;
        if (pos >= n) continue;
        const int j = perm[pos];
        if ((unsigned)j >= (unsigned)n) {
            atomicOr(err, DEV_ERR_CHECK);
            continue;
        }
        const double y0 = y[2 * (size_t)j], y1 = y[2 * (size_t)j + 1];
        long long X0, X1;
        if (grid_fixed31(y0, g, X0) && grid_fixed31(y1, g, X1)) {
            const int b = (int)(X1 >> 31) * side + (int)(X0 >> 31);
            if (bin_holds(box_start, b, (int)pos, n)) {
                tj[r] = j;
                tb[r] = b;
                t1[r] = cell_offset31(X0) * dcell;
                t2[r] = cell_offset31(X1) * dcell;
            }
        }
        if (tb[r] < 0) {  // not in the box of its coordinates: the box the binning assigns, offset in FP64
            const int b = bin_find(box_start, nbox, (int)pos, n);
            if (b >= 0) {
                tj[r] = j;
                tb[r] = b;
                t1[r] = (float)((y0 * side - ((b & (side - 1)) + 0.5)) / side * inv_scale);
                t2[r] = (float)((y1 * side - ((b >> g) + 0.5)) / side * inv_scale);
            } else {  // box_start does not bin [0, n)
                atomicOr(err, DEV_ERR_CHECK);
            }
        }
    }
    if constexpr (SPLIT > 1) {
        constexpr int B = P / SPLIT;
        if (tb[0] >= 0) {
            t2p_sum<P, B, 1, VEC>(C + (size_t)tb[0] * P * P + part * B * P, t1, t2, out);
            for (int k = 0; k < part * B; ++k) out[0] *= t1[0];
        }
#pragma unroll
        for (int o = 1; o < SPLIT; o <<= 1) out[0] += __shfl_xor_sync(0xffffffffu, out[0], o);
        if (tj[0] >= 0 && part == 0) G[tj[0]] = accumulate ? G[tj[0]] + out[0] : out[0];
        return;
    }
    const int b0 = __shfl_sync(0xffffffffu, tb[0], 0);
    bool same = b0 >= 0;
#pragma unroll
    for (int r = 0; r < ROWS; ++r) same &= tb[r] == b0 || base + 32 * r + lane >= n;
    if (__all_sync(0xffffffffu, same)) {
        t2p_sum<P, P, ROWS, VEC>(C + (size_t)b0 * P * P, t1, t2, out);
    } else {
#pragma unroll
        for (int r = 0; r < ROWS; ++r)
            if (tb[r] >= 0) t2p_sum<P, P, 1, VEC>(C + (size_t)tb[r] * P * P, t1 + r, t2 + r, out + r);
    }
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
        if (tj[r] >= 0) G[tj[r]] = accumulate ? G[tj[r]] + out[r] : out[r];
}

template <int P>
static int t2p_binned_p(int g, double sigma, const float* C, int n, const double* y, const int* perm,
                        const int* box_start, float* G, bool acc, int* err, cudaStream_t st)
{
    const double inv_scale = 1.0 / (sqrt(2.0) * sigma);
    const float dcell = (float)(ldexp(1.0, -g) * inv_scale);
    const bool vec = ((uintptr_t)C & 15) == 0;
    const int per = n >= kT2pWide ? 4 * kT2pThreads : n >= kT2pSplit ? kT2pThreads : kT2pThreads / 4;  // targets a block
    const unsigned grid = bin_blocks(n, per, (int64_t)1 << (2 * g), kT2pThreads);
    auto kern = n >= kT2pWide    ? (vec ? fgt_t2p_binned_kernel<P, true, 4, 1> : fgt_t2p_binned_kernel<P, false, 4, 1>)
                : n >= kT2pSplit ? (vec ? fgt_t2p_binned_kernel<P, true, 1, 1> : fgt_t2p_binned_kernel<P, false, 1, 1>)
                                 : (vec ? fgt_t2p_binned_kernel<P, true, 1, 4> : fgt_t2p_binned_kernel<P, false, 1, 4>);
    FMM_CUDA_TRY(launch_after(kern, grid, kT2pThreads, 0, st, g, inv_scale, dcell, C, n, y, perm, box_start, G, acc ? 1 : 0,
                              err));
    return FMM_OK;
}

}  // namespace fmmgb

using namespace fmmgb;

extern "C" int fgt_t2p_binned(int32_t grid_log2, int32_t p, double sigma, const float* C, const double* y, int64_t n,
                              const int32_t* perm, const int32_t* box_start, float* G, int32_t flags, void* stream)
{
    clear_error();
    if (grid_log2 < 0 || grid_log2 > 10)
        return fail(FMM_EINVAL, "fgt_t2p_binned: grid_log2 %d outside 0..10", grid_log2);
    if (!fgt_supported(p)) return fail(FMM_EINVAL, "fgt_t2p_binned: unsupported p = %d (4, 8, 12, 16)", p);
    if (!(sigma > 0.0) || !(sigma < 1e300)) return fail(FMM_EINVAL, "fgt_t2p_binned: sigma must be positive and finite");
    if (n < 0 || n > INT32_MAX) return fail(FMM_EINVAL, "fgt_t2p_binned: n = %lld outside 0..2^31-1", (long long)n);
    if (!C || !box_start || (n > 0 && (!y || !G || !perm))) return fail(FMM_EINVAL, "fgt_t2p_binned: NULL pointer");
    if (((uintptr_t)C & 3) || ((uintptr_t)y & 7) || ((uintptr_t)G & 3) || ((uintptr_t)perm & 3) ||
        ((uintptr_t)box_start & 3))
        return fail(FMM_EINVAL, "fgt_t2p_binned: misaligned pointer");
    if (flags & ~FMM_ACCUMULATE) return fail(FMM_EINVAL, "fgt_t2p_binned: unknown flags 0x%x", flags);
    if (n == 0) return FMM_OK;
    int* err = nullptr;
    if (int rc = device_error_word(&err)) return rc;
    const bool acc = (flags & FMM_ACCUMULATE) != 0;
    cudaStream_t st = (cudaStream_t)stream;
    const int nn = (int)n;
    switch (p) {
        case 4: return t2p_binned_p<4>(grid_log2, sigma, C, nn, y, perm, box_start, G, acc, err, st);
        case 8: return t2p_binned_p<8>(grid_log2, sigma, C, nn, y, perm, box_start, G, acc, err, st);
        case 12: return t2p_binned_p<12>(grid_log2, sigma, C, nn, y, perm, box_start, G, acc, err, st);
        default: return t2p_binned_p<16>(grid_log2, sigma, C, nn, y, perm, box_start, G, acc, err, st);
    }
}

extern "C" int fgt_t2p(int32_t grid_log2, int32_t p, double sigma, const float* C, const double* y, int64_t n,
                       float* G, int32_t flags, void* stream)
{
    clear_error();
    if (grid_log2 < 0 || grid_log2 > 12) return fail(FMM_EINVAL, "fgt_t2p: grid_log2 %d outside 0..12", grid_log2);
    if (!fgt_supported(p)) return fail(FMM_EINVAL, "fgt_t2p: unsupported p = %d (4, 8, 12, 16)", p);
    if (!(sigma > 0.0) || !(sigma < 1e300)) return fail(FMM_EINVAL, "fgt_t2p: sigma must be positive and finite");
    if (n < 0) return fail(FMM_EINVAL, "fgt_t2p: n < 0");
    if (!C || (n > 0 && (!y || !G))) return fail(FMM_EINVAL, "fgt_t2p: NULL pointer");
    if (((uintptr_t)C & 15) || ((uintptr_t)y & 7) || ((uintptr_t)G & 3))
        return fail(FMM_EINVAL, "fgt_t2p: misaligned pointer (C 16 bytes, y 8, G 4)");
    if (flags & ~FMM_ACCUMULATE) return fail(FMM_EINVAL, "fgt_t2p: unknown flags 0x%x", flags);
    if (n == 0) return FMM_OK;
    const bool acc = (flags & FMM_ACCUMULATE) != 0;
    cudaStream_t st = (cudaStream_t)stream;
    switch (p) {
        case 4: return t2p_p<4>(grid_log2, sigma, C, n, y, G, acc, st);
        case 8: return t2p_p<8>(grid_log2, sigma, C, n, y, G, acc, st);
        case 12: return t2p_p<12>(grid_log2, sigma, C, n, y, G, acc, st);
        default: return t2p_p<16>(grid_log2, sigma, C, n, y, G, acc, st);
    }
}
