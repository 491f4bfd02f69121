// fgt_hermite.cuh -- device pieces shared by the FP32 and tensor-core forms of
// the FGT Hermite evaluation (Sec. 4.2, Eq. hermite).
#pragma once

#include "common.cuh"

namespace fmmgb {

// h_n(t) = exp(-t^2) H_n(t), n < P, by the three-term recurrence
// h_{n+1} = 2t h_n - 2n h_{n-1} (h_0 = exp(-t^2), h_1 = 2t exp(-t^2)).
template <int P>
__device__ __forceinline__ void hermite_functions(float t, float (&h)[P])
{
    const float tt = t + t;
    h[0] = __expf(-t * t);
    if (P > 1) h[1] = tt * h[0];
#pragma unroll
    for (int m = 1; m + 1 < P; ++m) h[m + 1] = fmaf(tt, h[m], -(float)(2 * m) * h[m - 1]);
}

// Binned targets taken by place rather than by box.  bin_check (all threads of the grid): a box
// whose start or end lies outside [0, n] or that ends before it starts sets the error word.
__device__ __forceinline__ bool bin_range_ok(int first, int end, int n) { return 0 <= first && first <= end && end <= n; }
__device__ __forceinline__ void bin_check(const int* box_start, int nbox, int n, int* err)
{
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < nbox; b += (int64_t)gridDim.x * blockDim.x)
        if (!bin_range_ok(box_start[b], box_start[b + 1], n)) atomicOr(err, DEV_ERR_CHECK);
}
// Whether place pos lies in box b's run.
__device__ __forceinline__ bool bin_holds(const int* box_start, int b, int pos, int n)
{
    const int f = box_start[b], e = box_start[b + 1];
    return bin_range_ok(f, e, n) && f <= pos && pos < e;
}
// The box whose run holds place pos (by bisection), -1 if none does.
__device__ __forceinline__ int bin_find(const int* box_start, int nbox, int pos, int n)
{
    int lo = 0, hi = nbox;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (box_start[mid] <= pos) lo = mid;
        else hi = mid;
    }
    return bin_holds(box_start, lo, pos, n) ? lo : -1;
}
// Blocks of `threads` for n places at `per` a block and a check of nbox boxes at 8 a thread.
inline unsigned bin_blocks(int64_t n, int64_t per, int64_t nbox, int64_t threads)
{
    const int64_t a = (n + per - 1) / per, b = (nbox + 8 * threads - 1) / (8 * threads);
    return (unsigned)(a > b ? a : b);
}

// The run of binned targets that claim k covers: claims[b] is the exclusive
// prefix over boxes of ceil(targets of b / ch) (launch_h2p_claims), so claim k
// belongs to the box b with claims[b] <= k < claims[b+1] and covers
// [box_start[b] + (k - claims[b]) ch, ... + ch) clipped to the box.  An
// inconsistent box_start gives first >= end.
__device__ __forceinline__ void h2p_claim_range(const int* __restrict__ claims, const int* __restrict__ box_start,
                                                int nbox, int n, int ch, int k, int* first, int* end, int* box)
{
    int lo = 0, hi = nbox;  // largest b with claims[b] <= k
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(claims + mid) <= k) lo = mid;
        else hi = mid;
    }
    const int f = __ldg(box_start + lo) + (k - __ldg(claims + lo)) * ch;
    const int e = min(min(f + ch, __ldg(box_start + lo + 1)), n);
    const bool ok = 0 <= f && f < e;
    *first = ok ? f : 0;
    *end = ok ? e : 0;
    *box = lo;
}

// The same with the claim table over the nlist boxes in `order` (position i holds box order[i]).
__device__ __forceinline__ void h2p_claim_range_ordered(const int* claims, const int* order,
                                                        const int* box_start, int nbox, int nlist, int n,
                                                        int ch, int k, int* first, int* end, int* box)
{
    int lo = 0, hi = nlist;  // largest position i with claims[i] <= k
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (claims[mid] <= k) lo = mid;
        else hi = mid;
    }
    const int b = order[lo];
    const bool inb = (unsigned)b < (unsigned)nbox;
    const int f = inb ? box_start[b] + (k - claims[lo]) * ch : 0;
    const int e = inb ? min(min(f + ch, box_start[b + 1]), n) : 0;
    const bool ok = inb && 0 <= f && f < e;
    *first = ok ? f : 0;
    *end = ok ? e : 0;
    *box = ok ? b : 0;
}

// ---------------------------------------------------------------------------
// Direct Hermite sums (a CTA of NT threads, R targets a thread)
// ---------------------------------------------------------------------------
constexpr int kH2pMaxCut = 16;
constexpr int kH2pMaxBoxes = (2 * kH2pMaxCut + 1) * (2 * kH2pMaxCut + 1);
constexpr int kH2pBatch = 8;                  // source boxes per shared-memory stage
constexpr int kH2pStages = 3;                 // ring depth (two batches in flight)

struct H2pSums {
    int g, ncut, n;
    double d;  // box side / (sqrt2 sigma)
    const float* A;
    const double* y;
    const int* perm;
    const int* box_start;
    const unsigned char* nz;  // per source box: any non-zero coefficient
    float* G;
    int accumulate;
    int* err;
};

template <int NT>
struct H2pShared {
    float off[2 * kH2pMaxCut + 1];  // k d, k = -ncut .. ncut
    short list[kH2pMaxBoxes];       // non-empty source boxes, row-major, as (dy + ncut) * 64 + dx + ncut
    int warp_cnt[NT / 32];
};
template <int P>
struct H2pSmem {  // the ring of coefficients [kH2pStages][kH2pBatch][P][P]
    static constexpr size_t bytes = (size_t)kH2pStages * kH2pBatch * P * P * sizeof(float);
};

template <int NT>
__device__ __forceinline__ void h2p_offsets(H2pShared<NT>& sh, const H2pSums& a)  // before h2p_run, with a barrier between
{
    if (threadIdx.x < 2 * a.ncut + 1) sh.off[threadIdx.x] = (float)((double)((int)threadIdx.x - a.ncut) * a.d);
}

__device__ __forceinline__ void cp_async_16(void* smem, const void* gmem)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// G of the binned targets [first, end) of `box`, at most NT R of them; all threads call it, with a barrier
// between two calls.
template <int P, int R, int NT>
__device__ __forceinline__ void h2p_run(const H2pSums& a, H2pShared<NT>& sh, float* sA, int first, int end, int box)
{
    constexpr int PP = P * P;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int side = 1 << a.g, tx = box & (side - 1), ty = box >> a.g;
    const int x0 = max(tx - a.ncut, 0), x1 = min(tx + a.ncut, side - 1);
    const int y0 = max(ty - a.ncut, 0), y1 = min(ty + a.ncut, side - 1);
    const int w = x1 - x0 + 1, nb = w * (y1 - y0 + 1);

    // ordered compaction of the neighbourhood's non-empty source boxes (row-major)
    int total = 0;
    for (int base = 0; base < nb; base += NT) {
        const int i = base + tid;
        bool keep = false;
        int code = 0;
        if (i < nb) {
            const int sx = x0 + i % w, sy = y0 + i / w;
            keep = a.nz[sy * side + sx] != 0;
            code = (sy - ty + a.ncut) * 64 + (sx - tx + a.ncut);
        }
        const unsigned bal = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) sh.warp_cnt[warp] = __popc(bal);
        __syncthreads();
        int off = total;
        for (int q = 0; q < warp; ++q) off += sh.warp_cnt[q];
        if (keep) sh.list[off + __popc(bal & ((1u << lane) - 1))] = (short)code;
        for (int q = 0; q < NT / 32; ++q) total += sh.warp_cnt[q];
        __syncthreads();
    }

    // this thread's targets and their offsets u within the box
    int tj[R];
    float u1[R], u2[R], acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int pos = first + warp * 32 * R + r * 32 + lane;  // a warp's 32 R targets
        tj[r] = -1;
        u1[r] = u2[r] = acc[r] = 0.f;
        if (pos < end) {
            const int j = a.perm[pos];
            if ((unsigned)j < (unsigned)a.n) {
                tj[r] = j;
                u1[r] = (float)((a.y[2 * (size_t)j] * side - (tx + 0.5)) * a.d);
                u2[r] = (float)((a.y[2 * (size_t)j + 1] * side - (ty + 0.5)) * a.d);
            } else {
                atomicOr(a.err, DEV_ERR_CHECK);
            }
        }
    }
    const bool active = first + warp * 32 * R < end;  // warp-uniform

    const int nbatch = (total + kH2pBatch - 1) / kH2pBatch;
    auto stage = [&](int k) {
        if (k < nbatch) {
            float4* dst = reinterpret_cast<float4*>(sA + (size_t)(k % kH2pStages) * kH2pBatch * PP);
            const int cnt = min(kH2pBatch, total - k * kH2pBatch) * (PP / 4);
            for (int i = tid; i < cnt; i += NT) {
                const int code = sh.list[k * kH2pBatch + i / (PP / 4)];
                const int sx = tx + (code & 63) - a.ncut, sy = ty + (code >> 6) - a.ncut;
                cp_async_16(dst + i, reinterpret_cast<const float4*>(a.A + ((size_t)sy * side + sx) * PP) +
                                         i % (PP / 4));
            }
        }
        cp_async_commit();  // an empty group past the end keeps the wait counts uniform
    };
    stage(0);
    stage(1);
    int cur_dy = -1;
    float h2[R][P];
    for (int k = 0; k < nbatch; ++k) {
        cp_async_wait<1>();
        __syncthreads();  // batch k landed; everyone is done with batch k - 1's stage
        stage(k + 2);
        if (active) {
            const float* sb = sA + (size_t)(k % kH2pStages) * kH2pBatch * PP;
            const int nk = min(kH2pBatch, total - k * kH2pBatch);
#pragma unroll 1
            for (int e = 0; e < nk; ++e) {
                const int code = sh.list[k * kH2pBatch + e];
                const int dy = code >> 6, dx = code & 63;  // source offset + ncut
                if (dy != cur_dy) {
                    cur_dy = dy;
#pragma unroll
                    for (int r = 0; r < R; ++r) hermite_functions<P>(u2[r] + sh.off[2 * a.ncut - dy], h2[r]);
                }
                // sum_a1 h_a1(t1) T[a1], T[a1] = sum_a2 A[a1][a2] h_a2(t2), by Clenshaw's backward
                // recurrence for h_{a+1} = 2t h_a - 2a h_{a-1}:
                //   c_a = T[a] + 2t c_{a+1} - 2(a+1) c_{a+2},  c_p = c_{p+1} = 0,  sum = h_0(t1) c_0,
                // two multiply-adds per a1 beside the p of T[a1] (the forward recurrence and the
                // accumulation take three)
                float c1[R], c2[R], tt[R], e0[R];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float t = u1[r] + sh.off[2 * a.ncut - dx];
                    tt[r] = t + t;
                    e0[r] = __expf(-t * t);
                    c1[r] = c2[r] = 0.f;
                }
                const float4* Ab = reinterpret_cast<const float4*>(sb + e * PP);
#pragma unroll
                for (int a1 = P - 1; a1 >= 0; --a1) {
                    float t[R];
#pragma unroll
                    for (int r = 0; r < R; ++r) t[r] = fmaf(tt[r], c1[r], -(float)(2 * (a1 + 1)) * c2[r]);
#pragma unroll
                    for (int qd = 0; qd < P / 4; ++qd) {
                        const float4 v = Ab[a1 * (P / 4) + qd];
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            t[r] = fmaf(v.x, h2[r][4 * qd], t[r]);
                            t[r] = fmaf(v.y, h2[r][4 * qd + 1], t[r]);
                            t[r] = fmaf(v.z, h2[r][4 * qd + 2], t[r]);
                            t[r] = fmaf(v.w, h2[r][4 * qd + 3], t[r]);
                        }
                    }
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        c2[r] = c1[r];
                        c1[r] = t[r];
                    }
                }
#pragma unroll
                for (int r = 0; r < R; ++r) acc[r] = fmaf(e0[r], c1[r], acc[r]);
            }
        }
    }
    cp_async_wait<0>();
    __syncthreads();  // the ring and the list are free for the next claim
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (tj[r] >= 0) a.G[tj[r]] = a.accumulate ? a.G[tj[r]] + acc[r] : acc[r];
}

// Boxes listed for direct summation: *count holds their number << 32 | their claims, claim[i] the
// first claim of box[i].
struct H2pList {
    unsigned long long* count;
    int* box;
    int* claim;
};

// Host: claims[0..nbox] for runs of ch targets (one CTA, on `st`).
int launch_h2p_claims(int nbox, const int* box_start, int ch, int* claims, int* err, cudaStream_t st);

// Host: the evaluation through per-box Chebyshev coefficients (fgt_cheb.cu);
// *done = false when its rule does not take the call (nothing launched).
int launch_fgt_h2p_cheb(int g, int ncut, int p, double d, const float* A, const double* y, int n, const int* perm,
                        const int* box_start, float* G, bool accumulate, int* err, cudaStream_t st, bool* done);

// Host: the tensor-core evaluation (p = 16); claims must have been built with ch = 128.
int launch_fgt_h2p_tc(int g, int ncut, double d, bool split, const float* A, const double* y, int n, const int* perm,
                      const int* box_start, const int* claims, float* G, bool accumulate, int* err, cudaStream_t st);

}  // namespace fmmgb
