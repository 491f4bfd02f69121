// shift.cu -- the translations between a box and its four children (M2M, L2L and their
// conjugate transposes, radius-scaled units; Sec. 2.1 stages 2-3) for the orders of the M2L
// path, with the children folded by symmetry.
//
// A child's offset is z_t = i^t (1 + i)/4, t = 0..3 for (right, up), (left, up), (left, down),
// (right, down), and (1 + i)^4 = -4, so with q = 4a + b
//   z_t^q = i^(tb) (-4)^a 4^-q (1 + i)^b:
// a real number shared by the children, times one of four rotations.  Up (M2M):
//   M_j = sum_k C(j,k) 2^-k sum_t z_t^(j-k) m_t,k = sum_k c_jk D_((j-k) mod 4),k,
//   D_b,k = (1 + i)^b sum_t i^(tb) m_t,k,
// a 4-point transform of the children per k and then one real-times-complex product per (j, k)
// instead of four complex-times-complex ones.  Down (L2L) is the transpose: per j the sums
//   B_b = sum_(n-j = b mod 4) c_nj L_n,   L_t,j = sum_b i^(tb) (1 + i)^b B_b.
// The conjugate transposes use conj z_t = z_(3-t): the children trade places in y; and
// coefficients 2^-k / 2 (L2L's, up) or 2^-k (M2M's, down).  Every coefficient is an integer
// below 2^24 times a power of 2, exact in FP32.
//
// Threads are (box, index) pairs in index order, so every read and write of a coefficient row is
// one coalesced run; a block's rows meet in shared memory.  Bound by memory at the finest levels and by the
// launch at the coarse ones, which run as one (the chain below: four launches a pass instead of seven).
// A 9-level tree at p = 16: M2M and L2L's transpose together 253 -> 57 us, L2L and M2M's transpose
// 207 -> 60 us (a thread per output with its own powers of z and a table read per term before).
#include <algorithm>

#include "common.cuh"

namespace fmmgb {

constexpr int kShiftThreads = 128;   // per block, at most
constexpr int kChainThreads = 1024;  // of a chain's CTAs
template <int P, int NT>
struct ShiftCfg {
    static constexpr int BOXES = NT / P;            // parents per block
    static constexpr int THREADS = BOXES * P;
    static constexpr int ROW = P + 1;               // float2 row stride in shared memory
};

// Coefficients C(n, m) (-4)^a 4^-q 2^-m, q = n - m >= 0, as s[m][n] (n >= m).
template <int P>
__device__ __forceinline__ void shift_coefficients(float (*s)[P + 1], float scale, int threads)
{
    for (int i = threadIdx.x; i < P * P; i += threads) {
        const int m = i / P, n = i % P, q = n - m;
        // (-4)^a 4^-q = +-2^(2a - 2q)
        if (q >= 0) s[m][n] = scale * kBinom.v[n * 64 + m] * (q & 4 ? -1.f : 1.f) * pow2_neg(2 * q - 2 * (q >> 2) + m);
    }
}

// child t's box column and row parity: (1,1), (0,1), (0,0), (1,0)
__device__ __forceinline__ int child_x(int t) { return t == 0 || t == 3; }
__device__ __forceinline__ int child_y(int t) { return t < 2; }

// Shared memory of a block: the coefficients and the rows that its threads exchange.
template <int P, int NT>
struct ShiftSmem {
    float c[P][P + 1];
    float2 d[ShiftCfg<P, NT>::BOXES][4][ShiftCfg<P, NT>::ROW];
};

// One block of parents: Out[parent][j] (+)= sum_t sum_k c_jk (z_t or conj z_t)^(j-k) In[child t][k].
// Loads go to the L2: in a chain of levels another block has just written them.
template <int P, int NT>
__device__ __forceinline__ void shift_up_block(ShiftSmem<P, NT>& sm, int child_level, const float2* In, float2* Out, int conj,
                                               int accumulate, int64_t block)
{
    using C = ShiftCfg<P, NT>;
    const int np = 1 << (child_level - 1), nc = 2 * np;
    const int pl = threadIdx.x / P, j = threadIdx.x % P;
    const int64_t pb = block * C::BOXES + pl;
    const bool ok = pb < (int64_t)np * np;
    float2 m[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        m[t] = make_float2(0.f, 0.f);
        if (ok) {
            const int px = (int)(pb & (np - 1)), py = (int)(pb >> (child_level - 1));
            m[t] = __ldcg(In + ((size_t)(2 * py + (child_y(t) ^ conj)) * nc + 2 * px + child_x(t)) * P + j);
        }
    }
    float2 old = make_float2(0.f, 0.f);
    if (ok && accumulate) old = __ldcg(Out + (size_t)pb * P + j);
    {
        const float2 e = make_float2(m[0].x + m[2].x, m[0].y + m[2].y), f = make_float2(m[1].x + m[3].x, m[1].y + m[3].y);
        const float2 o = make_float2(m[0].x - m[2].x, m[0].y - m[2].y), g = make_float2(m[1].x - m[3].x, m[1].y - m[3].y);
        const float x1 = o.x - g.y, y1 = o.y + g.x, x3 = o.x + g.y, y3 = o.y - g.x;  // sums of i^t m, (-i)^t m
        const float x2 = e.x - f.x, y2 = e.y - f.y;
        sm.d[pl][0][j] = make_float2(e.x + f.x, e.y + f.y);
        sm.d[pl][1][j] = make_float2(x1 - y1, x1 + y1);
        sm.d[pl][2][j] = make_float2(-2.f * y2, 2.f * x2);
        sm.d[pl][3][j] = make_float2(-2.f * (x3 + y3), 2.f * (x3 - y3));
    }
    __syncthreads();
    if (!ok) return;
    float2 s = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < P; ++k)
        if (k <= j) {
            const float2 d = sm.d[pl][(j - k) & 3][k];
            const float c = sm.c[k][j];
            s.x = fmaf(c, d.x, s.x);
            s.y = fmaf(c, d.y, s.y);
        }
    if (accumulate) {
        s.x += old.x;
        s.y += old.y;
    }
    Out[(size_t)pb * P + j] = s;
}

// One block of parents: Out[child t][j] (+)= sum_(n >= j) c_nj (z_t or conj z_t)^(n-j) In[parent][n].
template <int P, int NT>
__device__ __forceinline__ void shift_down_block(ShiftSmem<P, NT>& sm, int child_level, const float2* In, float2* Out,
                                                 int conj, int accumulate, int64_t block)
{
    using C = ShiftCfg<P, NT>;
    const int np = 1 << (child_level - 1), nc = 2 * np;
    const int pl = threadIdx.x / P, j = threadIdx.x % P;
    const int64_t pb = block * C::BOXES + pl;
    const bool ok = pb < (int64_t)np * np;
    float2* out[4];
    float2 old[4];
    const int px = (int)(pb & (np - 1)), py = (int)(pb >> (child_level - 1));
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        out[t] = Out + ((size_t)(2 * py + (child_y(t) ^ conj)) * nc + 2 * px + child_x(t)) * P + j;
        old[t] = make_float2(0.f, 0.f);
        if (ok && accumulate) old[t] = __ldcg(out[t]);
    }
    sm.d[pl][0][j] = ok ? __ldcg(In + (size_t)pb * P + j) : make_float2(0.f, 0.f);
    __syncthreads();
    if (!ok) return;
    float2 b[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) b[r] = make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < P; ++q)
        if (j + q < P) {
            const float2 l = sm.d[pl][0][j + q];
            const float c = sm.c[j][j + q];
            b[q & 3].x = fmaf(c, l.x, b[q & 3].x);
            b[q & 3].y = fmaf(c, l.y, b[q & 3].y);
        }
    // (1 + i)^r B_r
    const float2 v1 = make_float2(b[1].x - b[1].y, b[1].x + b[1].y), v2 = make_float2(-2.f * b[2].y, 2.f * b[2].x);
    const float2 v3 = make_float2(-2.f * (b[3].x + b[3].y), 2.f * (b[3].x - b[3].y));
    const float2 e = make_float2(b[0].x + v2.x, b[0].y + v2.y), f = make_float2(v1.x + v3.x, v1.y + v3.y);
    const float2 o = make_float2(b[0].x - v2.x, b[0].y - v2.y), g = make_float2(v1.x - v3.x, v1.y - v3.y);
    const float2 r[4] = {make_float2(e.x + f.x, e.y + f.y), make_float2(o.x - g.y, o.y + g.x),
                         make_float2(e.x - f.x, e.y - f.y), make_float2(o.x + g.y, o.y - g.x)};
#pragma unroll
    for (int t = 0; t < 4; ++t) *out[t] = make_float2(r[t].x + old[t].x, r[t].y + old[t].y);
}

template <int P, bool UP>
__global__ void __launch_bounds__(kShiftThreads)
    shift_kernel(int child_level, const float2* In, float2* Out, float scale, int conj, int accumulate)
{
    __shared__ ShiftSmem<P, kShiftThreads> sm;
    shift_coefficients<P>(sm.c, scale, ShiftCfg<P, kShiftThreads>::THREADS);
    after_wait();
    // visible to the block at the barrier inside
    if constexpr (UP)
        shift_up_block<P>(sm, child_level, In, Out, conj, accumulate, blockIdx.x);
    else
        shift_down_block<P>(sm, child_level, In, Out, conj, accumulate, blockIdx.x);
}

// A run of levels in one launch: one cluster of CTAs takes the blocks of each level in turn, with a
// cluster barrier (release / acquire) between the levels.  For the coarse levels, where a launch
// costs more than the level: child levels up to kChainMax (4,096 boxes: two rounds of the cluster
// at p = 16, and one for each coarser level).
constexpr int kChainMax = 6;
constexpr int kChainCtas = 8;  // portable cluster size
struct ShiftChain {
    float2* level[kChainMax + 1];
    int first, last;  // child levels, in the order they are taken
};

template <int P, bool UP>
__global__ void __cluster_dims__(kChainCtas, 1, 1) __launch_bounds__(kChainThreads)
    shift_chain_kernel(const __grid_constant__ ShiftChain ch, float scale, int conj, int accumulate)
{
    using C = ShiftCfg<P, kChainThreads>;
    __shared__ ShiftSmem<P, kChainThreads> sm;
    shift_coefficients<P>(sm.c, scale, C::THREADS);
    after_wait();
    for (int l = ch.first;; l += UP ? -1 : 1) {
        const int64_t parents = (int64_t)1 << (2 * (l - 1));
        for (int64_t b = blockIdx.x; b * C::BOXES < parents; b += kChainCtas) {
            if constexpr (UP)
                shift_up_block<P>(sm, l, ch.level[l], ch.level[l - 1], conj, accumulate, b);
            else
                shift_down_block<P>(sm, l, ch.level[l - 1], ch.level[l], conj, accumulate, b);
            __syncthreads();  // the exchanged rows have been read
        }
        if (l == ch.last) break;
        asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    }
}

template <int P>
static int shift_launch(bool up, int child_level, const float2* In, float2* Out, float scale, bool conj, bool acc,
                        cudaStream_t st)
{
    using C = ShiftCfg<P, kShiftThreads>;
    const int64_t parents = (int64_t)1 << (2 * (child_level - 1));
    const unsigned grid = (unsigned)((parents + C::BOXES - 1) / C::BOXES);
    auto kern = up ? shift_kernel<P, true> : shift_kernel<P, false>;
    FMM_CUDA_TRY(launch_after(kern, grid, C::THREADS, 0, st, child_level, In, Out, scale, conj, acc));
    return FMM_OK;
}

template <int P>
static int chain_launch(bool up, const ShiftChain& ch, float scale, bool conj, bool acc, cudaStream_t st)
{
    auto kern = up ? shift_chain_kernel<P, true> : shift_chain_kernel<P, false>;
    FMM_CUDA_TRY(launch_after(kern, kChainCtas, ShiftCfg<P, kChainThreads>::THREADS, 0, st, ch, scale, conj, acc));
    return FMM_OK;
}

bool shift_supported(int p) { return p == 6 || p == 8 || p == 12 || p == 16 || p == 24; }

// up: child -> parent, else parent -> child; scale multiplies C(n, m) 2^-m z^(n-m).
int launch_shift(bool up, int child_level, int p, const float2* In, float2* Out, float scale, bool conj, bool acc,
                 cudaStream_t st)
{
    switch (p) {
        case 6: return shift_launch<6>(up, child_level, In, Out, scale, conj, acc, st);
        case 8: return shift_launch<8>(up, child_level, In, Out, scale, conj, acc, st);
        case 12: return shift_launch<12>(up, child_level, In, Out, scale, conj, acc, st);
        case 16: return shift_launch<16>(up, child_level, In, Out, scale, conj, acc, st);
        case 24: return shift_launch<24>(up, child_level, In, Out, scale, conj, acc, st);
        default: return fail(FMM_EINVAL, "shift: unsupported p = %d", p);
    }
}

}  // namespace fmmgb

using namespace fmmgb;

static int launch_chain(bool up, int p, const ShiftChain& ch, float scale, bool conj, bool acc, cudaStream_t st)
{
    switch (p) {
        case 6: return chain_launch<6>(up, ch, scale, conj, acc, st);
        case 8: return chain_launch<8>(up, ch, scale, conj, acc, st);
        case 12: return chain_launch<12>(up, ch, scale, conj, acc, st);
        case 16: return chain_launch<16>(up, ch, scale, conj, acc, st);
        default: return chain_launch<24>(up, ch, scale, conj, acc, st);
    }
}

// A whole pass of fmm_m2m (op 0), fmm_l2l_adjoint (1, accumulating), fmm_l2l (2, accumulating) or
// fmm_m2m_adjoint (3, accumulating) over levels lmin..lmax, levels[i] the array of level lmin + i:
// the same sums as the per-level calls, the levels up to kChainMax in one launch.  Used by the
// Python layer, whose calls cost more than the coarse levels' kernels; not part of the public header.
extern "C" int fmmgb_shift_levels(int32_t op, int32_t p, int32_t lmin, int32_t lmax, void* const* levels, void* stream)
{
    clear_error();
    if (op < 0 || op > 3) return fail(FMM_EINVAL, "fmmgb_shift_levels: op %d", op);
    if (lmin < 0 || lmax > FMM_MAX_LEVEL || lmin > lmax)
        return fail(FMM_EINVAL, "fmmgb_shift_levels: levels %d..%d outside 0..%d", lmin, lmax, FMM_MAX_LEVEL);
    if (p < 1 || p > 64) return fail(FMM_EINVAL, "fmmgb_shift_levels: p = %d outside 1..64", p);
    if (!levels) return fail(FMM_EINVAL, "fmmgb_shift_levels: NULL level array");
    for (int i = 0; i <= lmax - lmin; ++i)
        if (!levels[i] || ((uintptr_t)levels[i] & 7))
            return fail(FMM_EINVAL, "fmmgb_shift_levels: level %d NULL or misaligned", lmin + i);
    const cudaStream_t st = (cudaStream_t)stream;
    const bool up = op < 2;
    // child levels lmin + 1 .. chain in one launch where there are at least two of them
    const int chain = shift_supported(p) && std::min(lmax, kChainMax) - lmin >= 2 ? std::min(lmax, kChainMax) : lmin;
    auto run_chain = [&]() -> int {
        if (chain == lmin) return FMM_OK;
        ShiftChain ch{};
        for (int l = lmin; l <= chain; ++l) ch.level[l] = (float2*)levels[l - lmin];
        ch.first = up ? chain : lmin + 1;
        ch.last = up ? lmin + 1 : chain;
        return launch_chain(up, p, ch, op == 1 || op == 2 ? 0.5f : 1.f, op & 1, op != 0, st);
    };
    auto one = [&](int l) -> int {
        float2 *child = (float2*)levels[l - lmin], *parent = (float2*)levels[l - 1 - lmin];
        switch (op) {
            case 0: return launch_m2m(l, p, child, parent, false, st);
            case 1: return launch_l2l(l, p, child, parent, true, true, st);
            case 2: return launch_l2l(l, p, parent, child, true, false, st);
            default: return launch_m2m_adjoint(l, p, parent, child, true, st);
        }
    };
    if (up) {
        for (int l = lmax; l > chain; --l)
            if (int rc = one(l)) return rc;
        return run_chain();
    }
    if (int rc = run_chain()) return rc;
    for (int l = chain + 1; l <= lmax; ++l)
        if (int rc = one(l)) return rc;
    return FMM_OK;
}
