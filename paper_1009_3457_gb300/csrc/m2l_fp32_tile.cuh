// m2l_fp32_tile.cuh -- the FP32 M2L work unit shared by the per-level stencil
// kernel (m2l_fp32.cu) and the batched persistent kernel (m2l_batched.cu):
// one CTA translates and reduces every interaction list of the 64 target boxes
// of a 4 x 4 tile of parent boxes of one uniform level (Sec. 4.1 steps 2-3,
// Eq. M2Lmat).
//
// Formulation (radius-scaled units, E = (x_s - x_t)/r the integer box offset):
//   L~_t[n] = a_n sum_{s in IL(t)} sum_k h_E[n+k] (b_k M~_s[k]),
//   h_E[j] = (-1)^(j+1) j! s^j E^-(j+1),
// so each translation is a Hankel matrix-vector product between two diagonal
// scalings that do not depend on the offset: b_k is applied once per source
// box while it is staged into shared memory, a_n once per target box at the
// store.
//
// Offsets folded by symmetry.  h depends on E through E^-(j+1) alone, so
//   h_{iE}[j] = (-i)^(j+1) h_E[j]   and   h_{conj E}[j] = conj h_E[j]:
// the sources at E, iE, -E, -iE (an orbit of the rotation) need one Hankel
// product of h_E with the combinations
//   C_r[k] = m_E + (-i)^r m_iE + (-1)^r m_-E + i^r m_-iE,   r = (n + k + 1) mod 4
// (a 4-point transform of the four sources per k, shared by every row n), and
// with the conjugate orbit beside it (P_r, Q_r of E and conj E)
//   h P + conj(h) Q = Re h (P + Q) + i Im h (P - Q),
// two real products instead of two complex ones.  On the real axis Im h = 0; on
// the diagonals h is a real number times e^(-i pi (j+1)/4), whose r = (j+1) mod 4
// part goes into the combination and whose sign goes into the table.  The 27
// offsets of a target are 16 that every child class has (Chebyshev distance 2:
// orbits of (2,0), of (2,2), and of (2,1) with its conjugate) and 11 on the side
// away from its own parent (offsets 3 sx or 3 sy with sx = +1 for an even box
// column and -1 for an odd one, sy the same in y): the pairs (3,0)-(0,3),
// (3,1)-(-1,3) with (3,-1)-(1,3), (3,2)-(-2,3) with (3,-2)-(2,3), and (3,3).
// The other classes are reflections of that set: the sources' positions are
// reflected, and the products' factors follow from two signs per target,
//   s = sx sy (the rotation's direction: C_1 and C_3 trade places) and
//   e = sx ((-1)^(j+1) = -(-1)^n (-1)^k: odd k times e, even rows times e).
//
// Cost per target: 10 p^2 packed multiply-adds and ~158 p additions instead of
// 54 p^2 packed multiply-adds: 3.6x fewer cycles of the FP32 pipe at p = 16 (3.0x
// at p = 8, 4.0x at p = 24).  Levels 2-8 of a 2^22-point tree (87,376 boxes):
// p = 16 79.9 -> 27.2 us back to back, where the pipe's own time for this count is
// 16.6 us (61 % of it; 68 % for levels 2-10, 391 us, where the launch, the first tile and
// the last wave weigh less).  The rest is latency: 16 warps an SM, with the short
// addition chains of the combinations between the multiply-adds.  The error
// against 64 bits falls as well (2.9e-7 -> 1.6e-7): fewer terms are summed.
//
// Work unit (replaces the paper's thread-per-row, source-centric kernel and its
// separate reduction kernel, Sec. 4.1.1):
//   - the parent halo (tile + 1 on each side, 12 x 12 boxes) holds every source
//     any of the 64 targets needs; each source ME is read once per tile
//     (coalesced 16-byte loads), scaled by b_k and reused by up to 27 targets;
//   - the halo is stored transposed, [k][12][12] boxes with a k stride of 145:
//     a target and an offset are one address, and both the staging stores and
//     the reads of a half-warp (8 boxes of a row, and of the row two below) touch
//     every bank once;
//   - one target per lane and all p rows of it.  With 128 threads two warps take
//     the 16 common offsets and the pair (3,0)-(0,3) of 32 targets each, two the
//     other 9 offsets (4032 and 3616 cycles a warp at p = 16; the halves trade
//     warps from tile to tile, so that the SM's four schedulers share them); with
//     64 each warp takes both.  The two sums of a target meet in shared memory,
//     from where the tile is written in whole rows of boxes.  Two warps a target
//     are faster where a launch has only a few tiles per SM (p = 16, levels 2-8:
//     31.1 against 33.6 us as ordinary launches), one where it has many (40 trees of depth 4-9 in one
//     launch: 317 against 354 us), so the level kernel runs 128 threads and the
//     batched one 64;
//   - k runs in blocks of 4 (one period of r), so the code stays in the
//     instruction cache; the operator's values are warp-uniform operands from
//     constant memory (as shared loads into a register window they cost 30
//     registers and 5 us of 36.6);
//   - every sum has a fixed order (no atomics: deterministic).
#pragma once

#include "common.cuh"

namespace fmmgb {

constexpr int kTile = 4;       // parent boxes per tile side
constexpr int kBoxes = 2 * kTile;             // target boxes per tile side
constexpr int kW = 2 * (kTile + 2);           // halo boxes per side
constexpr int kPlane = kW * kW + 1;           // float2 stride between k-planes (odd: conflict-free)
constexpr int kPartSkew = 8;                  // extra float2 after every second box row of a partial sum

// NT threads per CTA: 128 (the two sums of a target in two warps) or 64 (one after the other in
// one; the sums meet the same way, so the results agree bit for bit).
template <int P, int NT = 128>
struct M2LCfg {
    static constexpr int THREADS = NT;
    static constexpr int KB = P % 4 == 0 ? 4 : P;  // k steps per loop pass (residues of k mod 4 compile-time)
    static constexpr int HALO = P * kPlane;        // float2 of the halo
    static constexpr int PART = kBoxes * kBoxes * (P + 1) + 3 * kPartSkew;  // float2 of one partial sum
    static constexpr bool SOLO = THREADS == 64;
    static constexpr int PART2 = SOLO ? HALO : PART;  // where the second partial sum lies
    static constexpr int BUF = SOLO ? HALO + PART : (HALO > 2 * PART ? HALO : 2 * PART);  // the sums reuse the halo's room
    // resident CTAs (registers): levels 2-8 at p = 16 take 31.7 / 31.1 / 33.5 us as ordinary launches (4: 27.2
    // as a dependent one) with 3 / 4 / 5 CTAs of 128, p = 24 60.7 / 74.8 (spills) with 3 / 4, p = 12 24.4 / 23.8 / 23.2 with 3 / 4 / 5
    static constexpr int MIN_CTAS = (P <= 12 ? 5 : (P <= 16 ? 4 : 3)) * 128 / NT;
    // halo loads a thread keeps in flight while staging a tile
    static constexpr int LOADS = P <= 6 ? 2 : (P <= 8 ? 3 : 4);
    static constexpr size_t smem = sizeof(float2) * BUF + sizeof(float) * 2 * P;
};

// Operator values of the orbits, h_E[j] of each orbit's first offset E (see above), built at
// compile time in FP64: (h, h) on the real axis; on a diagonal the real factor (|h|, its sign,
// and 1/sqrt 2 of the odd eighths of a turn) twice; (Re h, Im h) otherwise.  In constant
// memory: every lane of a warp reads the same value, and an operand from there takes no vector
// register.
template <int P>
struct alignas(16) OrbitTable {
    float2 h[kM2LOrbits][2 * P];
};
template <int P>
constexpr OrbitTable<P> make_orbit_table()
{
    constexpr int ex[kM2LOrbits] = {2, 2, 2, 3, 3, 3, 3}, ey[kM2LOrbits] = {0, 2, 1, 0, 1, 2, 3};
    constexpr double root2 = 1.41421356237309504880;
    constexpr double s = m2l_balance(P);
    OrbitTable<P> t{};
    for (int o = 0; o < kM2LOrbits; ++o) {
        const double x = ex[o], y = ey[o], den = x * x + y * y;
        const bool diag = ey[o] == ex[o], gen = ey[o] != 0 && !diag;
        // -1/E, or -1/|E| where the angle is kept apart
        const double ir = gen ? -x / den : (diag ? -1.0 / (x * root2) : -1.0 / x), ii = gen ? y / den : 0.0;
        double hr = ir, hi = ii;
        for (int j = 0; j < 2 * P - 1; ++j) {
            if (j > 0) {
                const double f = j * s, nr = (hr * ir - hi * ii) * f;
                hi = (hr * ii + hi * ir) * f;
                hr = nr;
            }
            double v = hr;
            if (diag && ((j + 1) & 4)) v = -v;
            if (diag && ((j + 1) & 1)) v /= root2;
            t.h[o][j].x = (float)v;
            t.h[o][j].y = (float)(gen ? hi : v);
        }
    }
    return t;
}
template <int P>
__constant__ constexpr OrbitTable<P> kOrbits = make_orbit_table<P>();

// Packed two-lane FP32 (PTX f32x2): a 64-bit register pair holds two values.
typedef unsigned long long pk_t;
__device__ __forceinline__ pk_t pk2(float a, float b)
{
    pk_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 upk2(pk_t v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ pk_t fma2(pk_t a, pk_t b, pk_t c)
{
    pk_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
// Packed sums and differences of two complex numbers.
__device__ __forceinline__ float2 operator+(float2 a, float2 b)
{
    pk_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pk2(a.x, a.y)), "l"(pk2(b.x, b.y)));
    return upk2(d);
}
__device__ __forceinline__ float2 operator-(float2 a, float2 b)
{
    pk_t d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pk2(a.x, a.y)), "l"(pk2(b.x, b.y)));
    return upk2(d);
}

// Number of 4 x 4-parent tiles of a level (levels 0 and 1 have no lists).
__host__ __device__ inline int m2l_tiles(int level)
{
    if (level < 2) return 0;
    const int np = 1 << (level - 1);
    const int t = (np + kTile - 1) / kTile;
    return t * t;
}

// One tile of one level: its coefficient arrays, its first box and, on an
// adaptive level, which boxes exist (NULL: all of them).
struct TileGeom {
    const float2* M;
    float2* L;
    const uint8_t* exists;
    int side, X0, Y0;
    int swap;  // which half of the warps takes the common offsets
};

__device__ __forceinline__ TileGeom tile_geom_of(const float2* M, float2* L, const uint8_t* exists, int level, int t)
{
    TileGeom g;
    g.M = M;
    g.L = L;
    g.exists = exists;
    g.side = 1 << level;
    const int tpr = ((g.side >> 1) + kTile - 1) / kTile;
    g.X0 = (t % tpr) * kBoxes;
    g.Y0 = (t / tpr) * kBoxes;
    g.swap = t & 1;
    return g;
}

// Shared-memory layout of the work unit for order P.
template <int P, int NT>
struct TileSmem {
    float2* buf;  // [P][kPlane] halo, then the two partial sums
    float* as;    // [P] post-scale
    float* bs;    // [P] pre-scale
    __device__ __forceinline__ explicit TileSmem(unsigned char* raw)
    {
        using C = M2LCfg<P, NT>;
        buf = reinterpret_cast<float2*>(raw);
        as = reinterpret_cast<float*>(buf + C::BUF);
        bs = as + P;
    }
};

// Load the diagonal scalings of order P into shared memory.  The caller synchronises
// before the next m2l_tile.
template <int P, int NT>
__device__ __forceinline__ void m2l_load_operator(unsigned char* raw, const float* __restrict__ ascale,
                                                  const float* __restrict__ bscale)
{
    const TileSmem<P, NT> s(raw);
    for (int i = threadIdx.x; i < P; i += NT) {
        s.as[i] = ascale[i];
        s.bs[i] = bscale[i];
    }
}

// The four combinations of an orbit of four sources, r = 0..3 (see above).
__device__ __forceinline__ void rot4(const float2 m1, const float2 m2, const float2 m3, const float2 m4, float2 c[4])
{
    const float2 e = m1 + m3, o = m1 - m3, f = m2 + m4, q = m2 - m4;
    c[0] = e + f;
    c[2] = e - f;
    c[1] = make_float2(o.x + q.y, o.y - q.x);
    c[3] = make_float2(o.x - q.y, o.y + q.x);
}
// ... of a pair E, iE, in the rotation's direction s.
__device__ __forceinline__ void rot2(const float2 m1, const float2 m2, float s, float2 c[4])
{
    c[0] = m1 + m2;
    c[2] = m1 - m2;
    c[1] = make_float2(fmaf(s, m2.y, m1.x), fmaf(-s, m2.x, m1.y));
    c[3] = make_float2(fmaf(-s, m2.y, m1.x), fmaf(s, m2.x, m1.y));
}

// acc += one k step of a real orbit: operator (h, h), combination c_r, rows n = 0..P-1.
// w holds the window h[k .. ]; J is k's place in the block.
template <int P, int J>
__device__ __forceinline__ void fold_real(pk_t (&A)[P], const pk_t* w, const float2 c[4])
{
    pk_t x[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) x[r] = pk2(c[r].x, c[r].y);
#pragma unroll
    for (int n = 0; n < P; ++n) A[n] = fma2(w[n + J], x[(n + J + 1) & 3], A[n]);
}

// ... of an orbit pc_r and its conjugate qc_r: operator (Re h, Im h); A sums
// (Re h Re S, Im h Re T), B (Re h Im S, Im h Im T), S = P + Q, T = P - Q, and the
// rows' values are (A.x - B.y, A.y + B.x) (a real orbit's too, with B = 0).
template <int P, int J>
__device__ __forceinline__ void fold_conj(pk_t (&A)[P], pk_t (&B)[P], const pk_t* w, const float2 pc[4],
                                          const float2 qc[4])
{
    pk_t x[4], y[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        x[r] = pk2(pc[r].x + qc[r].x, pc[r].x - qc[r].x);
        y[r] = pk2(pc[r].y + qc[r].y, pc[r].y - qc[r].y);
    }
#pragma unroll
    for (int n = 0; n < P; ++n) {
        A[n] = fma2(w[n + J], x[(n + J + 1) & 3], A[n]);
        B[n] = fma2(w[n + J], y[(n + J + 1) & 3], B[n]);
    }
}

// The operator window of one k block of an orbit: h[k0 .. k0 + P + KB - 2], warp-uniform.
template <int P>
__device__ __forceinline__ void fold_window(pk_t (&w)[P + M2LCfg<P>::KB], int orbit, int k0)
{
    const ulonglong2* h4 = reinterpret_cast<const ulonglong2*>(&kOrbits<P>.h[orbit][k0]);
#pragma unroll
    for (int i = 0; i < (P + M2LCfg<P>::KB) / 2; ++i) {
        const ulonglong2 v = h4[i];
        w[2 * i] = v.x;
        w[2 * i + 1] = v.y;
    }
}

// Calls f(k step) for the steps of a block with the step as a constant.
template <int J>
struct KStep {
    static constexpr int value = J;
};
template <int N, int J = 0, class F>
__device__ __forceinline__ void k_steps(F f)
{
    if constexpr (J < N) {
        f(KStep<J>{});
        k_steps<N, J + 1>(f);
    }
}

// The 16 common offsets of a target whose box is `t` in the halo, and the pair (3,0)-(0,3) of
// its class (e on the odd r instead of on odd k and even rows).
template <int P>
__device__ __forceinline__ void fold_ring(pk_t (&A)[P], pk_t (&B)[P], const float2* t, int sx, int sy)
{
    const float s = (float)(sx * sy), e = (float)sx;
    const float2 *px = t + 3 * sx, *py = t + 3 * kW * sy;
    constexpr int KB = M2LCfg<P>::KB;
#pragma unroll 1
    for (int k0 = 0; k0 < P; k0 += KB, t += KB * kPlane, px += KB * kPlane, py += KB * kPlane) {
        {
            pk_t w[P + KB];
            fold_window<P>(w, 3, k0);
            k_steps<KB>([&](auto jj) {
                constexpr int J = decltype(jj)::value;
                float2 c[4];
                rot2(px[J * kPlane], py[J * kPlane], s, c);
                c[1] = make_float2(e * c[1].x, e * c[1].y);
                c[3] = make_float2(e * c[3].x, e * c[3].y);
                fold_real<P, J>(A, w, c);
            });
        }
        auto m = [&](int j, int dx, int dy) { return t[j * kPlane + dy * kW + dx]; };
        {
            pk_t w[P + KB];
            fold_window<P>(w, 0, k0);
            k_steps<KB>([&](auto jj) {
                constexpr int J = decltype(jj)::value;
                float2 c[4];
                rot4(m(J, 2, 0), m(J, 0, 2), m(J, -2, 0), m(J, 0, -2), c);
                fold_real<P, J>(A, w, c);
            });
        }
        {
            pk_t w[P + KB];
            fold_window<P>(w, 1, k0);
            k_steps<KB>([&](auto jj) {
                constexpr int J = decltype(jj)::value;
                float2 c[4], d[4];
                rot4(m(J, 2, 2), m(J, -2, 2), m(J, -2, -2), m(J, 2, -2), c);
                // times e^(-i pi r/4) (sqrt 2 of the odd ones in the table)
                d[0] = c[0];
                d[1] = make_float2(c[1].x + c[1].y, c[1].y - c[1].x);
                d[2] = make_float2(c[2].y, -c[2].x);
                d[3] = make_float2(c[3].y - c[3].x, -c[3].x - c[3].y);
                fold_real<P, J>(A, w, d);
            });
        }
        {
            pk_t w[P + KB];
            fold_window<P>(w, 2, k0);
            k_steps<KB>([&](auto jj) {
                constexpr int J = decltype(jj)::value;
                float2 p[4], q[4];
                rot4(m(J, 2, 1), m(J, -1, 2), m(J, -2, -1), m(J, 1, -2), p);
                rot4(m(J, 2, -1), m(J, 1, 2), m(J, -2, 1), m(J, -1, -2), q);
                fold_conj<P, J>(A, B, w, p, q);
            });
        }
    }
}

// The other 9 offsets of the target's own class, sx, sy = +-1 (see above).
template <int P>
__device__ __forceinline__ void fold_side(pk_t (&A)[P], pk_t (&B)[P], const float2* t, int sx, int sy)
{
    constexpr int KB = M2LCfg<P>::KB;
    const float s = (float)(sx * sy), e = (float)sx;
    const float2 *tx = t + 3 * sx, *ty = t + 3 * kW * sy;  // the columns at 3 sx, the rows at 3 sy
    const int ox = kW * sx, oy = sy;
#pragma unroll 1
    for (int k0 = 0; k0 < P; k0 += KB, tx += KB * kPlane, ty += KB * kPlane) {
        auto at = [&](const float2* b, int j, int off) {
            const float2 v = b[j * kPlane + off];
            return j & 1 ? make_float2(e * v.x, e * v.y) : v;
        };
        {
            pk_t w[P + KB];
            fold_window<P>(w, 6, k0);
            k_steps<KB>([&](auto jj) {
                constexpr int J = decltype(jj)::value;
                const float2 v = at(ty, J, 3 * sx);
                const float vx = s * v.x, vy = s * v.y;
                const float2 c[4] = {v, make_float2(v.x + vy, v.y - vx), make_float2(vy, -vx),
                                     make_float2(vy - v.x, -v.y - vx)};
                fold_real<P, J>(A, w, c);
            });
        }
#pragma unroll
        for (int d = 1; d <= 2; ++d) {
            pk_t w[P + KB];
            fold_window<P>(w, 3 + d, k0);
            k_steps<KB>([&](auto jj) {
                constexpr int J = decltype(jj)::value;
                float2 p[4], q[4];
                rot2(at(tx, J, d * ox), at(ty, J, -d * oy), s, p);
                rot2(at(tx, J, -d * ox), at(ty, J, d * oy), s, q);
                fold_conj<P, J>(A, B, w, p, q);
            });
        }
    }
}

// Translate and reduce one tile (ADAPTIVE and g.exists set: only existing
// sources are read and existing targets written).  Requires the operator of order P in shared
// memory (m2l_load_operator + a barrier) and no thread still reading the buffer
// of a previous tile (a barrier).  All NT threads call it.  cj = -1 conjugates
// the MEs and the LEs (the conjugate operator), sgn = -1 negates the LEs.
template <int P, int NT, bool ADAPTIVE = false, int UMAX = M2LCfg<P>::LOADS>
__device__ __forceinline__ void m2l_tile(unsigned char* raw, const TileGeom& g, int periodic, int accumulate,
                                         float sgn = 1.f, float cj = 1.f)
{
    using C = M2LCfg<P, NT>;
    constexpr int Q = P / 2;
    constexpr bool SOLO = C::SOLO;
    const TileSmem<P, NT> s(raw);
    const int tid = threadIdx.x;

    // Stage the halo boxes, pre-scaled by b_k; consecutive threads read consecutive
    // 16-byte chunks of a row of boxes (coalesced); zero outside the level.
    // Each thread first issues up to U (<= UMAX, a register budget) loads, then scales
    // and stores them, so that a tile's staging costs a memory round trip or two
    // instead of one per chunk.
    const float4* M4 = reinterpret_cast<const float4*>(g.M);
    constexpr int NCH = kW * kW * Q;  // 16-byte chunks of the halo
    constexpr int U = (NCH + C::THREADS - 1) / C::THREADS < UMAX ? (NCH + C::THREADS - 1) / C::THREADS : UMAX;
    for (int i0 = tid; i0 < NCH; i0 += U * C::THREADS) {
        float4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * C::THREADS;
            v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (i >= NCH) continue;
            const int q = i % Q, bxy = i / Q;
            int ix = g.X0 - 2 + bxy % kW, iy = g.Y0 - 2 + bxy / kW;
            bool in = ix >= 0 && iy >= 0 && ix < g.side && iy < g.side;
            if (periodic) {
                ix = (ix + 2 * g.side) % g.side;
                iy = (iy + 2 * g.side) % g.side;
                in = true;
            }
            if constexpr (ADAPTIVE)
                if (in && g.exists) in = g.exists[(size_t)iy * g.side + ix] != 0;  // V-list: existing sources only
            if (in) v[u] = __ldcg(M4 + ((size_t)iy * g.side + ix) * Q + q);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * C::THREADS;
            if (i >= NCH) continue;
            const int q = i % Q, bxy = i / Q;
            const float b0 = s.bs[2 * q], b1 = s.bs[2 * q + 1];
            s.buf[(2 * q) * kPlane + bxy] = make_float2(v[u].x * b0, v[u].y * (cj * b0));
            s.buf[(2 * q + 1) * kPlane + bxy] = make_float2(v[u].z * b1, v[u].w * (cj * b1));
        }
    }
    __syncthreads();

    // Warp (half, 32-target group): half 0 the common offsets, half 1 the class's own.
    // Lanes 0-7, 8-15, 16-23, 24-31 take rows 0, 2, 1, 3 of the group's 4 rows of 8 boxes.
    const int warp = tid >> 5, lane = tid & 31;
    const int half = SOLO ? 0 : (warp >> 1) ^ g.swap;
    const int tx = lane & 7, ty = 4 * (warp & 1) + ((lane >> 3 & 1) << 1) + (lane >> 4);
    const int ix = g.X0 + tx, iy = g.Y0 + ty;
    // On an adaptive level a warp whose targets are all absent skips the
    // translation; the vote is warp-uniform.
    bool work = true;
    if constexpr (ADAPTIVE) {
        bool target = ix < g.side && iy < g.side;
        if (target && g.exists) target = g.exists[(size_t)iy * g.side + ix] != 0;
        work = __any_sync(0xffffffffu, target);
    }
    pk_t A[P], B[P];
    auto clear = [&] {
#pragma unroll
        for (int n = 0; n < P; ++n) A[n] = B[n] = 0ull;
    };
    // this lane's sums into its half's partial sum; the class's own rows carry e = sx
    auto put = [&](float2* room, float e) {
        float2* part = room + (8 * ty + tx) * (P + 1) + (ty >> 1) * kPartSkew;
#pragma unroll
        for (int n = 0; n < P; ++n) {
            const float2 a = upk2(A[n]), b = upk2(B[n]);
            const float re = a.x - b.y, im = a.y + b.x;
            part[n] = n & 1 ? make_float2(re, im) : make_float2(e * re, e * im);
        }
    };
    clear();
    const float2* t = s.buf + (ty + 2) * kW + tx + 2;
    const int sx = 1 - 2 * (tx & 1), sy = 1 - 2 * (ty & 1);
    if (work && half == 0) fold_ring<P>(A, B, t, sx, sy);
    if constexpr (SOLO) {
        put(s.buf + C::HALO, 1.f);
        clear();
    }
    if (work && (SOLO || half)) fold_side<P>(A, B, t, sx, sy);
    __syncthreads();  // every warp is done with the halo: its room takes the partial sums
    if constexpr (SOLO)
        put(s.buf, (float)sx);
    else
        put(s.buf + half * C::PART, half ? (float)sx : 1.f);
    __syncthreads();

    // ---- store L~[n] = a_n * (sum of the two halves), whole rows of boxes ----
    for (int i = tid; i < kBoxes * kBoxes * Q; i += C::THREADS) {
        const int q = i % Q, b = i / Q;
        const int bx = g.X0 + (b & 7), by = g.Y0 + (b >> 3);
        if (bx >= g.side || by >= g.side) continue;
        const size_t box = (size_t)by * g.side + bx;
        if constexpr (ADAPTIVE)
            if (g.exists && !g.exists[box]) continue;
        const float2* part = s.buf + b * (P + 1) + (b >> 4) * kPartSkew + 2 * q;
        const float2 r0 = part[0] + part[C::PART2], r1 = part[1] + part[C::PART2 + 1];
        const float s0 = sgn * s.as[2 * q], s1 = sgn * s.as[2 * q + 1];
        float4 o = make_float4(s0 * r0.x, s0 * cj * r0.y, s1 * r1.x, s1 * cj * r1.y);
        float4* dst = reinterpret_cast<float4*>(g.L + box * P) + q;
        if (accumulate) {
            const float4 old = *dst;
            o.x += old.x;
            o.y += old.y;
            o.z += old.z;
            o.w += old.w;
        }
        *dst = o;
    }
}

// ---------------------------------------------------------------------------
// stencil kernel: every requested level in one launch, tiles ordered heaviest
// level first.  Persistent when `counter` is set: each resident CTA loads the
// diagonal scalings once (the operator lies in constant memory), takes its first
// tile by blockIdx and claims the next from the work counter (counter[0];
// counter[1] counts the CTAs that finished, and the last one resets both), so
// no second round of CTAs leaves SMs half empty at the end.  With counter == NULL the grid covers every tile, one CTA each.
// ---------------------------------------------------------------------------
template <int P, bool ADAPTIVE>
__global__ void __launch_bounds__(M2LCfg<P>::THREADS, M2LCfg<P>::MIN_CTAS)
    m2l_fp32_kernel(const __grid_constant__ M2LLaunch job, const float* ascale,
                    const float* bscale, int total, int* __restrict__ counter)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_next;
    m2l_load_operator<P, M2LCfg<P>::THREADS>(smem_raw, ascale, bscale);  // tables of long ago
    after_wait();
    int tile = blockIdx.x;
    while (tile < total) {
        int li = 0;
        while (li + 1 < job.nlev && tile >= job.lv[li + 1].tile_begin) ++li;
        const M2LLevel& lv = job.lv[li];
        int t = tile - lv.tile_begin;
        if constexpr (ADAPTIVE)
            if (lv.tiles) t = lv.tiles[t];  // the level's tiles that hold an existing box
        const TileGeom g = tile_geom_of(lv.M, lv.L, ADAPTIVE ? lv.exists : nullptr, lv.level, t);
        __syncthreads();  // operator visible; the previous tile is done with the buffer
        m2l_tile<P, M2LCfg<P>::THREADS, ADAPTIVE>(smem_raw, g, job.periodic, job.accumulate, job.sgn, job.cj);
        if (!counter) break;
        // every thread read s_next of the previous claim before the barriers inside m2l_tile
        if (threadIdx.x == 0) s_next = (int)gridDim.x + atomicAdd(counter, 1);
        __syncthreads();
        tile = s_next;
    }
    // the last CTA to finish returns the counter slot to zero for its next use
    if (counter && threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(counter + 1, 1) == (int)gridDim.x - 1) {
            atomicExch(counter, 0);
            atomicExch(counter + 1, 0);
        }
    }
}

}  // namespace fmmgb
