// Small dense matrices held by ONE WARP in the accumulator layout of mma.sync.m16n8k8, and the products, the blocked
// Cholesky factorisation and the vector operations that the Riccati step needs on them, without shared memory.
//
// Layout: a matrix of 8 RB x 8 CB elements is cut into 16 x 8 tiles; lane = 4 g + t holds of tile (mt, cb)
//     v[mt][cb][0], [1] = row 16 mt + g,     columns 8 cb + 2 t, + 1
//     v[mt][cb][2], [3] = row 16 mt + 8 + g, the same columns          (absent rows are zero when RB is odd)
// The instruction leaves the assignment of contraction indices to its k slots free as long as both operands agree.
// With slot t <-> column 2 t and slot t + 4 <-> column 2 t + 1 of an 8-wide chunk, the registers of a matrix X are the A
// operand of X as they stand, and also the B operand of X' (transposed).  So X * Y' needs no data movement, and the
// Riccati step can be written with such products only (P symmetric):
//     V = B'P = (B')(P)',  T = A'P,  S = R + (B')(V)',  Y' = (A')(V)',  A'PA = (A')(T)',  Z'Z = (Z')(Z')'
// Every product keeps float32-grade accuracy: operands are split into a tf32 part rounded to nearest and the remainder,
// three passes (lo*hi + hi*lo + hi*hi) accumulate in float32.  The dropped term and the truncation of the remainder are
// both about 2^-23 of the product on average, 2^-20 at most.  (A second set of products takes pairs of float16 numbers, for
// operands whose values permit it.)
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

namespace ttc {
namespace frag {

constexpr unsigned FULL = 0xffffffffu;

// Index of the warp in its CTA.  By way of a shuffle the compiler knows that it is the same in the whole warp and keeps what
// depends on it (the instance, the addresses of its operands and outputs) in uniform registers.  65536 instances, n = 16, H = 32,
// operands from memory: 2.68 -> 2.50 ms; 64 instances, n = 16, H = 1024 in pieces: 230 -> 214 us; 16384, n = 32, H = 64: 8.53 -> 8.39 ms.
__device__ __forceinline__ int warp_index() { return __shfl_sync(FULL, (int)(threadIdx.x >> 5), 0); }

template <int RB, int CB>
struct Mat {
    static constexpr int MT = (RB + 1) / 2;
    float v[MT][CB][4];
};
// hi / lo parts of a matrix
template <int RB, int CB>
struct Split {
    static constexpr int MT = (RB + 1) / 2;
    uint32_t h[MT][CB][4], l[MT][CB][4];
};

__device__ __forceinline__ void split1(float x, uint32_t& h, uint32_t& l)
{
    h = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;      // nearest tf32 (ties away from zero)
    l = __float_as_uint(x - __uint_as_float(h));           // exact; the tensor core ignores its lowest bits
}

__device__ __forceinline__ void split2(float x0, float x1, uint32_t& h0, uint32_t& h1, uint32_t& l0, uint32_t& l1)
{
    split1(x0, h0, l0);
    split1(x1, h1, l1);
}

__device__ __forceinline__ void mma(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// d = X Y' + c with c in other registers (or constant zero), which saves the copies that an in-place accumulation needs
__device__ __forceinline__ void mma(float (&d)[4], const float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                    uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}

template <int RB, int CB>
__device__ __forceinline__ void split(Split<RB, CB>& s, const Mat<RB, CB>& m)
{
#pragma unroll
    for (int mt = 0; mt < Mat<RB, CB>::MT; ++mt)
#pragma unroll
        for (int cb = 0; cb < CB; ++cb)
#pragma unroll
            for (int e = 0; e < 4; e += 2) {
                if (e >= 2 && 2 * mt + 1 >= RB) {           // rows that do not exist
                    s.h[mt][cb][e] = s.h[mt][cb][e + 1] = 0u;
                    s.l[mt][cb][e] = s.l[mt][cb][e + 1] = 0u;
                } else {
                    split2(m.v[mt][cb][e], m.v[mt][cb][e + 1], s.h[mt][cb][e], s.h[mt][cb][e + 1], s.l[mt][cb][e],
                           s.l[mt][cb][e + 1]);
                }
            }
}

// d = c + X * Y'   (X: 8 RB x 8 KB, Y: 8 CB x 8 KB; d: 8 RB x 8 CB; c null: zero; c may be d).  LOWER: only the tiles that
// touch the lower triangle, of a result whose upper one is not needed or follows from it.
template <int RB, int KB, int CB, bool LOWER = false>
__device__ __forceinline__ void product(Mat<RB, CB>& d, const Mat<RB, CB>* c, const Split<RB, KB>& x, const Split<CB, KB>& y)
{
    const float z[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int kb = 0; kb < KB; ++kb) {
        // pass-major order: the tiles of a pass are independent of one another
#pragma unroll
        for (int pass = 0; pass < 3; ++pass)
#pragma unroll
            for (int cb = 0; cb < CB; ++cb)
#pragma unroll
                for (int mt = 0; mt < Mat<RB, CB>::MT; ++mt) {
                    if (LOWER && cb > 2 * mt + 1)
                        continue;
                    const uint32_t(&a)[4] = pass == 0 ? x.l[mt][kb] : x.h[mt][kb];
                    const uint32_t(&b)[4] = pass == 1 ? y.l[cb / 2][kb] : y.h[cb / 2][kb];
                    const uint32_t b0 = b[2 * (cb & 1)], b1 = b[2 * (cb & 1) + 1];
                    if (kb || pass)
                        mma(d.v[mt][cb], a[0], a[2], a[1], a[3], b0, b1);
                    else if (c)
                        mma(d.v[mt][cb], c->v[mt][cb], a[0], a[2], a[1], a[3], b0, b1);
                    else
                        mma(d.v[mt][cb], z, a[0], a[2], a[1], a[3], b0, b1);
                }
    }
}

// Value of another lane: lane (B | own bits under KEEP).  The segment mask of the instruction keeps any set of own lane
// bits, so that the source needs no index register.
template <int B, int KEEP>
__device__ __forceinline__ float lane_value(float x)
{
    float r;
    asm volatile("shfl.sync.idx.b32 %0, %1, %2, %3, 0xffffffff;" : "=f"(r) : "f"(x), "n"(B), "n"((KEEP << 8) | 0x1f));
    return r;
}

__device__ __forceinline__ float rcp_fast(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

template <int J>
__device__ __forceinline__ void pivot8(float& a0, float& a1, int g, int t)
{
    const float sel = (J & 1) ? a1 : a0;
    const float d = lane_value<4 * J + (J >> 1), 0>(sel);
    const float col = lane_value<(J >> 1), 28>(sel);
    const float r0 = lane_value<4 * J, 3>(a0), r1 = lane_value<4 * J, 3>(a1);
    const float f = (g > J) ? -col * rcp_fast(d) : 0.f;
    a0 = fmaf(f, r0, a0);
    a1 = fmaf(f, r1, a1);
    if (g > J && t == (J >> 1)) {                          // column J is eliminated, the inverse's moves in
        if (J & 1)
            a1 = f;
        else
            a0 = f;
    }
}

// Two pivots at once (columns 2 K and 2 K + 1, which share a lane): the second reciprocal waits for the first one but not
// for a second round of shuffles, so the chain of a pair is about 130 cycles instead of 220.
template <int K>
__device__ __forceinline__ void pivot_pair8(float& a0, float& a1, int g, int t)
{
    constexpr int J = 2 * K;
    const float d0 = lane_value<4 * J + K, 0>(a0), e = lane_value<4 * J + 4 + K, 0>(a0), d11 = lane_value<4 * J + 4 + K, 0>(a1);
    const float c0 = lane_value<K, 28>(a0), c1 = lane_value<K, 28>(a1);
    const float r00 = lane_value<4 * J, 3>(a0), r01 = lane_value<4 * J, 3>(a1);
    const float r10 = lane_value<4 * J + 4, 3>(a0), r11 = lane_value<4 * J + 4, 3>(a1);
    const float i0 = rcp_fast(d0), l = e * i0, i1 = rcp_fast(fmaf(-l, e, d11));
    const float f0 = (g > J) ? -c0 * i0 : 0.f;
    const float f1 = (g > J + 1) ? -fmaf(f0, e, c1) * i1 : 0.f;
    a0 = fmaf(f1, fmaf(-l, r00, r10), fmaf(f0, r00, a0));
    a1 = fmaf(f1, fmaf(-l, r01, r11), fmaf(f0, r01, a1));
    if (t == K) {                                          // eliminated columns: the inverse's move in
        if (g > J)
            a0 = fmaf(-f1, l, f0);
        if (g > J + 1)
            a1 = f1;
    }
}

// Inverse of the Cholesky factor of one symmetric positive definite 8 x 8 block held as (a0, a1) = row g, columns 2 t,
// 2 t + 1.  Eliminates below the diagonal in place, the vacated column taking the column of the (unit) inverse, then
// scales row g by 1/sqrt(pivot g).  On return (a0, a1) = W = L^{-1} (lower triangular, exact zeros above the diagonal).
// Returns 0 or 1 + the index of the first non-positive pivot (the same on every lane; the pivots up to it are those of
// the elimination, what follows is meaningless).
// PAIR: two pivots at a time.  A quarter shorter as a chain and a quarter longer in instructions: for launches that leave
// the schedulers idle (one warp per SM walks a step of the n = 16 layer in 1.30 instead of 1.47 us; a batch that fills the
// machine takes 1.94 instead of 1.87 ms).
template <bool PAIR>
__device__ __forceinline__ int chol8_inverse(float& a0, float& a1, int lane)
{
    const int g = lane >> 2, t = lane & 3;
    if constexpr (PAIR) {
        pivot_pair8<0>(a0, a1, g, t);
        pivot_pair8<1>(a0, a1, g, t);
        pivot_pair8<2>(a0, a1, g, t);
    } else {
        pivot8<0>(a0, a1, g, t);
        pivot8<1>(a0, a1, g, t);
        pivot8<2>(a0, a1, g, t);
        pivot8<3>(a0, a1, g, t);
        pivot8<4>(a0, a1, g, t);
        pivot8<5>(a0, a1, g, t);
    }
    pivot8<6>(a0, a1, g, t);
    const float dg = __shfl_sync(FULL, (g & 1) ? a1 : a0, (lane & 28) | (g >> 1));
    const unsigned bad = __ballot_sync(FULL, !(dg > 0.f));
    float rs;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rs) : "f"(dg));
    a0 = (2 * t < g ? a0 : 2 * t == g ? 1.f : 0.f) * rs;
    a1 = (2 * t + 1 < g ? a1 : 2 * t + 1 == g ? 1.f : 0.f) * rs;
    return bad ? 1 + ((__ffs(bad) - 1) >> 2) : 0;
}

// transpose of an 8 x 8 block held as (row g, columns 2 t, 2 t + 1)
__device__ __forceinline__ void transpose8(float& y0, float& y1, float x0, float x1, int lane)
{
    const int g = lane >> 2, t = lane & 3, src = 8 * t + (g >> 1);
    const float p0 = __shfl_sync(FULL, x0, src), p1 = __shfl_sync(FULL, x1, src);
    const float q0 = __shfl_sync(FULL, x0, src + 4), q1 = __shfl_sync(FULL, x1, src + 4);
    y0 = (g & 1) ? p1 : p0;
    y1 = (g & 1) ? q1 : q0;
}

// the tiles above the diagonal that LOWER products leave out: transposes of those below
template <int NB>
__device__ __forceinline__ void mirror(Mat<NB, NB>& m, int lane)
{
#pragma unroll
    for (int i = 0; i < NB; ++i)
#pragma unroll
        for (int j = 2; j < NB; ++j)
            if (j >= 2 * (i / 2) + 2)
                transpose8(m.v[i / 2][j][2 * (i & 1)], m.v[i / 2][j][2 * (i & 1) + 1], m.v[j / 2][i][2 * (j & 1)],
                       m.v[j / 2][i][2 * (j & 1) + 1], lane);
}
// M <- (M + M')/2 on the diagonal blocks, and the blocks above the diagonal become the transposes of those below
template <int NB>
__device__ __forceinline__ void make_symmetric(Mat<NB, NB>& m, int lane)
{
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        float y0, y1;
        float& d0 = m.v[i / 2][i][2 * (i & 1)];
        float& d1 = m.v[i / 2][i][2 * (i & 1) + 1];
        transpose8(y0, y1, d0, d1, lane);
        d0 = 0.5f * (d0 + y0);
        d1 = 0.5f * (d1 + y1);
#pragma unroll
        for (int j = 1; j < NB; ++j)
            if (j > i)
                transpose8(m.v[i / 2][j][2 * (i & 1)], m.v[i / 2][j][2 * (i & 1) + 1], m.v[j / 2][i][2 * (j & 1)],
                       m.v[j / 2][i][2 * (j & 1) + 1], lane);
    }
}

// vectors: "row form" = element 8 b + g in every lane of row g; "column form" = elements 8 b + 2 t, + 1 in lane (., t)
__device__ __forceinline__ void row_to_col(float& c0, float& c1, float r, int lane)
{
    const int t = lane & 3;
    c0 = __shfl_sync(FULL, r, 8 * t);
    c1 = __shfl_sync(FULL, r, 8 * t + 4);
}
__device__ __forceinline__ float col_to_row(float c0, float c1, int lane)
{
    const int g = lane >> 2;
    const float p0 = __shfl_sync(FULL, c0, g >> 1), p1 = __shfl_sync(FULL, c1, g >> 1);
    return (g & 1) ? p1 : p0;
}
__device__ __forceinline__ float sum_over_t(float v)       // result in row form
{
    v += __shfl_xor_sync(FULL, v, 1);
    v += __shfl_xor_sync(FULL, v, 2);
    return v;
}
__device__ __forceinline__ float sum_over_g(float v)       // result in column form
{
    v += __shfl_xor_sync(FULL, v, 4);
    v += __shfl_xor_sync(FULL, v, 8);
    v += __shfl_xor_sync(FULL, v, 16);
    return v;
}

// one 16 x 8 tile: d += X Y' over one 8-wide chunk (x: four registers of X's tile, y: the two registers of Y's block)
struct Tile {
    uint32_t h[4], l[4];
};
__device__ __forceinline__ void split_tile(Tile& s, const float (&v)[4])
{
#pragma unroll
    for (int e = 0; e < 4; e += 2)
        split2(v[e], v[e + 1], s.h[e], s.h[e + 1], s.l[e], s.l[e + 1]);
}
__device__ __forceinline__ void mma3(float (&d)[4], const Tile& x, uint32_t yh0, uint32_t yh1, uint32_t yl0, uint32_t yl1,
                                     bool from_zero = false)
{
    const float z[4] = {0.f, 0.f, 0.f, 0.f};
    if (from_zero)
        mma(d, z, x.l[0], x.l[2], x.l[1], x.l[3], yh0, yh1);
    else
        mma(d, x.l[0], x.l[2], x.l[1], x.l[3], yh0, yh1);
    mma(d, x.h[0], x.h[2], x.h[1], x.h[3], yl0, yl1);
    mma(d, x.h[0], x.h[2], x.h[1], x.h[3], yh0, yh1);
}

// Factorisation of S = L L' (nS = -S, 8 MB x 8 MB) together with Z' = Y'L^{-T} (nY = -Y', 8 NB x 8 MB), panel by panel
// of eight columns: the diagonal block is factored and inverted in registers, everything else is a product with its
// inverse.  On return nS holds L below the diagonal blocks, z the split of Z', w[p] = W_p = inverse of the p-th diagonal
// block of L.  (Negated operands keep every update a plain accumulation.)  Returns 0 or 1 + the first bad pivot.
template <int NB, int MB, bool PAIR = false>
__device__ __forceinline__ int factor(Mat<MB, MB>& nS, Mat<NB, MB>& nY, Split<NB, MB>& z, float (&w)[MB][2], int lane)
{
    int bad = 0;
#pragma unroll
    for (int p = 0; p < MB; ++p) {
        float a0 = -nS.v[p / 2][p][2 * (p & 1)], a1 = -nS.v[p / 2][p][2 * (p & 1) + 1];
        const int b = chol8_inverse<PAIR>(a0, a1, lane);
        if (b && !bad)
            bad = 8 * p + b;
        w[p][0] = a0;
        w[p][1] = a1;
        uint32_t wh0, wh1, wl0, wl1;
        split2(-a0, -a1, wh0, wh1, wl0, wl1);
        Tile lt[Mat<MB, MB>::MT];
#pragma unroll
        for (int mt = 0; mt < Mat<MB, MB>::MT; ++mt) {
            if (mt >= p / 2 && p + 1 < MB && 2 * mt + 1 > p) {            // the tile holds rows below the diagonal block
                Tile x;
                split_tile(x, nS.v[mt][p]);
                float d[4];
                mma3(d, x, wh0, wh1, wl0, wl1, true);
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    nS.v[mt][p][e] = d[e];
                split_tile(lt[mt], d);
            }
        }
#pragma unroll
        for (int mt = 0; mt < Mat<NB, MB>::MT; ++mt) {
            Tile x;
            split_tile(x, nY.v[mt][p]);
            float d[4];
            mma3(d, x, wh0, wh1, wl0, wl1, true);
#pragma unroll
            for (int e = 0; e < 4; e += 2) {
                nY.v[mt][p][e] = d[e];                     // Z' (float32) replaces its column of -Y'
                nY.v[mt][p][e + 1] = d[e + 1];
                split2(d[e], d[e + 1], z.h[mt][p][e], z.h[mt][p][e + 1], z.l[mt][p][e], z.l[mt][p][e + 1]);
            }
        }
#pragma unroll
        for (int q = 1; q < MB; ++q) {
            if (q <= p)
                continue;
            const int e = 2 * (q & 1);
            const Tile y = lt[q / 2];
#pragma unroll
            for (int mt = 0; mt < Mat<MB, MB>::MT; ++mt)
                if (mt >= q / 2)
                    mma3(nS.v[mt][q], lt[mt], y.h[e], y.h[e + 1], y.l[e], y.l[e + 1]);
#pragma unroll
            for (int mt = 0; mt < Mat<NB, MB>::MT; ++mt) {
                Tile x;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    x.h[k] = z.h[mt][p][k];
                    x.l[k] = z.l[mt][p][k];
                }
                mma3(nY.v[mt][q], x, y.h[e], y.h[e + 1], y.l[e], y.l[e + 1]);
            }
        }
    }
    return bad;
}

// K' = -Z'L^{-1} (8 NB x 8 MB) from the results of factor(); zt is Z' in float32 and becomes K'.
// Block column p, last one first:  K'_p = (Z'_p + sum_{q > p} K'_q L_qp)(-W_p).
template <int NB, int MB>
__device__ __forceinline__ void gains(Mat<NB, MB>& zt, const Mat<MB, MB>& L, const float (&w)[MB][2], int lane)
{
    constexpr int MT = Mat<NB, MB>::MT;
#pragma unroll
    for (int p = MB - 1; p >= 0; --p) {
#pragma unroll
        for (int q = 1; q < MB; ++q) {
            if (q <= p)
                continue;
            float y0, y1;
            transpose8(y0, y1, L.v[q / 2][p][2 * (q & 1)], L.v[q / 2][p][2 * (q & 1) + 1], lane);
            uint32_t h0, h1, l0, l1;
            split2(y0, y1, h0, h1, l0, l1);
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                Tile x;
                split_tile(x, zt.v[mt][q]);
                mma3(zt.v[mt][p], x, h0, h1, l0, l1);
            }
        }
        float y0, y1;
        transpose8(y0, y1, -w[p][0], -w[p][1], lane);
        uint32_t h0, h1, l0, l1;
        split2(y0, y1, h0, h1, l0, l1);
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            Tile x;
            split_tile(x, zt.v[mt][p]);
            float d[4];
            mma3(d, x, h0, h1, l0, l1, true);
#pragma unroll
            for (int e = 0; e < 4; ++e)
                zt.v[mt][p][e] = d[e];
        }
    }
}

// ---- operands that stay the same over many products: their split parts in shared memory in register order, one
// 16-byte word per lane, tile and part, so that a product reads them without arithmetic
template <int RB, int CB>
struct Stored {
    static constexpr int MT = (RB + 1) / 2;
    uint4 q[MT][CB][2][32];
};
template <int RB, int CB>
__device__ __forceinline__ void keep(Stored<RB, CB>& st, const Mat<RB, CB>& m, int lane)
{
    Split<RB, CB> s;
    split(s, m);
#pragma unroll
    for (int mt = 0; mt < Mat<RB, CB>::MT; ++mt)
#pragma unroll
        for (int cb = 0; cb < CB; ++cb) {
            // in the order of the instruction's A registers, so that the loaded group is used as it is
            st.q[mt][cb][0][lane] = make_uint4(s.h[mt][cb][0], s.h[mt][cb][2], s.h[mt][cb][1], s.h[mt][cb][3]);
            st.q[mt][cb][1][lane] = make_uint4(s.l[mt][cb][0], s.l[mt][cb][2], s.l[mt][cb][1], s.l[mt][cb][3]);
        }
}
// d = c + X * Y' with X stored
template <int RB, int KB, int CB, bool LOWER = false>
__device__ __forceinline__ void product(Mat<RB, CB>& d, const Mat<RB, CB>* c, const Stored<RB, KB>& x, const Split<CB, KB>& y, int lane)
{
    const float z[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int kb = 0; kb < KB; ++kb) {
        uint4 a[Mat<RB, CB>::MT][2];
#pragma unroll
        for (int mt = 0; mt < Mat<RB, CB>::MT; ++mt) {
            a[mt][0] = x.q[mt][kb][0][lane];
            a[mt][1] = x.q[mt][kb][1][lane];
        }
#pragma unroll
        for (int pass = 0; pass < 3; ++pass)
#pragma unroll
            for (int cb = 0; cb < CB; ++cb)
#pragma unroll
                for (int mt = 0; mt < Mat<RB, CB>::MT; ++mt) {
                    if (LOWER && cb > 2 * mt + 1)
                        continue;
                    const uint4 v = a[mt][pass == 0];
                    const uint32_t(&b)[4] = pass == 1 ? y.l[cb / 2][kb] : y.h[cb / 2][kb];
                    const uint32_t b0 = b[2 * (cb & 1)], b1 = b[2 * (cb & 1) + 1];
                    if (kb || pass)
                        mma(d.v[mt][cb], v.x, v.y, v.z, v.w, b0, b1);
                    else if (c)
                        mma(d.v[mt][cb], c->v[mt][cb], v.x, v.y, v.z, v.w, b0, b1);
                    else
                        mma(d.v[mt][cb], z, v.x, v.y, v.z, v.w, b0, b1);
                }
    }
}
// the float32 matrix back from its parts (exact)
template <int RB, int CB>
__device__ __forceinline__ void unkeep(Mat<RB, CB>& m, const Stored<RB, CB>& st, int lane)
{
#pragma unroll
    for (int mt = 0; mt < Mat<RB, CB>::MT; ++mt)
#pragma unroll
        for (int cb = 0; cb < CB; ++cb) {
            const uint4 h = st.q[mt][cb][0][lane], l = st.q[mt][cb][1][lane];
            m.v[mt][cb][0] = __uint_as_float(h.x) + __uint_as_float(l.x);
            m.v[mt][cb][2] = __uint_as_float(h.y) + __uint_as_float(l.y);
            m.v[mt][cb][1] = __uint_as_float(h.z) + __uint_as_float(l.z);
            m.v[mt][cb][3] = __uint_as_float(h.w) + __uint_as_float(l.w);
        }
}
// d = c + X X' with a result that is symmetric bit for bit when c is: lo*hi and hi*lo start from zero, so that one is the
// transpose of the other, and are added to each other first
template <int NB, int KB>
__device__ __forceinline__ void product_symmetric(Mat<NB, NB>& d, const Split<NB, KB>& x)
{
    const float z[4] = {0.f, 0.f, 0.f, 0.f};
    constexpr int MT = Mat<NB, NB>::MT;
#pragma unroll
    for (int cb = 0; cb < NB; ++cb)
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            if (cb > 2 * mt + 1)
                continue;                                  // lower tiles only: mirror() fills the rest
            float e1[4], e2[4];
#pragma unroll
            for (int kb = 0; kb < KB; ++kb) {
                const uint32_t(&xh)[4] = x.h[mt][kb];
                const uint32_t(&xl)[4] = x.l[mt][kb];
                const uint32_t(&yh)[4] = x.h[cb / 2][kb];
                const uint32_t(&yl)[4] = x.l[cb / 2][kb];
                const int i = 2 * (cb & 1);
                if (kb == 0) {
                    mma(e1, z, xl[0], xl[2], xl[1], xl[3], yh[i], yh[i + 1]);
                    mma(e2, z, xh[0], xh[2], xh[1], xh[3], yl[i], yl[i + 1]);
                } else {
                    mma(e1, xl[0], xl[2], xl[1], xl[3], yh[i], yh[i + 1]);
                    mma(e2, xh[0], xh[2], xh[1], xh[3], yl[i], yl[i + 1]);
                }
                mma(d.v[mt][cb], xh[0], xh[2], xh[1], xh[3], yh[i], yh[i + 1]);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e)
                d.v[mt][cb][e] += e1[e] + e2[e];
        }
}

// ---- the same products on pairs of halves: one instruction takes sixteen contraction indices at the price of eight in tf32
// (8 cycles of a scheduler's pipe): half the instructions, half the operand registers.  An operand is split into
//     s x = h + 2^-11 l,    h = half(s x),  l = half(2^11 (s x - h)),    s a power of two,
// so that the remainder has the exponent of the number itself (Ootomo and Yokota, 2022) and l*h + h*l are summed first, from
// zero, and multiplied by 2^-11 before h*h goes on top.  A float16 keeps the eleven bits of a tf32 number: the pair represents
// s x to 2^-22 |s x| (tf32: 2^-21, the remainder is truncated) above 2^-14 and to 2^-36 below, which is 2^-21 |s x| down to
// 2^-15.  Who may use them, and when: riccati_frag.cuh.  The tiles of two neighbouring column blocks are the instruction's A
// operand as they stand, and the B operand of the transpose, as above.
template <int RB, int CB>
struct Halves {
    static constexpr int MT = (RB + 1) / 2;
    uint32_t h[MT][CB][2], l[MT][CB][2];                   // [..][0]: row g, columns 2 t and 2 t + 1; [..][1]: row g + 8
};
constexpr float HALF_LOW = 0x1p-15f, HALF_HIGH = 65504.f, REMAINDER = 2048.f;
__device__ __forceinline__ __half2 as_half2(uint32_t x) { return *reinterpret_cast<const __half2*>(&x); }
// (a, b) <- (c a, c b)
__device__ __forceinline__ void scale_pair(float& a, float& b, float c)
{
    asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%0, %1};\n\tmov.b64 y, {%2, %2};\n\tmul.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
        : "+f"(a), "+f"(b) : "f"(c));
}
__device__ __forceinline__ void split_halves(float x0, float x1, float s, uint32_t& h, uint32_t& l)
{
    float y0 = x0, y1 = x1;
    scale_pair(y0, y1, s);
    const __half2 hh = __floats2half2_rn(y0, y1);
    h = *reinterpret_cast<const uint32_t*>(&hh);
    scale_pair(y0, y1, REMAINDER);
    float l0, l1;                                           // 2^11 (s x - h), exact; the mixed fma saves converting h back
    asm("{\n\t.reg .b16 a, b;\n\tmov.b32 {a, b}, %2;\n\t"
        "fma.rn.f32.f16 %0, a, %5, %3;\n\tfma.rn.f32.f16 %1, b, %5, %4;\n\t}"
        : "=f"(l0), "=f"(l1) : "r"(h), "f"(y0), "f"(y1), "h"((unsigned short)0xe800));     // -2048
    const __half2 ll = __floats2half2_rn(l0, l1);
    l = *reinterpret_cast<const uint32_t*>(&ll);
}
template <int RB, int CB>
__device__ __forceinline__ void split(Halves<RB, CB>& x, const Mat<RB, CB>& m, float s)
{
#pragma unroll
    for (int mt = 0; mt < Mat<RB, CB>::MT; ++mt)
#pragma unroll
        for (int cb = 0; cb < CB; ++cb)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                if (e && 2 * mt + 1 >= RB)                  // rows that do not exist
                    x.h[mt][cb][e] = x.l[mt][cb][e] = 0u;
                else
                    split_halves(m.v[mt][cb][2 * e], m.v[mt][cb][2 * e + 1], s, x.h[mt][cb][e], x.l[mt][cb][e]);
            }
}
// true in the whole warp when at least `elements` of X are not below LOW and none is above the largest float16 or a NaN
template <int RB, int CB>
__device__ __forceinline__ bool in_range(const Halves<RB, CB>& x, float low, int elements)
{
    __half2 count = __float2half2_rn(0.f), top = __float2half2_rn(0.f);
#pragma unroll
    for (int mt = 0; mt < Halves<RB, CB>::MT; ++mt)
#pragma unroll
        for (int cb = 0; cb < CB; ++cb)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                if (e && 2 * mt + 1 >= RB)
                    continue;
                const __half2 v = __habs2(as_half2(x.h[mt][cb][e]));
                count = __hadd2(count, __hge2(v, __float2half2_rn(low)));
                top = __hmax2_nan(top, v);
            }
    const float2 c = __half22float2(count);
    return __reduce_add_sync(FULL, __hble2(top, __float2half2_rn(HALF_HIGH)) ? (int)(c.x + c.y) : -65536) >= elements;
}
// d = X Y' over sixteen contraction indices, or over eight
__device__ __forceinline__ void mma_halves(float (&d)[4], const float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                           uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}
__device__ __forceinline__ void mma_halves(float (&d)[4], const float (&c)[4], uint32_t a0, uint32_t a1, uint32_t b0)
{
    asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%7,%8,%9,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(b0), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}
// split parts in shared memory, two column blocks to a 16-byte word (in the order of the instruction's A registers)
template <int RB, int CB>
struct StoredHalves {
    static constexpr int MT = (RB + 1) / 2, CP = (CB + 1) / 2;
    uint4 q[MT][CP][2][32];
};
template <int RB, int CB>
__device__ __forceinline__ void keep(StoredHalves<RB, CB>& st, const Halves<RB, CB>& s, int lane)
{
#pragma unroll
    for (int mt = 0; mt < Mat<RB, CB>::MT; ++mt)
#pragma unroll
        for (int cb = 0; cb < CB; cb += 2) {
            const int c1 = cb + 1 < CB ? cb + 1 : cb;       // (an odd last block: the second half of the word is not read)
            st.q[mt][cb / 2][0][lane] = make_uint4(s.h[mt][cb][0], s.h[mt][cb][1], s.h[mt][c1][0], s.h[mt][c1][1]);
            st.q[mt][cb / 2][1][lane] = make_uint4(s.l[mt][cb][0], s.l[mt][cb][1], s.l[mt][c1][0], s.l[mt][c1][1]);
        }
}
// d = X Y' with X stored, scaled by the scales of both operands; LOWER as above
template <int RB, int KB, int CB, bool LOWER = false>
__device__ __forceinline__ void product_halves(Mat<RB, CB>& d, const StoredHalves<RB, KB>& x, const Halves<CB, KB>& y, int lane)
{
#pragma unroll
    for (int main = 0; main < 2; ++main) {                  // lo*hi + hi*lo, then hi*hi
#pragma unroll
        for (int kb = 0; kb < KB; kb += 2) {
#pragma unroll
            for (int pass = main ? 2 : 0; pass < (main ? 3 : 2); ++pass) {
                uint4 a[Mat<RB, CB>::MT];
#pragma unroll
                for (int mt = 0; mt < Mat<RB, CB>::MT; ++mt)
                    a[mt] = x.q[mt][kb / 2][pass == 0][lane];
#pragma unroll
                for (int cb = 0; cb < CB; ++cb)
#pragma unroll
                    for (int mt = 0; mt < Mat<RB, CB>::MT; ++mt) {
                        if (LOWER && cb > 2 * mt + 1)
                            continue;
                        float(&dd)[4] = d.v[mt][cb];
                        if (!kb && !pass)
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                dd[e] = 0.f;
                        const uint32_t b0 = pass == 1 ? y.l[cb / 2][kb][cb & 1] : y.h[cb / 2][kb][cb & 1];
                        if (kb + 1 < KB)
                            mma_halves(dd, dd, a[mt].x, a[mt].y, a[mt].z, a[mt].w, b0,
                                       pass == 1 ? y.l[cb / 2][kb + 1][cb & 1] : y.h[cb / 2][kb + 1][cb & 1]);
                        else
                            mma_halves(dd, dd, a[mt].x, a[mt].y, b0);
                    }
            }
        }
        if (!main)
#pragma unroll
            for (int cb = 0; cb < CB; ++cb)
#pragma unroll
                for (int mt = 0; mt < Mat<RB, CB>::MT; ++mt)
                    if (!(LOWER && cb > 2 * mt + 1)) {
                        scale_pair(d.v[mt][cb][0], d.v[mt][cb][1], 1.f / REMAINDER);
                        scale_pair(d.v[mt][cb][2], d.v[mt][cb][3], 1.f / REMAINDER);
                    }
    }
}

// z = L^{-1} v and k = -L^{-T} z for a vector in row form, from the results of factor(): z in column form, k in column form
template <int MB>
__device__ __forceinline__ void solve_vector(float (&zc)[MB][2], float (&kc)[MB][2], const float (&v)[MB], const Mat<MB, MB>& L,
                                             const float (&w)[MB][2], int lane)
{
    float zr[MB], kr[MB];
#pragma unroll
    for (int b = 0; b < MB; ++b) {
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < MB; ++k)
            if (k < b)
                s = fmaf(L.v[b / 2][k][2 * (b & 1)], zc[k][0], fmaf(L.v[b / 2][k][2 * (b & 1) + 1], zc[k][1], s));
        float c0, c1;
        row_to_col(c0, c1, b ? v[b] - sum_over_t(s) : v[b], lane);
        zr[b] = sum_over_t(fmaf(w[b][0], c0, w[b][1] * c1));
        row_to_col(zc[b][0], zc[b][1], zr[b], lane);
    }
#pragma unroll
    for (int b = MB - 1; b >= 0; --b) {                     // last block first
        float s0 = 0.f, s1 = 0.f;                           // (L_qb' k_q) in column form
#pragma unroll
        for (int q = 0; q < MB; ++q)
            if (q > b) {
                s0 = fmaf(L.v[q / 2][b][2 * (q & 1)], kr[q], s0);
                s1 = fmaf(L.v[q / 2][b][2 * (q & 1) + 1], kr[q], s1);
            }
        float x = zr[b];
        if (b + 1 < MB)
            x += col_to_row(sum_over_g(s0), sum_over_g(s1), lane);
        kc[b][0] = -sum_over_g(w[b][0] * x);
        kc[b][1] = -sum_over_g(w[b][1] * x);
        kr[b] = col_to_row(kc[b][0], kc[b][1], lane);
    }
}

} // namespace frag
} // namespace ttc
