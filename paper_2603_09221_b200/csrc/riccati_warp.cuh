// Building blocks of the kernels that spread the columns of a matrix over the lanes of a warp (scan over the horizon,
// sigma-product baseline): N lanes own one instance (two instances per warp when N = 16), lane c
// holds COLUMN c of every per-instance matrix, and rows are broadcast from the instance's scratch in shared memory (row
// stride N + 4 floats: 16-byte accesses by row owners and 4-byte accesses by column owners are both conflict-free).
#pragma once

#include "common.cuh"

namespace ttc {
namespace rwarp {

constexpr int WARPS = 4;
constexpr int THREADS = 32 * WARPS;

template <int N>
struct Shape {
    static constexpr int LD = N + 4;               // row stride in floats
    static constexpr int IPW = 32 / N;             // instances per warp
    static constexpr int SLOTS = WARPS * IPW;      // instances in flight per CTA = tokens per chunk
    static constexpr int MAT = N * LD;
};

// Cholesky of an N x N SPD matrix spread over N lanes (lane i = row i = column i).  On return s holds
// row `c` of L (entries right of the diagonal are meaningless), rs_own = 1 / L[c][c].  The trailing
// update uses s_ij s_cj / d_j so that the broadcast of column j does not wait for the reciprocal.
// Returns 0 or 1 + the index of the first non-positive pivot.
template <int N>
__device__ __forceinline__ int seg_chol(float (&s)[N], float& rs_own, int c)
{
    int bad = 0;
    rs_own = 1.f;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const float sj = s[j];
        float d = __shfl_sync(0xffffffffu, sj, j, N);
        if (!(d > 0.f)) {
            if (!bad)
                bad = j + 1;
            d = 1.f;
        }
        const float rinv = __frcp_rn(d);
        const float f = sj * rinv;
#pragma unroll
        for (int cc = j + 1; cc < N; ++cc) {
            const float lc = __shfl_sync(0xffffffffu, sj, cc, N);
            s[cc] = fmaf(-f, lc, s[cc]);
        }
        const float rs = rsqrtf(d);
        s[j] = sj * rs;
        if (c == j)
            rs_own = rs;
    }
    return bad;
}

template <int N>
__device__ __forceinline__ void load_row(float (&v)[N], const float* row)
{
#pragma unroll
    for (int q = 0; q < N / 4; ++q) {
        const float4 t = *reinterpret_cast<const float4*>(row + 4 * q);
        v[4 * q] = t.x; v[4 * q + 1] = t.y; v[4 * q + 2] = t.z; v[4 * q + 3] = t.w;
    }
}
template <int N>
__device__ __forceinline__ void store_row(float* row, const float (&v)[N])
{
#pragma unroll
    for (int q = 0; q < N / 4; ++q)
        *reinterpret_cast<float4*>(row + 4 * q) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
}
// ---- packed fp32 pairs: fma.rn.f32x2 does two FMAs per issued instruction (the dense loops are issue-bound)
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ void fma2(f32x2& acc, f32x2 a, f32x2 b)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
template <int N>
__device__ __forceinline__ void pack_row(f32x2 (&v2)[N / 2], const float (&v)[N])
{
#pragma unroll
    for (int i = 0; i < N / 2; ++i)
        v2[i] = pack2(v[2 * i], v[2 * i + 1]);
}
template <int N>
__device__ __forceinline__ void unpack_row(float (&v)[N], const f32x2 (&v2)[N / 2])
{
#pragma unroll
    for (int i = 0; i < N / 2; ++i)
        unpack2(v2[i], v[2 * i], v[2 * i + 1]);
}
// acc[l] += w * row[l], l = 0..N-1
template <int N>
__device__ __forceinline__ void axpy_row(f32x2 (&acc)[N / 2], float w, const float* row)
{
    const f32x2 ww = pack2(w, w);
#pragma unroll
    for (int q = 0; q < N / 4; ++q) {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(row + 4 * q);
        fma2(acc[2 * q], ww, t.x);
        fma2(acc[2 * q + 1], ww, t.y);
    }
}

// ---- 32 x 32 x 32 contractions on the tensor cores (n = 32): mma.sync m16n8k8, tf32 operands, fp32 accumulate, with the
// operands split into tf32 high and low parts and three passes (lo*hi + hi*lo + hi*hi), which keeps float32-grade
// accuracy (the 1e-4 tolerance of the float32 configurations rules out single-pass tf32).  One warp computes one
// product; operands are float32 matrices in shared memory with row stride LD32 = 36 floats.
//   acc[mt][nt][..] is the 16 x 8 tile (rows 16 mt.., columns 8 nt..) in the accumulator layout of the instruction:
//   lane = 4 g + t holds (g, 2t), (g, 2t + 1), (g + 8, 2t), (g + 8, 2t + 1).
__device__ __forceinline__ void mma_tf32(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void split_hi_lo(float x, uint32_t& hi, uint32_t& lo)
{
    hi = __float_as_uint(x) & 0xffffe000u;
    lo = __float_as_uint(x - __uint_as_float(hi));
}
constexpr int LD32 = 36;
// acc += A' * B with both operands stored k-major: A'[i][k] = Am[k * LD32 + i], B[k][j] = Bm[k * LD32 + j].
// The instruction leaves the assignment of contraction indices to its k slots free as long as A and B agree, so
// slot (t, half) of k-step ks takes k = 16 (ks / 2) + 8 half + 2 t + (ks % 2): with the row stride of 36 floats the
// 32 lanes of a fragment load then fall into 32 different banks (bank = 8 t + g + 4 (ks % 2)).
__device__ __forceinline__ void mma32_product(float (&acc)[2][4][4], const float* Am, const float* Bm, int lane)
{
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
        const int k0 = 16 * (ks >> 1) + 2 * t + (ks & 1);
        uint32_t ah[2][4], al[2][4], bh[4][2], bl[4][2];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
            const int i0 = 16 * mt + g;
            split_hi_lo(Am[k0 * LD32 + i0], ah[mt][0], al[mt][0]);
            split_hi_lo(Am[k0 * LD32 + i0 + 8], ah[mt][1], al[mt][1]);
            split_hi_lo(Am[(k0 + 8) * LD32 + i0], ah[mt][2], al[mt][2]);
            split_hi_lo(Am[(k0 + 8) * LD32 + i0 + 8], ah[mt][3], al[mt][3]);
        }
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            split_hi_lo(Bm[k0 * LD32 + 8 * nt + g], bh[nt][0], bl[nt][0]);
            split_hi_lo(Bm[(k0 + 8) * LD32 + 8 * nt + g], bh[nt][1], bl[nt][1]);
        }
        // pass-major order: the eight accumulator tiles of a pass are independent of one another
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
                mma_tf32(acc[mt][nt], al[mt][0], al[mt][1], al[mt][2], al[mt][3], bh[nt][0], bh[nt][1]);
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
                mma_tf32(acc[mt][nt], ah[mt][0], ah[mt][1], ah[mt][2], ah[mt][3], bl[nt][0], bl[nt][1]);
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
                mma_tf32(acc[mt][nt], ah[mt][0], ah[mt][1], ah[mt][2], ah[mt][3], bh[nt][0], bh[nt][1]);
    }
}
__device__ __forceinline__ void mma32_zero(float (&acc)[2][4][4])
{
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                acc[mt][nt][e] = 0.f;
}
// accumulator tiles -> row-major matrix in shared memory (8-byte stores)
__device__ __forceinline__ void mma32_store(float* Dm, const float (&acc)[2][4][4], int lane)
{
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            *reinterpret_cast<float2*>(Dm + (16 * mt + g) * LD32 + 8 * nt + 2 * t) = make_float2(acc[mt][nt][0], acc[mt][nt][1]);
            *reinterpret_cast<float2*>(Dm + (16 * mt + g + 8) * LD32 + 8 * nt + 2 * t) = make_float2(acc[mt][nt][2], acc[mt][nt][3]);
        }
}

// out[:] += sum_k coef[k] * row_k(M)      (M row-major in shared memory, row stride LD)
template <int N>
__device__ __forceinline__ void mix(f32x2 (&out)[N / 2], const float (&coef)[N], const float* M)
{
#pragma unroll
    for (int k = 0; k < N; ++k)
        axpy_row<N>(out, coef[k], M + k * Shape<N>::LD);
}
template <int N>
__device__ __forceinline__ void zero2(f32x2 (&v)[N / 2])
{
#pragma unroll
    for (int i = 0; i < N / 2; ++i)
        v[i] = 0ull;
}

} // namespace rwarp
} // namespace ttc
