// Building blocks of the sigma-product baseline, which spreads the columns of a matrix over the lanes of a warp: N lanes own
// one instance (two instances per warp when N = 16), lane c holds COLUMN c of every per-instance matrix, and rows are
// broadcast from the instance's scratch in shared memory (row stride N + 4 floats: 16-byte accesses by row owners and 4-byte
// accesses by column owners are both conflict-free).
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
