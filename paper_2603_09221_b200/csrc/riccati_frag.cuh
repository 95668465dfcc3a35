// Riccati-backward + rollout kernel, float32, for n, m up to 32 (any request) or 64 (time-invariant): one WARP per
// instance, every matrix of the step in registers in the mma.sync accumulator layout (frag.cuh), so that a step is a
// chain of tensor-core products, one eight-column factorisation panel per block of controls and a few shuffles, without
// barriers.  Other sizes than whole blocks are padded: R with the identity, everything else with zero.
//
// The recursion is carried in negated variables (nP = -P etc.): every update is then a plain accumulation.
//   V = B' nP,  T = A' nP,  nS = -R + B' V',  nY' = A' V',  nP_t = -Q + A' T' + Z' Z     (Prop. 3.1; Alg. 1)
// with S = L L', Z = L^{-1} Y and, when gains are wanted, K' = -Z' L^{-1} from the inverses of L's diagonal blocks.
// Above 16 states or controls the five products with A, B and P run on pairs of halves while the values permit it (below); Z'Z,
// the factorisation and everything up to 16 in three passes of tf32.
//
// What bounds it: at n = 16 a step is 96 tensor-core instructions (8 cycles on a scheduler's pipe, about 4 of its issue
// slots) in about 830, and five or six warps per scheduler hide most of the chain of five products and sixteen
// pivots.  At n = 32 it is 441 tensor-core instructions (657 in tf32), two warps per scheduler (all 255 registers); above, registers spill
// to local memory (0.2 KB per lane at 40 x 16, 1.6 KB at 40 x 40, which the first-level cache absorbs; 10.7 KB at 64 x 64,
// which it does not: only twice as fast as one CTA per instance there).
// The forms this replaced: rows broadcast from shared memory at n = 16 (load/store pipe at 88 %), products through shared
// memory at n = 32 (74 %), one CTA per instance with two barriers per pivot elsewhere.  Measured before -> now:
//   65536 instances n = 16, H = 32, operands from memory  4.26 -> 2.50 ms     4096, n = 16, H = 16, all outputs 188 -> 106 us
//   16384 instances n = 32, H = 64, all outputs           14.2 -> 6.87 ms     1155, n = 40, m = 12, H = 20     2428 -> 198 us
//   64 instances n = 8, H = 8, own dynamics               107 -> 11 us     1155, n = m = 60, H = 20            21.9 -> 10.3 ms
// The halves' part in that, against three passes of tf32 throughout: n = 32 8.41 -> 6.87 ms, 40 x 12 235 -> 198 us, time-varying
// n = 32, 2048 instances of 32 steps 0.54 -> 0.47 ms.  Problems outside the range take 235 us at 40 x 12, and at n = 32 what
// they took (1.10 ms on 4096 instances of 32 steps, 0.91 inside).
#pragma once

#include "common.cuh"
#include "frag.cuh"

namespace ttc {
namespace rfrag {

using namespace frag;

constexpr int MAX_WARPS = 4;

// element offsets of one instance's operands
struct Place {
    long long inst;
    long long i0, i1, i2;
    __device__ __forceinline__ long long off(const OperandDev& o) const { return i0 * o.s0 + i1 * o.s1 + i2 * o.s2; }
};
// w-th instance of the launch's window (all counts are below 2^31)
__device__ __forceinline__ Place place(const SolveParams& p, unsigned w)
{
    Place r;
    const unsigned tc = (unsigned)p.tcount, b1 = (unsigned)p.b1;
    const unsigned head = w / tc, i2 = w - head * tc;
    r.i2 = p.t0 + i2;
    r.i0 = head / b1;
    r.i1 = head - (unsigned)r.i0 * b1;
    r.inst = (long long)head * p.b2 + r.i2;
    return r;
}

// ---- operands of one time step of one instance, staged in the warp's shared memory by asynchronous copies ahead of
// their use.  A and B are read transposed (lane (g, t) takes row 2 t, column g): with rows of 8 k + 4 floats the 32 lanes
// fall into 32 banks.  Q and R are read as pairs along the rows.
constexpr int pair_stride(int blocks) { return 8 * blocks + (blocks == 2 ? 4 : blocks % 2 ? 0 : 8); }
template <int NB, int MB>
struct Operands {
    static constexpr int LA = 8 * NB + 4, LB = 8 * MB + 4, LQ = pair_stride(NB), LR = pair_stride(MB);
    float A[8 * NB * LA], B[8 * NB * LB], Q[8 * NB * LQ], R[8 * MB * LR];
};
// What a warp keeps in shared memory.  Time-varying and n <= 16: two buffers in turn, A and B split in registers in every
// step.  Otherwise A' and B' are split once per change and kept in register order; the raw matrices pass through the same
// place.  (For n = 32 a second buffer does not fit, and the splits of five products cost more than storing them.)
template <int NB, int MB, bool TWO>
struct WarpMem {
    Operands<NB, MB> op[2];
};
template <int NB, int MB>
struct WarpMem<NB, MB, false> {
    using Ops = Operands<NB, MB>;
    Stored<NB, NB> A;
    Stored<MB, NB> B;
    float Q[8 * NB * Ops::LQ], R[8 * MB * Ops::LR];
    __device__ __forceinline__ float* rawA() { return reinterpret_cast<float*>(&A); }
    __device__ __forceinline__ float* rawB() { return reinterpret_cast<float*>(&B); }
    __device__ __forceinline__ StoredHalves<NB, NB>& halvesA() { return reinterpret_cast<StoredHalves<NB, NB>&>(A); }
    __device__ __forceinline__ StoredHalves<MB, NB>& halvesB() { return reinterpret_cast<StoredHalves<MB, NB>&>(B); }
    static_assert(sizeof(StoredHalves<NB, NB>) <= sizeof(Stored<NB, NB>) && sizeof(StoredHalves<MB, NB>) <= sizeof(Stored<MB, NB>), "halves");
    static_assert(sizeof(Stored<NB, NB>) >= sizeof(Ops::A) && sizeof(Stored<MB, NB>) >= sizeof(Ops::B), "raw operand does not fit");
};

__device__ __forceinline__ void copy16(float* dst, const float* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy4(float* dst, const float* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_landed()
{
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
}
// rows x cols row-major matrix (rows <= 8 RB, cols <= 8 CB) -> dst with row length LD; elements outside stay as they are
template <int RB, int CB, int LD, bool PAD>
__device__ __forceinline__ void stage(float* dst, const OperandDev& o, long long off, int rows, int cols, int lane)
{
    if (o.dtype == TTC_BF16) {
#pragma unroll 4
        for (int e = lane; e < 64 * RB * CB; e += 32) {
            const int r = e / (8 * CB), c = e % (8 * CB);
            if (!PAD || (r < rows && c < cols))
                dst[r * LD + c] = load_elem(o, off + r * (PAD ? cols : 8 * CB) + c);
        }
        return;
    }
    const float* src = reinterpret_cast<const float*>(o.ptr) + off;
    if (PAD) {
#pragma unroll 4
        for (int e = lane; e < 64 * RB * CB; e += 32) {
            const int r = e / (8 * CB), c = e % (8 * CB);
            if (r < rows && c < cols)
                copy4(dst + r * LD + c, src + r * cols + c);
        }
    } else {
#pragma unroll
        for (int e = lane; e < 16 * RB * CB; e += 32)
            copy16(dst + (e / (2 * CB)) * LD + 4 * (e % (2 * CB)), src + 4 * e);
    }
}
// X = M' from shared memory (with PAD: zero outside the nk x ni matrix)
template <int RB, int CB, int LD, bool PAD>
__device__ __forceinline__ void load_transposed(Mat<RB, CB>& x, const float* M, int nk, int ni, int lane)
{
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int mt = 0; mt < Mat<RB, CB>::MT; ++mt)
#pragma unroll
        for (int cb = 0; cb < CB; ++cb)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int i = 16 * mt + g + ((e & 2) ? 8 : 0), k = 8 * cb + 2 * t + (e & 1);
                if (e >= 2 && 2 * mt + 1 >= RB)
                    x.v[mt][cb][e] = 0.f;
                else
                    x.v[mt][cb][e] = PAD && !(i < ni && k < nk) ? 0.f : M[k * LD + i];
            }
}
// the same from a row-major operand in global memory (element by element), zero outside
template <int RB, int CB>
__device__ __forceinline__ void load_transposed_global(Mat<RB, CB>& x, const OperandDev& o, long long off, int ld, int nk, int ni, int lane)
{
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int mt = 0; mt < Mat<RB, CB>::MT; ++mt)
#pragma unroll
        for (int cb = 0; cb < CB; ++cb)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int i = 16 * mt + g + ((e & 2) ? 8 : 0), k = 8 * cb + 2 * t + (e & 1);
                x.v[mt][cb][e] = i < ni && k < nk ? load_elem(o, off + k * ld + i) : 0.f;
            }
}
// x = -M of a square matrix in shared memory
template <int RB, int LD>
__device__ __forceinline__ void load_negated(Mat<RB, RB>& x, const float* M, int lane)
{
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int mt = 0; mt < Mat<RB, RB>::MT; ++mt)
#pragma unroll
        for (int cb = 0; cb < RB; ++cb)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float2 f = make_float2(0.f, 0.f);
                if (h == 0 || 2 * mt + 1 < RB)
                    f = *reinterpret_cast<const float2*>(M + (16 * mt + 8 * h + g) * LD + 8 * cb + 2 * t);
                x.v[mt][cb][2 * h] = -f.x;
                x.v[mt][cb][2 * h + 1] = -f.y;
            }
}
// x = c x - M
template <int RB, int LD, bool LOWER>
__device__ __forceinline__ void scale_and_subtract(Mat<RB, RB>& x, float c, const float* M, int lane)
{
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int mt = 0; mt < Mat<RB, RB>::MT; ++mt)
#pragma unroll
        for (int cb = 0; cb < RB; ++cb) {
            if (LOWER && cb > 2 * mt + 1)
                continue;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float2 f = make_float2(0.f, 0.f);
                if (h == 0 || 2 * mt + 1 < RB)
                    f = *reinterpret_cast<const float2*>(M + (16 * mt + 8 * h + g) * LD + 8 * cb + 2 * t);
                x.v[mt][cb][2 * h] = fmaf(c, x.v[mt][cb][2 * h], -f.x);
                x.v[mt][cb][2 * h + 1] = fmaf(c, x.v[mt][cb][2 * h + 1], -f.y);
            }
        }
}

// element pair (row i, columns k, k + 1) of a row-major output with row length ld
__device__ __forceinline__ void store_pair(float* base, long long idx, float a, float b, int bf16)
{
    if (bf16)
        *reinterpret_cast<__nv_bfloat162*>(reinterpret_cast<__nv_bfloat16*>(base) + idx) = __floats2bfloat162_rn(a, b);
    else
        *reinterpret_cast<float2*>(base + idx) = make_float2(a, b);
}
template <int RB, bool PAD>
__device__ __forceinline__ void store_negated(float* base, long long off, const Mat<RB, RB>& x, int d, int bf16, int lane)
{
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int mt = 0; mt < Mat<RB, RB>::MT; ++mt)
#pragma unroll
        for (int cb = 0; cb < RB; ++cb)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (h == 1 && 2 * mt + 1 >= RB)
                    continue;
                const int i = 16 * mt + 8 * h + g, k = 8 * cb + 2 * t;
                const float a = -x.v[mt][cb][2 * h], b = -x.v[mt][cb][2 * h + 1];
                if (!PAD) {
                    store_pair(base, off + i * (8 * RB) + k, a, b, bf16);
                } else if (i < d) {
                    if (k < d)
                        store_out(base, off + i * d + k, a, bf16);
                    if (k + 1 < d)
                        store_out(base, off + i * d + k + 1, b, bf16);
                }
            }
}
// K [m][n] from K' (rows: states, columns: controls): for each control, eight consecutive states per request
template <int NB, int MB, bool PAD>
__device__ __forceinline__ void store_gain(float* base, long long off, const Mat<NB, MB>& kt, int n, int m, int bf16, int lane)
{
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int cb = 0; cb < MB; ++cb)
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int mt = 0; mt < Mat<NB, MB>::MT; ++mt) {
                if (e >= 2 && 2 * mt + 1 >= NB)
                    continue;
                const int i = 16 * mt + g + ((e & 2) ? 8 : 0), j = 8 * cb + 2 * t + (e & 1);
                if (!PAD || (i < n && j < m))
                    store_out(base, off + j * (PAD ? n : 8 * NB) + i, kt.v[mt][cb][e], bf16);
            }
}

// ---- when the five products with A, B and P run on pairs of halves (frag.cuh)
// In tf32 every element of an operand is represented to 2^-21 of itself, which leaves an error of 2^-20 |X||Y'| in a product
// (|.| element by element).  The pairs run where they leave no more.  A', B' and P are multiplied by powers of two that bring
// the largest |A_ij|, the largest |B_ij| and the largest P_ii into [2^14, 2^15); the conditions, on the values so scaled, are
//     every |A'_ij| and |B'_ij| is at least 2^-15                                         (represented to 2^-21 of itself)
//     every row sum of |A'| is at least 2^-5 of the power of two above the largest one, and so of |B'|
//     every |P_ij| is at least 2^-9 and none above 65504; if no element is more than half of its row sum in |A'| and |B'|,
//     two of P (P_ij and P_ji) may be smaller
// B'P and A'P are divided by those powers of two, so that they cannot overflow.  Their elements are represented to 2^-22 of
// themselves or 2^-36, and (|A'||P|)_ij is at least 2^-9 2^-5 / 2 = 2^-15 after that division: 2^-21 of it.  (The allowance for
// two is for dense matrices, where an element that small is an accident, once in 2000 steps at n = 40, and where a step in
// tf32 costs a launch of one wave 18 %: 1155 instances 201 or 238 us by chance, without it.)  Z'Z stays in tf32, whose split of Z'
// the factorisation makes anyway; on halves, with a test of Z', it took 6.87 instead of 6.91 ms at n = 32 and 212 instead of 201 us
// at 40 x 12.  A step in which P fails runs in tf32, an instance whose operands fail (zeros, rows of other units) throughout.
constexpr float OPERAND_LOW = 0x1p-15f, ROW_LOW = 0x1p-5f, VALUE_LOW = 0x1p-9f;
__device__ __forceinline__ float power_of_two(int e) { return __int_as_float((127 + e) << 23); }
__device__ __forceinline__ int exponent(unsigned bits) { return (int)(bits >> 23) - 127; }
// what a split of A' or B' (rows x cols exist) is scaled by, 2^scale, and its products with P, 2^shift
struct Scaling {
    int scale, shift;
    bool fits, spread;                                      // (spread: no element is more than half of its row)
};
template <int RB, int CB, bool PAD>
__device__ __forceinline__ Scaling operand_scaling(const Mat<RB, CB>& x, int rows, int cols, int lane)
{
    const int g = lane >> 2, t = lane & 3;
    const float inf = __int_as_float(0x7f800000);
    float top = 0.f, least = inf, low = inf, high = 0.f;
    bool spread = true;
#pragma unroll
    for (int b = 0; b < RB; ++b) {
        const bool row = !PAD || 8 * b + g < rows;
        float sum = 0.f, most = 0.f;
#pragma unroll
        for (int cb = 0; cb < CB; ++cb)
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const float v = fabsf(x.v[b / 2][cb][2 * (b & 1) + k]);
                sum += v;
                most = fmaxf(most, v);
                least = fminf(least, row && (!PAD || 8 * cb + 2 * t + k < cols) ? v : inf);
            }
        sum = sum_over_t(sum);
        most = fmaxf(most, __shfl_xor_sync(FULL, most, 1));
        most = fmaxf(most, __shfl_xor_sync(FULL, most, 2));
        top = fmaxf(top, most);
        high = fmaxf(high, sum);
        low = fminf(low, row ? sum : inf);
        spread = spread && 2.f * most <= sum;
    }
    const int et = exponent(__reduce_max_sync(FULL, __float_as_uint(top)));
    const int eh = exponent(__reduce_max_sync(FULL, __float_as_uint(high))) + 1;          // 2^eh is above every row sum
    Scaling r;
    r.scale = 14 - et;
    r.shift = -(eh + r.scale);
    r.spread = __all_sync(FULL, spread);
    r.fits = et >= -20 && eh <= 34;                         // (keeps every power of two below a normal number)
    if (r.fits)
        r.fits = __all_sync(FULL, least >= OPERAND_LOW * power_of_two(-r.scale) && low >= ROW_LOW * power_of_two(eh));
    return r;
}
// the scale of P: false when there is none
template <int NB>
__device__ __forceinline__ bool value_scaling(int& scale, const Mat<NB, NB>& nP, int lane)
{
    const int g = lane >> 2, t = lane & 3;
    float top = 0.f;
#pragma unroll
    for (int b = 0; b < NB; ++b)
        top = fmaxf(top, -((g & 1) ? nP.v[b / 2][b][2 * (b & 1) + 1] : nP.v[b / 2][b][2 * (b & 1)]));
    scale = 14 - exponent(__reduce_max_sync(FULL, t == (g >> 1) ? __float_as_uint(top) : 0u));
    return scale >= -26 && scale <= 54;
}
// W consecutive elements of a row (16-byte loads), or with PAD element by element within [0, n)
template <int W, bool PAD>
__device__ __forceinline__ void load_part(float (&v)[W], const float* row, int c0, int n)
{
    if (PAD) {
#pragma unroll
        for (int k = 0; k < W; ++k)
            v[k] = c0 + k < n ? row[c0 + k] : 0.f;
    } else {
#pragma unroll
        for (int q = 0; q < W / 4; ++q) {
            const float4 f = *reinterpret_cast<const float4*>(row + c0 + 4 * q);
            v[4 * q] = f.x; v[4 * q + 1] = f.y; v[4 * q + 2] = f.z; v[4 * q + 3] = f.w;
        }
    }
}

// ---- gradients of a loss of u_0 (Thm 3.2), after the backward pass of the same instance --------------------------------
// Both rollouts share every load of K_t, A_t, B_t, both co-state recursions every load of A_t, Q_t; the outer products
//     dA_t = lam_{t+1} xd_t' + lamd_{t+1} x_t'      dB_t = lam_{t+1} ud_t' + lamd_{t+1} u_t'
//     dQ_t = 1/2 (x_t xd_t' + xd_t x_t')            dR_t = 1/2 (u_t ud_t' + ud_t u_t')          lam_t = A_t'lam_{t+1} + Q_t x_t
// leave the registers as soon as the co-states of their step are known.  Row i of a matrix belongs to LPR lanes.  The
// gains and sequences that this warp wrote a moment ago come back from the second-level cache.
// What a step reads comes through a ring of asynchronous copies several steps ahead: by the time the gains are read again
// the stores of the other warps may have pushed them out to HBM.  Matrices keep rows of N floats with the 16-byte chunks
// of a row exchanged (chunk q of row r at q ^ swizzle(r)), which makes row and column reads conflict-free.
template <int N>
struct GradRing {
    static constexpr int FWD = 3 * N * N, BWD = 2 * N * N + 4 * N;         // floats per stage: K, A, B / A, Q, four vectors
    static constexpr int FS = N == 16 ? 3 : 2, BS = N == 16 ? 4 : 2;       // stages (no more than the backward pass needs anyway)
    static constexpr int VEC = 8 * N;                                      // vectors in front of the stages
    static constexpr size_t BYTES = sizeof(float) * (VEC + (FS * FWD > BS * BWD ? FS * FWD : BS * BWD));
    static __device__ __forceinline__ int swizzle(int r) { return N == 16 ? (r >> 1) & 3 : r & 7; }
    static __device__ __forceinline__ void copy(float* dst, const float* src, int lane)
    {
#pragma unroll
        for (int e = lane; e < N * N / 4; e += 32) {
            const int r = e / (N / 4), q = e % (N / 4);
            copy16(dst + r * N + 4 * (q ^ swizzle(r)), src + 4 * e);
        }
    }
    // W consecutive elements of row r from column c0
    template <int W>
    static __device__ __forceinline__ void row(float (&v)[W], const float* M, int r, int c0)
    {
#pragma unroll
        for (int q = 0; q < W / 4; ++q) {
            const float4 f = *reinterpret_cast<const float4*>(M + r * N + 4 * ((c0 / 4 + q) ^ swizzle(r)));
            v[4 * q] = f.x; v[4 * q + 1] = f.y; v[4 * q + 2] = f.z; v[4 * q + 3] = f.w;
        }
    }
    static __device__ __forceinline__ float at(const float* M, int r, int c) { return M[r * N + 4 * ((c >> 2) ^ swizzle(r)) + (c & 3)]; }
};
__device__ __forceinline__ void commit_copies() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int K>
__device__ __forceinline__ void wait_copies()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(K) : "memory");
    __syncwarp();
}
template <int W>
__device__ __forceinline__ void load_stream(float (&v)[W], const float* src)
{
#pragma unroll
    for (int q = 0; q < W / 4; ++q) {
        const float4 f = __ldg(reinterpret_cast<const float4*>(src) + q);
        v[4 * q] = f.x; v[4 * q + 1] = f.y; v[4 * q + 2] = f.z; v[4 * q + 3] = f.w;
    }
}
// row segment a v' + b w' (scaled by half, products rounded before they are added, when symmetric)
template <int W, bool SYM>
__device__ __forceinline__ void store_outer(float* dst, float a, const float (&v)[W], float b, const float (&w)[W])
{
#pragma unroll
    for (int q = 0; q < W / 4; ++q) {
        float r[4];
#pragma unroll
        for (int e = 0; e < 4; ++e)
            r[e] = SYM ? 0.5f * __fadd_rn(__fmul_rn(a, v[4 * q + e]), __fmul_rn(b, w[4 * q + e]))
                       : fmaf(a, v[4 * q + e], b * w[4 * q + e]);
        __stcs(reinterpret_cast<float4*>(dst) + q, make_float4(r[0], r[1], r[2], r[3]));
    }
}
template <int NB>
__device__ __forceinline__ void grad_tail(const SolveParams& p, const Place& pl, const float (&xr)[NB], const float (&k0)[NB][2],
                                          float* sm, int lane)
{
    constexpr int N = 8 * NB, LPR = N <= 16 ? 2 : 1, W = N / LPR;
    const int H = p.H, i = lane / LPR, c0 = (lane % LPR) * W, g = lane >> 2, t = lane & 3;
    const bool writer = lane % LPR == 0;
    const long long inst = pl.inst;
    const float* Ag = reinterpret_cast<const float*>(p.A.ptr) + pl.off(p.A);
    const float* Bg = reinterpret_cast<const float*>(p.B.ptr) + pl.off(p.B);
    const float* Qg = reinterpret_cast<const float*>(p.Q.ptr) + pl.off(p.Q);
    const float* Qfg = p.Qf.ptr ? reinterpret_cast<const float*>(p.Qf.ptr) + pl.off(p.Qf) : Qg;
    const float* Kg = p.K + inst * (long long)H * N * N;
    float* X = p.seq + inst * (long long)(4 * (H + 1)) * N;
    float* Xd = X + (long long)(H + 1) * N;
    float* U = Xd + (long long)(H + 1) * N;
    float* Ud = U + (long long)(H + 1) * N;
    using Ring = GradRing<N>;
    constexpr int FS = Ring::FS, BS = Ring::BS;
    float *sx = sm, *sxd = sm + N, *su = sm + 2 * N, *sud = sm + 3 * N, *sk = sm + 4 * N, *ring = sm + Ring::VEC;
    __syncwarp();                                           // K_t stored by the other lanes are visible; the operands are done
    auto stage_fwd = [&](int ts) {
        if (ts < H) {
            float* d = ring + (ts % FS) * Ring::FWD;
            Ring::copy(d, Kg + (long long)ts * N * N, lane);
            Ring::copy(d + N * N, Ag + ts * p.A.st, lane);
            Ring::copy(d + 2 * N * N, Bg + ts * p.B.st, lane);
        }
        commit_copies();
    };
#pragma unroll
    for (int k = 0; k < FS - 1; ++k)
        stage_fwd(k);
    if (g == 0)
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            sk[8 * b + 2 * t] = k0[b][0];
            sk[8 * b + 2 * t + 1] = k0[b][1];
        }
    if (t == 0)
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            sx[8 * b + g] = xr[b];
            sxd[8 * b + g] = 0.f;
        }
    __syncwarp();
    auto sum = [](float v) { return LPR == 2 ? v + __shfl_xor_sync(FULL, v, 1) : v; };
    if (writer) {
        X[i] = sx[i];
        Xd[i] = 0.f;
    }
#pragma unroll 1
    for (int ts = 0; ts < H; ++ts) {
        wait_copies<FS - 2>();
        stage_fwd(ts + FS - 1);
        const float* st = ring + (ts % FS) * Ring::FWD;
        float v[W], vd[W], r[W];
        load_part<W, false>(v, sx, c0, N);
        load_part<W, false>(vd, sxd, c0, N);
        float us = 0.f, uds = 0.f, xs = 0.f, xds = 0.f;
        Ring::template row<W>(r, st, i, c0);
#pragma unroll
        for (int k = 0; k < W; ++k) {
            us = fmaf(r[k], v[k], us);
            uds = fmaf(r[k], vd[k], uds);
        }
        Ring::template row<W>(r, st + N * N, i, c0);
#pragma unroll
        for (int k = 0; k < W; ++k) {
            xs = fmaf(r[k], v[k], xs);
            xds = fmaf(r[k], vd[k], xds);
        }
        us = sum(us);
        uds = sum(uds) + (ts == 0 ? sk[i] : 0.f);
        if (writer) {
            su[i] = us;
            sud[i] = uds;
            U[(long long)ts * N + i] = us;
            Ud[(long long)ts * N + i] = uds;
            if (ts == 0 && p.u0)
                p.u0[inst * N + i] = us;
        }
        __syncwarp();
        load_part<W, false>(v, su, c0, N);
        load_part<W, false>(vd, sud, c0, N);
        Ring::template row<W>(r, st + 2 * N * N, i, c0);
#pragma unroll
        for (int k = 0; k < W; ++k) {
            xs = fmaf(r[k], v[k], xs);
            xds = fmaf(r[k], vd[k], xds);
        }
        xs = sum(xs);
        xds = sum(xds);
        if (writer) {
            sx[i] = xs;
            sxd[i] = xds;
            X[(long long)(ts + 1) * N + i] = xs;
            Xd[(long long)(ts + 1) * N + i] = xds;
        }
        __syncwarp();
    }
    auto stage_bwd = [&](int k) {                           // k-th step backwards
        const int ts = H - 1 - k;
        if (ts >= 0) {
            float* d = ring + (k % BS) * Ring::BWD;
            Ring::copy(d, Ag + ts * p.A.st, lane);
            Ring::copy(d + N * N, Qg + ts * p.Q.st, lane);
            if (lane < N)                                   // x_t, xd_t, u_t, ud_t
                copy16(d + 2 * N * N + 4 * lane, X + (long long)(lane / (N / 4)) * (H + 1) * N + (long long)ts * N + 4 * (lane % (N / 4)));
        }
        commit_copies();
    };
    wait_copies<0>();
#pragma unroll
    for (int k = 0; k < BS - 1; ++k)
        stage_bwd(k);
    // co-states of t = H, outer product of the terminal weight
    float lam = 0.f, lamd = 0.f;
    float *sl = su, *sld = sud;
    {
        float v[W], vd[W], q[W];
        load_part<W, false>(v, sx, c0, N);
        load_part<W, false>(vd, sxd, c0, N);
        load_stream<W>(q, Qfg + i * N + c0);
#pragma unroll
        for (int k = 0; k < W; ++k) {
            lam = fmaf(q[k], v[k], lam);
            lamd = fmaf(q[k], vd[k], lamd);
        }
        if (p.dQf)
            store_outer<W, true>(p.dQf + (inst * N + i) * N + c0, sx[i], vd, sxd[i], v);
    }
#pragma unroll 1
    for (int ts = H - 1; ts >= 0; --ts) {
        const int k0s = H - 1 - ts;
        wait_copies<BS - 2>();
        stage_bwd(k0s + BS - 1);
        const float* st = ring + (k0s % BS) * Ring::BWD;
        const float* vec = st + 2 * N * N;
        lam = sum(lam);
        lamd = sum(lamd);
        if (writer) {
            sl[i] = lam;
            sld[i] = lamd;
        }
        const long long o = (inst * (long long)H + ts) * N * N + i * N + c0;
        float v[W], vd[W];
        load_part<W, false>(v, vec + 2 * N, c0, N);
        load_part<W, false>(vd, vec + 3 * N, c0, N);
        if (p.dB)
            store_outer<W, false>(p.dB + o, lam, vd, lamd, v);
        if (p.dR)
            store_outer<W, true>(p.dR + o, vec[2 * N + i], vd, vec[3 * N + i], v);
        load_part<W, false>(v, vec, c0, N);
        load_part<W, false>(vd, vec + N, c0, N);
        if (p.dA)
            store_outer<W, false>(p.dA + o, lam, vd, lamd, v);
        if (p.dQ)
            store_outer<W, true>(p.dQ + o, vec[i], vd, vec[N + i], v);
        lam = lamd = 0.f;
        float r[W];
        Ring::template row<W>(r, st + N * N, i, c0);
#pragma unroll
        for (int k = 0; k < W; ++k) {
            lam = fmaf(r[k], v[k], lam);
            lamd = fmaf(r[k], vd[k], lamd);
        }
        __syncwarp();
        load_part<W, false>(v, sl, c0, N);
        load_part<W, false>(vd, sld, c0, N);
#pragma unroll
        for (int k = 0; k < W; ++k) {
            const float a = Ring::at(st, c0 + k, i);        // column i of A_t
            lam = fmaf(a, v[k], lam);
            lamd = fmaf(a, vd[k], lamd);
        }
    }
    wait_copies<0>();
    lamd = sum(lamd);
    if (writer && p.dx0)
        p.dx0[inst * N + i] = lamd;
}

template <int NB, int MB, bool TV, bool GRAD>
__host__ __device__ constexpr size_t warp_bytes()
{
    constexpr size_t a = sizeof(WarpMem<NB, MB, TV && NB <= 2>), b = GRAD ? GradRing<8 * NB>::BYTES : 0;
    return ((a > b ? a : b) + 15) & ~size_t(15);
}

// NB, MB: number of 8-blocks of the state and the control dimension.
// TV = time-varying request (time strides or a terminal weight); AFF = linear control cost r_t'u_t (implies TV);
// PAD = n < 8 NB or m < 8 MB, or strides that do not keep the vector loads aligned: guarded element-wise accesses, the
// missing part of R is the identity and everything else zero, which leaves the recursion of the existing part untouched.
// CH = one piece of the horizon of an instance (see SolveParams; time-invariant): it starts from the value matrix and the
// state at the piece's ends, writes its part of the outputs and leaves failures to the caller.
// GRAD = the gradients of the first control in the same kernel (n = m = 8 NB, float32 operands): see grad_tail().
// FEW = at most four warps per SM: the factorisation with the shorter chain (chol8_inverse).
// CTAs per SM at n <= 16: as many as shared memory (time-varying) or registers hold.  Time-invariant six of them: 32768 instances,
// n = 16, H = 16, all outputs 0.756 ms with four, 0.737 with five, 0.716 with six, 4096 instances 106.6, 106.4, 106.2 us.  Launches
// that cannot fill that many (FEW, the pieces of a scan) keep four.
template <int NB, int MB, bool TV, bool AFF, bool PAD, bool CH = false, bool GRAD = false, bool FEW = false>
__global__ void __launch_bounds__(32 * MAX_WARPS, NB > 2 ? 2 : AFF && !GRAD ? 4 : TV ? 5 : CH || FEW ? 4 : 6) riccati_frag_kernel(SolveParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int warp = warp_index();
    const long long widx = (long long)blockIdx.x * (blockDim.x >> 5) + warp;
    if (widx >= p.b0 * p.b1 * p.tcount * (CH ? p.chunks : 1))
        return;
    const int chunk = CH ? (int)(widx % p.chunks) : 0;
    const Place pl = place(p, (unsigned)(CH ? widx / p.chunks : widx));
    const long long inst = pl.inst;
    const int n = PAD ? p.n : 8 * NB, m = PAD ? p.m : 8 * MB, obf = p.out_bf16;
    const int Ht = p.H, tb = CH ? chunk * p.chunk_len : 0, H = CH ? min(p.chunk_len, Ht - tb) : Ht;      // steps tb .. tb + H - 1 of Ht
    const bool last_piece = tb + H == Ht, first_ok = chunk == 0 || !p.first_only;
    const bool need_K_all = p.K != nullptr || p.x != nullptr || (p.u != nullptr && !p.first_only);
    const bool want_u0 = p.u != nullptr && p.first_only && !need_K_all;
    const bool need_k_all = AFF && p.kff != nullptr;
    float* const Kbase = (p.K && !obf) ? p.K : p.Kws;       // float32 gains (the rollout reads them)
    const long long Koff = (inst * (long long)Ht + tb) * m * n;
    const long long Poff = (inst * (long long)(p.first_only ? 1 : Ht + 1) + (p.first_only ? 0 : tb)) * n * n;
    using Ops = Operands<NB, MB>;
    constexpr bool TWO = TV && NB <= 2;
    using Mem = WarpMem<NB, MB, TWO>;
    Mem& mem = *reinterpret_cast<Mem*>(smem_raw + warp * warp_bytes<NB, MB, TV, GRAD>());
    const long long oA = pl.off(p.A), oB = pl.off(p.B), oR = pl.off(p.R), oQ = pl.off(p.Q);
    Mat<NB, NB> nP;
    if constexpr (PAD) {                                    // what does not exist: R is the identity, the rest zero
        for (int e = lane; e < (int)(sizeof(Mem) / sizeof(float)); e += 32)
            reinterpret_cast<float*>(&mem)[e] = 0.f;
        __syncwarp();
        for (int i = m + lane; i < 8 * MB; i += 32) {
            if constexpr (TWO)
                mem.op[0].R[i * Ops::LR + i] = mem.op[1].R[i * Ops::LR + i] = 1.f;
            else
                mem.R[i * Ops::LR + i] = 1.f;
        }
    }
    {
        const long long last = TV ? H - 1 : 0;
        if constexpr (TWO) {
            if (p.Qf.ptr) {                                 // P_H = Q_f, by way of the second buffer
                stage<NB, NB, Ops::LQ, PAD>(mem.op[1].Q, p.Qf, pl.off(p.Qf), n, n, lane);
                copies_landed();
                load_negated<NB, Ops::LQ>(nP, mem.op[1].Q, lane);
                __syncwarp();
            }
#pragma unroll
            for (int b = 0; b < 2; ++b) {                   // the second buffer: what does not change with time
                if (b == 0 || !p.A.st) stage<NB, NB, Ops::LA, PAD>(mem.op[b].A, p.A, oA + last * p.A.st, n, n, lane);
                if (b == 0 || !p.B.st) stage<NB, MB, Ops::LB, PAD>(mem.op[b].B, p.B, oB + last * p.B.st, n, m, lane);
                if (b == 0 || !p.R.st) stage<MB, MB, Ops::LR, PAD>(mem.op[b].R, p.R, oR + last * p.R.st, m, m, lane);
                if (b == 0 || !p.Q.st) stage<NB, NB, Ops::LQ, PAD>(mem.op[b].Q, p.Q, oQ + last * p.Q.st, n, n, lane);
            }
            copies_landed();
            if (!p.Qf.ptr)
                load_negated<NB, Ops::LQ>(nP, mem.op[0].Q, lane);
        } else {
            OperandDev end = TV && p.Qf.ptr ? p.Qf : p.Q;   // P_H
            long long oend = TV && p.Qf.ptr ? pl.off(p.Qf) : oQ + last * p.Q.st;
            const bool inner = CH && chunk < p.coarse;
            if (inner) {
                end.ptr = p.Pc;
                end.dtype = TTC_F32;
                oend = (inst * (p.coarse + 1) + chunk + 1) * (long long)n * n;
            }
            stage<NB, NB, Ops::LQ, PAD>(mem.Q, end, oend, n, n, lane);
            stage<NB, NB, Ops::LA, PAD>(mem.rawA(), p.A, oA + last * p.A.st, n, n, lane);
            stage<NB, MB, Ops::LB, PAD>(mem.rawB(), p.B, oB + last * p.B.st, n, m, lane);
            stage<MB, MB, Ops::LR, PAD>(mem.R, p.R, oR + last * p.R.st, m, m, lane);
            copies_landed();
            load_negated<NB, Ops::LQ>(nP, mem.Q, lane);
            if ((TV && p.Qf.ptr) || inner) {
                __syncwarp();
                stage<NB, NB, Ops::LQ, PAD>(mem.Q, p.Q, oQ + last * p.Q.st, n, n, lane);
            }
        }
    }
    if (p.P && !p.first_only && last_piece)
        store_negated<NB, PAD>(p.P, Poff + (long long)H * n * n, nP, n, obf, lane);

    auto start_state = [&](int i) {
        if (CH && p.xc)
            return p.xc[(inst * (p.coarse + 1) + chunk) * (long long)n + i];
        return p.x0.ptr ? load_elem(p.x0, pl.off(p.x0) + i) : 0.f;
    };
    float xr[NB];                                           // x_0 in row form
#pragma unroll
    for (int b = 0; b < NB; ++b)
        xr[b] = 8 * b + g < n ? start_state(8 * b + g) : 0.f;

    float pr[NB];                                           // affine term: p_{t+1} in row form
    float kc0[MB][2];                                       // k_t in column form
    if (AFF) {
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            pr[b] = 0.f;
            if (p.pvec && !p.first_only && t == 0 && 8 * b + g < n)
                p.pvec[(inst * (H + 1) + H) * (long long)n + 8 * b + g] = 0.f;
        }
    }

    int fail = 0;
    float gr[MB], ap[NB];                                   // affine: B'p + r and A'p in row form
    auto affine_part = [&](const Mat<NB, NB>& At, const Mat<MB, NB>& Bt, const int ts) {
        float pc[NB][2];
#pragma unroll
        for (int b = 0; b < NB; ++b)
            row_to_col(pc[b][0], pc[b][1], pr[b], lane);
        const long long orv = pl.off(p.r) + ts * p.r.st;
#pragma unroll
        for (int b = 0; b < MB; ++b) {
            float s = 0.f;
#pragma unroll
            for (int k = 0; k < NB; ++k)
                s = fmaf(Bt.v[b / 2][k][2 * (b & 1)], pc[k][0], fmaf(Bt.v[b / 2][k][2 * (b & 1) + 1], pc[k][1], s));
            gr[b] = sum_over_t(s) + (8 * b + g < m ? load_elem(p.r, orv + 8 * b + g) : 0.f);
        }
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            float s = 0.f;
#pragma unroll
            for (int k = 0; k < NB; ++k)
                s = fmaf(At.v[b / 2][k][2 * (b & 1)], pc[k][0], fmaf(At.v[b / 2][k][2 * (b & 1) + 1], pc[k][1], s));
            ap[b] = sum_over_t(s);
        }
    };
    // Form in which the operands lie in the warp's memory.  They are split in place, so that a change between the two split
    // forms stages the raw ones again.  After a failed attempt to run on halves, or the end of one, `rest` steps in tf32 pass
    // before the next: none the first time (a diagonal terminal weight), then one, three, seven ...
    // HALF: up to 16 the scaling and the tests take back most of what the products gain (4096 instances, H = 16: 100 us in the range
    // and 110 out of it, against 106 in tf32); above, see the head of this file.
    constexpr bool HALF = NB > 2;
    enum { RAW, TF32, HALVES };
    int formA = RAW, formB = RAW, scaleP = 0, rest = 0, pause = 0;
    Scaling sA = {}, sB = {};
    bool okP = HALF && value_scaling<NB>(scaleP, nP, lane);
    auto failed = [&]() {
        rest = pause;
        pause = pause < 1 << 20 ? 2 * pause + 1 : pause;
    };
    auto raw_instead_of = [&](int form, int ts) {           // what lies there in that form: the raw operand once more
        if constexpr (HALF) {
            if (formA != form && formB != form)
                return;
            const long long now = TV ? ts : 0;
            __syncwarp();
            if (formA == form) stage<NB, NB, Ops::LA, PAD>(mem.rawA(), p.A, oA + now * p.A.st, n, n, lane);
            if (formB == form) stage<NB, MB, Ops::LB, PAD>(mem.rawB(), p.B, oB + now * p.B.st, n, m, lane);
            copies_landed();
            formA = formA == form ? RAW : formA;
            formB = formB == form ? RAW : formB;
        }
    };
    auto begin_step = [&](const int ts) {
        if constexpr (!TWO) {
            if (TV || ts == H - 1)                          // (what CH stages for P_H is followed by Q)
                copies_landed();
            if (TV && p.A.st)
                formA = RAW;
            if (TV && p.B.st)
                formB = RAW;
            if (AFF && ts < p.r_count) {                    // from the float32 operands, before they are split in place
                Mat<NB, NB> At;
                Mat<MB, NB> Bt;
                if (formA == RAW)
                    load_transposed<NB, NB, Ops::LA, PAD>(At, mem.rawA(), n, n, lane);
                else
                    load_transposed_global<NB, NB>(At, p.A, oA, n, n, n, lane);
                if (formB == RAW)
                    load_transposed<MB, NB, Ops::LB, PAD>(Bt, mem.rawB(), n, m, lane);
                else
                    load_transposed_global<MB, NB>(Bt, p.B, oB, m, n, m, lane);
                affine_part(At, Bt, ts);
            }
        }
    };
    auto stage_next = [&](const int ts) {                   // operands of the next step, in flight while this one is factored
        if constexpr (TV && !TWO) {
            if (ts == 0)
                return;
            __syncwarp();
            if (p.A.st) stage<NB, NB, Ops::LA, PAD>(mem.rawA(), p.A, oA + (ts - 1) * p.A.st, n, n, lane);
            if (p.B.st) stage<NB, MB, Ops::LB, PAD>(mem.rawB(), p.B, oB + (ts - 1) * p.B.st, n, m, lane);
            if (p.R.st) stage<MB, MB, Ops::LR, PAD>(mem.R, p.R, oR + (ts - 1) * p.R.st, m, m, lane);
            if (p.Q.st) stage<NB, NB, Ops::LQ, PAD>(mem.Q, p.Q, oQ + (ts - 1) * p.Q.st, n, n, lane);
        }
    };
    // whether the raw operand permits halves, and the operand on halves, in place (time-varying: when it does)
    auto fits_A = [&](const Mat<NB, NB>& At) {
        sA = operand_scaling<NB, NB, PAD>(At, n, n, lane);
        return sA.fits;
    };
    auto fits_B = [&](const Mat<MB, NB>& Bt) {
        sB = operand_scaling<MB, NB, PAD>(Bt, m, n, lane);
        return sB.fits;
    };
    auto install_halves = [&]() -> bool {
        if constexpr (HALF) {
            if (formB == RAW) {
                Mat<MB, NB> Bt;
                load_transposed<MB, NB, Ops::LB, PAD>(Bt, mem.rawB(), n, m, lane);
                if (TV && !fits_B(Bt))
                    return false;
                Halves<MB, NB> bs;
                split(bs, Bt, power_of_two(sB.scale));
                __syncwarp();
                keep(mem.halvesB(), bs, lane);
                formB = HALVES;
            }
            if (formA == RAW) {
                Mat<NB, NB> At;
                load_transposed<NB, NB, Ops::LA, PAD>(At, mem.rawA(), n, n, lane);
                if (TV && !fits_A(At))
                    return false;
                Halves<NB, NB> as;
                split(as, At, power_of_two(sA.scale));
                __syncwarp();
                keep(mem.halvesA(), as, lane);
                formA = HALVES;
            }
            __syncwarp();
        }
        return true;
    };
    // the rest of a step, from S, Y' (Zt) and -Q - A'PA (nP)
    auto finish_step = [&](const int ts, Mat<MB, MB>& S, Mat<NB, MB>& Zt) {
        Split<NB, MB> zs;
        float w[MB][2];
        const int bad = factor<NB, MB, FEW || (NB > 2)>(S, Zt, zs, w, lane);  // Zt becomes Z', S the blocks of L
        if (bad && !fail)
            fail = ts * m + bad;
        product<NB, MB, NB, true>(nP, &nP, zs, zs);                              // -P_t = -Q - A'PA + Z'Z
        const bool gain = need_K_all || need_k_all || (want_u0 && ts == 0);
        if (AFF) {
            // z = L^{-1}(B'p + r);  p_t = A'p - Z'z;  k_t = -L^{-T} z   (all zero while p and r are)
            if (ts < p.r_count) {
                float zc[MB][2];
                solve_vector<MB>(zc, kc0, gr, S, w, lane);
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    float s = 0.f;
#pragma unroll
                    for (int k = 0; k < MB; ++k)
                        s = fmaf(Zt.v[b / 2][k][2 * (b & 1)], zc[k][0], fmaf(Zt.v[b / 2][k][2 * (b & 1) + 1], zc[k][1], s));
                    pr[b] = ap[b] - sum_over_t(s);
                }
            } else {
#pragma unroll
                for (int b = 0; b < MB; ++b)
                    kc0[b][0] = kc0[b][1] = 0.f;
            }
#pragma unroll
            for (int b = 0; b < MB; ++b)
#pragma unroll
                for (int e = 0; e < 2; ++e)
                    if (need_k_all && g == 0 && 8 * b + 2 * t + e < m)
                        p.kff[(inst * H + ts) * (long long)m + 8 * b + 2 * t + e] = kc0[b][e];
            if (p.pvec && (!p.first_only || ts == 0) && t == 0)
#pragma unroll
                for (int b = 0; b < NB; ++b)
                    if (8 * b + g < n)
                        p.pvec[(inst * (p.first_only ? 1 : H + 1) + (p.first_only ? 0 : ts)) * (long long)n + 8 * b + g] = pr[b];
        }
        if (gain) {
            gains<NB, MB>(Zt, S, w, lane);                  // Zt = K_t'
            if (need_K_all) {
                const long long off = Koff + (long long)ts * m * n;
                store_gain<NB, MB, PAD>(Kbase, off, Zt, n, m, 0, lane);
                if (obf && p.K)
                    store_gain<NB, MB, PAD>(p.K, off, Zt, n, m, 1, lane);
            } else if (want_u0 && ts == 0) {                // u_0 = K_0 x_0 + k_0 in column form
                const bool ok = fail == 0;
#pragma unroll
                for (int b = 0; b < MB; ++b)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        float s = 0.f;
#pragma unroll
                        for (int i = 0; i < NB; ++i)
                            s = fmaf(Zt.v[i / 2][b][2 * (i & 1) + e], xr[i], s);
                        s = sum_over_g(s);
                        if (AFF)
                            s += kc0[b][e];
                        if (ok && g == 0 && 8 * b + 2 * t + e < m)
                            store_out(p.u, inst * (long long)m + 8 * b + 2 * t + e, s, obf);
                    }
            }
        }
        // Q and Z'Z are symmetric, but the rounding of A'(PA) is not, and since the next step reads P through one
        // orientation only, the antisymmetric part E obeys E <- -A'E A: it grows along an open-loop unstable A however
        // well the closed loop is damped.
        if constexpr (HALF)
            okP = value_scaling<NB>(scaleP, nP, lane);      // (the diagonal stays)
        make_symmetric<NB>(nP, lane);
        if (p.P && first_ok && (!p.first_only || ts == 0))
            store_negated<NB, PAD>(p.P, Poff + (long long)(p.first_only ? 0 : ts) * n * n, nP, n, obf, lane);
    };
    int ts = H - 1;
#pragma unroll 1
    while (ts >= 0) {
        Mat<NB, MB> Zt;
        Mat<MB, MB> S;
        if constexpr (TWO) {
            const Ops& op = mem.op[(H - 1 - ts) & 1];
            if (ts < H - 1)
                copies_landed();                            // also: every lane is done with the other buffer
            if (ts > 0) {                                   // operands of the next step
                Ops& nx = mem.op[(H - ts) & 1];
                if (p.A.st) stage<NB, NB, Ops::LA, PAD>(nx.A, p.A, oA + (ts - 1) * p.A.st, n, n, lane);
                if (p.B.st) stage<NB, MB, Ops::LB, PAD>(nx.B, p.B, oB + (ts - 1) * p.B.st, n, m, lane);
                if (p.R.st) stage<MB, MB, Ops::LR, PAD>(nx.R, p.R, oR + (ts - 1) * p.R.st, m, m, lane);
                if (p.Q.st) stage<NB, NB, Ops::LQ, PAD>(nx.Q, p.Q, oQ + (ts - 1) * p.Q.st, n, n, lane);
            }
            Mat<NB, NB> At, T;
            Mat<MB, NB> Bt, V;
            Mat<MB, MB> nR;
            load_negated<MB, Ops::LR>(nR, op.R, lane);
            load_transposed<NB, NB, Ops::LA, false>(At, op.A, n, n, lane);
            load_transposed<MB, NB, Ops::LB, false>(Bt, op.B, n, m, lane);
            Split<NB, NB> as, ps;
            Split<MB, NB> bs, vs;
            split(ps, nP);
            split(as, At);
            split(bs, Bt);
            product<MB, NB, NB>(V, nullptr, bs, ps);        // V = B' nP
            product<NB, NB, NB>(T, nullptr, as, ps);        // T = A' nP
            split(vs, V);
            product<MB, NB, MB, true>(S, &nR, bs, vs);      // -S = -R + B' V'
            product<NB, NB, MB>(Zt, nullptr, as, vs);       // -Y' = A' V'
            split(ps, T);
            load_negated<NB, Ops::LQ>(nP, op.Q, lane);
            product<NB, NB, NB, true>(nP, &nP, as, ps);     // -Q - A'P A
            if (AFF && ts < p.r_count)
                affine_part(At, Bt, ts);
        } else {
            begin_step(ts);
            if constexpr (HALF && !TV)
                if (ts == H - 1) {                          // operands that do not change are looked at once
                    Mat<MB, NB> Bt;
                    load_transposed<MB, NB, Ops::LB, PAD>(Bt, mem.rawB(), n, m, lane);
                    bool fits = fits_B(Bt);
                    if (fits) {
                        Mat<NB, NB> At;
                        load_transposed<NB, NB, Ops::LA, PAD>(At, mem.rawA(), n, n, lane);
                        fits = fits_A(At);
                    }
                    rest = fits ? 0 : 1 << 30;
                }
            if constexpr (HALF) {
                if (rest > 0) {
                    --rest;
                } else {
                    bool installed = false;                 // operands that do not change, on halves
#pragma unroll 1
                    while (true) {
                        {
                            Halves<NB, NB> ps;
                            split(ps, nP, power_of_two(okP ? scaleP : 0));
                            if (!in_range(ps, VALUE_LOW, n * n - (!TV && sA.spread && sB.spread ? 2 : 0)) || !okP) {
                                failed();
                                break;
                            }
                            if (!installed) {
                                raw_instead_of(TF32, ts);
                                if (!install_halves()) {
                                    failed();
                                    break;
                                }
                                installed = !TV;
                            }
                            Mat<MB, NB> V;
                            Mat<NB, NB> T;
                            Halves<MB, NB> vs;
                            Halves<NB, NB> tsp;
                            product_halves<MB, NB, NB>(V, mem.halvesB(), ps, lane);
                            product_halves<NB, NB, NB>(T, mem.halvesA(), ps, lane);
                            split(vs, V, power_of_two(sB.shift));
                            split(tsp, T, power_of_two(sA.shift));
                            product_halves<MB, NB, MB, true>(S, mem.halvesB(), vs, lane);
                            scale_and_subtract<MB, Ops::LR, true>(S, power_of_two(-(2 * sB.scale + sB.shift + scaleP)), mem.R, lane);
                            product_halves<NB, NB, MB>(Zt, mem.halvesA(), vs, lane);
                            const float c = power_of_two(-(sA.scale + sB.scale + sB.shift + scaleP));
#pragma unroll
                            for (int mt = 0; mt < Mat<NB, MB>::MT; ++mt)
#pragma unroll
                                for (int cb = 0; cb < MB; ++cb)
#pragma unroll
                                    for (int e = 0; e < 4; e += 2)
                                        scale_pair(Zt.v[mt][cb][e], Zt.v[mt][cb][e + 1], c);
                            product_halves<NB, NB, NB, true>(nP, mem.halvesA(), tsp, lane);
                            scale_and_subtract<NB, Ops::LQ, true>(nP, power_of_two(-(2 * sA.scale + sA.shift + scaleP)), mem.Q, lane);
                        }
                        stage_next(ts);
                        finish_step(ts, S, Zt);
                        if (--ts < 0)
                            break;
                        begin_step(ts);
                    }
                    if (ts < 0)
                        break;
                }
            }
            if constexpr (HALF)
                raw_instead_of(HALVES, ts);
            if (formA == RAW) {                             // raw -> split, in place
                Mat<NB, NB> At;
                load_transposed<NB, NB, Ops::LA, PAD>(At, mem.rawA(), n, n, lane);
                __syncwarp();
                keep(mem.A, At, lane);
            }
            if (formB == RAW) {
                Mat<MB, NB> Bt;
                load_transposed<MB, NB, Ops::LB, PAD>(Bt, mem.rawB(), n, m, lane);
                __syncwarp();
                keep(mem.B, Bt, lane);
            }
            formA = formB = TF32;
            __syncwarp();
            Mat<MB, NB> V;
            Mat<NB, NB> T;
            Mat<MB, MB> nR;
            load_negated<MB, Ops::LR>(nR, mem.R, lane);
            {
                Split<NB, NB> ps;
                split(ps, nP);
                product<MB, NB, NB>(V, nullptr, mem.B, ps, lane);
                product<NB, NB, NB>(T, nullptr, mem.A, ps, lane);
            }
            {
                Split<MB, NB> vs;
                split(vs, V);
                product<MB, NB, MB, true>(S, &nR, mem.B, vs, lane);
                product<NB, NB, MB>(Zt, nullptr, mem.A, vs, lane);
            }
            load_negated<NB, Ops::LQ>(nP, mem.Q, lane);
            {
                Split<NB, NB> tsp;
                split(tsp, T);
                product<NB, NB, NB, true>(nP, &nP, mem.A, tsp, lane);
            }
            stage_next(ts);
        }
        finish_step(ts, S, Zt);
        --ts;
    }
    if (CH) {
        if (lane == 0)
            p.piece_info[widx] = fail;
    } else if (p.info && lane == 0) {
        p.info[inst] = fail;
    }
    if (CH && fail)
        return;
    if (fail) {                                             // uniform over the warp
        const float qn = quiet_nan();
        __syncwarp();
        if (p.K && !GRAD)
            for (long long e = lane; e < (long long)H * m * n; e += 32)
                store_out(p.K, Koff + e, qn, obf);
        if (p.P) {
            const long long cnt = (long long)(p.first_only ? 1 : H + 1) * n * n;
            for (long long e = lane; e < cnt; e += 32)
                store_out(p.P, Poff + e, qn, obf);
        }
        if (p.x)
            for (long long e = lane; e < (long long)(H + 1) * n; e += 32)
                store_out(p.x, inst * (long long)(H + 1) * n + e, qn, obf);
        if (p.u) {
            const long long cnt = p.first_only ? m : (long long)H * m;
            for (long long e = lane; e < cnt; e += 32)
                store_out(p.u, inst * cnt + e, qn, obf);
        }
        if (AFF && p.pvec) {
            const long long cnt = (long long)(p.first_only ? 1 : H + 1) * n;
            for (long long e = lane; e < cnt; e += 32)
                p.pvec[inst * cnt + e] = qn;
        }
        if (GRAD) {
            auto fill = [&](float* base, long long cnt) {
                if (base)
                    for (long long e = lane; e < cnt; e += 32)
                        base[inst * cnt + e] = qn;
            };
            fill(p.dA, (long long)H * n * n);
            fill(p.dB, (long long)H * n * m);
            fill(p.dQ, (long long)H * n * n);
            fill(p.dQf, (long long)n * n);
            fill(p.dR, (long long)H * m * m);
            fill(p.dx0, n);
            fill(p.u0, m);
        }
        if (need_k_all)
            for (long long e = lane; e < (long long)H * m; e += 32)
                p.kff[inst * (long long)H * m + e] = qn;
        return;
    }
    if constexpr (GRAD) {
        grad_tail<NB>(p, pl, xr, kc0, reinterpret_cast<float*>(&mem), lane);
        return;
    }
    if (want_u0 || !(p.x || p.u))
        return;

    // ---- forward loop of Alg. 1: LPR lanes per row and RPL rows per lane, the vectors in the warp's memory (whose
    // operands are no longer needed); the rows of K_{t+1} (and of A_{t+1}, B_{t+1}) are in flight while step t is summed
    constexpr int D = 8 * (NB > MB ? NB : MB), LPR = D <= 16 ? 2 : 1, RPL = D <= 32 ? 1 : 2, WN = 8 * NB / LPR, WM = 8 * MB / LPR;
    static_assert(D <= 64, "rows");
    const float* Ag = reinterpret_cast<const float*>(p.A.ptr) + oA;
    const float* Bg = reinterpret_cast<const float*>(p.B.ptr) + oB;
    float* const sx = reinterpret_cast<float*>(&mem);
    float* const su = sx + 64;
    const int row0 = lane / LPR, c0n = (lane % LPR) * WN, c0m = (lane % LPR) * WM;
    const bool writer = lane % LPR == 0;
    float x0v[RPL];
#pragma unroll
    for (int q = 0; q < RPL; ++q) {
        const int i = row0 + 32 * q;
        x0v[q] = i < n ? start_state(i) : 0.f;
    }
    __syncwarp();                                           // also: K_t stored by the other lanes are visible
#pragma unroll
    for (int q = 0; q < RPL; ++q)
        if (writer) {
            sx[row0 + 32 * q] = x0v[q];
            su[row0 + 32 * q] = 0.f;
        }
    __syncwarp();
    const float* Kr = Kbase + Koff;
    float kr[RPL][WN], ar[RPL][WN], br[RPL][WM], kt[RPL];
    auto load_rows = [&](int ts, bool dynamics) {
#pragma unroll
        for (int q = 0; q < RPL; ++q) {
            const int i = row0 + 32 * q, ri = i < n ? i : 0, rj = i < m ? i : 0;
            load_part<WN, PAD>(kr[q], Kr + ((long long)ts * m + rj) * n, c0n, n);
            if (dynamics || (TV && p.A.st)) load_part<WN, PAD>(ar[q], Ag + ts * p.A.st + ri * n, c0n, n);
            if (dynamics || (TV && p.B.st)) load_part<WM, PAD>(br[q], Bg + ts * p.B.st + ri * m, c0m, m);
            if (AFF && p.kff)
                kt[q] = p.kff[(inst * H + ts) * (long long)m + rj];
        }
    };
    load_rows(0, true);
    if (AFF && !p.kff) {                                    // only u_0 is wanted: k_0 is still in registers
#pragma unroll
        for (int q = 0; q < RPL; ++q) {
            const int i = row0 + 32 * q;
            kt[q] = 0.f;
#pragma unroll
            for (int b = 0; b < MB; ++b) {
                const float e0 = __shfl_sync(FULL, kc0[b][0], (i & 7) >> 1), e1 = __shfl_sync(FULL, kc0[b][1], (i & 7) >> 1);
                if (i / 8 == b)
                    kt[q] = (i & 1) ? e1 : e0;
            }
        }
    }
    const int steps = (p.x || !p.first_only) ? H : 1;
    const long long xoff = (inst * (long long)(Ht + 1) + tb) * n, uoff = p.first_only ? inst * m : (inst * (long long)Ht + tb) * m;
#pragma unroll
    for (int q = 0; q < RPL; ++q)
        if (p.x && writer && row0 + 32 * q < n)
            store_out(p.x, xoff + row0 + 32 * q, x0v[q], obf);
#pragma unroll 1
    for (int ts = 0; ts < steps; ++ts) {
        float us[RPL], xs[RPL];
        {
            float xv[WN];
            load_part<WN, false>(xv, sx, c0n, 64);
#pragma unroll
            for (int q = 0; q < RPL; ++q) {
                us[q] = xs[q] = 0.f;
#pragma unroll
                for (int k = 0; k < WN; ++k) {
                    us[q] = fmaf(kr[q][k], xv[k], us[q]);
                    xs[q] = fmaf(ar[q][k], xv[k], xs[q]);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < RPL; ++q) {
            const int i = row0 + 32 * q;
            if (LPR == 2)
                us[q] += __shfl_xor_sync(FULL, us[q], 1);
            if (AFF)
                us[q] += kt[q];
            if (writer) {
                su[i] = i < m ? us[q] : 0.f;
                if (p.u && i < m && first_ok && (!p.first_only || ts == 0))
                    store_out(p.u, uoff + (p.first_only ? 0 : (long long)ts * m) + i, us[q], obf);
            }
        }
        __syncwarp();
        {
            float uv[WM];
            load_part<WM, false>(uv, su, c0m, 64);
#pragma unroll
            for (int q = 0; q < RPL; ++q)
#pragma unroll
                for (int k = 0; k < WM; ++k)
                    xs[q] = fmaf(br[q][k], uv[k], xs[q]);
        }
        if (ts + 1 < steps)
            load_rows(ts + 1, false);
#pragma unroll
        for (int q = 0; q < RPL; ++q) {
            const int i = row0 + 32 * q;
            if (LPR == 2)
                xs[q] += __shfl_xor_sync(FULL, xs[q], 1);
            if (writer) {
                sx[i] = i < n ? xs[q] : 0.f;
                if (p.x && i < n && (!CH || last_piece || ts + 1 < H))
                    store_out(p.x, xoff + (long long)(ts + 1) * n + i, xs[q], obf);
            }
        }
        __syncwarp();
    }
}

template <int NB, int MB, bool TV, bool AFF, bool PAD, bool CH = false, bool GRAD = false>
inline cudaError_t launch_one(const SolveParams& p, int sm_count, cudaStream_t st)
{
    // up to 16 states a CTA is four warps, unless the instances are so few that one warp each spreads them over more SMs;
    // above, the operands of a warp fill 7 to 60 KB and CTAs of one warp pack best
    const long long nwin = p.b0 * p.b1 * p.tcount * (CH ? p.chunks : 1);
    const int warps = NB > 2 || nwin <= 4ll * sm_count ? 1 : MAX_WARPS;
    const size_t smem = warps * warp_bytes<NB, MB, TV, GRAD>();
    // (above 16 states two warps per scheduler leave it idle at any batch: the shorter chain always)
    constexpr bool CAN = NB <= 2 && !AFF && !CH && !GRAD;
    // by the size of the whole batch: the windows of a sliced call have to give the same bits as one call
    void (*kern)(SolveParams) = CAN && p.N <= 4ll * sm_count ? riccati_frag_kernel<NB, MB, TV, AFF, PAD, CH, GRAD, CAN>
                                                  : riccati_frag_kernel<NB, MB, TV, AFF, PAD, CH, GRAD, false>;
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess)
            return e;
    }
    kern<<<(unsigned)((nwin + warps - 1) / warps), 32 * warps, smem, st>>>(p);
    return cudaGetLastError();
}

} // namespace rfrag
} // namespace ttc
