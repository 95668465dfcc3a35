// Riccati-backward + rollout kernel for n, m <= 16, float32: one WARP per instance, every matrix of the step in registers
// in the mma.sync accumulator layout (frag.cuh), so that a step is a chain of tensor-core products, two or one
// eight-column factorisation panels and a few shuffles, without shared memory and without barriers.
//
// The recursion is carried in negated variables (nP = -P etc.): every update is then a plain accumulation.
//   V = B' nP,  T = A' nP,  nS = -R + B' V',  nY' = A' V',  nP_t = -Q + A' T' + Z' Z     (Prop. 3.1; Alg. 1)
// with S = L L', Z = L^{-1} Y and, when gains are wanted, K' = -Z' L^{-1} from the inverses of L's diagonal blocks.
//
// What bounds it: a step is 87 tensor-core instructions (8 cycles each on a scheduler's pipe) in about 830, and four
// warps per scheduler (128 registers) hide most of the chain of five products and sixteen pivots.  Columns of the
// matrices spread over the lanes of a warp with rows broadcast from shared memory (the form this replaced) ran at 88 %
// of the load/store pipe and 4.3 us per step for a single instance; this one takes about 2 us.
// 65536 instances, H = 32, operands from memory: 4.26 -> 2.84 ms (tensor pipe 46 %, issue slots 55 %); 4096 instances,
// H = 16, all outputs: 188 -> 109 us; 64 instances of n = m = 8, H = 8: 107 -> 22 us (generic kernel before).
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

// ---- operands of one time step of one instance, staged in the warp's shared memory by asynchronous copies one step
// ahead of their use: the registers they would occupy for a whole step go to a fifth CTA per SM instead.
// A and B are read transposed (lane (g, t) takes row 2 t, column g): with rows of 8 NB + 4 floats the 32 lanes fall into
// 32 banks.  Q and R are read as pairs along the rows (20 floats per row: five CTAs with two buffers each fit an SM).
template <int NB, int MB>
struct Operands {
    static constexpr int LA = 8 * NB + 4, LB = 8 * MB + 4, LQ = NB == 1 ? 8 : 20, LR = MB == 1 ? 8 : 20;
    float A[8 * NB * LA], B[8 * NB * LB], Q[8 * NB * LQ], R[8 * MB * LR];
};
// time-invariant form: A' and B' once more, split and in register order
template <int NB, int MB>
struct Fixed {
    Stored<NB, NB> A;
    Stored<MB, NB> B;
};
// what a warp keeps in shared memory
template <int NB, int MB, bool TV>
struct WarpMem {
    Operands<NB, MB> op[2];
};
template <int NB, int MB>
struct WarpMem<NB, MB, false> {
    Operands<NB, MB> op[1];
    Fixed<NB, MB> fixed;
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
// X = M' from shared memory
template <int RB, int CB, int LD>
__device__ __forceinline__ void load_transposed(Mat<RB, CB>& x, const float* M, int lane)
{
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int mt = 0; mt < Mat<RB, CB>::MT; ++mt)
#pragma unroll
        for (int cb = 0; cb < CB; ++cb)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                x.v[mt][cb][e] = e >= 2 && 2 * mt + 1 >= RB ? 0.f : M[(8 * cb + 2 * t + (e & 1)) * LD + 16 * mt + g + ((e & 2) ? 8 : 0)];
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

// `cnt` = 4 W consecutive elements of a row (16-byte loads), or with PAD element by element within [0, n)
template <int W, bool PAD>
__device__ __forceinline__ void load_half_row(float (&v)[4 * W], const float* row, int c0, int n)
{
    if (PAD) {
#pragma unroll
        for (int k = 0; k < 4 * W; ++k)
            v[k] = c0 + k < n ? row[c0 + k] : 0.f;
    } else {
#pragma unroll
        for (int q = 0; q < W; ++q) {
            const float4 f = *reinterpret_cast<const float4*>(row + c0 + 4 * q);
            v[4 * q] = f.x; v[4 * q + 1] = f.y; v[4 * q + 2] = f.z; v[4 * q + 3] = f.w;
        }
    }
}

struct Scratch {
    float x[16], u[16];
};

// NB, MB: number of 8-blocks of the state and the control dimension.
// TV = time-varying request (time strides or a terminal weight); AFF = linear control cost r_t'u_t (implies TV);
// PAD = n < 8 NB or m < 8 MB, or strides that do not keep the vector loads aligned: guarded element-wise accesses, the
// missing part of R is the identity and everything else zero, which leaves the recursion of the existing part untouched.
template <int NB, int MB, bool TV, bool AFF, bool PAD>
__global__ void __launch_bounds__(32 * MAX_WARPS, TV && !AFF ? 5 : 4) riccati_frag_kernel(SolveParams p)
{
    __shared__ __align__(16) Scratch scratch[MAX_WARPS];
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const long long widx = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (widx >= p.b0 * p.b1 * p.tcount)
        return;
    Scratch& sc = scratch[threadIdx.x >> 5];
    const Place pl = place(p, (unsigned)widx);
    const long long inst = pl.inst;
    const int n = PAD ? p.n : 8 * NB, m = PAD ? p.m : 8 * MB, H = p.H, obf = p.out_bf16;
    const bool need_K_all = p.K != nullptr || p.x != nullptr || (p.u != nullptr && !p.first_only);
    const bool want_u0 = p.u != nullptr && p.first_only && !need_K_all;
    const bool need_k_all = AFF && p.kff != nullptr;
    float* const Kbase = (p.K && !obf) ? p.K : p.Kws;       // float32 gains (the rollout reads them)
    const long long Koff = inst * (long long)H * m * n;
    const long long Poff = inst * (long long)(p.first_only ? 1 : H + 1) * n * n;
    using Ops = Operands<NB, MB>;
    WarpMem<NB, MB, TV>* const ops = reinterpret_cast<WarpMem<NB, MB, TV>*>(smem_raw) + (threadIdx.x >> 5);
    const long long oA = pl.off(p.A), oB = pl.off(p.B), oR = pl.off(p.R), oQ = pl.off(p.Q);
    Mat<NB, NB> nP;
    {
        if (PAD) {                                          // what does not exist: R is the identity, the rest zero
            for (int e = lane; e < (int)(sizeof(Ops) / sizeof(float)) * (TV ? 2 : 1); e += 32)
                reinterpret_cast<float*>(ops->op)[e] = 0.f;
            __syncwarp();
            for (int i = m + lane; i < 8 * MB; i += 32) {
                ops->op[0].R[i * Ops::LR + i] = 1.f;
                if (TV)
                    ops->op[1].R[i * Ops::LR + i] = 1.f;
            }
        }
        const long long last = TV ? H - 1 : 0;
        if (TV && p.Qf.ptr) {                               // P_H = Q_f, by way of the second buffer
            stage<NB, NB, Ops::LQ, PAD>(ops->op[TV].Q, p.Qf, pl.off(p.Qf), n, n, lane);
            copies_landed();
            load_negated<NB, Ops::LQ>(nP, ops->op[TV].Q, lane);
            __syncwarp();
        }
#pragma unroll
        for (int b = 0; b < (TV ? 2 : 1); ++b) {            // the second buffer: what does not change with time
            if (b == 0 || !p.A.st) stage<NB, NB, Ops::LA, PAD>(ops->op[b].A, p.A, oA + last * p.A.st, n, n, lane);
            if (b == 0 || !p.B.st) stage<NB, MB, Ops::LB, PAD>(ops->op[b].B, p.B, oB + last * p.B.st, n, m, lane);
            if (b == 0 || !p.R.st) stage<MB, MB, Ops::LR, PAD>(ops->op[b].R, p.R, oR + last * p.R.st, m, m, lane);
            if (b == 0 || !p.Q.st) stage<NB, NB, Ops::LQ, PAD>(ops->op[b].Q, p.Q, oQ + last * p.Q.st, n, n, lane);
        }
        copies_landed();
        if constexpr (!TV) {
            Mat<NB, NB> At;
            Mat<MB, NB> Bt;
            load_transposed<NB, NB, Ops::LA>(At, ops->op[0].A, lane);
            load_transposed<MB, NB, Ops::LB>(Bt, ops->op[0].B, lane);
            keep(ops->fixed.A, At, lane);
            keep(ops->fixed.B, Bt, lane);
            __syncwarp();
        }
        if (!(TV && p.Qf.ptr))
            load_negated<NB, Ops::LQ>(nP, ops->op[0].Q, lane);  // P_H = Q
    }
    if (p.P && !p.first_only)
        store_negated<NB, PAD>(p.P, Poff + (long long)H * n * n, nP, n, obf, lane);

    float xr[NB];                                           // x_0 in row form
#pragma unroll
    for (int b = 0; b < NB; ++b)
        xr[b] = (p.x0.ptr && 8 * b + g < n) ? load_elem(p.x0, pl.off(p.x0) + 8 * b + g) : 0.f;

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
#pragma unroll 1
    for (int ts = H - 1; ts >= 0; --ts) {
        const Ops& op = ops->op[TV ? (H - 1 - ts) & 1 : 0];
        if (TV && ts < H - 1)
            copies_landed();                                // also: every lane is done with the other buffer
        if (TV && ts > 0) {                                 // operands of the next step
            Ops& nx = ops->op[(H - ts) & 1];
            if (p.A.st) stage<NB, NB, Ops::LA, PAD>(nx.A, p.A, oA + (ts - 1) * p.A.st, n, n, lane);
            if (p.B.st) stage<NB, MB, Ops::LB, PAD>(nx.B, p.B, oB + (ts - 1) * p.B.st, n, m, lane);
            if (p.R.st) stage<MB, MB, Ops::LR, PAD>(nx.R, p.R, oR + (ts - 1) * p.R.st, m, m, lane);
            if (p.Q.st) stage<NB, NB, Ops::LQ, PAD>(nx.Q, p.Q, oQ + (ts - 1) * p.Q.st, n, n, lane);
        }
        Mat<NB, NB> At, T;
        Mat<MB, NB> Bt, V;
        Mat<NB, MB> Zt;
        Mat<MB, MB> S, nR;
        load_negated<MB, Ops::LR>(nR, op.R, lane);
        Split<NB, NB> ps;
        Split<MB, NB> vs;
        split(ps, nP);
        if constexpr (TV) {
            load_transposed<NB, NB, Ops::LA>(At, op.A, lane);
            load_transposed<MB, NB, Ops::LB>(Bt, op.B, lane);
            Split<NB, NB> as;
            Split<MB, NB> bs;
            split(as, At);
            split(bs, Bt);
            product<MB, NB, NB>(V, nullptr, bs, ps);        // V = B' nP
            product<NB, NB, NB>(T, nullptr, as, ps);        // T = A' nP
            split(vs, V);
            product<MB, NB, MB>(S, &nR, bs, vs);            // -S = -R + B' V'
            product<NB, NB, MB>(Zt, nullptr, as, vs);       // -Y' = A' V'
            split(ps, T);
            load_negated<NB, Ops::LQ>(nP, op.Q, lane);
            product<NB, NB, NB>(nP, &nP, as, ps);           // -Q - A'P A
        } else {
            const Fixed<NB, MB>& fx = ops->fixed;
            product<MB, NB, NB>(V, nullptr, fx.B, ps, lane);
            product<NB, NB, NB>(T, nullptr, fx.A, ps, lane);
            split(vs, V);
            product<MB, NB, MB>(S, &nR, fx.B, vs, lane);
            product<NB, NB, MB>(Zt, nullptr, fx.A, vs, lane);
            split(ps, T);
            load_negated<NB, Ops::LQ>(nP, op.Q, lane);
            product<NB, NB, NB>(nP, &nP, fx.A, ps, lane);
        }
        float gr[MB], ap[NB];                               // affine: B'p + r and A'p in row form
        if (AFF && ts < p.r_count) {
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
        }
        Split<NB, MB> zs;
        float w[MB][2];
        const int bad = factor<NB, MB>(S, Zt, zs, w, lane);  // Zt becomes Z', S the blocks of L
        if (bad && !fail)
            fail = ts * m + bad;
        product<NB, MB, NB>(nP, &nP, zs, zs);                              // -P_t = -Q - A'PA + Z'Z
        const bool gain = need_K_all || need_k_all || (want_u0 && ts == 0);
        if (AFF) {
            // z = L^{-1}(B'p + r);  p_t = A'p - Z'z;  k_t = -L^{-T} z   (all zero while p and r are)
            if (ts < p.r_count) {
                float zc[MB][2], zr[MB];
#pragma unroll
                for (int b = 0; b < MB; ++b) {
                    float s = 0.f;
#pragma unroll
                    for (int k = 0; k < b; ++k)
                        s = fmaf(S.v[b / 2][k][2 * (b & 1)], zc[k][0], fmaf(S.v[b / 2][k][2 * (b & 1) + 1], zc[k][1], s));
                    float c0, c1;
                    row_to_col(c0, c1, b ? gr[b] - sum_over_t(s) : gr[b], lane);
                    zr[b] = sum_over_t(fmaf(w[b][0], c0, w[b][1] * c1));
                    row_to_col(zc[b][0], zc[b][1], zr[b], lane);
                }
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    float s = 0.f;
#pragma unroll
                    for (int k = 0; k < MB; ++k)
                        s = fmaf(Zt.v[b / 2][k][2 * (b & 1)], zc[k][0], fmaf(Zt.v[b / 2][k][2 * (b & 1) + 1], zc[k][1], s));
                    pr[b] = ap[b] - sum_over_t(s);
                }
                float kr[MB];                               // k_t in row form, last block first
#pragma unroll
                for (int b = MB - 1; b >= 0; --b) {
                    float s0 = 0.f, s1 = 0.f;               // (L_qb' k_q) in column form
#pragma unroll
                    for (int q = b + 1; q < MB; ++q) {
                        s0 = fmaf(S.v[q / 2][b][2 * (q & 1)], kr[q], s0);
                        s1 = fmaf(S.v[q / 2][b][2 * (q & 1) + 1], kr[q], s1);
                    }
                    float v = zr[b];
                    if (b + 1 < MB)
                        v += col_to_row(sum_over_g(s0), sum_over_g(s1), lane);
                    kc0[b][0] = -sum_over_g(w[b][0] * v);
                    kc0[b][1] = -sum_over_g(w[b][1] * v);
                    kr[b] = col_to_row(kc0[b][0], kc0[b][1], lane);
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
        make_symmetric<NB>(nP, lane);
        if (p.P && (!p.first_only || ts == 0))
            store_negated<NB, PAD>(p.P, Poff + (long long)(p.first_only ? 0 : ts) * n * n, nP, n, obf, lane);
    }
    if (p.info && lane == 0)
        p.info[inst] = fail;
    if (fail) {                                             // uniform over the warp
        const float qn = quiet_nan();
        __syncwarp();
        if (p.K)
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
        if (need_k_all)
            for (long long e = lane; e < (long long)H * m; e += 32)
                p.kff[inst * (long long)H * m + e] = qn;
        return;
    }
    if (want_u0 || !(p.x || p.u))
        return;

    // ---- forward loop of Alg. 1: two lanes per row, the vectors in the warp's scratch; the rows of K_{t+1} (and of
    // A_{t+1}, B_{t+1}) are in flight while step t is summed
    const float* Ag = reinterpret_cast<const float*>(p.A.ptr) + oA;
    const float* Bg = reinterpret_cast<const float*>(p.B.ptr) + oB;
    const int i = lane >> 1, c0n = (lane & 1) * 4 * NB, c0m = (lane & 1) * 4 * MB;
    if ((lane & 1) == 0) {
        sc.x[i] = (i < n && p.x0.ptr) ? load_elem(p.x0, pl.off(p.x0) + i) : 0.f;
        sc.u[i] = 0.f;
    }
    __syncwarp();                                           // also: K_t stored by the other lanes are visible
    const bool xo = p.x && (lane & 1) == 0 && i < n, uo = p.u && (lane & 1) == 0 && i < m;
    const long long xoff = inst * (long long)(H + 1) * n + i, uoff = inst * (long long)(p.first_only ? m : H * m) + i;
    const int ri = i < n ? i : 0, rj = i < m ? i : 0;
    const float* Kr = Kbase + Koff + (long long)rj * n;
    float kr[4 * NB], ar[4 * NB], br[4 * MB], kt = 0.f;
    load_half_row<NB, PAD>(kr, Kr, c0n, n);
    load_half_row<NB, PAD>(ar, Ag + ri * n, c0n, n);
    load_half_row<MB, PAD>(br, Bg + ri * m, c0m, m);
    if (AFF && p.kff)
        kt = p.kff[inst * (long long)H * m + rj];
    else if (AFF) {                                         // only u_0 is wanted: k_0 is still in registers
#pragma unroll
        for (int b = 0; b < MB; ++b) {
            const float e0 = __shfl_sync(FULL, kc0[b][0], (i & 7) >> 1), e1 = __shfl_sync(FULL, kc0[b][1], (i & 7) >> 1);
            if (i / 8 == b)
                kt = (i & 1) ? e1 : e0;
        }
    }
    const int steps = (p.x || !p.first_only) ? H : 1;
    if (xo)
        store_out(p.x, xoff, sc.x[i], obf);
#pragma unroll 1
    for (int ts = 0; ts < steps; ++ts) {
        float xv[4 * NB], uv[4 * MB];
        load_half_row<NB, false>(xv, sc.x, c0n, 16);
        float us = 0.f, xs = 0.f;
#pragma unroll
        for (int k = 0; k < 4 * NB; ++k) {
            us = fmaf(kr[k], xv[k], us);
            xs = fmaf(ar[k], xv[k], xs);
        }
        us += __shfl_xor_sync(FULL, us, 1);
        if (AFF)
            us += kt;
        if ((lane & 1) == 0)
            sc.u[i] = i < m ? us : 0.f;
        if (uo && (!p.first_only || ts == 0))
            store_out(p.u, uoff + (p.first_only ? 0 : (long long)ts * m), us, obf);
        __syncwarp();
        load_half_row<MB, false>(uv, sc.u, c0m, 16);
#pragma unroll
        for (int k = 0; k < 4 * MB; ++k)
            xs = fmaf(br[k], uv[k], xs);
        if (ts + 1 < steps) {
            load_half_row<NB, PAD>(kr, Kr + (long long)(ts + 1) * m * n, c0n, n);
            if (TV && p.A.st) load_half_row<NB, PAD>(ar, Ag + (ts + 1) * p.A.st + ri * n, c0n, n);
            if (TV && p.B.st) load_half_row<MB, PAD>(br, Bg + (ts + 1) * p.B.st + ri * m, c0m, m);
            if (AFF && p.kff)
                kt = p.kff[(inst * H + ts + 1) * (long long)m + rj];
        }
        xs += __shfl_xor_sync(FULL, xs, 1);
        if ((lane & 1) == 0)
            sc.x[i] = i < n ? xs : 0.f;
        if (xo)
            store_out(p.x, xoff + (long long)(ts + 1) * n, xs, obf);
        __syncwarp();
    }
}

// Launch for n, m <= 16.  `exact`: the strides keep the vector loads aligned (rows of Q, Qf, R and of K, A, B in the
// rollout).  Few instances get a CTA each so that they spread over the SMs.
inline cudaError_t launch_riccati_frag(const SolveParams& p, bool time_varying, bool affine, bool exact, int sm_count, cudaStream_t st)
{
    const long long nwin = p.b0 * p.b1 * p.tcount;
    void (*kern)(SolveParams);
    size_t per_warp = sizeof(WarpMem<2, 2, false>);
    const bool sq8 = p.n <= 8 && p.m <= 8, m8 = p.m <= 8;
    const bool pad8 = !(exact && p.n == 8 && p.m == 8), pad16 = !(exact && p.n == 16 && p.m == 16);
    if (affine || time_varying) {
        per_warp = sizeof(WarpMem<2, 2, true>);
        if (affine)
            kern = pad16 ? riccati_frag_kernel<2, 2, true, true, true> : riccati_frag_kernel<2, 2, true, true, false>;
        else
            kern = pad16 ? riccati_frag_kernel<2, 2, true, false, true> : riccati_frag_kernel<2, 2, true, false, false>;
    } else if (sq8) {
        kern = pad8 ? riccati_frag_kernel<1, 1, false, false, true> : riccati_frag_kernel<1, 1, false, false, false>;
        per_warp = sizeof(WarpMem<1, 1, false>);
    } else if (m8) {
        kern = riccati_frag_kernel<2, 1, false, false, true>;
        per_warp = sizeof(WarpMem<2, 1, false>);
    } else {
        kern = pad16 ? riccati_frag_kernel<2, 2, false, false, true> : riccati_frag_kernel<2, 2, false, false, false>;
    }
    const int warps = nwin <= 4ll * sm_count ? 1 : MAX_WARPS;
    kern<<<(unsigned)((nwin + warps - 1) / warps), 32 * warps, warps * per_warp, st>>>(p);
    return cudaGetLastError();
}

} // namespace rfrag
} // namespace ttc
