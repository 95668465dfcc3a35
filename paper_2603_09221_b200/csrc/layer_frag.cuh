// One Test-Time Control layer evaluation per (token, head): the LQR parameters are synthesised inside the kernel from
// the coefficient vectors (Contextualization / Parameterization paragraphs of the TTC-Net section) and the backward
// Riccati recursion (Prop. A.1 / Alg. 1) runs on them; nothing time-dependent is written to HBM.  Paper indices t = 1..T:
//     A_t = I + diag(exp(-t g_A) a)                 (diagonal)
//     B_t = Bbar diag(exp(-t g_B)),                 Bbar = sum_i s_B[i] B^(i)
//     Q_t = diag(exp(-t g_Q)) Qbar diag(exp(-t g_Q)),  Qbar = sum_i s_Q[i] Q^(i),  Q_0 = 0,
//     Q_T = sum_i s_Qf[i] Q^(i)                     (terminal override)
//     R_t = diag(1 / r_inv)
// and the layer output is the first optimal control u_1* = K_1 h_0.
//
// One warp per instance, matrices in registers (frag.cuh).  Step s = t - 1 (s = T-1 .. 0), P = P_{s+1}, with
// a = diag(A_t), g = exp(-t g_B), q = exp(-s g_Q), in negated variables (nP = -P):
//     V   = G Bbar' nP               one product; Bbar' sits split in shared memory in register order
//     nS  = G Bbar' V' - R           one product, rows scaled
//     nY' = A V'                     V transposed by shuffles: with a diagonal A_t no product is needed
//     nP  = a_i a_j nP_ij - q_i q_j Qbar_ij + (Z'Z)_ij      elementwise and one product, symmetric bit for bit
// so that a step is 51 tensor-core instructions against 87 of the dense one.
//
// n = 16 is bound by the instructions it issues (about 690 per step, of which 220 are the sixteen pivots and 144 the
// splitting of operands): 65536 instances, T = 32: 2.28 -> 1.87 ms against the broadcast-row form with two columns per
// lane; 16 instances (one decoded token of 16 heads) are one dependent chain per SM: 98 -> 41 us.
// n = 32 needs all 255 registers for its eight 16 x 8 tiles per matrix and keeps two warps per scheduler: 16384
// instances, T = 32: 5.45 -> 3.2 ms (products through shared memory before).
#pragma once

#include "frag.cuh"
#include "ttc_layer.cuh"

namespace ttc {
namespace lfrag {

using namespace frag;
using layer::LayerParams;

constexpr int MAX_WARPS = 4;

template <int NB>
struct Slot {
    static constexpr int N = 8 * NB;
    Stored<NB, NB> B;                                // Bbar'
    float4 Q[(NB + 1) / 2][NB][32];                  // Qbar, register order
    float a[2][N], g[2][N], q[2][N];                 // diagonals of a step, two steps in turn
};

// accumulates sum_i coef_i M^(i) for the basis matrices of Bbar, Qbar and Q_T
template <int NB>
__device__ __forceinline__ void synthesise(Mat<NB, NB>& B, Mat<NB, NB>& Q, Mat<NB, NB>& F, const LayerParams& p, long long inst, int lane)
{
    constexpr int N = 8 * NB, MT = Mat<NB, NB>::MT;
    const int g = lane >> 2, t = lane & 3, r = p.r;
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int cb = 0; cb < NB; ++cb)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                B.v[mt][cb][e] = Q.v[mt][cb][e] = F.v[mt][cb][e] = 0.f;
    for (int k0 = 0; k0 < r; k0 += 32) {
        const bool have = k0 + lane < r;
        const float cb_ = have ? __ldg(p.s_b + inst * r + k0 + lane) : 0.f;
        const float cq = have ? __ldg(p.s_q + inst * r + k0 + lane) : 0.f;
        const float cf = have ? __ldg(p.s_qf + inst * r + k0 + lane) : 0.f;
        const int cnt = min(32, r - k0);
#pragma unroll 2
        for (int k = 0; k < cnt; ++k) {
            const float wb = __shfl_sync(FULL, cb_, k), wq = __shfl_sync(FULL, cq, k), wf = __shfl_sync(FULL, cf, k);
            const float* Bi = p.B_basis + (long long)(k0 + k) * N * N;
            const float* Qi = p.Q_basis + (long long)(k0 + k) * N * N;
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int cb = 0; cb < NB; ++cb)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int o = (16 * mt + 8 * h + g) * N + 8 * cb + 2 * t;
                        const float2 bv = __ldg(reinterpret_cast<const float2*>(Bi + o));
                        const float2 qv = __ldg(reinterpret_cast<const float2*>(Qi + o));
                        B.v[mt][cb][2 * h] = fmaf(wb, bv.x, B.v[mt][cb][2 * h]);
                        B.v[mt][cb][2 * h + 1] = fmaf(wb, bv.y, B.v[mt][cb][2 * h + 1]);
                        Q.v[mt][cb][2 * h] = fmaf(wq, qv.x, Q.v[mt][cb][2 * h]);
                        Q.v[mt][cb][2 * h + 1] = fmaf(wq, qv.y, Q.v[mt][cb][2 * h + 1]);
                        F.v[mt][cb][2 * h] = fmaf(wf, qv.x, F.v[mt][cb][2 * h]);
                        F.v[mt][cb][2 * h + 1] = fmaf(wf, qv.y, F.v[mt][cb][2 * h + 1]);
                    }
        }
    }
}

template <int NB>
__device__ __forceinline__ void transpose(Mat<NB, NB>& y, const Mat<NB, NB>& x, int lane)
{
#pragma unroll
    for (int i = 0; i < NB; ++i)
#pragma unroll
        for (int j = 0; j < NB; ++j)
            transpose8(y.v[j / 2][i][2 * (j & 1)], y.v[j / 2][i][2 * (j & 1) + 1], x.v[i / 2][j][2 * (i & 1)],
                       x.v[i / 2][j][2 * (i & 1) + 1], lane);
}

// decay rates of the instance: n = 16 spreads the three vectors over the two halves of the warp, n = 32 takes one
// component per lane
template <int NB>
struct Rates {
    float k1, k2, k3, sa;
    __device__ __forceinline__ void load(const LayerParams& p, long long inst, int lane)
    {
        constexpr int N = 8 * NB;
        const int c = lane % N;
        const bool first = lane < N;
        sa = __ldg(p.s_a + inst * N + c);
        k1 = __ldg((first ? p.s_ga : p.s_gb) + inst * N + c);
        k2 = __ldg(p.s_gq + inst * N + c);
        k3 = N == 32 ? __ldg(p.s_gb + inst * N + c) : 0.f;
    }
    // diagonals of step s into the slot
    __device__ __forceinline__ void step(Slot<NB>& sl, int s, int lane) const
    {
        constexpr int N = 8 * NB;
        const float tt = (float)(s + 1);
        const float e1 = __expf(-tt * k1);
        float* a = sl.a[s & 1];
        float* g = sl.g[s & 1];
        if (lane < N) {
            a[lane] = fmaf(e1, sa, 1.f);
            sl.q[s & 1][lane] = s >= 1 ? __expf(-(float)s * k2) : 0.f;      // Q_0 = 0
        }
        if (N == 32)
            g[lane] = __expf(-tt * k3);
        else if (lane >= N && lane < 2 * N)
            g[lane - N] = e1;
    }
};

// parameters of one instance: Bbar' and Qbar into the slot, nP = -P_T = -Q_T
template <int NB>
__device__ __forceinline__ void prepare(Slot<NB>& sl, Mat<NB, NB>& nP, const LayerParams& p, long long inst, int lane)
{
    Mat<NB, NB> B, Q, Bt;
    synthesise<NB>(B, Q, nP, p, inst, lane);
    transpose<NB>(Bt, B, lane);
    keep(sl.B, Bt, lane);
#pragma unroll
    for (int mt = 0; mt < Mat<NB, NB>::MT; ++mt)
#pragma unroll
        for (int cb = 0; cb < NB; ++cb) {
            sl.Q[mt][cb][lane] = make_float4(Q.v[mt][cb][0], Q.v[mt][cb][1], Q.v[mt][cb][2], Q.v[mt][cb][3]);
#pragma unroll
            for (int e = 0; e < 4; ++e)
                nP.v[mt][cb][e] = -nP.v[mt][cb][e];
        }
}

// The backward recursion of one instance.  nP comes in as -P_T and goes out as -P_0; `on_step(s, Zt, S, w)` is called
// with what gains() needs after each factorisation.  Returns 0 or s n + j + 1 for the first bad pivot.
template <int NB, bool PAIR, typename F>
__device__ __forceinline__ int backward(Mat<NB, NB>& nP, Slot<NB>& sl, const Rates<NB>& rates, const float (&rd)[NB], int T, int lane,
                                        F&& on_step)
{
    constexpr int N = 8 * NB, MT = Mat<NB, NB>::MT;
    const int g = lane >> 2, t = lane & 3;
    int fail = 0;
    rates.step(sl, T - 1, lane);
#pragma unroll 1
    for (int s = T - 1; s >= 0; --s) {
        __syncwarp();
        const float* av = sl.a[s & 1];
        const float* gv = sl.g[s & 1];
        const float* qv = sl.q[s & 1];
        if (s > 0)
            rates.step(sl, s - 1, lane);
        Mat<NB, NB> V, S, Zt;
        {
            Split<NB, NB> ps;
            split(ps, nP);
            product<NB, NB, NB>(V, nullptr, sl.B, ps, lane);         // Bbar' nP
        }
        float gr[NB], ar[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            gr[b] = gv[8 * b + g];
            ar[b] = av[8 * b + g];
        }
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int cb = 0; cb < NB; ++cb)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    V.v[mt][cb][e] *= gr[2 * mt + (e >> 1)];
        {
            Split<NB, NB> vs;
            split(vs, V);
            product<NB, NB, NB, true>(S, nullptr, sl.B, vs, lane);         // Bbar' V'
        }
        transpose<NB>(Zt, V, lane);
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int cb = 0; cb < NB; ++cb)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int b = 2 * mt + (e >> 1);
                    Zt.v[mt][cb][e] *= ar[b];               // -Y' = A V'
                    // -S = G Bbar' V' - R (lower tiles)
                    if (cb > 2 * mt + 1)
                        continue;
                    if (cb == b)
                        S.v[mt][cb][e] = fmaf(S.v[mt][cb][e], gr[b], t == (g >> 1) && (e & 1) == (g & 1) ? -rd[b] : 0.f);
                    else
                        S.v[mt][cb][e] *= gr[b];
                }
        {
            float ac[NB][2], qc[NB][2], qr[NB];
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const float2 a2 = *reinterpret_cast<const float2*>(av + 8 * b + 2 * t);
                const float2 q2 = *reinterpret_cast<const float2*>(qv + 8 * b + 2 * t);
                ac[b][0] = a2.x; ac[b][1] = a2.y;
                qc[b][0] = q2.x; qc[b][1] = q2.y;
                qr[b] = qv[8 * b + g];
            }
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int cb = 0; cb < NB; ++cb) {
                    const float4 q4 = sl.Q[mt][cb][lane];
                    const float qq[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int b = 2 * mt + (e >> 1);
                        nP.v[mt][cb][e] = fmaf(-qq[e], qr[b] * qc[cb][e & 1], nP.v[mt][cb][e] * (ar[b] * ac[cb][e & 1]));
                    }
                }
        }
        Split<NB, NB> zs;
        float w[NB][2];
        const int bad = factor<NB, NB, PAIR>(S, Zt, zs, w, lane);
        if (bad && !fail)
            fail = s * N + bad;
        product_symmetric<NB, NB>(nP, zs);
        mirror<NB>(nP, lane);
        on_step(s, Zt, S, w);
    }
    return fail;
}

// FEW: at most four warps per SM, see chol8_inverse
template <int NB, bool FEW>
__global__ void __launch_bounds__(32 * MAX_WARPS, NB == 2 ? 5 : 2) layer_frag_kernel(LayerParams p)
{
    constexpr int N = 8 * NB, MT = Mat<NB, NB>::MT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    // (n = 32, T = 32, through a shuffle as at n = 16: 1024 instances 180.2 instead of 179.6 us, 8192 instances 1198 instead of 1195 us;
    // n = 16: 41.0 to 1872 us with it, 41.2 to 1872 without)
    const int warp = NB > 2 ? (int)(threadIdx.x >> 5) : warp_index();
    const long long inst = (long long)blockIdx.x * (blockDim.x >> 5) + warp;
    if (inst >= p.N)
        return;
    Slot<NB>& sl = reinterpret_cast<Slot<NB>*>(smem_raw)[warp];
    Mat<NB, NB> nP;
    prepare<NB>(sl, nP, p, inst, lane);
    Rates<NB> rates;
    rates.load(p, inst, lane);
    float rd[NB], hr[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        rd[b] = 1.f / __ldg(p.r_inv + inst * N + 8 * b + g);
        hr[b] = __ldg(p.h0 + inst * N + 8 * b + g);
    }
    float u[NB][2];
#pragma unroll
    for (int b = 0; b < NB; ++b)
        u[b][0] = u[b][1] = 0.f;
    const int fail = backward<NB, FEW>(nP, sl, rates, rd, p.T, lane, [&](int s, Mat<NB, NB>& Zt, const Mat<NB, NB>& S, const float(&w)[NB][2]) {
        if (s == 0 && p.u1) {                               // u_1* = K_1 h_0
            gains<NB, NB>(Zt, S, w, lane);
#pragma unroll
            for (int b = 0; b < NB; ++b)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    float v = 0.f;
#pragma unroll
                    for (int i = 0; i < NB; ++i)
                        v = fmaf(Zt.v[i / 2][b][2 * (i & 1) + e], hr[i], v);
                    u[b][e] = sum_over_g(v);
                }
        }
    });
    const float qn = quiet_nan();
    if (p.P0) {
        float* P0 = p.P0 + inst * (long long)N * N;
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int cb = 0; cb < NB; ++cb)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float x = -nP.v[mt][cb][2 * h], y = -nP.v[mt][cb][2 * h + 1];
                    *reinterpret_cast<float2*>(P0 + (16 * mt + 8 * h + g) * N + 8 * cb + 2 * t) =
                        make_float2(fail ? qn : x, fail ? qn : y);
                }
    }
    if (p.u1 && g == 0) {
#pragma unroll
        for (int b = 0; b < NB; ++b)
            *reinterpret_cast<float2*>(p.u1 + inst * N + 8 * b + 2 * t) = make_float2(fail ? qn : u[b][0], fail ? qn : u[b][1]);
    }
    if (p.info && lane == 0)
        p.info[inst] = fail;
}

// Few instances get a CTA each so that they spread over the SMs.
template <int NB>
inline cudaError_t launch_layer_frag(const LayerParams& p, int sm_count, cudaStream_t st)
{
    const int warps = p.N <= 4ll * sm_count ? 1 : MAX_WARPS;
    void (*kern)(LayerParams) = p.few ? layer_frag_kernel<NB, true> : layer_frag_kernel<NB, false>;
    const size_t smem = sizeof(Slot<NB>) * warps;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess)
            return e;
    }
    kern<<<(unsigned)((p.N + warps - 1) / warps), 32 * warps, smem, st>>>(p);
    return cudaGetLastError();
}

} // namespace lfrag
} // namespace ttc
