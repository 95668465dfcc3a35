// Gradients of the contextualised layer's output u_1* with respect to what the coefficient layers hand over
// (Thm 3.2, then the chain rule through the Contextualization / Parameterization paragraphs), without ever forming
// the per-step matrices dA_t, dB_t, dQ_t, dR_t: every outer product of the theorem is reduced on the fly onto
// s_A, s_GammaA, s_GammaB, s_GammaQ, R^{-1}, h_0 and onto three d x d matrices per instance (the gradients of
// Bbar = sum_k s_B[k] B^(k), Qbar = sum_k s_Q[k] Q^(k) and Q_T), which are then contracted with the bases.
//
// Launches: (1) layer_grad_kernel<NB>, one warp per instance from beginning to end: backward Riccati pass in registers
// (layer_frag.cuh) that writes every gain K_s, both rollouts (primal from h_0; dual from 0 with first control
// k_0 = -S_0^{-1} g), both co-state recursions backwards, and the reductions; (2) basis_reduce_kernel:
// dB^(k) = sum_i s_B[i][k] dBbar_i etc.
//
// Step s = t - 1 (library indexing) uses a_s = 1 + e^{-(s+1) gA} sA (diagonal of A_{s+1}), B_s = Bbar diag(e^{-(s+1) gB}),
// R = diag(1 / r_inv), state weight Q_s = G Qbar G with G = diag(e^{-s gQ}) for s >= 1, Q_0 = 0, terminal weight Q_T.
//   dA_s[i,i] = lam_{s+1}[i] xd_s[i] + lamd_{s+1}[i] x_s[i]          -> d sA, d gA
//   dB_s      = lam_{s+1} ud_s' + lamd_{s+1} u_s'                    -> d Bbar (column-scaled), d gB
//   dQ_s      = 1/2 (x_s xd_s' + xd_s x_s')  (1 <= s <= T-1; s = T: Q_T) -> d Qbar (scaled both sides), d gQ, d Q_T
//   dR_s[j,j] = u_s[j] ud_s[j]                                        -> d r_inv = -dR / r_inv^2;   d h_0 = lamd_0
// The co-states obey lam_s = a_s lam_{s+1} + Q_s x_s, which amplifies rounding by the open-loop a_s (up to about 1.9).
// Since R u_s + B_s'lam_{s+1} = 0, the same lam_s is
//     lam_s = a_s lam_{s+1} + Q_s x_s + K_s'(R u_s + B_s'lam_{s+1}),
// whose errors are propagated by the damped closed loop (A + B K)'.  It needs the gains only; the value matrices are not
// kept, which halves the workspace against lam_s = P_s x_s.
#pragma once

#include "layer_frag.cuh"
#include "riccati_frag.cuh"

namespace ttc {
namespace lgrad {

using namespace frag;

struct LayerGradParams {
    layer::LayerParams lp;       // inputs; g, u1; Kws [N][T][n][n]
    float* seq;                  // [N][4][T + 1][n]: x | xd | u | ud
    int* info;                   // [N]: status (failed instances give NaN gradients)
    float *d_sa, *d_ga, *d_gb, *d_gq, *d_ri, *d_h0;     // [N][n], each may be null
    float *d_sb, *d_sq, *d_sqf;                         // [N][r], each may be null
    float *GB, *GQ, *GF;         // [N][n][n] per-instance gradients of Bbar, Qbar, Q_T for the basis reduction, or null
};

template <int NB>
struct Tail {
    static constexpr int N = 8 * NB, LD = N + 4, STAGES = N == 16 ? 4 : 2;
    float B[N * LD], Q[N * LD], F[N * LD];          // rows of Bbar, Qbar, Q_T
    float K[STAGES][N * N];                         // ring of gains, chunks exchanged as in GradRing
    float v[8][N];                                  // vectors that travel between lanes
    float seq[STAGES][4 * N];                       // ring of x_s, xd_s, u_s, ud_s
};
template <int NB>
__host__ __device__ constexpr size_t warp_bytes()
{
    constexpr size_t a = sizeof(lfrag::Slot<NB>), b = sizeof(Tail<NB>);
    return ((a > b ? a : b) + 15) & ~size_t(15);
}

template <int NB>
__device__ __forceinline__ void store_ld(float* dst, const Mat<NB, NB>& x, int lane)
{
    constexpr int LD = Tail<NB>::LD;
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int mt = 0; mt < Mat<NB, NB>::MT; ++mt)
#pragma unroll
        for (int cb = 0; cb < NB; ++cb)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                *reinterpret_cast<float2*>(dst + (16 * mt + 8 * h + g) * LD + 8 * cb + 2 * t) =
                    make_float2(x.v[mt][cb][2 * h], x.v[mt][cb][2 * h + 1]);
}

// PART 0: everything; 1: the backward pass only; 2: the rest, from the gains, k_0 and status of a PART 1 launch
// (Persistent warps that take instance after instance through one slot of the workspace measured 4.19 against 3.90 ms.  Five
// CTAs per SM for the whole, 96 registers without spills: 3.89 -> 3.79 ms on 65536 instances of n = 16, T = 32.)
template <int NB, int PART>
__global__ void __launch_bounds__(32 * lfrag::MAX_WARPS, NB > 2 ? 2 : PART == 0 ? 5 : 4) layer_grad_kernel(LayerGradParams q)
{
    constexpr int N = 8 * NB, LPR = N <= 16 ? 2 : 1, W = N / LPR, LD = N + 4;
    using Ring = rfrag::GradRing<N>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const layer::LayerParams& p = q.lp;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, T = p.T, r = p.r;
    const int warp = NB > 2 ? (int)(threadIdx.x >> 5) : warp_index();       // (as in layer_frag_kernel)
    const long long inst = (long long)blockIdx.x * (blockDim.x >> 5) + warp;
    if (inst >= p.N)
        return;
    unsigned char* const mem = smem_raw + warp * warp_bytes<NB>();
    float* const Kg = p.Kws + inst * (long long)T * N * N;
    float k0[NB][2];                                        // first control of the dual problem, column form
    int fail;
    if constexpr (PART == 2) {
        fail = q.info[inst];
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const float2 k2 = *reinterpret_cast<const float2*>(p.k0 + inst * N + 8 * b + 2 * t);
            k0[b][0] = k2.x;
            k0[b][1] = k2.y;
        }
    } else {
        lfrag::Slot<NB>& sl = *reinterpret_cast<lfrag::Slot<NB>*>(mem);
        Mat<NB, NB> nP;
        lfrag::prepare<NB>(sl, nP, p, inst, lane);
        lfrag::Rates<NB> rates;
        rates.load(p, inst, lane);
        float rd[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            rd[b] = 1.f / __ldg(p.r_inv + inst * N + 8 * b + g);
            k0[b][0] = k0[b][1] = 0.f;
        }
        fail = lfrag::backward<NB, PART == 1>(nP, sl, rates, rd, T, lane, [&](int s, Mat<NB, NB>& Zt, const Mat<NB, NB>& S, const float(&w)[NB][2]) {
            if (s == 0) {
                float gv[NB], zc[NB][2];
#pragma unroll
                for (int b = 0; b < NB; ++b)
                    gv[b] = __ldg(p.g + inst * N + 8 * b + g);
                solve_vector<NB>(zc, k0, gv, S, w, lane);
            }
            gains<NB, NB>(Zt, S, w, lane);
            rfrag::store_gain<NB, NB, false>(Kg, (long long)s * N * N, Zt, N, N, 0, lane);
        });
    }
    if (PART != 2 && q.info && lane == 0)
        q.info[inst] = fail;
    if constexpr (PART == 1) {
        if (g == 0)
#pragma unroll
            for (int b = 0; b < NB; ++b)
                *reinterpret_cast<float2*>(p.k0 + inst * N + 8 * b + 2 * t) = make_float2(k0[b][0], k0[b][1]);
        return;
    }
    __syncwarp();                                           // gains stored by the other lanes are visible; the slot is free
    Tail<NB>& tl = *reinterpret_cast<Tail<NB>*>(mem);
    {
        Mat<NB, NB> B, Q, F;
        lfrag::synthesise<NB>(B, Q, F, p, inst, lane);
        store_ld<NB>(tl.B, B, lane);
        store_ld<NB>(tl.Q, Q, lane);
        store_ld<NB>(tl.F, F, lane);
    }
    // ---- forward: primal rollout from h_0, dual rollout from 0 with the first control k_0 (Prop. A.1, r_0 = g).  Row i
    // of every matrix and component i of every vector belong to LPR lanes.
    const int i = lane / LPR, c0 = (lane % LPR) * W;
    const bool writer = lane % LPR == 0;
    auto sum = [](float v) { return LPR == 2 ? v + __shfl_xor_sync(FULL, v, 1) : v; };
    auto part = [&](float (&v)[W], const float* src) { rfrag::load_part<W, false>(v, src, c0, N); };
    float* const X = q.seq + inst * (long long)(4 * (T + 1)) * N;         // x_s | xd_s | u_s | ud_s, (T + 1) rows of N each
    const long long SQ = (long long)(T + 1) * N;
    const float sa = __ldg(p.s_a + inst * N + i), ga = __ldg(p.s_ga + inst * N + i), gb = __ldg(p.s_gb + inst * N + i);
    const float gq = __ldg(p.s_gq + inst * N + i), rinv = __ldg(p.r_inv + inst * N + i), rdiag = 1.f / rinv;
    constexpr int ST = Tail<NB>::STAGES;
    auto stage_gain = [&](int k, int s) {
        if (s >= 0 && s < T)
            Ring::copy(tl.K[k % ST], Kg + (long long)s * N * N, lane);
    };
#pragma unroll
    for (int k = 0; k < ST - 1; ++k) {
        stage_gain(k, k);
        rfrag::commit_copies();
    }
    if (g == 0)
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            tl.v[4][8 * b + 2 * t] = k0[b][0];
            tl.v[4][8 * b + 2 * t + 1] = k0[b][1];
        }
    float xi = __ldg(p.h0 + inst * N + i), xdi = 0.f;
    if (writer) {
        tl.v[0][i] = xi;
        tl.v[1][i] = 0.f;
        X[i] = xi;
        X[SQ + i] = 0.f;
    }
    __syncwarp();
    const float k0i = tl.v[4][i];
    {
        float br[W];
        part(br, tl.B + i * LD);
#pragma unroll 1
        for (int s = 0; s < T; ++s) {
            rfrag::wait_copies<ST - 2>();
            stage_gain(s + ST - 1, s + ST - 1);
            rfrag::commit_copies();
            float kr[W], v[W], vd[W];
            part(v, tl.v[0]);
            part(vd, tl.v[1]);
            Ring::template row<W>(kr, tl.K[s % ST], i, c0);
            float us = 0.f, uds = 0.f, xs = 0.f, xds = 0.f;
#pragma unroll
            for (int k = 0; k < W; ++k) {
                us = fmaf(kr[k], v[k], us);
                uds = fmaf(kr[k], vd[k], uds);
            }
            us = sum(us);
            uds = sum(uds) + (s == 0 ? k0i : 0.f);
            const float tt = (float)(s + 1), gi = __expf(-tt * gb), ai = fmaf(__expf(-tt * ga), sa, 1.f);
            if (writer) {
                tl.v[2][i] = gi * us;
                tl.v[3][i] = gi * uds;
                X[2 * SQ + (long long)s * N + i] = us;
                X[3 * SQ + (long long)s * N + i] = uds;
                if (s == 0 && p.u1)
                    p.u1[inst * N + i] = fail ? quiet_nan() : us;
            }
            __syncwarp();
            part(v, tl.v[2]);
            part(vd, tl.v[3]);
#pragma unroll
            for (int k = 0; k < W; ++k) {
                xs = fmaf(br[k], v[k], xs);
                xds = fmaf(br[k], vd[k], xds);
            }
            xi = fmaf(ai, xi, sum(xs));                     // a_s x_s + Bbar (g .* u)
            xdi = fmaf(ai, xdi, sum(xds));
            if (writer) {
                tl.v[0][i] = xi;
                tl.v[1][i] = xdi;
                X[(long long)(s + 1) * N + i] = xi;
                X[SQ + (long long)(s + 1) * N + i] = xdi;
            }
            __syncwarp();
        }
    }
    // ---- backward: co-states of both problems, every outer product of Thm 3.2 reduced as it appears
    auto stage_bwd = [&](int k) {                           // k-th step backwards
        const int s = T - 1 - k;
        stage_gain(k, s);
        if (s >= 0 && lane < N)
            rfrag::copy16(tl.seq[k % ST] + 4 * lane, X + (lane / (N / 4)) * SQ + (long long)s * N + 4 * (lane % (N / 4)));
        rfrag::commit_copies();
    };
    rfrag::wait_copies<0>();
#pragma unroll
    for (int k = 0; k < ST - 1; ++k)
        stage_bwd(k);
    float dB[W], dQ[W], dF[W];                              // this lane's part of row i of the gradients of Bbar, Qbar, Q_T
    float d_sa = 0.f, d_ga = 0.f, d_gb = 0.f, d_gq = 0.f, d_ri = 0.f, lam = 0.f, lamd = 0.f;
    {
        float v[W], vd[W], fr[W];
        part(v, tl.v[0]);
        part(vd, tl.v[1]);
        part(fr, tl.F + i * LD);
#pragma unroll
        for (int k = 0; k < W; ++k) {
            lam = fmaf(fr[k], v[k], lam);                   // lam_T = Q_T x_T
            lamd = fmaf(fr[k], vd[k], lamd);
            dF[k] = 0.5f * (xi * vd[k] + xdi * v[k]);
            dB[k] = dQ[k] = 0.f;
        }
        lam = sum(lam);
        lamd = sum(lamd);
    }
    constexpr bool HOLD = NB <= 2;                          // row i of Qbar and column i of Bbar in registers
    float qrow[HOLD ? W : 1], bcol[HOLD ? W : 1];
    if constexpr (HOLD) {
        part(qrow, tl.Q + i * LD);
#pragma unroll
        for (int k = 0; k < W; ++k)
            bcol[k] = tl.B[(c0 + k) * LD + i];
    }
#pragma unroll 1
    for (int s = T - 1; s >= 0; --s) {
        const int k0s = T - 1 - s;
        rfrag::wait_copies<ST - 2>();                       // also: the vectors of the previous step are read
        stage_bwd(k0s + ST - 1);
        const float* sq = tl.seq[k0s % ST];
        const float tt = (float)(s + 1), ea = __expf(-tt * ga), gi = __expf(-tt * gb), ai = fmaf(ea, sa, 1.f);
        const float ei = s >= 1 ? __expf(-(float)s * gq) : 0.f;          // Q_0 = 0: no state cost at s = 0
        const float x = sq[i], xd = sq[N + i], u = sq[2 * N + i], ud = sq[3 * N + i];
        const float dA = fmaf(lam, xd, lamd * x);           // dA_s[i][i]
        d_sa = fmaf(ea, dA, d_sa);
        d_ga = fmaf(-tt * ea * sa, dA, d_ga);
        d_ri = fmaf(-u, ud, d_ri);
        if (writer) {
            tl.v[0][i] = lam;
            tl.v[1][i] = lamd;
            tl.v[2][i] = gi * u;
            tl.v[3][i] = gi * ud;
            tl.v[4][i] = ei * x;
            tl.v[5][i] = ei * xd;
        }
        __syncwarp();
        float v[W], vd[W];
        part(v, tl.v[0]);
        part(vd, tl.v[1]);
        float bl = 0.f, bld = 0.f;                          // (Bbar'lam)[i], (Bbar'lamd)[i]
#pragma unroll
        for (int k = 0; k < W; ++k) {
            float b;
            if constexpr (HOLD)
                b = bcol[k];
            else
                b = tl.B[(c0 + k) * LD + i];
            bl = fmaf(b, v[k], bl);
            bld = fmaf(b, vd[k], bld);
        }
        bl = sum(bl);
        bld = sum(bld);
        d_gb = fmaf(-tt * gi, fmaf(ud, bl, u * bld), d_gb);
        part(v, tl.v[2]);
        part(vd, tl.v[3]);
#pragma unroll
        for (int k = 0; k < W; ++k)
            dB[k] += fmaf(lam, vd[k], lamd * v[k]);
        if (s >= 1) {
            part(v, tl.v[4]);
            part(vd, tl.v[5]);
            float qx = 0.f, qxd = 0.f;                      // (Q_s x_s)[i], (Q_s xd_s)[i]
            const float h = 0.5f * ei;
            if constexpr (!HOLD) {
#pragma unroll
                for (int k4 = 0; k4 < W / 4; ++k4) {
                    const float4 f = *reinterpret_cast<const float4*>(tl.Q + i * LD + c0 + 4 * k4);
                    qx = fmaf(f.x, v[4 * k4], qx); qx = fmaf(f.y, v[4 * k4 + 1], qx);
                    qx = fmaf(f.z, v[4 * k4 + 2], qx); qx = fmaf(f.w, v[4 * k4 + 3], qx);
                    qxd = fmaf(f.x, vd[4 * k4], qxd); qxd = fmaf(f.y, vd[4 * k4 + 1], qxd);
                    qxd = fmaf(f.z, vd[4 * k4 + 2], qxd); qxd = fmaf(f.w, vd[4 * k4 + 3], qxd);
                }
            }
#pragma unroll
            for (int k = 0; k < W; ++k) {
                if constexpr (HOLD) {
                    qx = fmaf(qrow[k], v[k], qx);
                    qxd = fmaf(qrow[k], vd[k], qxd);
                }
                dQ[k] = fmaf(h, fmaf(x, vd[k], xd * v[k]), dQ[k]);
            }
            qx = ei * sum(qx);
            qxd = ei * sum(qxd);
            d_gq = fmaf(-(float)s, fmaf(x, qxd, xd * qx), d_gq);
            if (writer) {                                   // R u_s + B_s'lam_{s+1}: zero but for rounding
                tl.v[6][i] = fmaf(gi, bl, rdiag * u);
                tl.v[7][i] = fmaf(gi, bld, rdiag * ud);
            }
            __syncwarp();
            part(v, tl.v[6]);
            part(vd, tl.v[7]);
            float kw = 0.f, kwd = 0.f;
#pragma unroll
            for (int k = 0; k < W; ++k) {
                const float kk = Ring::at(tl.K[k0s % ST], c0 + k, i);
                kw = fmaf(kk, v[k], kw);
                kwd = fmaf(kk, vd[k], kwd);
            }
            lam = fmaf(ai, lam, qx + sum(kw));
            lamd = fmaf(ai, lamd, qxd + sum(kwd));
        } else {
            lamd = ai * lamd;                               // lamd_0 = A_1'lamd_1 (Q_0 = 0, xd_0 = 0): the gradient of h_0
        }
    }
    rfrag::wait_copies<0>();
    d_ri *= rdiag * rdiag;
    // ---- outputs; contraction of the three matrices with the bases
    const float qn = quiet_nan();
    if (writer) {
        const long long o = inst * N + i;
        if (q.d_sa) q.d_sa[o] = fail ? qn : d_sa;
        if (q.d_ga) q.d_ga[o] = fail ? qn : d_ga;
        if (q.d_gb) q.d_gb[o] = fail ? qn : d_gb;
        if (q.d_gq) q.d_gq[o] = fail ? qn : d_gq;
        if (q.d_ri) q.d_ri[o] = fail ? qn : d_ri;
        if (q.d_h0) q.d_h0[o] = fail ? qn : lamd;
    }
    if (q.GB) {
        // (NaN of a failed instance must not meet the zero coefficient that the reduction gives it)
        const long long o = (inst * N + i) * N + c0;
#pragma unroll
        for (int k = 0; k < W; k += 4) {
            *reinterpret_cast<float4*>(q.GB + o + k) = fail ? make_float4(0.f, 0.f, 0.f, 0.f) : make_float4(dB[k], dB[k + 1], dB[k + 2], dB[k + 3]);
            *reinterpret_cast<float4*>(q.GQ + o + k) = fail ? make_float4(0.f, 0.f, 0.f, 0.f) : make_float4(dQ[k], dQ[k + 1], dQ[k + 2], dQ[k + 3]);
            *reinterpret_cast<float4*>(q.GF + o + k) = fail ? make_float4(0.f, 0.f, 0.f, 0.f) : make_float4(dF[k], dF[k + 1], dF[k + 2], dF[k + 3]);
        }
    }
    if (q.d_sb || q.d_sq || q.d_sqf) {
#pragma unroll 1
        for (int k = 0; k < r; ++k) {
            const float4* Bk = reinterpret_cast<const float4*>(p.B_basis + (long long)k * N * N + i * N + c0);
            const float4* Qk = reinterpret_cast<const float4*>(p.Q_basis + (long long)k * N * N + i * N + c0);
            float pb = 0.f, pq = 0.f, pf = 0.f;
#pragma unroll
            for (int c = 0; c < W / 4; ++c) {
                const float4 b4 = __ldg(Bk + c), q4 = __ldg(Qk + c);
                const float bb[4] = {b4.x, b4.y, b4.z, b4.w}, qq[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    pb = fmaf(dB[4 * c + e], bb[e], pb);
                    pq = fmaf(dQ[4 * c + e], qq[e], pq);
                    pf = fmaf(dF[4 * c + e], qq[e], pf);
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                pb += __shfl_xor_sync(FULL, pb, o);
                pq += __shfl_xor_sync(FULL, pq, o);
                pf += __shfl_xor_sync(FULL, pf, o);
            }
            if (lane == 0) {
                if (q.d_sb) q.d_sb[inst * r + k] = fail ? qn : pb;
                if (q.d_sq) q.d_sq[inst * r + k] = fail ? qn : pq;
                if (q.d_sqf) q.d_sqf[inst * r + k] = fail ? qn : pf;
            }
        }
    }
}

// dBasis[k][e] += sum over instances of coef[i][k] * G[i][e]: a product with the instances as the long dimension.  A CTA
// takes 256 elements (two per thread) and 16 coefficients; the coefficients of 64 instances at a
// time sit in shared memory, so that a 16-byte broadcast feeds eight multiply-adds (one broadcast load per multiply-add
// before).  Partial sums of the CTAs meet in float atomics.  Up to two (coefficient, matrix) pairs go to the same
// destination (Q^(k) collects s_Q[k] dQbar and s_Qf[k] dQ_T).
constexpr int RED_THREADS = 128, RED_INST = 64, RED_K = 16;
__global__ void __launch_bounds__(RED_THREADS) basis_reduce_kernel(long long N, int r, int nn, const int* info, const float* c0, const float* G0,
                                                                   const float* c1, const float* G1, float* dst)
{
    __shared__ __align__(16) float coef[2][RED_INST][RED_K];
    const int e = (blockIdx.y * RED_THREADS + threadIdx.x) * 2, k0 = blockIdx.z * RED_K;
    const long long per = (N + gridDim.x - 1) / gridDim.x;
    const long long i0 = per * blockIdx.x, i1 = i0 + per < N ? i0 + per : N;
    float acc[RED_K][2];
#pragma unroll
    for (int k = 0; k < RED_K; ++k)
        acc[k][0] = acc[k][1] = 0.f;
    for (long long ib = i0; ib < i1; ib += RED_INST) {
        const int cnt = (int)(i1 - ib < RED_INST ? i1 - ib : RED_INST);
        __syncthreads();
        for (int j = threadIdx.x; j < RED_INST * RED_K; j += RED_THREADS) {
            const int ii = j / RED_K, k = j % RED_K;
            const bool ok = ii < cnt && k0 + k < r && info[ib + ii] == 0;       // failed instances count for nothing
            coef[0][ii][k] = ok ? __ldg(c0 + (ib + ii) * r + k0 + k) : 0.f;
            coef[1][ii][k] = ok && c1 ? __ldg(c1 + (ib + ii) * r + k0 + k) : 0.f;
        }
        __syncthreads();
#pragma unroll 1
        for (int m = 0; m < (G1 ? 2 : 1); ++m) {
            const float* G = (m ? G1 : G0) + ib * nn + e;
#pragma unroll 4
            for (int ii = 0; ii < cnt; ++ii) {
                const float2 v = __ldcs(reinterpret_cast<const float2*>(G + (long long)ii * nn));
#pragma unroll
                for (int q4 = 0; q4 < RED_K / 4; ++q4) {
                    const float4 c = *reinterpret_cast<const float4*>(&coef[m][ii][4 * q4]);
                    acc[4 * q4][0] = fmaf(c.x, v.x, acc[4 * q4][0]);
                    acc[4 * q4][1] = fmaf(c.x, v.y, acc[4 * q4][1]);
                    acc[4 * q4 + 1][0] = fmaf(c.y, v.x, acc[4 * q4 + 1][0]);
                    acc[4 * q4 + 1][1] = fmaf(c.y, v.y, acc[4 * q4 + 1][1]);
                    acc[4 * q4 + 2][0] = fmaf(c.z, v.x, acc[4 * q4 + 2][0]);
                    acc[4 * q4 + 2][1] = fmaf(c.z, v.y, acc[4 * q4 + 2][1]);
                    acc[4 * q4 + 3][0] = fmaf(c.w, v.x, acc[4 * q4 + 3][0]);
                    acc[4 * q4 + 3][1] = fmaf(c.w, v.y, acc[4 * q4 + 3][1]);
                }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < RED_K; ++k)
        if (k0 + k < r) {
            atomicAdd(dst + (long long)(k0 + k) * nn + e, acc[k][0]);
            atomicAdd(dst + (long long)(k0 + k) * nn + e + 1, acc[k][1]);
        }
}
inline cudaError_t launch_basis_reduce(long long N, int r, int nn, const int* info, const float* c0, const float* G0, const float* c1, const float* G1,
                                       float* dst, int sm_count, cudaStream_t st)
{
    // nn is 256 or 1024: one CTA covers 256 elements; about 8 CTAs per SM over slices of at least 16 instances
    const unsigned ny = nn / (2 * RED_THREADS), nz = (r + RED_K - 1) / RED_K;
    long long nx = (long long)sm_count * 8 / (ny * nz);
    if (nx > (N + 15) / 16) nx = (N + 15) / 16;
    if (nx < 1) nx = 1;
    basis_reduce_kernel<<<dim3((unsigned)nx, ny, nz), RED_THREADS, 0, st>>>(N, r, nn, info, c0, G0, c1, G1, dst);
    return cudaGetLastError();
}

template <int NB, int PART>
inline cudaError_t launch_part(const LayerGradParams& q, int warps, cudaStream_t st)
{
    const size_t smem = warp_bytes<NB>() * warps;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(layer_grad_kernel<NB, PART>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess)
            return e;
    }
    layer_grad_kernel<NB, PART><<<(unsigned)((q.lp.N + warps - 1) / warps), 32 * warps, smem, st>>>(q);
    return cudaGetLastError();
}
// One kernel for batches that fill the machine: its phases are bound by different units and overlap across warps.  With
// at most four instances per SM there is nothing to overlap with and the two parts stay separate launches.
template <int NB>
inline cudaError_t launch_layer_grad(const LayerGradParams& q, int sm_count, cudaStream_t st, int* launches)
{
    if (q.lp.N > 4ll * sm_count) {
        *launches = 1;
        return launch_part<NB, 0>(q, NB > 2 ? 1 : lfrag::MAX_WARPS, st);
    }
    *launches = 2;
    const cudaError_t e = launch_part<NB, 1>(q, 1, st);
    return e ? e : launch_part<NB, 2>(q, 1, st);
}

} // namespace lgrad
} // namespace ttc
