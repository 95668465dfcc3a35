// Scan over the horizon for n = m = 16 / 32, time-invariant problems.
//
// Element of the scan: the symplectic transition matrix of Thm A.2 kept inverse-free as e = (A, G, J) with C = G G'
// (C = B R^{-1} B', J = Q for one step).  Both of its operations are Riccati-type steps whose only solve is a Cholesky
// factorisation of S = I + G'(.)G >= I:
//     apply(e, P) = J + A'P A - Y'S^{-1}Y,   Y = G'P A                     (Prop. 3.1 with B = G, R = I, Q = J)
//     e o e :  S = I + G'J G = L L',  Z = L^{-1} G'J A,  U = A G L^{-T}
//              A2 = A A - U Z,   J2 = J + A'J A - Z'Z,   C2 = C + U U',   G2 = chol(C2)
// (with W = (I + C J)^{-1}: A W A = A A - U Z by Woodbury, and W C = G S^{-1} G', so C2 is a sum of squares).
//
// The horizon is cut into pieces of L = 2^k steps, L near sqrt(H):
//   power    one warp per instance squares the element k times: e^L
//   tail     the H mod L last steps give the value matrix at the last boundary (absent when L divides H)
//   coarse   the boundaries are themselves an LQR problem with A = A_L, B = G_L, R = I, Q = J_L over H / L steps: the
//            recursion kernel gives the value matrix AND the state at every boundary
//   pieces   every piece is then an independent problem of L steps: the recursion kernel again, N H / L warps
//   finish   status words, NaN fill of failed instances
// The chain of an instance is about k squarings + H/L + L steps instead of H, and the work about 1.1 times the
// recursion's.  64 instances, n = 16, H = 1024: see the launcher.
#pragma once

#include "riccati_dispatch.cuh"

namespace ttc {
namespace scanf {

using namespace frag;

template <int NB>
struct PowerMem {
    Stored<NB, NB> At, A, Gt;                       // A', A, G' split, in register order
    float C[(NB + 1) / 2][NB][4][32];
};

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
template <int NB>
__device__ __forceinline__ void store_rows(float* dst, const Mat<NB, NB>& x, int lane)
{
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int mt = 0; mt < Mat<NB, NB>::MT; ++mt)
#pragma unroll
        for (int cb = 0; cb < NB; ++cb)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                *reinterpret_cast<float2*>(dst + (16 * mt + 8 * h + g) * 8 * NB + 8 * cb + 2 * t) =
                    make_float2(x.v[mt][cb][2 * h], x.v[mt][cb][2 * h + 1]);
}
// matrix in global memory, any element stride alignment
template <int NB>
__device__ __forceinline__ void load_rows(Mat<NB, NB>& x, const OperandDev& o, long long off, int lane)
{
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int mt = 0; mt < Mat<NB, NB>::MT; ++mt)
#pragma unroll
        for (int cb = 0; cb < NB; ++cb)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                x.v[mt][cb][e] = load_elem(o, off + (16 * mt + g + ((e & 2) ? 8 : 0)) * 8 * NB + 8 * cb + 2 * t + (e & 1));
}
template <int NB>
__device__ __forceinline__ void negate(Mat<NB, NB>& y, const Mat<NB, NB>& x)
{
#pragma unroll
    for (int mt = 0; mt < Mat<NB, NB>::MT; ++mt)
#pragma unroll
        for (int cb = 0; cb < NB; ++cb)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                y.v[mt][cb][e] = -x.v[mt][cb][e];
}

// Lower factor of a positive SEMI-definite matrix (nC = -C, lower tiles; destroyed): a pivot that is not larger than
// `tiny` gives a zero column (the matrix has no weight in that direction).  Never fails; NaN input gives NaN output.
template <int NB>
__device__ __forceinline__ void factor_psd(Mat<NB, NB>& G, Mat<NB, NB>& nC, float tiny, int lane)
{
    constexpr int MT = Mat<NB, NB>::MT;
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int p = 0; p < NB; ++p) {
        float a0 = -nC.v[p / 2][p][2 * (p & 1)], a1 = -nC.v[p / 2][p][2 * (p & 1) + 1];
#pragma unroll
        for (int j = 0; j < 7; ++j) {                       // as chol8_inverse, with the pivot test
            const float sel = (j & 1) ? a1 : a0;
            const float d = __shfl_sync(FULL, sel, 4 * j + (j >> 1));
            const float col = __shfl_sync(FULL, sel, (lane & 28) | (j >> 1));
            const float r0 = __shfl_sync(FULL, a0, 4 * j + t), r1 = __shfl_sync(FULL, a1, 4 * j + t);
            const float f = (g > j && d > tiny) ? -col * rcp_fast(d) : 0.f;
            a0 = fmaf(f, r0, a0);
            a1 = fmaf(f, r1, a1);
            if (g > j && t == (j >> 1)) {
                if (j & 1)
                    a1 = f;
                else
                    a0 = f;
            }
        }
        const float dg = __shfl_sync(FULL, (g & 1) ? a1 : a0, (lane & 28) | (g >> 1));
        const float rs = dg > tiny ? rsqrtf(dg) : dg <= tiny ? 0.f : dg;       // NaN stays
        a0 = (2 * t < g ? a0 : 2 * t == g ? 1.f : 0.f) * rs;
        a1 = (2 * t + 1 < g ? a1 : 2 * t + 1 == g ? 1.f : 0.f) * rs;
        uint32_t h0, h1, l0, l1;
        split2(-a0, -a1, h0, h1, l0, l1);
        Tile lt[MT];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            float d[4] = {0.f, 0.f, 0.f, 0.f};
            if (mt >= p / 2) {
                Tile x;
                split_tile(x, nC.v[mt][p]);
                mma3(d, x, h0, h1, l0, l1, true);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int b = 2 * mt + (e >> 1);
                // nothing above the diagonal: whole blocks, and the upper half of the diagonal one
                G.v[mt][p][e] = b < p || (b == p && 2 * t + (e & 1) > g) ? 0.f : d[e];
                d[e] = b <= p ? 0.f : d[e];
            }
            split_tile(lt[mt], d);
        }
#pragma unroll
        for (int q = 1; q < NB; ++q) {
            if (q <= p)
                continue;
            const int e = 2 * (q & 1);
            const Tile y = lt[q / 2];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
                if (mt >= q / 2)
                    mma3(nC.v[mt][q], lt[mt], y.h[e], y.h[e + 1], y.l[e], y.l[e + 1]);
        }
    }
}

// e^(2^squarings) of every instance: elem [N][3][n][n] = A | G | J; eye [n][n] receives the identity (R of the coarse
// problem); fail [N].
template <int NB>
__global__ void __launch_bounds__(32) scan_power_kernel(SolveParams p, int squarings, float* elem, float* eye, int* fail)
{
    constexpr int N = 8 * NB, MT = Mat<NB, NB>::MT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PowerMem<NB>& mem = *reinterpret_cast<PowerMem<NB>*>(smem_raw);
    const int lane = threadIdx.x & 31;
    const rfrag::Place pl = rfrag::place(p, blockIdx.x);
    if (blockIdx.x == 0)
        for (int e = lane; e < N * N; e += 32)
            eye[e] = e / N == e % N ? 1.f : 0.f;
    int bad = 0;
    Mat<NB, NB> J, G;                                       // J positive; G in the end
    {
        Mat<NB, NB> A, At, B, S;
        load_rows<NB>(A, p.A, pl.off(p.A), lane);
        transpose<NB>(At, A, lane);
        keep(mem.A, A, lane);
        keep(mem.At, At, lane);
        load_rows<NB>(J, p.Q, pl.off(p.Q), lane);
        load_rows<NB>(B, p.B, pl.off(p.B), lane);
        load_rows<NB>(S, p.R, pl.off(p.R), lane);
        negate<NB>(S, S);
        negate<NB>(G, B);
        Split<NB, NB> gs;
        float w[NB][2];
        bad = factor<NB, NB, true>(S, G, gs, w, lane);            // G = B L_R^{-T}
        Mat<NB, NB> Gt, C;
        transpose<NB>(Gt, G, lane);
        keep(mem.Gt, Gt, lane);
        product<NB, NB, NB>(C, nullptr, gs, gs);            // C = G G'
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int cb = 0; cb < NB; ++cb)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    mem.C[mt][cb][e][lane] = C.v[mt][cb][e];
        __syncwarp();
    }
#pragma unroll 1
    for (int k = 0; k < squarings; ++k) {
        Mat<NB, NB> S;
        Mat<2 * NB, NB> rhs;                                // -Y' over -A G; then Z' over U
        {
            Mat<NB, NB> V, T, AG;
            {
                Split<NB, NB> js;
                split(js, J);
                product<NB, NB, NB>(V, nullptr, mem.Gt, js, lane);      // V = G'J
                product<NB, NB, NB>(T, nullptr, mem.At, js, lane);      // T = A'J
            }
            {
                Split<NB, NB> vs;
                split(vs, V);
                product<NB, NB, NB>(S, nullptr, mem.Gt, vs, lane);      // G'J G
                product<NB, NB, NB>(V, nullptr, mem.At, vs, lane);      // Y' = A'J G
            }
            {
                Split<NB, NB> ts;
                split(ts, T);
                negate<NB>(J, J);
                product<NB, NB, NB>(T, nullptr, mem.At, ts, lane);      // A'J A
            }
            {
                Mat<NB, NB> Gt;
                unkeep(Gt, mem.Gt, lane);
                Split<NB, NB> gs;
                split(gs, Gt);
                product<NB, NB, NB>(AG, nullptr, mem.A, gs, lane);      // A G
            }
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int cb = 0; cb < NB; ++cb)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        J.v[mt][cb][e] -= T.v[mt][cb][e];               // -J - A'J A
                        rhs.v[mt][cb][e] = -V.v[mt][cb][e];
                        rhs.v[mt + MT][cb][e] = -AG.v[mt][cb][e];
                        const int g = lane >> 2, t = lane & 3, b = 2 * mt + (e >> 1);
                        S.v[mt][cb][e] = -S.v[mt][cb][e] - (cb == b && t == (g >> 1) && (e & 1) == (g & 1) ? 1.f : 0.f);
                    }
        }
        Split<2 * NB, NB> zs;
        float w[NB][2];
        const int b = factor<2 * NB, NB, true>(S, rhs, zs, w, lane);
        if (b && !bad)
            bad = b;
        Split<NB, NB> us, z1;                               // U and Z'
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int cb = 0; cb < NB; ++cb)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    z1.h[mt][cb][e] = zs.h[mt][cb][e];
                    z1.l[mt][cb][e] = zs.l[mt][cb][e];
                    us.h[mt][cb][e] = zs.h[mt + MT][cb][e];
                    us.l[mt][cb][e] = zs.l[mt + MT][cb][e];
                }
        product<NB, NB, NB>(J, &J, z1, z1);                 // -J2 = -J - A'J A + Z'Z
        make_symmetric<NB>(J, lane);
        negate<NB>(J, J);
        Mat<NB, NB> A2, UZ;
        product<NB, NB, NB>(UZ, nullptr, us, z1);           // U Z
        {
            Mat<NB, NB> At;
            unkeep(At, mem.At, lane);
            Split<NB, NB> as;
            split(as, At);
            product<NB, NB, NB>(A2, nullptr, mem.A, as, lane);          // A A
        }
        Mat<NB, NB> C;
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int cb = 0; cb < NB; ++cb)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    A2.v[mt][cb][e] -= UZ.v[mt][cb][e];
                    C.v[mt][cb][e] = mem.C[mt][cb][e][lane];
                }
        product<NB, NB, NB>(C, &C, us, us);                 // C2 = C + U U'
        make_symmetric<NB>(C, lane);
        __syncwarp();
        float dmax = 0.f;
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int cb = 0; cb < NB; ++cb)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    mem.C[mt][cb][e][lane] = C.v[mt][cb][e];
                    const int g = lane >> 2, t = lane & 3, bb = 2 * mt + (e >> 1);
                    if (cb == bb && t == (g >> 1) && (e & 1) == (g & 1))
                        dmax = fmaxf(dmax, C.v[mt][cb][e]);
                }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            dmax = fmaxf(dmax, __shfl_xor_sync(FULL, dmax, o));
        negate<NB>(C, C);
        factor_psd<NB>(G, C, 1e-7f * dmax, lane);
        {
            Mat<NB, NB> t;
            keep(mem.A, A2, lane);
            transpose<NB>(t, A2, lane);
            keep(mem.At, t, lane);
            transpose<NB>(t, G, lane);
            keep(mem.Gt, t, lane);
        }
        __syncwarp();
    }
    float* E = elem + pl.inst * (3 * N * N);
    {
        Mat<NB, NB> A;
        unkeep(A, mem.A, lane);
        store_rows<NB>(E, A, lane);
    }
    store_rows<NB>(E + N * N, G, lane);
    store_rows<NB>(E + 2 * N * N, J, lane);
    if (lane == 0)
        fail[pl.inst] = bad;
}

// Status of every instance from the words of its stages; a failed instance loses its outputs.
__global__ void __launch_bounds__(128) scan_finish_kernel(SolveParams p, const int* stage_fail, int stages, const int* piece_fail, int pieces)
{
    const int lane = threadIdx.x & 31;
    const long long w = (long long)blockIdx.x * 4 + (threadIdx.x >> 5);
    if (w >= p.b0 * p.b1 * p.tcount)
        return;
    const long long inst = rfrag::place(p, (unsigned)w).inst;
    int bad = 0;
    for (int k = lane; k < stages; k += 32)
        bad = max(bad, stage_fail[k * p.N + inst]);
    for (int k = lane; k < pieces; k += 32)
        bad = max(bad, piece_fail[w * pieces + k]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        bad = max(bad, __shfl_xor_sync(FULL, bad, o));
    if (p.info && lane == 0)
        p.info[inst] = bad;
    if (!bad)
        return;
    const float qn = quiet_nan();
    const long long n = p.n, m = p.m, H = p.H;
    auto fill = [&](float* base, long long cnt) {
        if (base)
            for (long long e = lane; e < cnt; e += 32)
                base[inst * cnt + e] = qn;
    };
    fill(p.K, H * m * n);
    fill(p.P, (p.first_only ? 1 : H + 1) * n * n);
    fill(p.x, (H + 1) * n);
    fill(p.u, p.first_only ? m : H * m);
}

// Sizes of the stages for a horizon of H steps.
struct Cut {
    int squarings, len, coarse, tail;
};
// The chain is about 2 squarings' worth per doubling of L, plus H / L + L steps: L = 2^k nearest to sqrt(H).  Horizons
// below eight steps are one piece (the plain recursion).
inline Cut cut_horizon(int H)
{
    Cut c = {0, H, 0, 0};
    if (H < 8)
        return c;
    while ((2ll << c.squarings) * (1ll << c.squarings) < H)            // L^2 < H / 2  ->  double
        ++c.squarings;
    c.len = 1 << c.squarings;
    c.coarse = H / c.len;
    c.tail = H - c.coarse * c.len;
    return c;
}
// floats per launch of the handle's element workspace for N instances of n states
inline size_t workspace_floats(long long N, int n, int H)
{
    const Cut c = cut_horizon(H);
    const size_t nn = (size_t)n * n;
    return nn + (size_t)N * (3 * nn + nn + (c.coarse + 1) * (nn + n) + c.coarse * nn);
}
inline size_t flag_words(long long N, int H)
{
    const Cut c = cut_horizon(H);
    return (size_t)N * (3 + c.coarse + 1);
}

// p.Kws holds the gains when the rollout needs them and K is not wanted.
template <int NB>
inline cudaError_t launch_scan_frag(const SolveParams& p, float* ws, int* flags, bool exact, int sm_count, cudaStream_t st, int* launches)
{
    constexpr int N = 8 * NB;
    const Cut c = cut_horizon(p.H);
    const long long nwin = p.b0 * p.b1 * p.tcount, nn = N * N;
    cudaError_t e;
    *launches = 0;
    SolveParams q = p;
    q.Qf.ptr = nullptr;
    if (c.coarse == 0) {                                    // one piece
        *launches = 1;
        return rfrag::launch_riccati_frag(p, false, false, exact, sm_count, st);
    }
    float* eye = ws;
    float* elem = eye + nn;
    float* tailP = elem + p.N * 3 * nn;
    float* Pc = tailP + p.N * nn;
    float* Kc = Pc + p.N * (c.coarse + 1) * nn;
    float* xc = Kc + p.N * c.coarse * nn;
    int* stage = flags;                                     // power | coarse | tail
    int* piece = flags + 3 * p.N;
    const size_t smem = sizeof(PowerMem<NB>);
    if (smem > 48 * 1024 &&
        (e = cudaFuncSetAttribute(scan_power_kernel<NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem))) return e;
    scan_power_kernel<NB><<<(unsigned)nwin, 32, smem, st>>>(p, c.squarings, elem, eye, stage);
    if ((e = cudaGetLastError())) return e;
    ++*launches;
    if (c.tail) {
        q.H = c.tail;
        q.K = q.x = q.u = q.Kws = nullptr;
        q.P = tailP;
        q.info = stage + 2 * p.N;
        q.first_only = 1;
        if ((e = rfrag::launch_riccati_frag(q, false, false, exact, sm_count, st))) return e;
        ++*launches;
    }
    const bool rollout = p.x || p.u, need_all = p.K || p.x || (p.u && !p.first_only) || (p.P && !p.first_only);
    auto dense = [&](const float* ptr, long long stride) {
        OperandDev o;
        o.ptr = ptr; o.dtype = TTC_F32; o.st = 0;
        o.s2 = stride; o.s1 = stride * p.b2; o.s0 = o.s1 * p.b1;
        return o;
    };
    q = p;
    q.H = c.coarse;
    q.A = dense(elem, 3 * nn);
    q.B = dense(elem + nn, 3 * nn);
    q.Q = dense(elem + 2 * nn, 3 * nn);
    q.R = dense(eye, 0);
    q.Qf = c.tail ? dense(tailP, nn) : p.Q;
    q.Qf.st = 0;
    q.K = nullptr;
    q.Kws = rollout ? Kc : nullptr;
    q.P = Pc;
    q.x = rollout && need_all ? xc : nullptr;
    q.u = nullptr;
    q.info = stage + p.N;
    q.first_only = 0;
    q.n = q.m = N;
    if ((e = rfrag::launch_riccati_frag(q, true, false, exact, sm_count, st))) return e;
    ++*launches;
    q = p;
    q.chunk_len = c.len;
    q.coarse = c.coarse;
    q.chunks = need_all ? c.coarse + (c.tail ? 1 : 0) : 1;
    q.Pc = Pc;
    q.xc = rollout && need_all ? xc : nullptr;
    q.piece_info = piece;
    if (!need_all)                                          // only P_0 / u_0: a horizon that ends at the first boundary
        q.H = c.len;
    if ((e = exact ? rfrag::launch_one<NB, NB, false, false, false, true>(q, sm_count, st)
                   : rfrag::launch_one<NB, NB, false, false, true, true>(q, sm_count, st))) return e;
    ++*launches;
    scan_finish_kernel<<<(unsigned)((nwin + 3) / 4), 128, 0, st>>>(p, stage, c.tail ? 3 : 2, piece, q.chunks);
    if ((e = cudaGetLastError())) return e;
    ++*launches;
    return cudaSuccess;
}

} // namespace scanf
} // namespace ttc
