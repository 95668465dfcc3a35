// Which variant of the one-warp recursion (riccati_frag.cuh) a request takes.
#pragma once

#include "riccati_frag.cuh"

namespace ttc {
namespace rfrag {

// Sizes this kernel serves: up to 32 x 32 for every request, all of them for time-invariant ones.
inline bool riccati_frag_serves(int n, int m, bool time_varying)
{
    return !time_varying || (n <= 32 && m <= 32);
}

// Most variants are instantiated in sources of their own (riccati_frag_*.cu), which compile beside the rest.
cudaError_t launch_affine(const SolveParams& p, int kb, bool full16, bool full32, int sm_count, cudaStream_t st);
cudaError_t launch_time_varying(const SolveParams& p, int kb, bool full16, bool full32, int sm_count, cudaStream_t st);
cudaError_t launch_blocks_3_4(const SolveParams& p, int kb, int mb, bool full32, int sm_count, cudaStream_t st);
cudaError_t launch_blocks_5(const SolveParams& p, int mb, int sm_count, cudaStream_t st);
cudaError_t launch_blocks_6(const SolveParams& p, int mb, int sm_count, cudaStream_t st);
cudaError_t launch_blocks_8_wide(const SolveParams& p, int mb, int sm_count, cudaStream_t st);
cudaError_t launch_blocks_8(const SolveParams& p, int mb, int sm_count, cudaStream_t st);

// `exact`: the strides keep the vector loads aligned (rows of Q, Qf, R and of K, A, B in the rollout).
// Time-invariant requests: a step's products are linear in the number of control blocks, so every number of them has a
// variant up to five blocks of states, and every even one above, where the numbers of state blocks are even too (registers
// spill there, and a variant takes several seconds to compile).  1155 instances of 20 steps, padded to the next variant ->
// with their own: n = 24, m = 12 148 -> 111 us, n = 32, m = 20 266 -> 225, n = 40, m = 28 1090 -> 812, n = 56, m = 48 from
// 10.7 to 6.6 ms.
inline cudaError_t launch_riccati_frag(const SolveParams& p, bool time_varying, bool affine, bool exact, int sm_count, cudaStream_t st)
{
    const int nb = (p.n + 7) / 8, mb = (p.m + 7) / 8, kb = nb > mb ? nb : mb;
    const bool full16 = exact && p.n == 16 && p.m == 16, full32 = exact && p.n == 32 && p.m == 32;
    if (affine)
        return launch_affine(p, kb, full16, full32, sm_count, st);
    if (time_varying)
        return launch_time_varying(p, kb, full16, full32, sm_count, st);
    switch (kb) {
    case 1:
        return exact && p.n == 8 && p.m == 8 ? launch_one<1, 1, false, false, false>(p, sm_count, st)
                                             : launch_one<1, 1, false, false, true>(p, sm_count, st);
    case 2:
        return full16 ? launch_one<2, 2, false, false, false>(p, sm_count, st)
             : mb == 1 ? launch_one<2, 1, false, false, true>(p, sm_count, st) : launch_one<2, 2, false, false, true>(p, sm_count, st);
    case 3:
    case 4:
        return launch_blocks_3_4(p, kb, mb, full32, sm_count, st);
    case 5:
        return launch_blocks_5(p, mb, sm_count, st);
    case 6:
        return launch_blocks_6(p, mb, sm_count, st);
    default:
        return mb <= 4 ? launch_blocks_8(p, mb, sm_count, st) : launch_blocks_8_wide(p, mb, sm_count, st);
    }
}

// Gradients of the first control, everything in one kernel: n = m = 16 / 32, float32 operands with aligned strides.
cudaError_t launch_grad_frag(const SolveParams& p, int sm_count, cudaStream_t st);

} // namespace rfrag
} // namespace ttc
