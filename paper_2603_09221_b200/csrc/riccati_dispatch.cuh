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

// The variants of five, six and eight blocks of states take half of the build time: they are instantiated in sources of their
// own (riccati_frag_5_6.cu, riccati_frag_8.cu), which compile beside the rest.
cudaError_t launch_blocks_5_6(const SolveParams& p, int kb, int mb, int sm_count, cudaStream_t st);
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
    if (affine) {
        if (kb <= 2)
            return full16 ? launch_one<2, 2, true, true, false>(p, sm_count, st) : launch_one<2, 2, true, true, true>(p, sm_count, st);
        return full32 ? launch_one<4, 4, true, true, false>(p, sm_count, st) : launch_one<4, 4, true, true, true>(p, sm_count, st);
    }
    if (time_varying) {
        if (kb <= 2)
            return full16 ? launch_one<2, 2, true, false, false>(p, sm_count, st) : launch_one<2, 2, true, false, true>(p, sm_count, st);
        return full32 ? launch_one<4, 4, true, false, false>(p, sm_count, st) : launch_one<4, 4, true, false, true>(p, sm_count, st);
    }
    switch (kb) {
    case 1:
        return exact && p.n == 8 && p.m == 8 ? launch_one<1, 1, false, false, false>(p, sm_count, st)
                                             : launch_one<1, 1, false, false, true>(p, sm_count, st);
    case 2:
        return full16 ? launch_one<2, 2, false, false, false>(p, sm_count, st)
             : mb == 1 ? launch_one<2, 1, false, false, true>(p, sm_count, st) : launch_one<2, 2, false, false, true>(p, sm_count, st);
    case 3:
        return mb == 1 ? launch_one<3, 1, false, false, true>(p, sm_count, st)
             : mb == 2 ? launch_one<3, 2, false, false, true>(p, sm_count, st) : launch_one<3, 3, false, false, true>(p, sm_count, st);
    case 4:
        return full32 ? launch_one<4, 4, false, false, false>(p, sm_count, st)
             : mb == 1 ? launch_one<4, 1, false, false, true>(p, sm_count, st)
             : mb == 2 ? launch_one<4, 2, false, false, true>(p, sm_count, st)
             : mb == 3 ? launch_one<4, 3, false, false, true>(p, sm_count, st) : launch_one<4, 4, false, false, true>(p, sm_count, st);
    case 5:
    case 6:
        return launch_blocks_5_6(p, kb, mb, sm_count, st);
    default:
        return launch_blocks_8(p, mb, sm_count, st);
    }
}

// Gradients of the first control, everything in one kernel: n = m = 16 / 32, float32 operands with aligned strides.
inline cudaError_t launch_grad_frag(const SolveParams& p, int sm_count, cudaStream_t st)
{
    return p.n == 16 ? launch_one<2, 2, true, true, false, false, true>(p, sm_count, st)
                     : launch_one<4, 4, true, true, false, false, true>(p, sm_count, st);
}

} // namespace rfrag
} // namespace ttc
