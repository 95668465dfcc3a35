// One-warp recursion with seven or eight blocks of states and at most four of controls (riccati_frag.cuh: time-invariant requests).
#include "riccati_frag.cuh"

namespace ttc {
namespace rfrag {

cudaError_t launch_blocks_8(const SolveParams& p, int mb, int sm_count, cudaStream_t st)
{
    return mb <= 2 ? launch_one<8, 2, false, false, true>(p, sm_count, st) : launch_one<8, 4, false, false, true>(p, sm_count, st);
}

} // namespace rfrag
} // namespace ttc
