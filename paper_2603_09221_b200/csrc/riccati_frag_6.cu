// One-warp recursion with six blocks of states (riccati_frag.cuh: time-invariant requests, any strides).
#include "riccati_frag.cuh"

namespace ttc {
namespace rfrag {

cudaError_t launch_blocks_6(const SolveParams& p, int mb, int sm_count, cudaStream_t st)
{
    return mb <= 2 ? launch_one<6, 2, false, false, true>(p, sm_count, st)
         : mb <= 4 ? launch_one<6, 4, false, false, true>(p, sm_count, st) : launch_one<6, 6, false, false, true>(p, sm_count, st);
}

} // namespace rfrag
} // namespace ttc
