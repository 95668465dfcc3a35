// One-warp recursion with five blocks of states (riccati_frag.cuh: time-invariant requests, any strides).
#include "riccati_frag.cuh"

namespace ttc {
namespace rfrag {

cudaError_t launch_blocks_5(const SolveParams& p, int mb, int sm_count, cudaStream_t st)
{
    return mb == 1 ? launch_one<5, 1, false, false, true>(p, sm_count, st)
         : mb == 2 ? launch_one<5, 2, false, false, true>(p, sm_count, st)
         : mb == 3 ? launch_one<5, 3, false, false, true>(p, sm_count, st)
         : mb == 4 ? launch_one<5, 4, false, false, true>(p, sm_count, st) : launch_one<5, 5, false, false, true>(p, sm_count, st);
}

} // namespace rfrag
} // namespace ttc
