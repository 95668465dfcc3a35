// One-warp recursion with three or four blocks of states (riccati_frag.cuh: time-invariant requests).
#include "riccati_frag.cuh"

namespace ttc {
namespace rfrag {

cudaError_t launch_blocks_3_4(const SolveParams& p, int kb, int mb, bool full32, int sm_count, cudaStream_t st)
{
    if (kb == 3)
        return mb == 1 ? launch_one<3, 1, false, false, true>(p, sm_count, st)
             : mb == 2 ? launch_one<3, 2, false, false, true>(p, sm_count, st) : launch_one<3, 3, false, false, true>(p, sm_count, st);
    return full32 ? launch_one<4, 4, false, false, false>(p, sm_count, st)
         : mb == 1 ? launch_one<4, 1, false, false, true>(p, sm_count, st)
         : mb == 2 ? launch_one<4, 2, false, false, true>(p, sm_count, st)
         : mb == 3 ? launch_one<4, 3, false, false, true>(p, sm_count, st) : launch_one<4, 4, false, false, true>(p, sm_count, st);
}

} // namespace rfrag
} // namespace ttc
