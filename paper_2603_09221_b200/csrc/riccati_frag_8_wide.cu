// One-warp recursion with seven or eight blocks of states or controls (riccati_frag.cuh: time-invariant requests, any strides).
#include "riccati_frag.cuh"

namespace ttc {
namespace rfrag {

cudaError_t launch_blocks_8_wide(const SolveParams& p, int mb, int sm_count, cudaStream_t st)
{
    return mb <= 6 ? launch_one<8, 6, false, false, true>(p, sm_count, st) : launch_one<8, 8, false, false, true>(p, sm_count, st);
}

} // namespace rfrag
} // namespace ttc
