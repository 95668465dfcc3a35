// One-warp recursion for time-varying and affine requests, and the gradients of the first control (riccati_frag.cuh).
#include "riccati_frag.cuh"

namespace ttc {
namespace rfrag {

cudaError_t launch_affine(const SolveParams& p, int kb, bool full16, bool full32, int sm_count, cudaStream_t st)
{
    if (kb <= 2)
        return full16 ? launch_one<2, 2, true, true, false>(p, sm_count, st) : launch_one<2, 2, true, true, true>(p, sm_count, st);
    return full32 ? launch_one<4, 4, true, true, false>(p, sm_count, st) : launch_one<4, 4, true, true, true>(p, sm_count, st);
}

cudaError_t launch_time_varying(const SolveParams& p, int kb, bool full16, bool full32, int sm_count, cudaStream_t st)
{
    if (kb <= 2)
        return full16 ? launch_one<2, 2, true, false, false>(p, sm_count, st) : launch_one<2, 2, true, false, true>(p, sm_count, st);
    return full32 ? launch_one<4, 4, true, false, false>(p, sm_count, st) : launch_one<4, 4, true, false, true>(p, sm_count, st);
}

cudaError_t launch_grad_frag(const SolveParams& p, int sm_count, cudaStream_t st)
{
    return p.n == 16 ? launch_one<2, 2, true, true, false, false, true>(p, sm_count, st)
                     : launch_one<4, 4, true, true, false, false, true>(p, sm_count, st);
}

} // namespace rfrag
} // namespace ttc
