// Expansion of a factored state cost (ttc_lqr_solve_lowrank_q).
#pragma once

#include "common.cuh"

namespace ttc {

// Q = scale * U U' + diag(d) written out densely (float32, [N][n][n]) for the instances of the launch's token window:
// the state cost of the TTC layer is a combination of a few basis directions plus a diagonal (Parameterization
// paragraph), so a caller can hand over U [n][r] and d [n] instead of n x n numbers per instance.  One CTA per
// instance at a time; U', d staged in shared memory.
__global__ void __launch_bounds__(256) expand_lowrank_q_kernel(SolveParams p, OperandDev U, OperandDev d, int r, float scale,
                                                               float* Qdense)
{
    extern __shared__ float sm_u[];          // U' [r][n] then d [n]
    const int n = p.n;
    const long long nwin = p.b0 * p.b1 * p.tcount;
    for (long long w = blockIdx.x; w < nwin; w += gridDim.x) {
        const long long inst = window_instance(p, w);
        const long long ou = operand_offset(U, inst, p.b1, p.b2), od = operand_offset(d, inst, p.b1, p.b2);
        __syncthreads();
        for (int e = threadIdx.x; e < n * r; e += blockDim.x)
            sm_u[(e % r) * n + e / r] = load_elem(U, ou + e);
        for (int e = threadIdx.x; e < n; e += blockDim.x)
            sm_u[r * n + e] = load_elem(d, od + e);
        __syncthreads();
        float* dst = Qdense + inst * (long long)n * n;
        for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
            const int i = e / n, j = e % n;
            float acc = 0.f;
            for (int k = 0; k < r; ++k)
                acc = fmaf(sm_u[k * n + i], sm_u[k * n + j], acc);
            acc *= scale;
            if (i == j)
                acc += sm_u[r * n + i];
            dst[e] = acc;
        }
    }
}

} // namespace ttc
