// Arguments of one contextualised layer evaluation, as the kernels take them (layer_frag.cuh, layer_grad.cuh and the
// baseline in sigma_product.cuh).
#pragma once

namespace ttc {
namespace layer {

struct LayerParams {
    long long N;                 // instances
    bool few;                    // the whole batch (of which this may be a slice) has at most four instances per SM
    int T, r;
    const float *s_a, *s_ga, *s_gb, *s_gq;   // [N][n]
    const float *s_b, *s_q, *s_qf;           // [N][r]
    const float *r_inv, *h0;                 // [N][n]
    const float *B_basis, *Q_basis;          // [r][n][n]
    float* u1;                   // [N][n] or null
    float* P0;                   // [N][n][n] or null
    int* info;                   // [N] or null
    // gradient path only
    float* Kws;                  // [N][T][n][n]: K of step s = t - 1
    const float* g;              // [N][n]: dl/du_1*
    float* k0;                   // [N][n]: -S_0^{-1} g
};

} // namespace layer
} // namespace ttc
