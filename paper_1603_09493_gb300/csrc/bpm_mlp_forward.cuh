// One-kernel forward pass of the surrogate: declarations shared with bpm_mlp.cu.
#pragma once
#include "bpm_internal.cuh"

namespace bpm {

constexpr int kMaxMlpLayers = 7;     // depth 6 and the output layer

// Layer l: rows of W_l as the tensor map's box (n_mma: whole hidden layers, the output layer's rows
// rounded up to 16), k_pad columns; n_pad is the padded width of its output, n_real the real one.
struct MlpForward {
    CUtensorMap w[kMaxMlpLayers];
    const float* bias[kMaxMlpLayers];
    int k_pad[kMaxMlpLayers], n_pad[kMaxMlpLayers], n_mma[kMaxMlpLayers], n_real[kMaxMlpLayers];
    int L, n_in, sigmoid;
    long long N;
    const float* X;                  // [N][n_in]
    float* out;                      // [N][n_real of the last layer]: logits, or probabilities with sigmoid
};
bool mlp_forward_fits(int L, const int* k_pad, const int* n_pad);
int mlp_forward_launch(cudaStream_t s, const MlpForward& p, int sm_count, int* err);

}  // namespace bpm
