// What the MLP's fused training launches (mlp_tc.cu) share with its entry points (mlp.cu).
#pragma once

#include <cuda_bf16.h>

#include "common.cuh"

namespace gs {

// One split's shares of the gradients: dW^T of the four layers ([in][out], padded; a
// TMEM lane is an output neuron, so a warp writes whole lines), then the bias gradients.
constexpr int kMlpPartW0 = 0, kMlpPartW1 = kMlpPartW0 + 128 * 208, kMlpPartW2 = kMlpPartW1 + 128 * 128;
constexpr int kMlpPartW3 = kMlpPartW2 + 128 * 128, kMlpPartB0 = kMlpPartW3 + 16 * 128, kMlpPartB1 = kMlpPartB0 + 128;
constexpr int kMlpPartB2 = kMlpPartB1 + 128, kMlpPartB3 = kMlpPartB2 + 128, kMlpPart = kMlpPartB3 + 128;

struct MlpTrainBufs {
    __nv_bfloat16* Xt;     // [208][Mp]
    float* G[3];           // [128][Mp]
    __nv_bfloat16* Ht[3];  // [128][Mp]
    float* Z3;             // [Mp][16]
    __nv_bfloat16* Wt[3];  // [128][128], [128][128], [128][16]
    float* part;           // [ceil(Mp / 256)][kMlpPart]
    float* loss_part;      // [ceil(Mp / 256)]
};

int mlp_train_fused(const float* const* w, const float* const* b, const float* image, int W, int H,
                    const MlpTrainBufs& t, int64_t M, int64_t Mp, const float* targets, float w_depth, float w_scale,
                    float* out, cudaStream_t s);

}  // namespace gs
