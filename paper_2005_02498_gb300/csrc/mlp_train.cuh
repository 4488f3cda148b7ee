// mlp_train.cuh -- one minibatch of surrogate training in two launches
// (mlp_train.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace ptadd {

// Padded layer sizes (inputs 30 -> 32, outputs 6 -> 16).
__host__ __device__ constexpr int din_p(int l) { return l == 0 ? 32 : 256; }
__host__ __device__ constexpr int dout_p(int l) { return l == 3 ? 16 : 256; }

struct TrainArgs {
    // the minibatch: sample idx[r] (or r) of xn [. x 30], yn [. x 6] for r < n; rows = n rounded up to 16
    const float *xn = nullptr, *yn = nullptr;
    const int32_t* idx = nullptr;
    int64_t n = 0, rows = 0;
    // parameters: BF16 copies (W row-major, W^T), FP32 masters, Adam's moments
    __nv_bfloat16 *Wb[4] = {}, *Wt[4] = {};
    float *W[4] = {}, *b[4] = {}, *mW[4] = {}, *vW[4] = {}, *mb[4] = {}, *vb[4] = {};
    float *gW[4] = {}, *gb[4] = {};  // gradients out (adam = 0)
    // work: activations and their gradients, transposed: [. x rows] in tiles of 128 x 64 (mlp_train.cu),
    // both padded to full tiles
    __nv_bfloat16 *Xt = nullptr, *Ht[3] = {}, *dYt = nullptr, *dZt[3] = {};
    float* loss_part = nullptr;  // [ceil(rows / 128)]
    int adam = 0;                // 1: update the parameters, 0: write the gradients
    float lr = 0, b1 = 0, b2 = 0, eps = 0, c1 = 0, c2 = 0;
    int* err = nullptr;  // set to 1 if a wait for the tensor core gave up
};

// Forward, loss and backward of the minibatch; then the weight gradients with the update.  Two launches.
cudaError_t launch_mlp_train(const TrainArgs& g, cudaStream_t s);

}  // namespace ptadd
