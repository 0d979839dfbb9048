// Training layers of the snapshot codec (ae_train.cu).
#pragma once

#include "ae_internal.h"

namespace rtm {

// bytes of the packed bf16 weights of one training step (16-byte aligned)
constexpr int kAePackedBytes = (27 * 64 + 32 * 128 + 64 * 64 + 14 * 128) * 16;

cudaError_t ae_pack_weights(const float* P, void* packed, cudaStream_t s);
// forward layers; h and l are the half- and quarter-resolution grids
cudaError_t ae_train_e2(const float* P, const void* W, const ae::bf16* h1, ae::bf16* lat, ae::Dims3 h,
                        ae::Dims3 l, int* status, cudaStream_t s);
cudaError_t ae_train_d1(const float* P, const void* W, const ae::bf16* lat, ae::bf16* g1, ae::Dims3 h,
                        ae::Dims3 l, int* status, cudaStream_t s);
// data gradients
cudaError_t ae_train_d1_grad(const void* W, const ae::bf16* ga3, ae::bf16* glat, ae::Dims3 h,
                             ae::Dims3 l, int* status, cudaStream_t s);
cudaError_t ae_train_e2_grad(const void* W, const ae::bf16* glat, const ae::bf16* h1, ae::bf16* ga1,
                             ae::Dims3 h, ae::Dims3 l, int* status, cudaStream_t s);
// weight (and bias) gradients, added to grad: W3; W2 and b2; W1, b1, W4 and b3
cudaError_t ae_train_d1_weights(const ae::bf16* lat, const ae::bf16* ga3, float* grad, ae::Dims3 h,
                                ae::Dims3 l, int* status, cudaStream_t s);
cudaError_t ae_train_e2_weights(const ae::bf16* h1, const ae::bf16* glat, float* grad, ae::Dims3 h,
                                ae::Dims3 l, int* status, cudaStream_t s);
cudaError_t ae_train_patch_weights(const ae::bf16* xq, const ae::bf16* ga1, const ae::bf16* gy,
                                   const ae::bf16* g1, const ae::bf16* ga3, float* grad,
                                   ae::Dims3 h, ae::Dims3 l, int* status, cudaStream_t s);

}  // namespace rtm
