// pd_net_train.cuh — loss and parameter gradients of the learned network.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace pd {
namespace nettrain {

// bytes of the bf16 weight images of one step
size_t image_bytes();
// bytes of the bf16 h2 and dz3 rows of max_batch hits
size_t h2_bytes(uint32_t max_batch);
size_t dz3_bytes(uint32_t max_batch);
// bytes of the blocks' gradient sums
size_t slice_bytes(uint32_t max_batch, int sms);
// Gradient of every parameter into grads (overwritten; 8-byte aligned) and
// the loss added to *loss (if not NULL) for n >= 1 patches x[n][25] with
// float32 parameters w.  img, h2, dz3, slices: scratch of the sizes above
// (16-byte aligned).  n_reg: the offset loss's divisor.  sms: the device's SMs.
cudaError_t gradients(const float* w, const float* x, const uint8_t* counts, const float* targets,
                      const uint8_t* mask, uint32_t n, float n_reg, float lambda, uint4* img,
                      uint16_t* h2, uint16_t* dz3, float* slices, float* grads, float* loss,
                      int sms, cudaStream_t s);

}  // namespace nettrain
}  // namespace pd
