// Tensor-core (tcgen05) forward products of the warm-start network: shared between the network's
// entry points (cnn.cu) and the kernel (cnn_tc.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace celeste {
namespace cnn_tc {

// D[M x N] = A[M x K] B[K x N]: A the layer input (im2col of a 3x3, padding-1 convolution over an
// NHWC tensor, or [M][K]), B the weights [N][K] (K-major), bias [N]; D stored as BF16 after ReLU into
// out [M][N], or as FP32 into out_f [M][N] (times scale plus shift when scale is set).  The kernels are
// built for the network's layers.
enum LayerId { CONV1, CONV2, CONV3, CONV4, DENSE1, DENSE2 };
struct Args {
  int M, N, B;                   // rows and columns of D, patches
  const __nv_bfloat16* in;
  const __nv_bfloat16* w;
  const float* bias;
  __nv_bfloat16* out;
  float* out_f;
  const float* scale;
  const float* shift;
  int* err;                      // error word, set when a bounded wait runs out
  long long wait_budget;         // SM cycles a wait may take (negative: every wait gives up at once)
};

}  // namespace cnn_tc

// n_sm: SMs of the current device.
cudaError_t tc_forward(cnn_tc::LayerId layer, const cnn_tc::Args& a, int n_sm, cudaStream_t st);

}  // namespace celeste
