// k_conv.cu -- the stride-1 convolutions of the ResNet-1D data summary (Sec. 4) as
// implicit GEMMs on the tensor cores: no im2col matrix and no transposed copy is
// materialised, forward or backward.
//   forward:         z[b][t][o]  = sum_{j,c} x[b][t + j - p][c] W[o][j C + c]
//   input gradient:  dx[b][t][c] = sum_{j,o} dz[b][t - (j - p)][o] W[o][j C + c]
//                    (the same implicit form, taps mirrored, W read as it lies)
//   weight gradient: dW[o][j C + c] = sum_{b,t} dz[b][t][o] x[b][t + j - p][c]
//                    (both operands read as they lie, the times of a tap shifted by the box)
// (p = (k - 1)/2, zero outside [0, T)); the products run in k_gemm.cu's kernel, whose tiles
// come from 3-D tensor maps of the channels-last activations.
#include <cuda_bf16.h>

#include "gwx_internal.h"

namespace gwx {

namespace {

size_t al256(size_t v) { return (v + 255) / 256 * 256; }

}  // namespace

// Workspace of conv_backward: dz in bfloat16 [B T][O] and the split-K partial products of dW.
size_t conv_backward_ws(int64_t Bn, int64_t T, int C, int O, int k) {
  const int64_t M = Bn * T;
  return al256((size_t)M * O * 2) + al256(wgrad_ws(O, (int64_t)k * C, M, 1));
}

cudaError_t launch_conv_forward(const void* x, int64_t Bn, int64_t T, int C, int k, const void* W, int O,
                                const float* addend, float* z, cudaStream_t s) {
  return launch_conv_gemm(x, Bn, T, C, k, +1, W, O, z, addend, s);
}

// dx [B][T][C] (+ addend) and dW [O][k C] of the stride-1 convolution z = conv(x, W) given
// dz [B][T][O] in bfloat16; ws holds the split-K partial products.
cudaError_t launch_conv_backward_dz(const void* dz16, const void* x, const void* W, int64_t Bn, int64_t T, int C, int O,
                                    int k, const float* addend, float* dx, float* dW, void* ws, cudaStream_t s) {
  // the input gradient: dz as the implicit A (channels O), taps mirrored
  cudaError_t e = dx ? launch_conv_gemm(dz16, Bn, T, O, k, -1, W, C, dx, addend, s) : cudaSuccess;
  if (e != cudaSuccess || !dW) return e;
  return launch_conv_wgrad(dz16, x, dW, Bn, T, C, O, k, reinterpret_cast<float*>(ws), s);
}

// The same from FP32 dz.
cudaError_t launch_conv_backward(const float* dz, const void* x, const void* W, int64_t Bn, int64_t T, int C, int O,
                                 int k, const float* addend, float* dx, float* dW, void* ws, cudaStream_t s) {
  const int64_t M = Bn * T;
  const cudaError_t e = launch_dz_rows(dz, nullptr, M, O, ws, nullptr, s);
  if (e != cudaSuccess) return e;
  return launch_conv_backward_dz(ws, x, W, Bn, T, C, O, k, addend, dx, dW,
                                 reinterpret_cast<char*>(ws) + al256((size_t)M * O * 2), s);
}

}  // namespace gwx
