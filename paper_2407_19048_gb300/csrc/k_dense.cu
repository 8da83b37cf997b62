// k_dense.cu -- backward pass of the dense layer Y = act(X W^T + b) of the learned part
// (the embedding network of Sec. 4 and the flow of Sec. 5), by the chain rule:
//   dZ = dY * act'(Z),  dX = dZ W,  dW = dZ^T X,  db = sum over rows of dZ,
// with both products on the tensor cores (k_gemm.cu), which reads dZ, W and X as they lie:
// no transposed copies.  Where the derivative needs Z, the product that recomputes it writes
// dZ itself; where a ReLU layer's output is at hand, or there is no activation, one pass over
// dY does.  dW is split along the batch when its N x K output has few tiles.  This file holds
// that pass and the column-sum reduction.  (4096 x 1968 -> 512, ReLU, forward and backward:
// 130 us with Z in memory and transposes of dZ, X and W, now 65 to 78 with the host's issue.)
#include <cuda_bf16.h>

#include <algorithm>

#include "gwx_internal.h"
#include "pdl.cuh"
#include "sum2.cuh"

namespace gwx {

namespace {

constexpr int TT = 32;   // rows of a column-sum partial; columns of a k_colsum block

// dZ = dY (masked by Y > 0 when Y, the layer's bfloat16 ReLU output, is given: that is Z > 0,
// since a positive float never rounds to a bfloat16 zero short of 1e-40) in bfloat16, and the
// FP32 column sums of every 32 rows into part.  HBM bound: a warp takes 32 rows x 64 columns,
// 256-byte row segments in (sixteen in flight), 128-byte segments out.
__global__ void __launch_bounds__(256) k_dz_rows(const float* dY, const __nv_bfloat16* Y,
                                                 int64_t M, int N, __nv_bfloat16* __restrict__ dZ,
                                                 float* __restrict__ part) {
  pdl_enter();
  const int units = (N + 63) / 64;
  const int64_t u = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int64_t p = u / units;
  const int col = (int)(u - p * units) * 64 + 2 * (threadIdx.x & 31);
  const int64_t m0 = p * TT;
  if (m0 >= M || col >= N) return;
  const int rows = (int)(M - m0 < TT ? M - m0 : TT);
  const bool pairs = ((uintptr_t)dY & 7u) == 0;   // dY comes with 4-byte alignment only
  float s0 = 0.f, s1 = 0.f;
  for (int r0 = 0; r0 < rows; r0 += 16) {
    float2 v[16];
    __nv_bfloat162 y[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int64_t at = (m0 + min(r0 + i, rows - 1)) * N + col;
      v[i] = pairs ? *reinterpret_cast<const float2*>(dY + at) : make_float2(dY[at], dY[at + 1]);
      if (Y != nullptr) y[i] = *reinterpret_cast<const __nv_bfloat162*>(Y + at);
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      if (r0 + i >= rows) break;
      if (Y != nullptr) {
        v[i].x = __low2float(y[i]) > 0.f ? v[i].x : 0.f;
        v[i].y = __high2float(y[i]) > 0.f ? v[i].y : 0.f;
      }
      *reinterpret_cast<__nv_bfloat162*>(dZ + (m0 + r0 + i) * N + col) = __floats2bfloat162_rn(v[i].x, v[i].y);
      s0 += v[i].x;
      s1 += v[i].y;
    }
  }
  if (part != nullptr) *reinterpret_cast<float2*>(part + p * N + col) = make_float2(s0, s1);
}

// db[n] = sum_p part[p][n] (two-float accumulation of the FP32 tile sums), in two
// deterministic passes: block (32 columns, slice y of the partials) has row lane ty sum
// partials ty, ty + 32, ... of its slice, then warp ty the 32 lanes of column ty into
// part2[y][n]; then k_colsum_finish adds the slices in order.  With one slice the first pass
// writes db itself (db non-null), rounded once.  (FP64 sums and one thread a column over the
// 32 lanes: 6.3 us for 128 partials of 512 columns, 3.7 now.)
constexpr int CS_MAX_SLICES = 64;

int colsum_slices(int64_t P) { return (int)std::min<int64_t>(CS_MAX_SLICES, std::max<int64_t>(1, (P + 255) / 256)); }

__global__ void __launch_bounds__(1024) k_colsum(const float* part, int P, int N,
                                                 double* __restrict__ part2, float* __restrict__ db) {
  pdl_enter();
  __shared__ float2 red[TT][TT + 1];
  const int n = blockIdx.x * TT + threadIdx.x;
  const int per = (P + gridDim.y - 1) / gridDim.y, p0 = blockIdx.y * per, p1 = min(P, p0 + per);
  Sum2 s;
  if (n < N)
#pragma unroll 4
    for (int p = p0 + threadIdx.y; p < p1; p += TT) s.add(part[(int64_t)p * N + n]);
  red[threadIdx.y][threadIdx.x] = make_float2(s.h, s.l);
  __syncthreads();
  const float2 v = red[threadIdx.x][threadIdx.y];
  s.h = v.x;
  s.l = v.y;
  const int c = blockIdx.x * TT + threadIdx.y;
  warp_total(s, part + (int64_t)p0 * N + c, p1 - p0, N, c < N, [&](auto t) {
    if (db) db[c] = t.rounded();
    else part2[(int64_t)blockIdx.y * N + c] = t.value();
  });
}

__global__ void k_colsum_finish(const double* part2, int slices, int N, float* __restrict__ db) {
  pdl_enter();
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  double t = 0.0;
  for (int y = 0; y < slices; ++y) t += part2[(int64_t)y * N + n];
  db[n] = (float)t;
}

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

}  // namespace

cudaError_t launch_dz_rows(const float* dY, const void* Y, int64_t M, int N, void* dZ, float* part, cudaStream_t s) {
  const int64_t units = (M + TT - 1) / TT * ((N + 63) / 64);
  pdl_launch(k_dz_rows, dim3((unsigned)((units + 7) / 8)), dim3(256), 0, s, dY,
             reinterpret_cast<const __nv_bfloat16*>(Y), M, N, reinterpret_cast<__nv_bfloat16*>(dZ), part);
  return cudaGetLastError();
}

size_t dense_backward_ws(int64_t M, int64_t N, int64_t K) {
  const int64_t P = (M + TT - 1) / TT;
  return align256((size_t)M * N * 2)                 // dZ
         + align256((size_t)P * N * 4)               // column-sum partials
         + align256((size_t)CS_MAX_SLICES * N * 8)   // their slice sums
         + align256(wgrad_ws(N, K, M, 1));           // split-K slices of dW
}

// dX = dZ W and dW = dZ^T X from dZ in bfloat16; ws holds the split-K partial products.
cudaError_t launch_dense_backward_dz(const void* dZ16, const void* X, const void* W, int64_t M, int64_t N, int64_t K,
                                     float* dX, float* dW, void* ws, cudaStream_t s) {
  const cudaError_t e = dX ? launch_gemm_nn(dZ16, W, dX, M, K, N, s) : cudaSuccess;
  if (e != cudaSuccess || !dW) return e;
  return launch_wgrad(dZ16, X, dW, N, K, M, reinterpret_cast<float*>(ws), s);
}

cudaError_t launch_dense_backward(const void* X, const void* W, const float* bias, const float* dY, int64_t M,
                                  int64_t N, int64_t K, int act, float* dX, float* dW, float* db, void* ws, int group,
                                  cudaStream_t s, const void* Y) {
  char* w = reinterpret_cast<char*>(ws);
  void* dZ = w;
  w += align256((size_t)M * N * 2);
  float* part = reinterpret_cast<float*>(w);
  const int64_t P = (M + TT - 1) / TT;
  w += align256((size_t)P * N * 4);
  double* part2 = reinterpret_cast<double*>(w);
  w += align256((size_t)CS_MAX_SLICES * N * 8);
  float* kpart = reinterpret_cast<float*>(w);
  // only the activation derivative needs Z = X W^T + b, and a ReLU layer whose output Y is
  // given takes its mask from Y instead
  const void* Y16 = act == GWX_ACT_RELU ? Y : nullptr;
  cudaError_t e = act == GWX_ACT_NONE || Y16 != nullptr
                      ? launch_dz_rows(dY, Y16, M, (int)N, dZ, part, s)
                      : launch_gemm_dact(X, W, bias, dY, act, M, N, K, dZ, part, group, s);
  if (e != cudaSuccess) return e;
  if ((e = launch_dense_backward_dz(dZ, X, W, M, N, K, dX, dW, kpart, s)) != cudaSuccess) return e;
  if (db) {
    const int slices = colsum_slices(P);
    pdl_launch(k_colsum, dim3((unsigned)((N + TT - 1) / TT), (unsigned)slices), dim3(TT, TT), 0, s, part, (int)P,
               (int)N, part2, slices == 1 ? db : nullptr);
    if (slices > 1) pdl_launch(k_colsum_finish, dim3((unsigned)((N + 127) / 128)), dim3(128), 0, s, part2, slices,
                               (int)N, db);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace gwx
