// flow_tile.cuh -- what the fused coupling-flow kernels share: a CTA holds 128 rows of the
// flow; activations lie in shared memory as K-blocks of 128 rows x 64 bfloat16 columns in the
// 128-byte-swizzle layout that TMA and the tensor core read, accumulators in tensor memory.
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include "gwx_internal.h"
#include "tc05.cuh"

namespace gwx {
namespace flowt {

using namespace tc;

constexpr int FM = 128;                                  // rows per tile
constexpr int F_THREADS = 320;                           // warp 0 TMA, warp 1 MMA, warps 2-9 rows
constexpr uint32_t KB_BYTES = FM * 128;                  // one 128-row x 64-column bfloat16 K-block: 16 KiB
constexpr uint32_t X_BYTES = 2 * KB_BYTES;               // conditioner input, 8 + C <= 128 columns
constexpr uint32_t G_BYTES = 4 * KB_BYTES;               // hidden activations, H <= 256 columns
constexpr uint32_t SLOT_BYTES = 2 * 256 * 128;           // two K-blocks of a 256-row weight tile
constexpr uint32_t F_WAIT = 1u << 22;
constexpr float S_MAX = 3.f;

// Split p of the eight coordinates: conditioning half a_j = A(p, j), transformed half
// b_j = Bc(p, j) (the flow's four fixed splits; compile-time so v[] stays in registers).
__host__ __device__ constexpr int A(int p, int j) {
  return p == 0 ? j : p == 1 ? 4 + j : p == 2 ? 2 * j : 2 * j + 1;
}
__host__ __device__ constexpr int Bc(int p, int j) {
  return p == 0 ? 4 + j : p == 1 ? j : p == 2 ? 2 * j + 1 : 2 * j;
}

// Byte offset of 16-byte chunk j of row r inside a 128-row K-block (128-byte swizzle).
__device__ __forceinline__ uint32_t swz(int r, int j) {
  return (uint32_t)((r >> 3) * 1024 + (r & 7) * 128 + ((j ^ (r & 7)) << 4));
}

__device__ __forceinline__ uint32_t pack2(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}

// The same of max(a, 0), max(b, 0): the maximum is taken on the rounded pair in one instruction
// (rounding is monotonic and keeps zero, so the values are the same; a NaN gives 0 as fmaxf does).
__device__ __forceinline__ uint32_t pack2_relu(float a, float b) {
  __nv_bfloat162 h = __hmax2(__floats2bfloat162_rn(a, b), __floats2bfloat162_rn(0.f, 0.f));
  return *reinterpret_cast<uint32_t*>(&h);
}

__device__ __forceinline__ void proxy_fence() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Box at (x, y, z) of a tensor map from shared memory, as one bulk group of this thread.
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, uint32_t src, int x, int y, int z) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(x), "r"(y), "r"(z), "r"(src)
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// This thread's stores have read their shared memory / have completed.
__device__ __forceinline__ void tma_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

template <int P>
__device__ __forceinline__ void pack_half(const float* v, uint32_t& w0, uint32_t& w1) {
  w0 = pack2(v[A(P, 0)], v[A(P, 1)]);
  w1 = pack2(v[A(P, 2)], v[A(P, 3)]);
}

inline PFN_cuTensorMapEncodeTiled_v12000 encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// bfloat16 [layers][rows][cols] with the layers lstride elements apart; boxes of 64 columns
// x box_rows rows x one layer.
inline bool layer_map(CUtensorMap* map, const void* base, int64_t cols, int64_t rows, int64_t layers, int64_t lstride,
                      uint32_t box_rows) {
  auto enc = encoder();
  if (!enc) return false;
  cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)layers};
  cuuint64_t strides[2] = {(cuuint64_t)cols * 2, (cuuint64_t)lstride * 2};
  cuuint32_t box[3] = {64, box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace flowt
}  // namespace gwx
