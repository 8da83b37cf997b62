// flow_tile.cuh -- what the fused coupling-flow kernels share: a CTA holds 128 rows of the
// flow; activations lie in shared memory as K-blocks of 128 rows x 64 bfloat16 columns in the
// 128-byte-swizzle layout that TMA and the tensor core read, accumulators in tensor memory.
#pragma once

#include <stddef.h>

#include <cuda.h>
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

// ---- the forward conditioner of one layer after another (sampling and density)
// Warp 0 streams weights and biases (fwd_produce), warp 1 issues the products (fwd_multiply),
// warps 2-17 own the rows; what each holds where is described in k_flow_fused.cu.
constexpr int ROW_WARPS = 16;                              // four warps a tensor-memory lane quarter
constexpr int FWD_THREADS = 64 + 32 * ROW_WARPS;
constexpr uint32_t V3_BYTES = 16 * 256 * 2;
constexpr uint32_t FWD_BYTES = X_BYTES + 2 * SLOT_BYTES + V3_BYTES;   // X, weight ring, V3: 1024-byte aligned
constexpr uint32_t ACC2 = 256, ACC3 = 16;                  // tensor-memory columns of the second and third products

struct FwdRing {
  uint64_t full[3], empty[3], xready, gready[2], acc1f, acc2f, acc3f, biasf[2], cplf[4], drained;
  alignas(16) float sb[2][2 * 256 + 8];                    // biases of a layer: first, second, third product (bulk copies)
  float s_new[4][FM], s_log[4][FM];                        // the rows' transformed coordinates and log scales
  uint32_t tmem_slot;
  uint32_t fills[3];                                       // the producer's, once it has stopped: weight slots, V3, biases
  int abort_flag;
};

static_assert(offsetof(FwdRing, sb) % 16 == 0 && sizeof(FwdRing::sb[0]) % 16 == 0 && alignof(FwdRing) == 16,
              "bulk copies start on 16 bytes");

struct FwdWeights {
  const CUtensorMap *v1, *v2, *v3;
  const float *e1, *e2, *e3;                               // layer-0 biases; layer l at + l * lstride
  int64_t lstride;
  int C, H, K, tiles;
  bool reverse;                                            // layers K - 1 .. 0
};

// Barriers and tensor memory; all threads, ends in __syncthreads.  Returns the tensor memory.
__device__ __forceinline__ uint32_t fwd_begin(FwdRing& rg) {
  if (threadIdx.x == 0) {
    for (int s = 0; s < 3; ++s) {
      mbar_init(su32(&rg.full[s]), 1);
      mbar_init(su32(&rg.empty[s]), 1);
    }
    mbar_init(su32(&rg.xready), ROW_WARPS);
    for (int r = 0; r < 2; ++r) {
      mbar_init(su32(&rg.gready[r]), ROW_WARPS);
      mbar_init(su32(&rg.biasf[r]), 1);
    }
    mbar_init(su32(&rg.acc1f), 1);
    mbar_init(su32(&rg.acc2f), 1);
    mbar_init(su32(&rg.acc3f), 1);
    for (int q = 0; q < 4; ++q) mbar_init(su32(&rg.cplf[q]), 4);
    mbar_init(su32(&rg.drained), 1);
    rg.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (threadIdx.x >> 5 == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&rg.tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  return rg.tmem_slot;
}

// ring_drain of two slots filled in turn, n fills so far.
__device__ __forceinline__ void pair_drain(const uint64_t* full, uint32_t n, uint32_t limit) {
  ring_drain(full, 2, n & 1u, ((n >> 1) & 1u) ^ 1u, limit);
}

// Lets the copies and products in flight end; all threads (a call: the registers it would take are
// those of the row warps' loops).
static __device__ __noinline__ void fwd_drain(FwdRing& rg) {
  if (threadIdx.x >> 5 == 0) {
    pair_drain(rg.full, rg.fills[0], F_WAIT);
    ring_drain(rg.full + 2, 1, 0u, (rg.fills[1] & 1u) ^ 1u, F_WAIT);   // one slot
    pair_drain(rg.biasf, rg.fills[2], F_WAIT);
  }
  if (threadIdx.x >> 5 == 1) mma_drain(&rg.drained, F_WAIT);
  __syncthreads();
}

// Records a given-up wait in *status, lets what is in flight end then, and frees the tensor memory;
// all threads.
__device__ __forceinline__ void fwd_end(FwdRing& rg, uint32_t tmem, int* status) {
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (*(volatile int*)&rg.abort_flag) {
    if (threadIdx.x == 0) atomicExch(status, 1);
    fwd_drain(rg);
  }
  if (threadIdx.x >> 5 == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

__device__ __forceinline__ void fwd_produce(FwdRing& rg, const FwdWeights& w, uint32_t sw) {
  const int lane = threadIdx.x & 31, H = w.H, NP = 2 + H / 128;   // weight parts per layer
  uint32_t it = 0, li = 0, thirds = 0, biases = 0;
  bool ok = true;
  for (int t = blockIdx.x; t < w.tiles && ok; t += gridDim.x)
    for (int n = 0; n < w.K && ok; ++n, ++li)
      for (int p = 0; p < NP; ++p) {
        const int l = w.reverse ? w.K - 1 - n : n;
        const bool last = p == NP - 1;
        const uint32_t s = last ? 2u : it & 1u;
        if (!mbar_wait_warp(su32(&rg.empty[s]), ((last ? li : it >> 1) & 1u) ^ 1u, F_WAIT) ||
            __any_sync(0xffffffffu, *(volatile int*)&rg.abort_flag)) {
          ok = false;
          break;
        }
        const uint32_t dst = sw + s * SLOT_BYTES, bar = su32(&rg.full[s]);
        if (elect_one()) {
          if (p == 0) {
            // the slot just freed was filled in the layer before (two parts back), so the rows
            // are through the one before that, whose biases these replace
            const uint32_t bb = su32(&rg.biasf[li & 1u]), d = su32(rg.sb[li & 1u]);
            mbar_expect_tx(bb, (uint32_t)H * 8u + 32u);
            bulk_load(d, w.e1 + l * w.lstride, (uint32_t)H * 4u, bb);
            bulk_load(d + 1024u, w.e2 + l * w.lstride, (uint32_t)H * 4u, bb);
            bulk_load(d + 2048u, w.e3 + l * w.lstride, 32u, bb);
          }
          if (last) {
            mbar_expect_tx(bar, (uint32_t)H * 32u);
            for (int kb = 0; kb < H / 64; ++kb) tma_load_3d(dst + 2048u * kb, w.v3, 64 * kb, 0, l, bar);
          } else {
            const CUtensorMap* m = p == 0 ? w.v1 : w.v2;
            const int kb0 = p == 0 ? 0 : 2 * (p - 1);
            mbar_expect_tx(bar, (uint32_t)H * 256u);
            tma_load_3d(dst, m, 64 * kb0, 0, l, bar);
            tma_load_3d(dst + (uint32_t)H * 128u, m, 64 * (kb0 + 1), 0, l, bar);
          }
        }
        __syncwarp();
        it += !last;
        thirds += last;
        biases += p == 0;
      }
  if (lane == 0) {
    rg.fills[0] = it;
    rg.fills[1] = thirds;
    rg.fills[2] = biases;
    if (!ok) atomicExch(&rg.abort_flag, 1);
  }
}

__device__ __forceinline__ void fwd_multiply(FwdRing& rg, const FwdWeights& w, uint32_t tmem, uint32_t sx, uint32_t sw) {
  const int lane = threadIdx.x & 31, H = w.H, NR = H / 128;       // 128-column rounds
  const uint32_t sv3 = sw + 2 * SLOT_BYTES;
  const uint32_t id_h = idesc_bf16(FM, (uint32_t)H), id_16 = idesc_bf16(FM, 16);
  uint32_t it = 0, li = 0;
  bool ok = true;
  const int xk = (8 + w.C + 15) / 16;                      // K steps of X that hold values
  auto wait_on = [&](uint64_t* bar, uint32_t parity) -> bool {
    const bool got = mbar_wait_warp(su32(bar), parity, F_WAIT);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    return got;
  };
  for (int t = blockIdx.x; t < w.tiles && ok; t += gridDim.x)
    for (int n = 0; n < w.K && ok; ++n, ++li) {
      // acc1 = X V1^T
      uint32_t slot = it & 1u, wb = sw + slot * SLOT_BYTES;
      if (!(ok = wait_on(&rg.full[slot], (it >> 1) & 1u) && wait_on(&rg.xready, li & 1u))) break;
      if (elect_one()) {
        const uint64_t da = sw128_desc(sx), db = sw128_desc(wb);
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)
          if (kk < xk)
            mma_bf16(tmem, da + (KB_BYTES * (kk >> 2) + 32u * (kk & 3)) / 16,
                     db + ((uint32_t)H * 128u * (kk >> 2) + 32u * (kk & 3)) / 16, id_h, kk != 0);
        mma_commit(su32(&rg.acc1f));
        mma_commit(su32(&rg.empty[slot]));
      }
      __syncwarp();
      ++it;
      // acc2 = g1 V2^T: K round pr (g1 columns 128 pr ..) once the rows have written it
      for (int pr = 0; pr < NR; ++pr) {
        slot = it & 1u, wb = sw + slot * SLOT_BYTES;
        if (!(ok = wait_on(&rg.full[slot], (it >> 1) & 1u) && wait_on(&rg.gready[pr], 0u))) break;
        if (elect_one()) {
          const uint64_t db = sw128_desc(wb);
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            mma_bf16_ts(tmem + ACC2, tmem + 128u * pr + 32u * (kk >> 1) + 8u * (kk & 1),
                        db + ((uint32_t)H * 128u * (kk >> 2) + 32u * (kk & 3)) / 16, id_h, (pr | kk) != 0);
          if (pr == NR - 1) mma_commit(su32(&rg.acc2f));
          mma_commit(su32(&rg.empty[slot]));
        }
        __syncwarp();
        ++it;
      }
      if (!ok) break;
      // acc3 = g2 V3^T (16 rows, 8 of them the conditioner's outputs)
      if (!(ok = wait_on(&rg.full[2], li & 1u))) break;
      for (int r = 0; r < NR; ++r) {
        if (!(ok = wait_on(&rg.gready[r], 1u))) break;
        if (elect_one()) {
          const uint64_t db = sw128_desc(sv3 + 4096u * r);
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            mma_bf16_ts(tmem + ACC3, tmem + ACC2 + 128u * r + 32u * (kk >> 1) + 8u * (kk & 1),
                        db + (2048u * (kk >> 2) + 32u * (kk & 3)) / 16, id_16, (r | kk) != 0);
          if (r == NR - 1) {
            mma_commit(su32(&rg.acc3f));
            mma_commit(su32(&rg.empty[2]));
          }
        }
        __syncwarp();
      }
    }
  if (!ok && lane == 0) atomicExch(&rg.abort_flag, 1);
}

// A row warp's arrival and wait (all lanes; false: given up).
__device__ __forceinline__ void row_arrive(uint64_t* bar) {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(su32(bar));
}
__device__ __forceinline__ bool row_wait(uint64_t* bar, uint32_t parity) {
  const bool got = mbar_wait(su32(bar), parity, F_WAIT);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  return __all_sync(0xffffffffu, got);
}
// The same, false as well when another warp has given up (the flag as one vote of the warp).
__device__ __forceinline__ bool row_wait(uint64_t* bar, uint32_t parity, const int* abort_flag) {
  const bool got = mbar_wait(su32(bar), parity, F_WAIT);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  return !__any_sync(0xffffffffu, !got || *(volatile const int*)abort_flag != 0);
}

// bias + ReLU of the 32 accumulator columns from `at` on (bias: theirs), written over the first
// 16 of them as bfloat16 pairs.  In the fragment shape a thread holds 8 columns of 4 rows and
// reads 8 biases (32 columns of one row would be 32 biases: 512 cycles of shared-memory reads
// a round, of 540): w[k][2 i + e] is row 16 k + 8 e + lane / 4, columns 8 i + 2 (lane % 4) + {0, 1}.
__device__ __forceinline__ void fwd_hidden(uint32_t at, const float* bias, uint32_t w[2][8]) {
  const int lane = threadIdx.x & 31;
  uint32_t raw[32];
  tmem_ld_frag_async(at, raw);
  tmem_ld_frag_async(at + (16u << 16), raw + 16);
  float2 b[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) b[i] = *reinterpret_cast<const float2*>(bias + 8 * i + 2 * (lane & 3));
  tmem_wait_ld32(raw);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float2 s =
          add2(make_float2(__uint_as_float(raw[16 * k + 2 * i]), __uint_as_float(raw[16 * k + 2 * i + 1])), b[i / 2]);
      w[k][i] = pack2_relu(s.x, s.y);
    }
    tmem_st_frag(at + ((uint32_t)(16 * k) << 16), w[k]);
  }
  tmem_wait_st();
}

// Coordinate j of the transformed half, and v[Bc(P, j)] = x[j] for all of them.
template <int P>
__device__ __forceinline__ float half_at(const float* v, int j) {
  return j == 0 ? v[Bc(P, 0)] : j == 1 ? v[Bc(P, 1)] : j == 2 ? v[Bc(P, 2)] : v[Bc(P, 3)];
}
__device__ __forceinline__ float half_at(int p, const float* v, int j) {
  switch (p) {
    case 0: return half_at<0>(v, j);
    case 1: return half_at<1>(v, j);
    case 2: return half_at<2>(v, j);
    default: return half_at<3>(v, j);
  }
}
template <int P>
__device__ __forceinline__ void set_half(float* v, const float* x) {
#pragma unroll
  for (int j = 0; j < 4; ++j) v[Bc(P, j)] = x[j];
}
__device__ __forceinline__ void set_half(int p, float* v, const float* x) {
  switch (p) {
    case 0: set_half<0>(v, x); break;
    case 1: set_half<1>(v, x); break;
    case 2: set_half<2>(v, x); break;
    default: set_half<3>(v, x); break;
  }
}
__device__ __forceinline__ void pack_half(int p, const float* v, uint32_t& w0, uint32_t& w1) {
  switch (p) {
    case 0: pack_half<0>(v, w0, w1); break;
    case 1: pack_half<1>(v, w0, w1); break;
    case 2: pack_half<2>(v, w0, w1); break;
    default: pack_half<3>(v, w0, w1); break;
  }
}

// bfloat16 [layers][rows][cols] with the layers lstride elements apart; boxes of box_cols (64, or
// 32) columns x box_rows rows x one layer, the row of a box as wide as its swizzle.
inline bool layer_map(CUtensorMap* map, const void* base, int64_t cols, int64_t rows, int64_t layers, int64_t lstride,
                      uint32_t box_rows, uint32_t box_cols = 64) {
  auto enc = tensor_map_encoder();
  if (!enc) return false;
  cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)layers};
  cuuint64_t strides[2] = {(cuuint64_t)cols * 2, (cuuint64_t)lstride * 2};
  cuuint32_t box[3] = {box_cols, box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, box_cols == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace flowt
}  // namespace gwx
