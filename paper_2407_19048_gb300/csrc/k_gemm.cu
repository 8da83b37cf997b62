// k_gemm.cu -- C = A B^T with bfloat16 operands and FP32 accumulation on the fifth-
// generation tensor cores: the dense layers of the learned part (the embedding network
// of Sec. 4 and the normalizing flow of Sec. 5) are products of this form.
//
// Persistent CTAs (one per SM) walk the 128 x 256 tiles of C; per CTA:
// - warp 0 streams 128 x 64 (A) and 256 x 64 (B) bfloat16 tiles into shared memory with
//   TMA (cp.async.bulk.tensor, 128-byte swizzle), 192 KiB of stages deep, each stage completing
//   on a "full" mbarrier;
// - warp 1 allocates 512 tensor-memory columns and issues tcgen05.mma (M 128, N 256,
//   K 16; four per stage) into one of two 256-column FP32 accumulators, committing each
//   stage to an "empty" mbarrier (the stage goes back to the producer) and each tile to a
//   "tfull" mbarrier;
// - warps 2-9 drain the accumulator of the previous tile with tcgen05.ld (lane quarter
//   warp % 4 = rows 32 q .. 32 q + 31; two warps per quarter, 128 columns each) and
//   store C, while the next tile accumulates.  Eight draining warps keep the fused
//   epilogue (bias, activation, conversion, stores) off the critical path of products
//   with a short K, where it, not the MMA, sets the time per tile.
// Every mbarrier wait is bounded: on expiry the CTA records a status, stops storing, lets its
// copies and products in flight end (bounded again), frees its tensor memory and returns.
//
// Wide tiles (MW = 2, large products): a CTA computes a 256 x 256 tile of C as two
// M 128 x N 256 products that share each B tile, from three 64 KiB stages (A 256 x 64 in
// one TMA box, B 256 x 64).  Per flop this moves a third less operand data from L2 into
// shared memory than the 128 x 256 tile (the 128 x 256 kernel's operand stream, ~84 B per
// cycle and SM at full tensor rate, is what holds its tensor pipe near 70 %).  The two
// accumulators fill the 512 tensor-memory columns, so a tile's epilogue no longer overlaps
// the next tile's products (~2 % at K = 8192); the eight draining warps take one
// accumulator half each.
//
// Operand layouts (OPS): besides A [M][K] and B [N][K] (both K-major), B or both operands
// can be read as they lie when K is their row index ("MN-major": boxes of 64 columns x 64
// rows, transposed by the tensor core's operand descriptors), so that the products of a
// dense layer's backward, dX = dZ W and dW = dZ^T X, need no transposed copies.
//
// Split K: a product with few tiles and a long K (the weight gradients dW = dZ^T X, whose
// K is the batch) would run on a handful of SMs.  There the work list is (tile, K slice)
// pairs: slice s covers K blocks [s kbs, (s + 1) kbs) and stores its FP32 partial product
// at C + s M N; a second kernel sums the slices in a fixed order (deterministic).
#include <cuda.h>
#include <cuda_bf16.h>

#include "gwx_internal.h"
#include "pdl.cuh"
#include "tc05.cuh"

namespace gwx {

namespace {

using namespace tc;

constexpr int GM = 128, GN = 256, GK = 64;               // GN: the dense products' tile width
constexpr int EPI_WARPS = 8;                            // two per tensor-memory lane quarter
constexpr int GEMM_THREADS = 64 + 32 * EPI_WARPS;
constexpr uint32_t WAIT_POLLS = 1u << 22;
constexpr uint32_t EPI_BUF_BYTES = 32 * 32 * 4;         // per epilogue warp: a 32 x 32 FP32 transpose tile

// Per tile width TN_ (64, 128 or 256 columns of C) and M-tiles per CTA MW (1, or 2 with
// TN_ = 256): B tile, stage and accumulator sizes.  MW = 1: two accumulators of TN_
// columns alternate between tiles; MW = 2: one pair (rows 0-127, 128-255) per tile.
template <int TN_, int MW = 1>
struct Tile {
  static_assert(MW == 1 || (MW == 2 && TN_ == 256), "wide tiles are 256 x 256");
  static constexpr int ROWS = GM * MW;                     // rows of C per tile
  static constexpr uint32_t A_TILE = (uint32_t)ROWS * GK * 2;
  static constexpr uint32_t B_BYTES = TN_ * GK * 2;
  static constexpr uint32_t BLOCK_BYTES = A_TILE + B_BYTES;
  // K blocks per stage: a stage costs the issuing warp ~250 cycles of wait, poll and commit
  // besides its MMAs (~130 cycles a K block at 64 columns), so the narrowest tiles take two at
  // a time (128 x 64 tiles at K = 3968: 22.4 us with lane-wise issue, 17.6, 14.6)
  static constexpr int KPS = TN_ == 64 ? 2 : 1;
  static constexpr uint32_t STAGE_BYTES = KPS * BLOCK_BYTES;
  // 192 KiB of stages: a narrow tile's K blocks are small, and a product with few tiles and a
  // long K is bound by the latency of its stages, so it keeps more of them in flight
  static constexpr int NSTAGE = 192 * 1024 / (int)STAGE_BYTES;
  static constexpr int NACC = MW == 1 ? 2 : 1;             // accumulator sets in tensor memory
  static constexpr uint32_t TMEM_COLS = TN_;              // FP32 columns of one accumulator
  static constexpr size_t SMEM = (size_t)NSTAGE * STAGE_BYTES + (size_t)EPI_WARPS * EPI_BUF_BYTES + 1024;
};

// Implicit-GEMM convolution geometry (conv mode): A is the channels-last activation
// x [B][T][Cin] as a 3-D tensor map; M tile tm covers times 128 (tm mod T/128) ..
// + 127 of sample tm div (T/128), and K block kb covers tap kb div KC, channels
// 64 (kb mod KC) .. + 63, read at time t + dir (tap - pad) (zero outside [0, T)).
struct ConvGeo {
  int T;     // time steps per sample (a multiple of 128)
  int KC;    // Cin / 64
  int pad;   // (k - 1) / 2
  int dir;   // +1: convolution; -1: its input gradient (taps mirrored)
};

// Operand layouts of the kernel.
enum : int {
  OP_KK = 0,       // A [M][K], B [N][K]
  OP_NN = 1,       // A [M][K], B [K][N]
  OP_TN = 2,       // A [groups][K][M], B [groups][K][N]
  OP_CONV = 3,     // A an implicit im2col tile (ConvGeo), B [N][K]
  OP_CONV_NN = 4,  // A an implicit im2col tile, B [K / k][k N] (tap-major columns: the input gradient's weights)
  OP_CONV_TN = 5   // A [K][M] rows of times, B the implicit im2col rows [K][N], N = k Cin (the weight gradient)
};
constexpr bool op_a_mn(int op) { return op == OP_TN || op == OP_CONV_TN; }
constexpr bool op_b_mn(int op) { return op == OP_NN || op == OP_TN || op == OP_CONV_NN || op == OP_CONV_TN; }
constexpr bool op_conv_a(int op) { return op == OP_CONV || op == OP_CONV_NN; }

// What the epilogue writes: FP32, bfloat16, or dZ = dY act'(Z) in bfloat16 for the product
// Z = A B^T + bias, with the FP32 column sums of every 32 rows.
enum : int { OUT_F32 = 0, OUT_BF16 = 1, OUT_DACT = 2 };

__device__ __forceinline__ float act_grad(float z, int act) {
  if (act == 1) return z > 0.f ? 1.f : 0.f;
  if (act == 2)   // GELU: Phi(z) + z phi(z)
    return 0.5f * erfcf(-0.70710678118654752f * z) + z * 0.39894228040143268f * expf(-0.5f * z * z);
  return 1.f;
}

__device__ int g_gemm_status;

// Four consecutive floats from p (n of them exist; vec: p is 16-byte aligned and n >= 4).
__device__ __forceinline__ float4 load4(const float* p, int n, bool vec) {
  if (vec) return *reinterpret_cast<const float4*>(p);
  return make_float4(p[0], n > 1 ? p[1] : 0.f, n > 2 ? p[2] : 0.f, n > 3 ? p[3] : 0.f);
}

__device__ __forceinline__ float act_of(float z, int act) {
  if (act == 1) return fmaxf(z, 0.f);
  if (act == 2) return 0.5f * z * erfcf(-0.70710678118654752f * z);
  return z;
}

// Division by a number known at launch: q = floor(n m / 2^32) with m = floor(2^32 / d) + 1 is
// the quotient or one more for every 32-bit n (m d - 2^32 <= d).
struct Div {
  uint32_t d, m;   // m = 0: d = 1
};
inline Div make_div(int64_t d) { return d <= 1 ? Div{1u, 0u} : Div{(uint32_t)d, 0xffffffffu / (uint32_t)d + 1u}; }
__device__ __forceinline__ int divide(const Div& v, int n, int& rem) {
  uint32_t q = v.m ? __umulhi((uint32_t)n, v.m) : (uint32_t)n;
  int r = n - (int)(q * v.d);
  if (r < 0) {
    --q;
    r += (int)v.d;
  }
  rem = r;
  return (int)q;
}

// Work item w of a persistent CTA -> K slice, group z and tile (tm, tn), tile fastest; the tiles
// in bands of `group` tile-rows, columns fastest within a band, so that the CTAs working at
// the same time share a few A and B panels in L2.  (Plain divisions cost every role of the
// kernel 640 cycles a tile, as much as four K blocks.)
constexpr int DEFAULT_GROUP = 16;
struct WorkMap {
  Div per, tiles, band, group, last;   // last: the rows of the last band
  int TM;
};
inline WorkMap make_work_map(int64_t TM, int64_t TN, int group, int groups) {
  const int64_t rest = TM % group;
  return WorkMap{make_div(TM * TN * groups), make_div(TM * TN), make_div(group * TN), make_div(group),
                 make_div(rest ? rest : group), (int)TM};
}
struct WorkItem {
  int tm, tn, z, slice;
};
__device__ __forceinline__ WorkItem work_item(const WorkMap& m, int w) {
  WorkItem i;
  int r, t;
  i.slice = divide(m.per, w, r);
  i.z = divide(m.tiles, r, t);
  const int first = divide(m.band, t, r) * (int)m.group.d;
  i.tn = divide(first + (int)m.group.d <= m.TM ? m.group : m.last, r, i.tm);
  i.tm += first;
  return i;
}

// The epilogue of a turned 32 x 32 tile at (row0, c0) whose rows are not multiples of four values: a
// lane keeps P values of a row, W / P lanes a row (W = 8 in a narrow product), value by value to
// memory, bfloat16 pairs whole where N is even.  Eight values are read, finished and written at a
// time.  (8192 x 1001 x 512: four columns a lane 30.8 us FP32 and 30.7 bfloat16, value by value 24.6
// and 24.7, now 18.2 and 18.6; 20000 x 7 x 128 8.3, now 6.3.)
template <int OUT, int W>
__device__ __forceinline__ void ragged_rows(uint32_t ebuf, void* out, const float* bias, int act, int row0, int c0, int M,
                                            int N) {
  constexpr int P = OUT == OUT_F32 ? 1 : 2, L = W / P, RPI = 32 / L;   // lanes a row, rows an iteration
  int lane = threadIdx.x & 31;
  asm volatile("" : "+r"(lane));   // (what follows from it is not kept in registers across the other path's loop)
  const int cl = P * (lane % L), col = c0 + cl, rl = lane / L;
  const bool in0 = col < N, in1 = P == 2 && col + 1 < N, pairs = N % 2 == 0;
  const float b0 = bias != nullptr && in0 ? bias[col] : 0.f, b1 = bias != nullptr && in1 ? bias[col + 1] : 0.f;
  constexpr int U = L < 8 ? L : 8;
  int64_t at = (int64_t)(row0 + rl) * N + col;
#pragma unroll 1
  for (int k0 = 0; k0 < L; k0 += U) {
    float v0[U], v1[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int r = RPI * (k0 + k) + rl;
      const uint32_t src = ebuf + 128u * r + (uint32_t)(((cl >> 2) ^ (r & 7)) << 4) + 4u * (cl & 3);
      if constexpr (P == 1) v0[k] = lds32(src);
      else lds64(src, v0[k], v1[k]);
    }
    if (bias != nullptr) {
#pragma unroll
      for (int k = 0; k < U; ++k) {
        v0[k] += b0;
        if (P == 2) v1[k] += b1;
      }
    }
    if (act != 0) {
#pragma unroll
      for (int k = 0; k < U; ++k) {
        v0[k] = act_of(v0[k], act);
        if (P == 2) v1[k] = act_of(v1[k], act);
      }
    }
#pragma unroll
    for (int k = 0; k < U; ++k, at += (int64_t)RPI * N) {
      if (row0 + RPI * (k0 + k) + rl >= M || !in0) continue;
      if constexpr (P == 1) {
        reinterpret_cast<float*>(out)[at] = v0[k];
      } else {
        __nv_bfloat16* o = reinterpret_cast<__nv_bfloat16*>(out) + at;
        if (pairs) {
          *reinterpret_cast<__nv_bfloat162*>(o) = __floats2bfloat162_rn(v0[k], v1[k]);
        } else {
          o[0] = __float2bfloat16_rn(v0[k]);
          if (in1) o[1] = __float2bfloat16_rn(v1[k]);
        }
      }
    }
  }
}

// Persistent, warp-specialised: warp 0 produces (TMA), warp 1 allocates tensor memory and
// issues the MMAs, one elected lane of their uniform loops each; warps 2-9 drain accumulators.  MW = 1: two
// TN_-column accumulators alternate between tiles, so a tile's epilogue overlaps the next
// tile's main loop; MW = 2 (256 x 256 tiles): the two accumulators are the tile's two
// 128-row halves and the next tile waits for both to drain.  "tfull" (MMA commit) and
// "tempty" (one arrival per epilogue warp) hand them over.
// TN_: tile width; OPS: operand layouts.  extra: with OUT_DACT the dY of C = dY act'(Z)
// (N % 8 == 0, 4-byte aligned); of a convolution an optional addend (N % 64 == 0, 16-byte
// aligned): C = A B^T + addend.  colsum (OUT_DACT): [ceil(M/32)][N], 16-byte aligned.
// groups: independent products (OP_TN; map coordinate z), group g's C at + g cstride; with
// splits > 1 the slice's partial product of group g at C + (slice groups + g) M N.
template <int OUT, int TN_, int OPS, int MW = 1>
__global__ void __launch_bounds__(GEMM_THREADS, 1)
    k_gemm_bf16(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb, void* __restrict__ C,
                const float* bias, int act, const WorkMap map, int M, int N, int K, int kbs, int splits,
                const float* extra, float* __restrict__ colsum, int groups, int64_t cstride,
                ConvGeo geo) {
  static_assert(MW == 1 || OPS == OP_KK, "wide tiles are for plain products");
  constexpr bool A_MN = op_a_mn(OPS), B_MN = op_b_mn(OPS);
  constexpr uint32_t CHUNK = 64 * GK * 2;   // one 64-column box of an MN-major operand
  constexpr int GN = TN_;
  using TL = Tile<TN_, MW>;
  constexpr int GMT = TL::ROWS;
  constexpr int STAGES = TL::NSTAGE;
  constexpr int NACC = TL::NACC;
  constexpr uint32_t A_BYTES = TL::A_TILE;
  constexpr uint32_t STAGE_BYTES = TL::STAGE_BYTES, BLOCK_BYTES = TL::BLOCK_BYTES;
  constexpr int KPS = TL::KPS;
  constexpr uint32_t TMEM_COLS = TL::TMEM_COLS;
  constexpr uint32_t IDESC = idesc_bf16(GM, TN_, A_MN, B_MN);
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES], tfull[2], tempty[2], drained;
  __shared__ uint32_t tmem_slot, fill_stage, fill_phase;   // (of the producer's next fill, once it has stopped)
  __shared__ int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t base = (su32(smem_raw) + 1023u) & ~1023u;   // 1024-byte aligned stages
  const int KB = (K + GK - 1) / GK;
  const int work = (int)map.per.d * splits;   // (tile, group, K slice) triples, tile fastest

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(su32(&full[s]), 1);
      mbar_init(su32(&empty[s]), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(su32(&tfull[a]), 1);
      mbar_init(su32(&tempty[a]), EPI_WARPS);
    }
    mbar_init(su32(&drained), 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&tmem_slot)),
                 "r"(2 * TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  pdl_enter();

  if (warp == 0) {
    uint32_t s = 0, ph = 1;   // stage and the parity of its "empty" phase (the first round finds them free)
    bool ok = true, ready = true;
    for (int w = blockIdx.x; w < work && ok; w += gridDim.x) {
      const WorkItem item = work_item(map, w);
      const int tm = item.tm, tn = item.tn, z = item.z;
      const int kb0 = item.slice * kbs, kb1 = min(KB, kb0 + kbs);
      for (int k0 = kb0; k0 < kb1; k0 += KPS) {
        if (!__all_sync(0xffffffffu, ready) && !mbar_wait_warp(su32(&empty[s]), ph, WAIT_POLLS)) {
          ok = false;
          break;
        }
        const uint32_t st = base + s * STAGE_BYTES, bar = su32(&full[s]);
        const int nk = min(KPS, kb1 - k0);
        if (++s == STAGES) {
          s = 0;
          ph ^= 1u;
        }
        // the next stage's poll overlaps the copies' issue (not with the wide tiles, whose
        // 1024 cycles of MMAs a stage hide it)
        ready = MW == 1 && mbar_test(su32(&empty[s]), ph);
        if (elect_one()) {
          mbar_expect_tx(bar, (uint32_t)nk * BLOCK_BYTES);
#pragma unroll
          for (int j = 0; j < KPS; ++j) {
            if (j >= nk) break;
            const int kb = k0 + j;
            const uint32_t sa = st + (uint32_t)j * BLOCK_BYTES, sb = sa + A_BYTES;
            if constexpr (op_conv_a(OPS)) {
              const int tpb = geo.T / GM;   // M tiles per sample
              const int tap = kb / geo.KC, cb = kb - tap * geo.KC;
              tma_load_3d(sa, &ta, cb * GK, (tm % tpb) * GM + geo.dir * (tap - geo.pad), tm / tpb, bar);
              if constexpr (B_MN) {   // rows cb GK .. of [K / k][k N], columns of tap `tap`
#pragma unroll
                for (int c = 0; c < TN_ / 64; ++c)
                  tma_load_2d(sb + c * CHUNK, &tb, tap * N + min(tn * GN + 64 * c, N - 64), cb * GK, bar);
              }
            } else if constexpr (A_MN) {
#pragma unroll
              for (int c = 0; c < GM / 64; ++c)
                tma_load_3d(sa + c * CHUNK, &ta, tm * GM + 64 * c, kb * GK, z, bar);
            } else {
              tma_load_2d(sa, &ta, kb * GK, tm * GMT, bar);   // one box of GMT rows
            }
            if constexpr (OPS == OP_CONV_TN) {
              // 64 times of one sample (T % 128 == 0); columns past N repeat the last 64
              const int row = kb * GK, b = row / geo.T, t0 = row - b * geo.T;
#pragma unroll
              for (int c = 0; c < TN_ / 64; ++c) {
                const int col = min(tn * GN + 64 * c, N - 64) / 64, tap = col / geo.KC;
                tma_load_3d(sb + c * CHUNK, &tb, (col - tap * geo.KC) * 64, t0 + tap - geo.pad, b, bar);
              }
            } else if constexpr (OPS == OP_TN) {
#pragma unroll
              for (int c = 0; c < TN_ / 64; ++c)
                tma_load_3d(sb + c * CHUNK, &tb, tn * GN + 64 * c, kb * GK, z, bar);
            } else if constexpr (OPS == OP_NN) {
#pragma unroll
              for (int c = 0; c < TN_ / 64; ++c)
                tma_load_2d(sb + c * CHUNK, &tb, tn * GN + 64 * c, kb * GK, bar);
            } else if constexpr (!B_MN) {
              tma_load_2d(sb, &tb, kb * GK, tn * GN, bar);
            }
          }
        }
        __syncwarp();
      }
      if (*(volatile int*)&abort_flag) ok = false;
      ok = __all_sync(0xffffffffu, ok);
    }
    if (lane == 0) {
      fill_stage = s;
      fill_phase = ph;
      if (!ok) atomicExch(&abort_flag, 1);
    }
  } else if (warp == 1) {
    uint32_t s = 0, ph = 0, tl = 0;
    bool ok = true;
    for (int w = blockIdx.x; w < work && ok; w += gridDim.x, ++tl) {
      const uint32_t acc = tl % NACC;
      int unused;
      const int kb0 = divide(map.per, w, unused) * kbs, kb1 = min(KB, kb0 + kbs);
      if (tl >= NACC && !mbar_wait_warp(su32(&tempty[acc]), ((tl / NACC) - 1) & 1u, WAIT_POLLS)) {
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t d = tmem + acc * TMEM_COLS;
      bool ready = false;   // the coming stage's poll, taken while the MMAs before it are issued
      for (int k0 = kb0; k0 < kb1; k0 += KPS) {
        if (!__all_sync(0xffffffffu, ready) && !mbar_wait_warp(su32(&full[s]), ph, WAIT_POLLS)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t st = base + s * STAGE_BYTES, done = su32(&empty[s]);
        const int nk = min(KPS, kb1 - k0);
        if (++s == STAGES) {
          s = 0;
          ph ^= 1u;
        }
        ready = MW == 1 && k0 + KPS < kb1 && mbar_test(su32(&full[s]), ph);
        if (elect_one()) {
#pragma unroll
          for (int j = 0; j < KPS; ++j) {
            if (j >= nk) break;
            const uint32_t sa = st + (uint32_t)j * BLOCK_BYTES, sb = sa + A_BYTES;
#pragma unroll
            for (int kk = 0; kk < GK / 16; ++kk) {   // 16 bfloat16 = 32 bytes along K per instruction
              // M-tile m: rows 128 m .. of the A box (16 KiB apart), accumulator columns m TN_ ..
#pragma unroll
              for (int m = 0; m < MW; ++m)
                mma_bf16(d + (uint32_t)m * TMEM_COLS,
                         A_MN ? sw128_mn_desc(sa + 2048u * kk, CHUNK)
                              : sw128_desc(sa + (uint32_t)m * (GM * GK * 2) + 32u * kk),
                         B_MN ? sw128_mn_desc(sb + 2048u * kk, CHUNK) : sw128_desc(sb + 32u * kk), IDESC,
                         k0 + j != kb0 || kk != 0);
            }
          }
          mma_commit(done);
        }
        __syncwarp();
      }
      if (elect_one()) mma_commit(su32(&tfull[acc]));   // arrives once the tile's MMAs have completed
      __syncwarp();
      if (*(volatile int*)&abort_flag) ok = false;
      ok = __all_sync(0xffffffffu, ok);
    }
    if (!ok && lane == 0) atomicExch(&abort_flag, 1);
  } else {
    // epilogue warps 2-9; tensor-memory lane quarter (warp % 4) = tile rows 32 q .. 32 q + 31;
    // (warp - 2) / 4 picks the column half (MW = 1) or the M-tile (MW = 2, all columns)
    const int q = warp & 3;
    const int hsel = (warp - 2) >> 2;
    const int c_lo = MW == 1 ? hsel * (GN / 64) : 0, c_hi = MW == 1 ? c_lo + GN / 64 : GN / 32;
    const int msel = MW == 1 ? 0 : hsel;
    const uint32_t ebuf = base + STAGES * STAGE_BYTES + (uint32_t)(warp - 2) * EPI_BUF_BYTES;
    uint32_t tl = 0;
    for (int w = blockIdx.x; w < work; w += gridDim.x, ++tl) {
      const WorkItem item = work_item(map, w);
      const int tm = item.tm, tn = item.tn;
      const size_t slice = splits > 1 ? (size_t)(item.slice * groups + item.z) * (size_t)M * (size_t)N
                                      : (size_t)item.z * (size_t)cstride;
      const uint32_t acc = tl % NACC;
      const bool have = mbar_wait(su32(&tfull[acc]), (tl / NACC) & 1u, WAIT_POLLS);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (__any_sync(0xffffffffu, !have || *(volatile int*)&abort_flag != 0)) {
        if (lane == 0) atomicExch(&abort_flag, 1);
        break;
      }
      // Each warp turns 32 rows x 32 columns around in a shared tile (16-byte chunk j of row r at
      // chunk j ^ (r mod 8): conflict-free both ways), after which a lane holds four consecutive
      // columns of rows 4 k + lane / 8: bias, addend and dY are read, and C written, four values
      // at a time and four whole row segments an instruction.  (One value at a time, with the
      // bias read by every row, the epilogue of one tile took 8000 cycles at 128 columns of
      // bfloat16, 25000 with dY, 16000 at 256 columns of FP32: as long as the products.)
      const int row0 = tm * GMT + GM * msel + 32 * q;
      const int c_end = row0 < M ? min(c_hi, (N - tn * GN + 31) / 32) : c_lo;
      const uint32_t tcol = tmem + ((uint32_t)(32 * q) << 16) + (acc + (uint32_t)msel) * TMEM_COLS;
      // Rows that are not multiples of four values (plain products alone; the others' N is a
      // multiple of 8 and their C 16-byte aligned): ragged_rows.
      constexpr int ESZ = OUT == OUT_F32 ? 4 : 2;
      uint8_t* out = reinterpret_cast<uint8_t*>(C) + slice * ESZ;
      constexpr bool EXTRA = OUT == OUT_DACT || op_conv_a(OPS);
      constexpr bool RAGGED = OPS == OP_KK && OUT != OUT_DACT;
      const bool vec = !RAGGED || (N % 4 == 0 && (uintptr_t)out % (4 * ESZ) == 0);
      const bool vec_b = (uintptr_t)bias % 16 == 0, vec_x = N % 4 == 0 && (uintptr_t)extra % 16 == 0;
      const int rl = lane >> 3, jc = lane & 7;
      uint32_t raw[32];
      if (c_lo < c_end) tmem_ld32_async(tcol + 32u * c_lo, raw);
#pragma unroll 1
      for (int c = c_lo; c < c_end; ++c) {
        const int col = tn * GN + 32 * c + 4 * jc, left = N - col;   // this lane's columns
        // the rows' addend or dY, and the bias, before the accumulator, so that their latency
        // overlaps the tensor-memory load
        float4 x[8], b4 = make_float4(0.f, 0.f, 0.f, 0.f);
        if (EXTRA && extra != nullptr) {
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const int r = row0 + 4 * k + rl;
            x[k] = r < M && left > 0 ? load4(extra + (int64_t)r * N + col, left, vec_x) : make_float4(0.f, 0.f, 0.f, 0.f);
          }
        }
        if (bias != nullptr && vec && left > 0) b4 = load4(bias + col, left, vec_b && left >= 4);
        tmem_wait_ld32(raw);
#pragma unroll
        for (int j = 0; j < 8; ++j)
          sts128(ebuf + 128u * lane + (uint32_t)((j ^ (lane & 7)) << 4), raw[4 * j], raw[4 * j + 1], raw[4 * j + 2],
                 raw[4 * j + 3]);
        __syncwarp();
        if (RAGGED && !vec) {
          const int c0 = tn * GN + 32 * c;
          if (N - c0 > 8) ragged_rows<OUT, 32>(ebuf, out, bias, act, row0, c0, M, N);
          else ragged_rows<OUT, 8>(ebuf, out, bias, act, row0, c0, M, N);
          __syncwarp();
          if (c + 1 < c_end) tmem_ld32_async(tcol + 32u * (c + 1), raw);
          continue;
        }
        if (c + 1 < c_end) tmem_ld32_async(tcol + 32u * (c + 1), raw);
        float4 sum = make_float4(0.f, 0.f, 0.f, 0.f), vk[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int r = 4 * k + rl;
          vk[k] = lds128(ebuf + 128u * r + (uint32_t)((jc ^ (r & 7)) << 4));
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int grow = row0 + 4 * k + rl;
          float4 v = vk[k];
          if (EXTRA && OUT != OUT_DACT && extra != nullptr) {
            v.x += x[k].x;
            v.y += x[k].y;
            v.z += x[k].z;
            v.w += x[k].w;
          }
          if (bias != nullptr) {
            v.x += b4.x;
            v.y += b4.y;
            v.z += b4.z;
            v.w += b4.w;
          }
          if constexpr (OUT == OUT_DACT) {
            float4 a = x[k];
            if (act != 0) {
              a.x *= act_grad(v.x, act);
              a.y *= act_grad(v.y, act);
              a.z *= act_grad(v.z, act);
              a.w *= act_grad(v.w, act);
            }
            v = a;
            sum.x += a.x;
            sum.y += a.y;
            sum.z += a.z;
            sum.w += a.w;
          } else if (act != 0) {
            v = make_float4(act_of(v.x, act), act_of(v.y, act), act_of(v.z, act), act_of(v.w, act));
          }
          if (grow >= M || left <= 0) continue;
          if constexpr (OUT == OUT_F32) {
            *reinterpret_cast<float4*>(reinterpret_cast<float*>(out) + (int64_t)grow * N + col) = v;
          } else {
            const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
            *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(out) + (int64_t)grow * N + col) =
                make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
          }
        }
        if constexpr (OUT == OUT_DACT) {
#pragma unroll
          for (int o = 16; o >= 8; o >>= 1) {
            sum.x += __shfl_xor_sync(0xffffffffu, sum.x, o);
            sum.y += __shfl_xor_sync(0xffffffffu, sum.y, o);
            sum.z += __shfl_xor_sync(0xffffffffu, sum.z, o);
            sum.w += __shfl_xor_sync(0xffffffffu, sum.w, o);
          }
          if (rl == 0 && left > 0) {
            *reinterpret_cast<float4*>(colsum + (int64_t)(row0 / 32) * N + col) = sum;
          }
        }
        __syncwarp();
      }
      // the accumulator is drained: hand it back to the MMA issuer
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(su32(&tempty[acc]));
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (*(volatile int*)&abort_flag) {
    if (threadIdx.x == 0) atomicExch(&g_gemm_status, 1);
    if (warp == 0) ring_drain(full, STAGES, fill_stage, fill_phase, WAIT_POLLS);
    if (warp == 1) mma_drain(&drained, WAIT_POLLS);
    __syncthreads();
  }
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * TMEM_COLS) : "memory");
}

// Row-major bfloat16 [groups][rows][cols], groups gstride elements apart, as a 3-D tensor
// map with boxes of 64 columns x 64 rows (an MN-major operand).
bool make_map_mn(CUtensorMap* map, const void* ptr, int64_t rows, int64_t cols, int64_t groups, int64_t gstride) {
  auto enc = tensor_map_encoder();
  if (!enc) return false;
  cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)groups};
  cuuint64_t strides[2] = {(cuuint64_t)cols * 2, (cuuint64_t)gstride * 2};
  cuuint32_t box[3] = {64, (cuuint32_t)GK, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Row-major bfloat16 [rows][K] as a 2-D tensor map with boxes of box_rows x 64.
bool make_map(CUtensorMap* map, const void* ptr, int64_t rows, int64_t K, uint32_t box_rows) {
  auto enc = tensor_map_encoder();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)K * 2};
  cuuint32_t box[2] = {(cuuint32_t)GK, box_rows};
  cuuint32_t estr[2] = {1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// out[g][i] = sum over s of part[s][g][i] for i < n (a multiple of 4, 16-byte aligned); groups
// of out ostride apart.  Four elements a thread; LANES threads share them, lane y taking slices
// y, y + LANES, ... in order, then the lanes in order: deterministic.  Eight lanes for many
// slices of a small result (64 of 64 x 320: 21 us one thread an element, 5 with eight lanes),
// one for few slices of a large one (4 of 512 x 1968), where idle lanes only cost.
template <int LANES>
__global__ void __launch_bounds__(256) k_split_reduce(const float4* part, int splits, int64_t n4,
                                                      int64_t ostride4, float4* __restrict__ out) {
  pdl_enter();
  constexpr int X = 256 / LANES;
  __shared__ float4 red[LANES][X];
  const int x = threadIdx.x % X, y = threadIdx.x / X;
  const int64_t i = (int64_t)blockIdx.x * X + x;
  const int64_t total = n4 * gridDim.y;
  const float4* p = part + (int64_t)blockIdx.y * n4 + i;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  auto add = [&acc](float4 v) {
    acc.x += v.x;
    acc.y += v.y;
    acc.z += v.z;
    acc.w += v.w;
  };
  if (i < n4) {
#pragma unroll 4
    for (int s = y; s < splits; s += LANES) add(p[(int64_t)s * total]);
  }
  if constexpr (LANES > 1) {
    red[y][x] = acc;
    __syncthreads();
    if (y != 0) return;
#pragma unroll
    for (int k = 1; k < LANES; ++k) add(red[k][x]);
  }
  if (i < n4) out[(int64_t)blockIdx.y * ostride4 + i] = acc;
}

// Everything of a launch but the operands.
struct GemmCall {
  void* C;
  int64_t M, N, K;
  const float* bias = nullptr;
  int act = 0;
  int group = DEFAULT_GROUP;
  int splits = 1;
  const float* extra = nullptr;
  float* colsum = nullptr;
  int groups = 1;
  int64_t cstride = 0;
  ConvGeo geo{0, 0, 0, 0};
};

cudaError_t sm_count(int* sms) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
  return e;
}

template <int OUT, int TN_, int OPS, int MW = 1>
cudaError_t run_gemm(const CUtensorMap& ta, const CUtensorMap& tb, const GemmCall& c, int sms, cudaStream_t s) {
  const int KB = (int)((c.K + GK - 1) / GK);
  const int kbs = (KB + c.splits - 1) / c.splits;   // every slice has at least one K block
  const int splits = (KB + kbs - 1) / kbs;
  const int64_t TM = (c.M + Tile<TN_, MW>::ROWS - 1) / Tile<TN_, MW>::ROWS, TN = (c.N + TN_ - 1) / TN_;
  const int64_t work = TM * TN * splits * c.groups;
  const unsigned grid = (unsigned)(work < sms ? work : sms);   // persistent: one CTA per SM
  constexpr size_t smem = Tile<TN_, MW>::SMEM;
  auto kern = k_gemm_bf16<OUT, TN_, OPS, MW>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  pdl_launch(kern, dim3(grid), dim3(GEMM_THREADS), smem, s, ta, tb, c.C, c.bias, c.act,
             make_work_map(TM, TN, c.group, c.groups), (int)c.M, (int)c.N, (int)c.K, kbs, splits, c.extra, c.colsum,
             c.groups, c.cstride, c.geo);
  return cudaGetLastError();
}

// The same at a tile width chosen at run time.
template <int OUT, int OPS>
cudaError_t run_gemm_at(int tn, const CUtensorMap& ta, const CUtensorMap& tb, const GemmCall& c, int sms,
                        cudaStream_t s) {
  if (tn == 64) return run_gemm<OUT, 64, OPS>(ta, tb, c, sms, s);
  if (tn == 128) return run_gemm<OUT, 128, OPS>(ta, tb, c, sms, s);
  return run_gemm<OUT, 256, OPS>(ta, tb, c, sms, s);
}

// Tile width of a product: 256 columns unless the 128 x 256 tiles would leave more than half
// of the SMs idle (the flow's conditioner products on a few hundred to a few thousand rows),
// then 128 or 64, so that more CTAs share the work; no wider than N needs (the stem's product
// has 64 columns).
int gemm_tile_width(int64_t M, int64_t N, int sms) {
  const int64_t tm = (M + GM - 1) / GM;
  for (int tn : {256, 128})
    if (2 * N > tn && tm * ((N + tn - 1) / tn) * 2 >= sms) return tn;
  return 64;
}

// Wide 256 x 256 tiles for large products: a K long enough that the epilogue
// (no longer overlapped) is a small part of a tile, at least one full wave of them, and no
// GELU (its erfc epilogue, unoverlapped, cost more than the wide tiles gained: 0.77 vs
// 0.73 ms for an 8192^3 dense layer).
bool gemm_wide(int64_t M, int64_t N, int64_t K, int act, int sms) {
  return K >= 1024 && act != GWX_ACT_GELU && ((M + 255) / 256) * ((N + 255) / 256) >= sms;
}

// C = A B^T with A [M][K], B [N][K]; OUT as in the kernel.
template <int OUT>
cudaError_t launch_gemm(const void* A, const void* B, GemmCall c, cudaStream_t s) {
  if (c.group < 1) c.group = DEFAULT_GROUP;
  int sms = 0;
  cudaError_t e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  CUtensorMap ta, tb;
  if constexpr (OUT != OUT_DACT) {
    if (gemm_wide(c.M, c.N, c.K, c.act, sms)) {
      if (!make_map(&ta, A, c.M, c.K, 2 * GM) || !make_map(&tb, B, c.N, c.K, 256)) return cudaErrorInvalidValue;
      return run_gemm<OUT, 256, OP_KK, 2>(ta, tb, c, sms, s);
    }
  }
  const int tn = gemm_tile_width(c.M, c.N, sms);
  if (!make_map(&ta, A, c.M, c.K, GM) || !make_map(&tb, B, c.N, c.K, (uint32_t)tn)) return cudaErrorInvalidValue;
  return run_gemm_at<OUT, OP_KK>(tn, ta, tb, c, sms, s);
}

// Channels-last bfloat16 x [Bn][T][C] as a 3-D tensor map with boxes of 64 channels x
// box_t times.
bool make_map_3d(CUtensorMap* map, const void* ptr, int64_t Bn, int64_t T, int64_t C, uint32_t box_t) {
  auto enc = tensor_map_encoder();
  if (!enc) return false;
  cuuint64_t dims[3] = {(cuuint64_t)C, (cuuint64_t)T, (cuuint64_t)Bn};
  cuuint64_t strides[2] = {(cuuint64_t)C * 2, (cuuint64_t)T * C * 2};
  cuuint32_t box[3] = {(cuuint32_t)GK, box_t, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

// Implicit-GEMM 1-D convolution, stride 1, "same" zero padding: out [Bn][T][N] (FP32) =
// sum over taps j < k and channels c of x[b][t + dir (j - (k-1)/2)][c] Wj[c][o], plus addend
// if given.  dir +1: Wj[c][o] = W[o][j C + c] for W [N][k C] (the convolution); dir -1:
// Wj[c][o] = W[c][j N + o] for W [C][k N] (its input gradient, C the output channels of the
// convolution, whose weights are read as they lie).  Tile width 64 / 128 / 256 by N.
// Shapes checked by the caller.
cudaError_t launch_conv_gemm(const void* x, int64_t Bn, int64_t T, int64_t C, int k, int dir, const void* W, int64_t N,
                             float* out, const float* addend, cudaStream_t s) {
  CUtensorMap ta, tb;
  GemmCall c{out, Bn * T, N, (int64_t)k * C};
  c.extra = addend;
  c.geo = ConvGeo{(int)T, (int)(C / GK), (k - 1) / 2, dir};
  const int tn = N <= 64 ? 64 : (N <= 128 ? 128 : 256);
  int sms = 0;
  cudaError_t e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  if (!make_map_3d(&ta, x, Bn, T, C, GM)) return cudaErrorInvalidValue;
  if (dir > 0) {
    if (!make_map(&tb, W, N, c.K, (uint32_t)tn)) return cudaErrorInvalidValue;
    return run_gemm_at<OUT_F32, OP_CONV>(tn, ta, tb, c, sms, s);
  }
  if (!make_map(&tb, W, C, (int64_t)k * N, GK)) return cudaErrorInvalidValue;   // boxes of 64 x 64
  return run_gemm_at<OUT_F32, OP_CONV_NN>(tn, ta, tb, c, sms, s);
}

cudaError_t launch_gemm_bf16(const void* A, const void* B, void* C, int64_t M, int64_t N, int64_t K, bool out_bf16,
                             const float* bias, int act, int group, cudaStream_t s) {
  GemmCall c{C, M, N, K};
  c.bias = bias;
  c.act = act;
  c.group = group;
  return out_bf16 ? launch_gemm<OUT_BF16>(A, B, c, s) : launch_gemm<OUT_F32>(A, B, c, s);
}

cudaError_t launch_gemm_dact(const void* X, const void* W, const float* bias, const float* dY, int act, int64_t M,
                             int64_t N, int64_t K, void* dZ, float* colsum, int group, cudaStream_t s) {
  GemmCall c{dZ, M, N, K};
  c.bias = bias;
  c.act = act;
  c.group = group;
  c.extra = dY;
  c.colsum = colsum;
  return launch_gemm<OUT_DACT>(X, W, c, s);
}

cudaError_t launch_gemm_nn(const void* A, const void* B, float* C, int64_t M, int64_t N, int64_t K, cudaStream_t s) {
  GemmCall c{C, M, N, K};
  int sms = 0;
  cudaError_t e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  CUtensorMap ta, tb;
  const int tn = gemm_tile_width(M, N, sms);
  if (!make_map(&ta, A, M, K, GM) || !make_map(&tb, B, K, N, GK)) return cudaErrorInvalidValue;
  return run_gemm_at<OUT_F32, OP_NN>(tn, ta, tb, c, sms, s);
}

// K slices of a weight gradient with `tiles` output tiles: ~128 work items, at least four K
// blocks per slice.
static int wgrad_splits_of(int64_t tiles, int64_t K) {
  const int64_t KB = (K + GK - 1) / GK;
  if (tiles >= 64) return 1;
  const int64_t sp = std::min<int64_t>(128 / tiles, KB / 4);
  if (sp <= 1) return 1;
  const int64_t kbs = (KB + sp - 1) / sp;
  return (int)((KB + kbs - 1) / kbs);
}

static int wgrad_width(int64_t N) { return N <= 64 ? 64 : (N <= 128 ? 128 : GN); }

int wgrad_splits(int64_t M, int64_t N, int64_t K, int64_t groups) {
  const int tn = wgrad_width(N);
  return wgrad_splits_of(((M + GM - 1) / GM) * ((N + tn - 1) / tn) * groups, K);
}

size_t wgrad_ws(int64_t M, int64_t N, int64_t K, int64_t groups) {
  const int sp = wgrad_splits(M, N, K, groups);
  return sp > 1 ? (size_t)sp * (size_t)groups * (size_t)M * (size_t)N * 4 : 0;
}

static cudaError_t wgrad_finish(const GemmCall& c, float* C, int64_t cstride, const float* part, cudaStream_t s) {
  if (c.splits <= 1) return cudaSuccess;
  const int64_t n4 = c.M * c.N / 4;   // N is a multiple of 8
  const auto* p = reinterpret_cast<const float4*>(part);
  auto* out = reinterpret_cast<float4*>(C);
  if (c.splits >= 16)
    pdl_launch(k_split_reduce<8>, dim3((unsigned)((n4 + 31) / 32), (unsigned)c.groups), dim3(256), 0, s, p, c.splits,
               n4, cstride / 4, out);
  else
    pdl_launch(k_split_reduce<1>, dim3((unsigned)((n4 + 255) / 256), (unsigned)c.groups), dim3(256), 0, s, p,
               c.splits, n4, cstride / 4, out);
  return cudaGetLastError();
}

cudaError_t launch_wgrad(const void* dZ, const void* X, float* dW, int64_t M, int64_t N, int64_t K, float* part,
                         cudaStream_t s, int64_t groups, int64_t dz_stride, int64_t x_stride, int64_t dw_stride) {
  GemmCall c{dW, M, N, K};
  c.groups = (int)groups;
  c.cstride = dw_stride;
  c.splits = wgrad_splits(M, N, K, groups);
  if (c.splits > 1) c.C = part;
  int sms = 0;
  cudaError_t e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  CUtensorMap ta, tb;
  if (!make_map_mn(&ta, dZ, K, M, groups, groups > 1 ? dz_stride : K * M) ||
      !make_map_mn(&tb, X, K, N, groups, groups > 1 ? x_stride : K * N))
    return cudaErrorInvalidValue;
  e = run_gemm_at<OUT_F32, OP_TN>(wgrad_width(N), ta, tb, c, sms, s);
  return e != cudaSuccess ? e : wgrad_finish(c, dW, dw_stride, part, s);
}

cudaError_t launch_conv_wgrad(const void* dz, const void* x, float* dW, int64_t Bn, int64_t T, int64_t C, int64_t O,
                              int k, float* part, cudaStream_t s) {
  GemmCall c{dW, O, (int64_t)k * C, Bn * T};
  c.splits = wgrad_splits(c.M, c.N, c.K, 1);
  if (c.splits > 1) c.C = part;
  c.geo = ConvGeo{(int)T, (int)(C / GK), (k - 1) / 2, +1};
  int sms = 0;
  cudaError_t e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  CUtensorMap ta, tb;
  if (!make_map_mn(&ta, dz, c.K, O, 1, c.K * O) || !make_map_3d(&tb, x, Bn, T, C, GK)) return cudaErrorInvalidValue;
  e = run_gemm_at<OUT_F32, OP_CONV_TN>(wgrad_width(c.N), ta, tb, c, sms, s);
  return e != cudaSuccess ? e : wgrad_finish(c, dW, 0, part, s);
}

// Self-test of the bounded waits: one thread waits on an mbarrier that nothing arrives at,
// gives up after `polls` polls and records the expiry in the status flag the tensor-core
// kernels use, as they do when their own copies never land.
__global__ void k_selftest_wait(uint32_t polls) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(su32(&bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x == 0 && !mbar_wait(su32(&bar), 0u, polls)) atomicExch(&g_gemm_status, 1);
}

cudaError_t launch_selftest_wait(uint32_t polls, cudaStream_t s) {
  k_selftest_wait<<<1, 32, 0, s>>>(polls);
  return cudaGetLastError();
}

cudaError_t gemm_status(int* status) {
  int zero = 0;
  cudaError_t e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = cudaMemcpyFromSymbol(status, g_gemm_status, sizeof(int));
  if (e == cudaSuccess && *status != 0) e = cudaMemcpyToSymbol(g_gemm_status, &zero, sizeof(int));
  return e;
}

}  // namespace gwx
