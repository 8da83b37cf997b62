// k_flow_train.cu -- the coupling flow's density direction and its backward as one persistent
// tensor-core kernel each (the training step of Sec. 5): a CTA takes 128 rows through all K
// coupling layers without leaving the SM.
//
// k_flow_density applies the layers K-1 .. 0 to x, with the roles of the sampling kernel
// (flow_tile.cuh, k_flow_fused.cu).  For training it also stores what the backward needs: each
// layer's output and conditioner output o (FP32), the conditioner's input X and hidden
// activations g1, g2 (bfloat16, row-major, by TMA stores), and the signs of g1, g2 as bits.
//
// k_flow_backward undoes layer 0 first, eight row warps, operands in shared memory.  Per layer
// the rows form dL/do in registers, and
// three products run as in the forward pass, each weight matrix read as it lies (K is its
// row index: MN-major descriptors), the ReLU masks and the FP32 column sums of every 32 rows
// (the bias gradients' partials) in the drain between them:
//   dg2 = dO V3,  dZ2 = dg2 [g2 > 0],  dg1 = dZ2 V2,  dZ1 = dg1 [g1 > 0],  dX = dZ1 V1;
// dO, dZ2 and dZ1 go to memory in bfloat16 for the weight gradients, which one grouped
// product per weight kind computes for all layers afterwards (k_gemm.cu).  The context's
// gradient stays in registers over the layers.
//
// Every value is rounded where, and summed in the order that, the layer-by-layer kernels
// do, so the results are theirs bit for bit (weight gradients: to the order of the batch
// sum).  Latency bound: one tile's chain MMA -> drain -> MMA, 6.4 us a layer of 256 in the
// density with what it keeps (3.8 without; 6.9 with the operands in shared memory), 7.9 in the
// backward; a batch of 4096 fills 32 SMs.  As ~370 launches of 3 to 13 us (each layer: input
// rows, three products, coupling step; backward 17 kernels) the step took 3.04 ms, now 0.44.
#include "flow_tile.cuh"
#include "pdl.cuh"
#include "sum2.cuh"

namespace gwx {

namespace {

using namespace flowt;

constexpr uint32_t STAGE_BYTES = 32 * 64;                // a row warp's 32 rows x 32 columns on their way out
constexpr size_t DENSITY_SMEM = (size_t)FWD_BYTES + ROW_WARPS * STAGE_BYTES + 1024;
constexpr size_t BACKWARD_SMEM = (size_t)KB_BYTES + G_BYTES + 2 * SLOT_BYTES + 1024;
constexpr double LN_2PI = 1.8378770664093454835606594728112353;

__device__ int g_train_status;

// Backward of the step w_b = (v_b - mu) e^-s, mu_j = o_j, s_j = 3 tanh(o_{4+j} / 3), given
// g = dL/dw and the weight of sum_s in the loss:
// d = dL/do, and g becomes dL/dv_in (without the conditioner's share).
template <int P>
__device__ __forceinline__ void uncouple_back(const float* w, const float* o, float* g, float row_weight, float* d) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int b = Bc(P, j);
    const float t = tanhf(o[4 + j] / S_MAX);
    const float e = expf(-S_MAX * t);
    d[j] = -g[b] * e;
    d[4 + j] = (row_weight - g[b] * w[b]) * (1.f - t * t);
    g[b] *= e;
  }
}

template <int P>
__device__ __forceinline__ void add_half(float* g, const float* d) {
#pragma unroll
  for (int j = 0; j < 4; ++j) g[A(P, j)] += d[j];
}

__device__ __forceinline__ void load8(const float* p, float* v) {
  const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void store8(float* p, const float* v) {
  reinterpret_cast<float4*>(p)[0] = make_float4(v[0], v[1], v[2], v[3]);
  reinterpret_cast<float4*>(p)[1] = make_float4(v[4], v[5], v[6], v[7]);
}

// Signs of 32 columns (pairs of non-negative bfloat16 values in the fragment shape of
// fwd_hidden) of row 16 (j / 2) + 8 (j % 2) + lane / 4, j = lane % 4: bit i for column 2 i,
// bit 16 + i for column 2 i + 1, set when the value is not zero.  Adding 0x7fff to a half-word
// in [0, 0x7fff] sets its top bit exactly when it is not zero, without a carry into the other.
__device__ __forceinline__ uint32_t sign_bits(const uint32_t w[2][8]) {
  const int j = threadIdx.x & 3;
  uint32_t own = 0;
#pragma unroll
  for (int k = 0; k < 2; ++k)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      uint32_t m = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        m |= ((((w[k][2 * i + e] & 0x7fff7fffu) + 0x7fff7fffu) & 0x80008000u) >> 15) << (4 * i);
      m <<= j;
      m |= __shfl_xor_sync(0xffffffffu, m, 1);
      m |= __shfl_xor_sync(0xffffffffu, m, 2);
      if (j == 2 * k + e) own = m;
    }
  return own;
}
__device__ __forceinline__ bool sign_of(uint32_t m, int col) { return (m >> ((col >> 1) + 16 * (col & 1))) & 1u; }

// Sums of 32 columns over the warp's 32 rows: v[c] of every lane in, the sum of column `lane`
// out (each step halves the columns a lane holds and doubles the rows they cover).
__device__ __forceinline__ float column_sums(float* v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1) {
#pragma unroll
    for (int i = 0; i < s; ++i) {
      const bool up = (lane & s) != 0;
      const float send = up ? v[i] : v[i + s], keep = up ? v[i + s] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
    }
  }
  return v[0];
}

struct DensityArgs {
  const float* x;                 // [n][8]
  const __nv_bfloat16* ctx;       // [rows or E][C]
  const int64_t* off;             // [E + 1] event offsets of global rows, or NULL: row r's own context row
  int64_t E, row0, n;
  int C, H, K;
  const float* e1;                // layer-0 biases; layer l at + l * lstride
  const float* e2;
  const float* e3;
  int64_t lstride;
  float* z_out;                   // [n][8] (density only; may be x)
  float* ss_out;                  // [n]    (density only)
  // training (save): layer l's output at xs + l n 8, conditioner output at o + l n 8, sign
  // bits of g1, g2 (mask_at), FP64 sums of the loss over every 32 rows
  int save;
  float* xs;
  float* o;
  uint32_t* m1;
  uint32_t* m2;
  double* loss_part;
};

// Word of rows 32 p .. (one a row) and columns 32 c .. of layer l among the sign bits, [K][P][H / 32][32].
__device__ __forceinline__ int64_t mask_at(int l, int64_t p, int64_t P, int chunks, int c) {
  return ((l * P + p) * chunks + c) * 32;
}

// Barriers, tensor memory and the weight ring of both kernels.
struct Ring {
  uint64_t full[2], empty[2], in_ready, gready[2], acc1f[2], acc2f[2], acc3f, drained;
};

__device__ __forceinline__ void ring_init(Ring* r, int* abort_flag) {
  for (int s = 0; s < 2; ++s) {
    mbar_init(su32(&r->full[s]), 1);
    mbar_init(su32(&r->empty[s]), 1);
    mbar_init(su32(&r->gready[s]), 8);
    mbar_init(su32(&r->acc1f[s]), 1);
    mbar_init(su32(&r->acc2f[s]), 1);
  }
  mbar_init(su32(&r->in_ready), 8);
  mbar_init(su32(&r->acc3f), 1);
  mbar_init(su32(&r->drained), 1);
  *abort_flag = 0;
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ bool wait_mma(uint64_t* bar, uint32_t parity) {   // the issuing warp's wait
  const bool got = mbar_wait_warp(su32(bar), parity, F_WAIT);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  return got;
}

// A row warp's arrival (its shared-memory writes made visible to the tensor core and to TMA).
__device__ __forceinline__ void arrive_rows(uint64_t* bar) {
  proxy_fence();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(su32(bar));
}

// As the sampling kernel with the layers the other way round and the coupling step undone; for
// training also what the backward needs goes out: the hidden activations by way of 2 KiB a row
// warp (the next product reads them from tensor memory, so that the stores are off its path).
__global__ void __launch_bounds__(FWD_THREADS, 1)
    k_flow_density(const __grid_constant__ CUtensorMap mv1, const __grid_constant__ CUtensorMap mv2,
                   const __grid_constant__ CUtensorMap mv3, const __grid_constant__ CUtensorMap sx_map,
                   const __grid_constant__ CUtensorMap s1_map, const __grid_constant__ CUtensorMap s2_map,
                   DensityArgs a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(16) FwdRing rg;
  __shared__ float s_o[8][FM];                                 // the rows' conditioner outputs
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t base = (su32(smem_raw) + 1023u) & ~1023u;
  const uint32_t sx = base, sw = base + X_BYTES;
  const int K = a.K, C = a.C, H = a.H, NR = H / 128;           // 128-column rounds of the hidden layers
  const int tiles = (int)((a.n + FM - 1) / FM);
  const FwdWeights wt{&mv1, &mv2, &mv3, a.e1, a.e2, a.e3, a.lstride, C, H, K, tiles, true};
  const uint32_t tmem = fwd_begin(rg);
  pdl_enter();

  if (warp == 0) {
    fwd_produce(rg, wt, sw);
  } else if (warp == 1) {
    fwd_multiply(rg, wt, tmem, sx, sw);
  } else {
    const int q = warp & 3;
    const int h = (warp - 2) >> 2;                             // which 32 of every 128 columns
    const int r = 32 * q + lane;                               // row of the tile = tensor-memory lane
    const uint32_t lane_addr = tmem + ((uint32_t)(32 * q) << 16);
    const uint32_t stage = base + FWD_BYTES + (uint32_t)(warp - 2) * STAGE_BYTES;
    uint32_t li = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
      const int64_t row = (int64_t)t * FM + r;
      const int wrow = t * FM + 32 * q;                        // first row of this warp
      const bool valid = row < a.n;
      const bool save = a.save != 0 && wrow < a.n;             // uniform over the warp
      float v[8], ss = 0.f;
      if (valid) {
        load8(a.x + row * 8, v);
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = 0.f;
      }
      // context: columns 8 .. 8 + C - 1 of the input row, zeros up to 128
      int64_t e = valid ? row : 0;
      if (valid && a.off != nullptr) {
        int64_t lo = 0, hi = a.E, s = a.row0 + row;
        while (hi - lo > 1) {
          const int64_t mid = (lo + hi) >> 1;
          if (a.off[mid] <= s) lo = mid; else hi = mid;
        }
        e = lo;
      }
      const uint4* crow = reinterpret_cast<const uint4*>(a.ctx + e * C);
      for (int g = h == 0 ? 1 : 4 * h; g < 4 * h + 4; ++g) {
        uint4 x = make_uint4(0u, 0u, 0u, 0u);
        if (valid && g <= C / 8) x = crow[g - 1];
        sts128(sx + KB_BYTES * (g >> 3) + swz(r, g & 7), x.x, x.y, x.z, x.w);
      }
      // chunk c (32 columns) of a hidden layer: signs and activations out, when the chunk before has
      // left this warp's buffer (4096 rows, 16 layers: 102 us; 125 with plain 16-byte stores, 109
      // with signs and rows by bulk copies as well; 61 of it the chain, the rest what is kept).
      auto keep = [&](const uint32_t w[2][8], int c, int l, const CUtensorMap* map, uint32_t* masks) {
        const uint32_t bits = sign_bits(w);
        if (lane == 0) tma_store_wait_read();
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int rr = 16 * k + 8 * (i & 1) + (lane >> 2);
            sts32(stage + 64u * rr + (uint32_t)((((i >> 1) ^ (rr >> 1)) & 3) << 4) + 4u * (lane & 3), w[k][i]);
          }
        proxy_fence();
        __syncwarp();
        if (lane == 0) tma_store_3d(map, stage, 32 * c, wrow, l);
        const int rj = 16 * ((lane & 3) >> 1) + 8 * (lane & 1) + (lane >> 2);
        masks[mask_at(l, wrow / 32, (a.n + 31) / 32, H / 32, c) + rj] = bits;
      };
      uint32_t w[2][2][8];                                     // this warp's chunks of a hidden layer
      for (int l = K - 1; l >= 0; --l, ++li) {
        const int p = l & 3;
        if (h == 0) {
          uint32_t w0, w1;
          pack_half(p, v, w0, w1);
          sts128(sx + swz(r, 0), w0, w1, 0u, 0u);
        }
        proxy_fence();
        row_arrive(&rg.xready);
        // what goes out does so while the tensor core works, a chunk at a time with a pause for the
        // buffer: the second chunk of the last layer's g2 here, g1 and the first of g2 below
        if (save && l < K - 1 && NR > 1) keep(w[1], 4 + h, l + 1, &s2_map, a.m2);
        const float* bl = rg.sb[li & 1u];
        if (!(ok = row_wait(&rg.biasf[li & 1u], (li >> 1) & 1u, &rg.abort_flag))) break;
        if (!(ok = row_wait(&rg.acc1f, li & 1u))) break;
#pragma unroll
        for (int rd = 0; rd < 2; ++rd) {
          if (rd >= NR) break;
          const int c = 4 * rd + h;
          fwd_hidden(lane_addr + 32u * c, bl + 32 * c, w[rd]);
          row_arrive(&rg.gready[rd]);
        }
        if (save) {
          keep(w[0], h, l, &s1_map, a.m1);
          if (NR > 1) keep(w[1], 4 + h, l, &s1_map, a.m1);
        }
        // the input rows (all four warps' columns: acc1 followed their arrivals)
        if (save && lane == 0 && (h == 0 || (h == 1 && 8 + C > 64)))
          tma_store_3d(&sx_map, sx + KB_BYTES * h + 4096u * q, 64 * h, wrow, l);
        if (!(ok = row_wait(&rg.acc2f, li & 1u))) break;
#pragma unroll
        for (int rd = 0; rd < 2; ++rd) {
          if (rd >= NR) break;
          const int c = 4 * rd + h;
          fwd_hidden(lane_addr + ACC2 + 32u * c, bl + 256 + 32 * c, w[rd]);
          row_arrive(&rg.gready[rd]);
        }
        if (save) keep(w[0], h, l, &s2_map, a.m2);
        // v_b <- (v_b - mu) e^-s with mu_j = o_j, s_j = 3 tanh(o_{4+j} / 3): coordinate j by warp
        // h = j of the quarter, handed to the others in shared memory
        if (!(ok = row_wait(&rg.acc3f, li & 1u))) break;
        uint32_t om = tmem_ld1_async(lane_addr + ACC3 + h), os = tmem_ld1_async(lane_addr + ACC3 + 4u + h);
        asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(om), "+r"(os)::"memory");
        const float mu = __uint_as_float(om) + bl[512 + h], ol = __uint_as_float(os) + bl[512 + 4 + h];
        const float s = S_MAX * tanhf(ol / S_MAX);
        rg.s_new[h][r] = (half_at(p, v, h) - mu) * expf(-s);
        rg.s_log[h][r] = s;
        if (save) {
          s_o[h][r] = mu;
          s_o[4 + h][r] = ol;
          // the input rows have been read before the quarter may write new ones
          if (lane == 0) tma_store_wait_read();
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(su32(&rg.cplf[q]));
        if (!(ok = row_wait(&rg.cplf[q], li & 1u))) break;
        float x[4], sl = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          x[j] = rg.s_new[j][r];
          sl += rg.s_log[j][r];
        }
        set_half(p, v, x);
        ss = l == K - 1 ? sl : ss + sl;
        if (save && valid && h == 0) store8(a.xs + ((int64_t)l * a.n + row) * 8, v);
        if (save && valid && h == 1) {
          float o[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) o[j] = s_o[j][r];
          store8(a.o + ((int64_t)l * a.n + row) * 8, o);
        }
      }
      if (!ok) break;
      if (save && NR > 1) keep(w[1], 4 + h, 0, &s2_map, a.m2);
      if (h != 0) continue;
      if (a.save == 0) {
        if (valid) {
          store8(a.z_out + row * 8, v);
          a.ss_out[row] = ss;
        }
      } else if (save) {
        // the rows' loss |z|^2 / 2 + 4 ln 2 pi + sum_s
        double lb = 0.0;
        if (valid) {
          double zz = 0.0;
#pragma unroll
          for (int i = 0; i < 8; ++i) zz += (double)v[i] * (double)v[i];
          lb = 0.5 * zz + 4.0 * LN_2PI + (double)ss;
        }
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) lb += __shfl_down_sync(0xffffffffu, lb, s);
        if (lane == 0) a.loss_part[wrow / 32] = lb;
      }
    }
    if (a.save != 0 && lane == 0) tma_store_wait();            // before the shared tiles go away
    if (!ok && lane == 0) atomicExch(&rg.abort_flag, 1);
  }
  fwd_end(rg, tmem, &g_train_status);
}

struct BackwardArgs {
  const float* xs;                // [K][n][8] layer outputs (xs[0] = z)
  const float* o;                 // [K][n][8]
  const uint32_t* m1;             // sign bits of g1, g2 (mask_at)
  const uint32_t* m2;
  int64_t n;
  int C, H, K;
  float inv_n;
  __nv_bfloat16* dO;              // [K][n][8]
  float* p1;                      // column sums of dZ1, dZ2 and dO over every 32 rows: [K][P][H], [K][P][H], [K][P][8]
  float* p2;
  float* p3;
  int64_t P;
  float* dctx;                    // [n][C]
};

__global__ void __launch_bounds__(F_THREADS, 1)
    k_flow_backward(const __grid_constant__ CUtensorMap mv1, const __grid_constant__ CUtensorMap mv2,
                    const __grid_constant__ CUtensorMap mv3, const __grid_constant__ CUtensorMap s1_map,
                    const __grid_constant__ CUtensorMap s2_map, BackwardArgs a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) Ring rg;
  __shared__ uint32_t tmem_slot, fills;                    // (the producer's, once it has stopped)
  __shared__ int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t base = (su32(smem_raw) + 1023u) & ~1023u;
  const uint32_t so = base, sg = base + KB_BYTES, sw = base + KB_BYTES + G_BYTES;
  const int H = a.H, K = a.K, C = a.C;
  const int NR = H / 128, NP = 2 + NR;                     // weight parts per layer: V3, NR row blocks of V2, V1
  const int NX = (8 + C + 15) / 16 * 16;                   // columns of dX
  const int tiles = (int)((a.n + FM - 1) / FM);
  const uint32_t id_128 = idesc_bf16(FM, 128, false, true), id_x = idesc_bf16(FM, (uint32_t)NX, false, true);

  if (threadIdx.x == 0) ring_init(&rg, &abort_flag);
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  pdl_enter();

  if (warp == 0) {
    uint32_t it = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x)
      for (int l = 0; l < K && ok; ++l)
        for (int p = 0; p < NP; ++p, ++it) {
          const uint32_t s = it & 1u;
          if (!mbar_wait_warp(su32(&rg.empty[s]), ((it >> 1) & 1u) ^ 1u, F_WAIT) ||
              __any_sync(0xffffffffu, *(volatile int*)&abort_flag)) {
            ok = false;
            break;
          }
          const uint32_t dst = sw + s * SLOT_BYTES, bar = su32(&rg.full[s]);
          if (elect_one()) {
            if (p == 0) {                                      // V3: 8 rows (16 with the zero fill) x H columns
              mbar_expect_tx(bar, (uint32_t)H * 32u);
              for (int c = 0; c < H / 64; ++c) tma_load_3d(dst + 2048u * c, &mv3, 64 * c, 0, l, bar);
            } else if (p < NP - 1) {                           // V2: rows 128 (p - 1) .., H columns
              mbar_expect_tx(bar, (uint32_t)H * 256u);
              for (int c = 0; c < H / 64; ++c) tma_load_3d(dst + 16384u * c, &mv2, 64 * c, 128 * (p - 1), l, bar);
            } else {                                           // V1: H rows, 8 + C columns
              const int nc = (8 + C + 63) / 64;
              mbar_expect_tx(bar, (uint32_t)H * 128u * nc);
              for (int c = 0; c < nc; ++c) tma_load_3d(dst + (uint32_t)H * 128u * c, &mv1, 64 * c, 0, l, bar);
            }
          }
          __syncwarp();
        }
    if (lane == 0) {
      fills = it;
      if (!ok) atomicExch(&abort_flag, 1);
    }
  } else if (warp == 1) {
    uint32_t it = 0, li = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x)
      for (int l = 0; l < K && ok; ++l, ++li) {
        // acc1 = dO V3: one K = 16 step (8 outputs and 8 zeros)
        uint32_t slot = it & 1u, wb = sw + slot * SLOT_BYTES;
        if (!(ok = wait_mma(&rg.full[slot], (it >> 1) & 1u) && wait_mma(&rg.in_ready, li & 1u))) break;
        if (elect_one()) {
          for (int np = 0; np < NR; ++np) {
            mma_bf16(tmem + 128u * np, sw128_desc(so), sw128_mn_desc(wb + 4096u * np, 2048u), id_128, 0u);
            mma_commit(su32(&rg.acc1f[np]));
          }
          mma_commit(su32(&rg.empty[slot]));
        }
        __syncwarp();
        ++it;
        // acc2 = dZ2 V2: K round pr (dZ2 columns 128 pr .., rows of V2) once the rows have written it
        for (int pr = 0; pr < NR; ++pr) {
          slot = it & 1u, wb = sw + slot * SLOT_BYTES;
          if (!(ok = wait_mma(&rg.full[slot], (it >> 1) & 1u) && wait_mma(&rg.gready[pr], 0u))) break;
          if (elect_one()) {
            for (int np = 0; np < NR; ++np) {
#pragma unroll
              for (int kk = 0; kk < 8; ++kk)
                mma_bf16(tmem + 256u + 128u * np, sw128_desc(sg + KB_BYTES * (2 * pr + (kk >> 2)) + 32u * (kk & 3)),
                         sw128_mn_desc(wb + 32768u * np + 2048u * kk, 16384u), id_128, (pr | kk) != 0);
              if (pr == NR - 1) mma_commit(su32(&rg.acc2f[np]));
            }
            mma_commit(su32(&rg.empty[slot]));
          }
          __syncwarp();
          ++it;
        }
        if (!ok) break;
        // acc3 = dZ1 V1
        slot = it & 1u, wb = sw + slot * SLOT_BYTES;
        if (!(ok = wait_mma(&rg.full[slot], (it >> 1) & 1u))) break;
        for (int r = 0; r < NR; ++r) {
          if (!(ok = wait_mma(&rg.gready[r], 1u))) break;
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
              const int ks = 8 * r + kk;
              mma_bf16(tmem, sw128_desc(sg + KB_BYTES * (ks >> 2) + 32u * (ks & 3)),
                       sw128_mn_desc(wb + 2048u * ks, (uint32_t)H * 128u), id_x, ks != 0);
            }
            if (r == NR - 1) {
              mma_commit(su32(&rg.acc3f));
              mma_commit(su32(&rg.empty[slot]));
            }
          }
          __syncwarp();
        }
        ++it;
      }
    if (!ok && lane == 0) atomicExch(&abort_flag, 1);
  } else {
    const int q = warp & 3;
    const int h = (warp - 2) >> 2;
    const int r = 32 * q + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(32 * q) << 16);
    uint32_t li = 0;
    bool ok = true;
    // 64 accumulator columns (chunk c), masked: bfloat16 into K-block c, FP32 column sums to part
    auto masked = [&](uint32_t col0, uint2 m, int c, float* part, bool in) {
      uint32_t raw[2][32];
      tmem_ld32_async(lane_addr + col0 + 64u * c, raw[0]);
      tmem_ld32_async(lane_addr + col0 + 64u * c + 32u, raw[1]);
      tmem_wait_ld();
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        const uint32_t mm = hh ? m.y : m.x;
        float f[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) f[i] = sign_of(mm, i) ? __uint_as_float(raw[hh][i]) : 0.f;
#pragma unroll
        for (int t4 = 0; t4 < 4; ++t4) {
          const int col = 64 * c + 32 * hh + 8 * t4;
          sts128(sg + KB_BYTES * (col >> 6) + swz(r, (col & 63) >> 3), pack2(f[8 * t4], f[8 * t4 + 1]),
                 pack2(f[8 * t4 + 2], f[8 * t4 + 3]), pack2(f[8 * t4 + 4], f[8 * t4 + 5]),
                 pack2(f[8 * t4 + 6], f[8 * t4 + 7]));
        }
#pragma unroll
        for (int i = 0; i < 32; ++i) raw[hh][i] = __float_as_uint(f[i]);
      }
      return [raw, part, c, in, lane]() mutable {              // the column sums, after the arrival
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          float f[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) f[i] = __uint_as_float(raw[hh][i]);
          const float s = column_sums(f);
          if (in) part[64 * c + 32 * hh + lane] = s;
        }
      };
    };
    // columns 8 .. 15 of dO's K-block stay zero (one K = 16 step reads 16 columns)
    if (h == 0) sts128(so + swz(r, 1), 0u, 0u, 0u, 0u);
    for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
      const int64_t row = (int64_t)t * FM + r;
      const int wrow = t * FM + 32 * q;
      const bool valid = row < a.n, in = wrow < a.n;           // `in`: uniform over the warp
      // context gradient: columns 8 + j of dX; the first half's warp holds j = 0 .. 23 (with
      // the eight input columns), the second's j = 24 .. 63
      float g[8], w[8], o[8], dctx[40];
#pragma unroll
      for (int i = 0; i < 8; ++i) g[i] = w[i] = o[i] = 0.f;
      if (h == 0 && valid) {
        load8(a.xs + row * 8, w);
        load8(a.o + row * 8, o);
#pragma unroll
        for (int i = 0; i < 8; ++i) g[i] = w[i] * a.inv_n;     // dL/dz = z / n
      }
      for (int l = 0; l < K; ++l, ++li) {
        const int p = l & 3;
        const int64_t at = (int64_t)l * a.n + row;
        const int64_t pr0 = (int64_t)l * a.P + wrow / 32;
        uint2 k1[2], k2[2];                                    // this thread's chunks of both masks
#pragma unroll
        for (int rd = 0; rd < 2; ++rd) {
          const bool have = valid && rd < NR;
          const int64_t m = mask_at(l, wrow / 32, a.P, H / 32, 2 * (2 * rd + h)) + lane;
          k2[rd] = have ? make_uint2(a.m2[m], a.m2[m + 32]) : make_uint2(0u, 0u);
          k1[rd] = have ? make_uint2(a.m1[m], a.m1[m + 32]) : make_uint2(0u, 0u);
        }
        if (h == 0) {
          float d[8];
          const float rw = valid ? a.inv_n : 0.f;
          switch (p) {
            case 0: uncouple_back<0>(w, o, g, rw, d); break;
            case 1: uncouple_back<1>(w, o, g, rw, d); break;
            case 2: uncouple_back<2>(w, o, g, rw, d); break;
            default: uncouple_back<3>(w, o, g, rw, d); break;
          }
          const uint4 dv = make_uint4(pack2(d[0], d[1]), pack2(d[2], d[3]), pack2(d[4], d[5]), pack2(d[6], d[7]));
          sts128(so + swz(r, 0), dv.x, dv.y, dv.z, dv.w);
          arrive_rows(&rg.in_ready);
          if (valid) *reinterpret_cast<uint4*>(a.dO + at * 8) = dv;
          // its column sums: lanes 4 j + .. hold column j after three halvings
#pragma unroll
          for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) d[i] += __shfl_xor_sync(0xffffffffu, d[i], s);
          if (in && lane == 0) store8(a.p3 + pr0 * 8, d);
        } else {
          arrive_rows(&rg.in_ready);                           // (it has read the last layer's dX)
        }
        for (int rd = 0; rd < NR && ok; ++rd) {
          if (!(ok = row_wait(&rg.acc1f[rd], li & 1u, &abort_flag))) break;
          const int c = 2 * rd + h;
          if (lane == 0) tma_store_wait_read();                // the last layer's dZ1 has been read
          __syncwarp();
          auto sums = masked(0u, k2[rd], c, a.p2 + pr0 * H, in);
          arrive_rows(&rg.gready[rd]);
          if (in && lane == 0) tma_store_3d(&s2_map, sg + KB_BYTES * c + 4096u * q, 64 * c, wrow, l);
          sums();
        }
        for (int rd = 0; rd < NR && ok; ++rd) {
          if (!(ok = row_wait(&rg.acc2f[rd], li & 1u, &abort_flag))) break;
          const int c = 2 * rd + h;
          if (lane == 0) tma_store_wait_read();                // dZ2 has been read
          __syncwarp();
          auto sums = masked(256u, k1[rd], c, a.p1 + pr0 * H, in);
          arrive_rows(&rg.gready[rd]);
          if (in && lane == 0) tma_store_3d(&s1_map, sg + KB_BYTES * c + 4096u * q, 64 * c, wrow, l);
          sums();
        }
        if (!ok) break;
        if (h == 0 && valid && l + 1 < K) {                    // the next layer's rows, before the wait
          load8(a.xs + (at + a.n) * 8, w);
          load8(a.o + (at + a.n) * 8, o);
        }
        if (!(ok = row_wait(&rg.acc3f, li & 1u, &abort_flag))) break;
        uint32_t raw[32];
        tmem_ld32_async(lane_addr + 32u * h, raw);
        if (h == 0) {
          tmem_wait_ld();
          float dx[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) dx[j] = __uint_as_float(raw[j]);
          switch (p) {
            case 0: add_half<0>(g, dx); break;
            case 1: add_half<1>(g, dx); break;
            case 2: add_half<2>(g, dx); break;
            default: add_half<3>(g, dx); break;
          }
#pragma unroll
          for (int i = 0; i < 24; ++i) {
            const float d = __uint_as_float(raw[8 + i]);
            dctx[i] = l == 0 ? d : dctx[i] + d;
          }
        } else {
          float hi[16];
          tmem_ld16(lane_addr + 64u, hi);                      // waits for both loads
#pragma unroll
          for (int i = 0; i < 40; ++i) {
            const float d = i < 32 ? __uint_as_float(raw[i & 31]) : hi[i & 15];
            dctx[i] = l == 0 ? d : dctx[i] + d;
          }
        }
      }
      if (!ok) break;
      if (valid) {
        const int j0 = h ? 24 : 0, j1 = h ? 64 : 24;
#pragma unroll
        for (int i = 0; i < 10; ++i)
          if (j0 + 4 * i < j1 && j0 + 4 * i < C)
            *reinterpret_cast<float4*>(a.dctx + row * C + j0 + 4 * i) =
                make_float4(dctx[4 * i], dctx[4 * i + 1], dctx[4 * i + 2], dctx[4 * i + 3]);
      }
    }
    if (lane == 0) tma_store_wait();
    if (!ok && lane == 0) atomicExch(&abort_flag, 1);
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (*(volatile int*)&abort_flag) {
    if (threadIdx.x == 0) atomicExch(&g_train_status, 1);
    if (warp == 0) pair_drain(rg.full, fills, F_WAIT);
    if (warp == 1) mma_drain(&rg.drained, F_WAIT);
    __syncthreads();
  }
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

// Bias gradients of every layer and the mean loss: block (c, l) sums 32 columns' partials
// (p1, p2, p3: H, H and 8 columns) of layer l, 32 row lanes and then a warp a column, in
// two-float arithmetic (FP64: 9.8 us for 16 layers of 256 and 128 partials, 6.0 now); the
// extra block (0, K) sums the loss in FP64.
__global__ void __launch_bounds__(1024) k_flow_bias_grads(const float* p1, const float* p2, const float* p3,
                                                          int64_t P, int H, int K,
                                                          float* __restrict__ g1, float* __restrict__ g2,
                                                          float* __restrict__ g3, int64_t lstride,
                                                          const double* loss_part, double n,
                                                          double* __restrict__ loss) {
  pdl_enter();
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, l = blockIdx.y;
  if (l == K) {
    __shared__ double red[32][33];
    if (blockIdx.x > 0) return;
    double s = 0.0;
    for (int64_t i = threadIdx.x; i < P; i += 1024) s += loss_part[i];
    red[ty][tx] = s;
    __syncthreads();
    if (ty != 0) return;
    double t = 0.0;
    for (int y = 0; y < 32; ++y) t += red[y][tx];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (tx == 0) *loss = t / n;
    return;
  }
  __shared__ float2 red[32][33];
  const int hc = H / 32, kind = (int)blockIdx.x < hc ? 0 : ((int)blockIdx.x < 2 * hc ? 1 : 2);
  const int col0 = 32 * ((int)blockIdx.x - kind * hc), cols = kind == 2 ? 8 : H;
  const float* p = (kind == 0 ? p1 : (kind == 1 ? p2 : p3)) + (int64_t)l * P * cols;
  Sum2 s;
  if (col0 + tx < cols)
#pragma unroll 4
    for (int64_t i = ty; i < P; i += 32) s.add(p[i * cols + col0 + tx]);
  red[ty][tx] = make_float2(s.h, s.l);
  __syncthreads();
  const float2 v = red[tx][ty];
  s.h = v.x;
  s.l = v.y;
  const int c = col0 + ty;
  warp_total(s, p + c, P, cols, c < cols,
             [&](auto t) { (kind == 0 ? g1 : (kind == 1 ? g2 : g3))[(int64_t)l * lstride + c] = t.rounded(); });
}

cudaError_t tile_grid(int64_t n, unsigned* grid) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t tiles = (n + FM - 1) / FM;
  *grid = (unsigned)(tiles < sms ? tiles : sms);
  return e;
}

cudaError_t run_density(const void* params_bf16, const float* params, const int64_t* off_t, DensityArgs a,
                        const CUtensorMap* stores, cudaStream_t s) {
  const __nv_bfloat16* p16 = reinterpret_cast<const __nv_bfloat16*>(params_bf16);
  const int C = a.C, H = a.H, K = a.K;
  a.lstride = K > 1 ? off_t[12] - off_t[6] : 64;   // one layer's tensors repeat every lstride elements
  a.e1 = params + off_t[7];
  a.e2 = params + off_t[9];
  a.e3 = params + off_t[11];
  CUtensorMap m1, m2, m3;
  if (!layer_map(&m1, p16 + off_t[6], 8 + C, H, K, a.lstride, (uint32_t)H) ||
      !layer_map(&m2, p16 + off_t[8], H, H, K, a.lstride, (uint32_t)H) ||
      !layer_map(&m3, p16 + off_t[10], H, 8, K, a.lstride, 16u))
    return cudaErrorInvalidValue;
  unsigned grid = 0;
  cudaError_t e = tile_grid(a.n, &grid);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_flow_density, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DENSITY_SMEM);
  if (e != cudaSuccess) return e;
  pdl_launch(k_flow_density, dim3(grid), dim3(FWD_THREADS), DENSITY_SMEM, s, m1, m2, m3, stores ? stores[0] : m1,
             stores ? stores[1] : m1, stores ? stores[2] : m1, a);
  return cudaGetLastError();
}

}  // namespace

// Widths the fused kernels cover: as the sampling kernel, with the context's gradient in registers, 24
// columns of it with one warp of a quarter and 40 with the other.
bool flow_fused_train_supported(int C, int H, int K) { return flow_fused_supported(C, H, K) && C <= 64; }

cudaError_t launch_flow_density(const void* params_bf16, const float* params, const int64_t* off_t, int C, int H, int K,
                                const float* x, const void* ctx, const int64_t* ev_off, int64_t E, int64_t row0,
                                int64_t n, float* z_out, float* ss_out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  DensityArgs a{};
  a.x = x;
  a.ctx = reinterpret_cast<const __nv_bfloat16*>(ctx);
  a.off = ev_off;
  a.E = E;
  a.row0 = row0;
  a.n = n;
  a.C = C;
  a.H = H;
  a.K = K;
  a.z_out = z_out;
  a.ss_out = ss_out;
  return run_density(params_bf16, params, off_t, a, nullptr, s);
}

FlowTrainBufs flow_train_bufs(int64_t n, int C, int H, int K, void* base, size_t* bytes) {
  char* b = reinterpret_cast<char*>(base);
  size_t used = 0;
  auto take = [&](size_t sz) {
    char* p = b ? b + used : nullptr;
    used += (sz + 255) & ~(size_t)255;
    return p;
  };
  FlowTrainBufs f;
  const size_t Kn = (size_t)K * (size_t)n, P = (size_t)((n + 31) / 32);
  f.X = take(Kn * (8 + C) * 2);
  f.g1 = take(Kn * H * 2);
  f.g2 = take(Kn * H * 2);
  f.dz1 = take(Kn * H * 2);
  f.dz2 = take(Kn * H * 2);
  f.dO = take(Kn * 8 * 2);
  f.m1 = take(K * P * H * 4);
  f.m2 = take(K * P * H * 4);
  f.o = reinterpret_cast<float*>(take(Kn * 8 * 4));
  f.p1 = reinterpret_cast<float*>(take(K * P * H * 4));
  f.p2 = reinterpret_cast<float*>(take(K * P * H * 4));
  f.p3 = reinterpret_cast<float*>(take(K * P * 8 * 4));
  f.loss_part = reinterpret_cast<double*>(take(P * 8));
  size_t ws = wgrad_ws(H, H, n, K);
  if (wgrad_ws(H, 8 + C, n, K) > ws) ws = wgrad_ws(H, 8 + C, n, K);
  if (wgrad_ws(8, H, n, K) > ws) ws = wgrad_ws(8, H, n, K);
  f.kpart = reinterpret_cast<float*>(take(ws));
  if (bytes) *bytes = used;
  return f;
}

cudaError_t launch_flow_train_fused(const void* params_bf16, const float* params, const int64_t* off_t, int C, int H,
                                    int K, float* xs, const void* ctx, int64_t n, float* grads, float* dctx,
                                    double* loss_mean, const FlowTrainBufs& f, cudaStream_t s) {
  const __nv_bfloat16* p16 = reinterpret_cast<const __nv_bfloat16*>(params_bf16);
  const int64_t lstride = K > 1 ? off_t[12] - off_t[6] : 64;
  // forward, with what the backward needs
  CUtensorMap st[3], b1, b2, w1, w2, w3;
  if (!layer_map(&st[0], f.X, 8 + C, n, K, n * (8 + C), 32u) || !layer_map(&st[1], f.g1, H, n, K, n * H, 32u, 32u) ||
      !layer_map(&st[2], f.g2, H, n, K, n * H, 32u, 32u) || !layer_map(&b1, f.dz1, H, n, K, n * H, 32u) ||
      !layer_map(&b2, f.dz2, H, n, K, n * H, 32u) ||
      !layer_map(&w1, p16 + off_t[6], 8 + C, H, K, lstride, (uint32_t)H) ||
      !layer_map(&w2, p16 + off_t[8], H, H, K, lstride, 128u) || !layer_map(&w3, p16 + off_t[10], H, 8, K, lstride, 16u))
    return cudaErrorInvalidValue;
  DensityArgs a{};
  a.x = xs + (int64_t)K * n * 8;
  a.ctx = reinterpret_cast<const __nv_bfloat16*>(ctx);
  a.n = n;
  a.C = C;
  a.H = H;
  a.K = K;
  a.save = 1;
  a.xs = xs;
  a.o = f.o;
  a.m1 = reinterpret_cast<uint32_t*>(f.m1);
  a.m2 = reinterpret_cast<uint32_t*>(f.m2);
  a.loss_part = f.loss_part;
  cudaError_t e = run_density(params_bf16, params, off_t, a, st, s);
  if (e != cudaSuccess) return e;
  // backward
  BackwardArgs b{};
  b.xs = xs;
  b.o = f.o;
  b.m1 = a.m1;
  b.m2 = a.m2;
  b.n = n;
  b.C = C;
  b.H = H;
  b.K = K;
  b.inv_n = 1.f / (float)n;
  b.dO = reinterpret_cast<__nv_bfloat16*>(f.dO);
  b.p1 = f.p1;
  b.p2 = f.p2;
  b.p3 = f.p3;
  b.P = (n + 31) / 32;
  b.dctx = dctx;
  unsigned grid = 0;
  e = tile_grid(n, &grid);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_flow_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BACKWARD_SMEM);
  if (e != cudaSuccess) return e;
  pdl_launch(k_flow_backward, dim3(grid), dim3(F_THREADS), BACKWARD_SMEM, s, w1, w2, w3, b1, b2, b);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // weight gradients of all layers, one grouped product per kind; bias gradients and the loss
  if ((e = launch_wgrad(f.dO, f.g2, grads + off_t[10], 8, H, n, f.kpart, s, K, n * 8, n * H, lstride)) != cudaSuccess ||
      (e = launch_wgrad(f.dz2, f.g1, grads + off_t[8], H, H, n, f.kpart, s, K, n * H, n * H, lstride)) !=
          cudaSuccess ||
      (e = launch_wgrad(f.dz1, f.X, grads + off_t[6], H, 8 + C, n, f.kpart, s, K, n * H, n * (8 + C), lstride)) !=
          cudaSuccess)
    return e;
  pdl_launch(k_flow_bias_grads, dim3((unsigned)(2 * (H / 32) + 1), (unsigned)(K + 1)), dim3(1024), 0, s, f.p1, f.p2,
             f.p3, b.P, H, K, grads + off_t[7], grads + off_t[9], grads + off_t[11], lstride, f.loss_part, (double)n,
             loss_mean);
  return cudaGetLastError();
}

cudaError_t flow_train_status(int* status) {
  int zero = 0;
  cudaError_t e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = cudaMemcpyFromSymbol(status, g_train_status, sizeof(int));
  if (e == cudaSuccess && *status != 0) e = cudaMemcpyToSymbol(g_train_status, &zero, sizeof(int));
  return e;
}

}  // namespace gwx
