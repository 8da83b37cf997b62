// k_flow_fused.cu -- the coupling flow's sampling pass as one persistent tensor-core
// kernel (the draw step of Sec. 5's posterior estimator).  Each CTA takes 128 draws at a
// time through all K coupling layers without leaving the SM:
//   - warp 0 streams each layer's conditioner weights from L2 with 3-D TMA boxes into a
//     two-slot ring (part 0: V1; parts 1..H/128: pairs of V2's 64-column K-blocks) and a
//     buffer for V3 (padded to 16 rows by the box's zero fill), and its biases;
//   - warp 1 issues tcgen05.mma: acc1 = X V1^T, acc2 = g1 V2^T, acc3 = g2 V3^T (FP32 in
//     tensor memory), acc2 and acc3 in rounds of 128 columns of their input, so that the
//     first round runs while the rows write the second's;
//   - warps 2-17 own one draw (row) per thread, four warps per tensor-memory lane quarter:
//     each writes a share of the context into the conditioner input X once per tile and
//     of the hidden activations g1, g2 (bias, ReLU, bfloat16), and applies the coupling step
//     to one of the four transformed coordinates; the first writes the conditioning half
//     of X once per layer.
// The activations stay in tensor memory: 32 accumulator columns are read, and 16 columns of
// bfloat16 pairs written over the first of them, from where the next product takes its A
// operand (columns 0..255 acc1, then g1; 256..511 acc2, then g2; acc3 in 16..31, which g1
// leaves free).  Per draw and layer only the weights (shared by all draws, L2-resident) move.
//
// Bound by one tile's chain MMA -> drain -> MMA -> drain -> MMA -> coupling: of ~6900 cycles a
// layer at H = 256 the products take 640 + 2048 + 256 and each hand-over ~300 more.  As
// 128-column MMAs (which cost nearly what 256 columns do) from g in shared memory, eight row
// warps and biases by every thread from L2, a layer took 9200: 20,000 draws of 16 layers
// 163 us, now 122 (157 tiles on 152 SMs, two rounds; A from tensor memory 147, biases staged
// 134, four warps a quarter and 256-column MMAs with the fragment-shaped drain 122).
// Every mbarrier wait is bounded; on expiry the CTA records a status, stops and frees its
// tensor memory.
#include "flow_tile.cuh"

namespace gwx {

namespace {

using namespace flowt;

constexpr uint32_t V3_BYTES = 16 * 256 * 2;
constexpr size_t FUSED_SMEM = (size_t)X_BYTES + 2 * SLOT_BYTES + V3_BYTES + 1024;
constexpr int ROW_WARPS = 16;                // four warps a tensor-memory lane quarter
constexpr int S_THREADS = 64 + 32 * ROW_WARPS;
constexpr uint32_t ACC2 = 256, ACC3 = 16;   // tensor-memory columns of the second and third products

__device__ int g_flow_status;

struct FusedArgs {
  const float* z;                 // [n][8] base draws of this chunk
  const __nv_bfloat16* ctx;       // [E][C] per-event context
  const int64_t* off;             // [E + 1] event offsets (global rows)
  int64_t E, row0, n;
  int C, H, K;
  const float* e1;                // layer-0 biases; layer l at + l * lstride
  const float* e2;
  const float* e3;
  int64_t lstride;                // elements between consecutive layers' tensors
  float* x_out;                   // [n][8]
  float* ss_out;                  // [n]
};

// Coordinate j of the transformed half, and v[Bc(P, j)] = x[j] for all of them.
template <int P>
__device__ __forceinline__ float half_at(const float* v, int j) {
  return j == 0 ? v[Bc(P, 0)] : j == 1 ? v[Bc(P, 1)] : j == 2 ? v[Bc(P, 2)] : v[Bc(P, 3)];
}
template <int P>
__device__ __forceinline__ void set_half(float* v, const float* x) {
#pragma unroll
  for (int j = 0; j < 4; ++j) v[Bc(P, j)] = x[j];
}

__global__ void __launch_bounds__(S_THREADS, 1)
    k_flow_sample_fused(const __grid_constant__ CUtensorMap mv1, const __grid_constant__ CUtensorMap mv2,
                        const __grid_constant__ CUtensorMap mv3, FusedArgs a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[3], empty[3], xready, gready[2], acc1f, acc2f, acc3f, biasf[2], cplf[4];
  __shared__ __align__(16) float sb[2][2 * 256 + 8];       // biases of a layer: first, second, third product
  __shared__ float s_new[4][FM], s_log[4][FM];              // the rows' transformed coordinates and log scales
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t base = (su32(smem_raw) + 1023u) & ~1023u;
  const uint32_t sx = base, sw = base + X_BYTES, sv3 = sw + 2 * SLOT_BYTES;
  const int H = a.H, K = a.K, C = a.C;
  const int NP = 2 + H / 128;                              // weight parts per layer
  const int NR = H / 128;                                  // 128-column parts and rounds
  const int tiles = (int)((a.n + FM - 1) / FM);
  const uint32_t id_h = idesc_bf16(FM, (uint32_t)H), id_16 = idesc_bf16(FM, 16);

  if (threadIdx.x == 0) {
    for (int s = 0; s < 3; ++s) {
      mbar_init(su32(&full[s]), 1);
      mbar_init(su32(&empty[s]), 1);
    }
    mbar_init(su32(&xready), ROW_WARPS);
    for (int r = 0; r < 2; ++r) {
      mbar_init(su32(&gready[r]), ROW_WARPS);
      mbar_init(su32(&biasf[r]), 1);
    }
    mbar_init(su32(&acc1f), 1);
    mbar_init(su32(&acc2f), 1);
    mbar_init(su32(&acc3f), 1);
    for (int q = 0; q < 4; ++q) mbar_init(su32(&cplf[q]), 4);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
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

  if (warp == 0) {
    uint32_t it = 0, li = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x)
      for (int l = 0; l < K && ok; ++l, ++li)
        for (int p = 0; p < NP; ++p) {
          const bool last = p == NP - 1;
          const uint32_t s = last ? 2u : it & 1u;
          if (!mbar_wait_warp(su32(&empty[s]), ((last ? li : it >> 1) & 1u) ^ 1u, F_WAIT) ||
              __any_sync(0xffffffffu, *(volatile int*)&abort_flag)) {
            ok = false;
            break;
          }
          const uint32_t dst = sw + s * SLOT_BYTES, bar = su32(&full[s]);
          if (elect_one()) {
            if (p == 0) {
              // the slot just freed was filled in the layer before (two parts back), so the rows
              // are through the one before that, whose biases these replace
              const uint32_t bb = su32(&biasf[li & 1u]), d = su32(sb[li & 1u]);
              mbar_expect_tx(bb, (uint32_t)H * 8u + 32u);
              bulk_load(d, a.e1 + l * a.lstride, (uint32_t)H * 4u, bb);
              bulk_load(d + 1024u, a.e2 + l * a.lstride, (uint32_t)H * 4u, bb);
              bulk_load(d + 2048u, a.e3 + l * a.lstride, 32u, bb);
            }
            if (last) {
              mbar_expect_tx(bar, (uint32_t)H * 32u);
              for (int kb = 0; kb < H / 64; ++kb) tma_load_3d(dst + 2048u * kb, &mv3, 64 * kb, 0, l, bar);
            } else {
              const CUtensorMap* m = p == 0 ? &mv1 : &mv2;
              const int kb0 = p == 0 ? 0 : 2 * (p - 1);
              mbar_expect_tx(bar, (uint32_t)H * 256u);
              tma_load_3d(dst, m, 64 * kb0, 0, l, bar);
              tma_load_3d(dst + (uint32_t)H * 128u, m, 64 * (kb0 + 1), 0, l, bar);
            }
          }
          __syncwarp();
          it += !last;
        }
    if (!ok && lane == 0) atomicExch(&abort_flag, 1);
  } else if (warp == 1) {
    uint32_t it = 0, li = 0;
    bool ok = true;
    const int xk = (8 + C + 15) / 16;                        // K steps of X that hold values
    auto wait_on = [&](uint64_t* bar, uint32_t parity) -> bool {
      const bool got = mbar_wait_warp(su32(bar), parity, F_WAIT);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      return got;
    };
    for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x)
      for (int l = 0; l < K && ok; ++l, ++li) {
        // acc1 = X V1^T
        uint32_t slot = it & 1u, wb = sw + slot * SLOT_BYTES;
        if (!(ok = wait_on(&full[slot], (it >> 1) & 1u) && wait_on(&xready, li & 1u))) break;
        if (elect_one()) {
          const uint64_t da = sw128_desc(sx), db = sw128_desc(wb);
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            if (kk < xk)
              mma_bf16(tmem, da + (KB_BYTES * (kk >> 2) + 32u * (kk & 3)) / 16,
                       db + ((uint32_t)H * 128u * (kk >> 2) + 32u * (kk & 3)) / 16, id_h, kk != 0);
          mma_commit(su32(&acc1f));
          mma_commit(su32(&empty[slot]));
        }
        __syncwarp();
        ++it;
        // acc2 = g1 V2^T: K round pr (g1 columns 128 pr ..) once the rows have written it
        for (int pr = 0; pr < NR; ++pr) {
          slot = it & 1u, wb = sw + slot * SLOT_BYTES;
          if (!(ok = wait_on(&full[slot], (it >> 1) & 1u) && wait_on(&gready[pr], 0u))) break;
          if (elect_one()) {
            const uint64_t db = sw128_desc(wb);
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
              mma_bf16_ts(tmem + ACC2, tmem + 128u * pr + 32u * (kk >> 1) + 8u * (kk & 1),
                          db + ((uint32_t)H * 128u * (kk >> 2) + 32u * (kk & 3)) / 16, id_h, (pr | kk) != 0);
            if (pr == NR - 1) mma_commit(su32(&acc2f));
            mma_commit(su32(&empty[slot]));
          }
          __syncwarp();
          ++it;
        }
        if (!ok) break;
        // acc3 = g2 V3^T (16 rows, 8 of them the conditioner's outputs)
        if (!(ok = wait_on(&full[2], li & 1u))) break;
        for (int r = 0; r < NR; ++r) {
          if (!(ok = wait_on(&gready[r], 1u))) break;
          if (elect_one()) {
            const uint64_t db = sw128_desc(sv3 + 4096u * r);
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
              mma_bf16_ts(tmem + ACC3, tmem + ACC2 + 128u * r + 32u * (kk >> 1) + 8u * (kk & 1),
                          db + (2048u * (kk >> 2) + 32u * (kk & 3)) / 16, id_16, (r | kk) != 0);
            if (r == NR - 1) {
              mma_commit(su32(&acc3f));
              mma_commit(su32(&empty[2]));
            }
          }
          __syncwarp();
        }
      }
    if (!ok && lane == 0) atomicExch(&abort_flag, 1);
  } else {
    const int q = warp & 3;
    const int h = (warp - 2) >> 2;                             // which 32 of every 128 columns
    const int r = 32 * q + lane;                               // row of the tile = tensor-memory lane
    const uint32_t lane_addr = tmem + ((uint32_t)(32 * q) << 16);
    uint32_t li = 0;
    bool ok = true;
    auto arrive = [&](uint64_t* bar) {
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(su32(bar));
    };
    auto wait_on = [&](uint64_t* bar, uint32_t parity) -> bool {
      const bool got = mbar_wait(su32(bar), parity, F_WAIT);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      return __all_sync(0xffffffffu, got);
    };
    // bias + ReLU of 32 accumulator columns (chunk c), written over the chunk's own first 16 as
    // bfloat16 pairs; round rd of a hidden layer is chunk 4 rd + h.  In the fragment shape a
    // thread holds 8 columns of 4 rows and reads 8 biases (32 columns of one row would be 32
    // biases: 512 cycles of shared-memory reads a round, of 540)
    auto hidden = [&](uint32_t col0, const float* bias, int c) {
      const uint32_t at = lane_addr + col0 + 32u * c;
      uint32_t raw[32], w[2][8];
      tmem_ld_frag_async(at, raw);
      tmem_ld_frag_async(at + (16u << 16), raw + 16);
      float2 b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) b[i] = *reinterpret_cast<const float2*>(bias + 32 * c + 8 * i + 2 * (lane & 3));
      tmem_wait_ld32(raw);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float2 s = add2(make_float2(__uint_as_float(raw[16 * k + 2 * i]), __uint_as_float(raw[16 * k + 2 * i + 1])), b[i / 2]);
          w[k][i] = pack2_relu(s.x, s.y);
        }
        tmem_st_frag(at + ((uint32_t)(16 * k) << 16), w[k]);
      }
      tmem_wait_st();
    };
    for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
      const int64_t row = (int64_t)t * FM + r;
      const bool valid = row < a.n;
      float v[8], ss = 0.f;
      if (valid) {
        const float4 z0 = reinterpret_cast<const float4*>(a.z + row * 8)[0];
        const float4 z1 = reinterpret_cast<const float4*>(a.z + row * 8)[1];
        v[0] = z0.x; v[1] = z0.y; v[2] = z0.z; v[3] = z0.w; v[4] = z1.x; v[5] = z1.y; v[6] = z1.z; v[7] = z1.w;
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = 0.f;
      }
      // context: columns 8 .. 8 + C - 1 of the input row, zeros up to 128
      int64_t e = 0;
      if (valid) {
        int64_t lo = 0, hi = a.E, s = a.row0 + row;
        while (hi - lo > 1) {
          const int64_t mid = (lo + hi) >> 1;
          if (__ldg(&a.off[mid]) <= s) lo = mid; else hi = mid;
        }
        e = lo;
      }
      const uint4* crow = reinterpret_cast<const uint4*>(a.ctx + e * C);
      for (int g = h == 0 ? 1 : 4 * h; g < 4 * h + 4; ++g) {
        uint4 d = make_uint4(0u, 0u, 0u, 0u);
        if (valid && g <= C / 8) d = __ldg(crow + (g - 1));
        sts128(sx + KB_BYTES * (g >> 3) + swz(r, g & 7), d.x, d.y, d.z, d.w);
      }
      for (int l = 0; l < K; ++l, ++li) {
        const int p = l & 3;
        if (h == 0) {
          uint32_t w0, w1;
          switch (p) {
            case 0: pack_half<0>(v, w0, w1); break;
            case 1: pack_half<1>(v, w0, w1); break;
            case 2: pack_half<2>(v, w0, w1); break;
            default: pack_half<3>(v, w0, w1); break;
          }
          sts128(sx + swz(r, 0), w0, w1, 0u, 0u);
        }
        proxy_fence();
        arrive(&xready);
        const float* bl = sb[li & 1u];
        if (!(ok = wait_on(&biasf[li & 1u], (li >> 1) & 1u) && !*(volatile int*)&abort_flag)) break;
        if (!(ok = wait_on(&acc1f, li & 1u))) break;
        for (int rd = 0; rd < NR; ++rd) {
          hidden(0u, bl, 4 * rd + h);
          arrive(&gready[rd]);
        }
        if (!(ok = wait_on(&acc2f, li & 1u))) break;
        for (int rd = 0; rd < NR; ++rd) {
          hidden(ACC2, bl + 256, 4 * rd + h);
          arrive(&gready[rd]);
        }
        // v_b <- v_b e^s + mu with mu_j = o_j + b3_j, s_j = 3 tanh((o_{4+j} + b3_{4+j}) / 3):
        // coordinate j by warp h = j of the quarter, handed to the others in shared memory
        if (!(ok = wait_on(&acc3f, li & 1u))) break;
        uint32_t om = tmem_ld1_async(lane_addr + ACC3 + h), os = tmem_ld1_async(lane_addr + ACC3 + 4u + h);
        asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(om), "+r"(os)::"memory");
        float vb;
        switch (p) {
          case 0: vb = half_at<0>(v, h); break;
          case 1: vb = half_at<1>(v, h); break;
          case 2: vb = half_at<2>(v, h); break;
          default: vb = half_at<3>(v, h); break;
        }
        const float s = S_MAX * tanhf((__uint_as_float(os) + bl[512 + 4 + h]) / S_MAX);
        s_new[h][r] = fmaf(vb, expf(s), __uint_as_float(om) + bl[512 + h]);
        s_log[h][r] = s;
        __syncwarp();
        if (lane == 0) mbar_arrive(su32(&cplf[q]));
        if (!(ok = wait_on(&cplf[q], li & 1u))) break;
        float x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          x[j] = s_new[j][r];
          ss += s_log[j][r];
        }
        switch (p) {
          case 0: set_half<0>(v, x); break;
          case 1: set_half<1>(v, x); break;
          case 2: set_half<2>(v, x); break;
          default: set_half<3>(v, x); break;
        }
      }
      if (!ok) break;
      if (valid && h == 0) {
        reinterpret_cast<float4*>(a.x_out + row * 8)[0] = make_float4(v[0], v[1], v[2], v[3]);
        reinterpret_cast<float4*>(a.x_out + row * 8)[1] = make_float4(v[4], v[5], v[6], v[7]);
        a.ss_out[row] = ss;
      }
    }
    if (!ok && lane == 0) atomicExch(&abort_flag, 1);
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && *(volatile int*)&abort_flag) atomicExch(&g_flow_status, 1);
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

}  // namespace

bool flow_fused_supported(int C, int H, int K) {
  return (H == 128 || H == 256) && C >= 8 && C % 8 == 0 && 8 + C <= 128 && K >= 1;
}

cudaError_t launch_flow_sample_fused(const void* params_bf16, const float* params, const int64_t* off_t, int C, int H,
                                     int K, const float* z, const void* ctx, const int64_t* ev_off, int64_t E,
                                     int64_t row0, int64_t n, float* x_out, float* ss_out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const __nv_bfloat16* p16 = reinterpret_cast<const __nv_bfloat16*>(params_bf16);
  // one layer's tensors repeat every lstride elements (a multiple of 64, so 128 bytes)
  const int64_t lstride = K > 1 ? off_t[12] - off_t[6] : 64;
  CUtensorMap m1, m2, m3;
  if (!layer_map(&m1, p16 + off_t[6], 8 + C, H, K, lstride, (uint32_t)H) ||
      !layer_map(&m2, p16 + off_t[8], H, H, K, lstride, (uint32_t)H) ||
      !layer_map(&m3, p16 + off_t[10], H, 8, K, lstride, 16u))
    return cudaErrorInvalidValue;
  FusedArgs a;
  a.z = z;
  a.ctx = reinterpret_cast<const __nv_bfloat16*>(ctx);
  a.off = ev_off;
  a.E = E;
  a.row0 = row0;
  a.n = n;
  a.C = C;
  a.H = H;
  a.K = K;
  a.e1 = params + off_t[7];
  a.e2 = params + off_t[9];
  a.e3 = params + off_t[11];
  a.lstride = lstride;
  a.x_out = x_out;
  a.ss_out = ss_out;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int64_t tiles = (n + FM - 1) / FM;
  const unsigned grid = (unsigned)(tiles < sms ? tiles : sms);
  e = cudaFuncSetAttribute(k_flow_sample_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FUSED_SMEM);
  if (e != cudaSuccess) return e;
  k_flow_sample_fused<<<grid, S_THREADS, FUSED_SMEM, s>>>(m1, m2, m3, a);
  return cudaGetLastError();
}

cudaError_t flow_fused_status(int* status) {
  int zero = 0;
  cudaError_t e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = cudaMemcpyFromSymbol(status, g_flow_status, sizeof(int));
  if (e == cudaSuccess && *status != 0) e = cudaMemcpyToSymbol(g_flow_status, &zero, sizeof(int));
  return e;
}

}  // namespace gwx
