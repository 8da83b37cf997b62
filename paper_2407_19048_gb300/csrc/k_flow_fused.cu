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
// Every mbarrier wait is bounded; on expiry the CTA records a status, stops, lets its copies and
// products in flight end and frees its tensor memory.
#include "flow_tile.cuh"
#include "pdl.cuh"

namespace gwx {

namespace {

using namespace flowt;

constexpr size_t FUSED_SMEM = FWD_BYTES + 1024;

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

__global__ void __launch_bounds__(FWD_THREADS, 1)
    k_flow_sample_fused(const __grid_constant__ CUtensorMap mv1, const __grid_constant__ CUtensorMap mv2,
                        const __grid_constant__ CUtensorMap mv3, FusedArgs a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(16) FwdRing rg;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t base = (su32(smem_raw) + 1023u) & ~1023u;
  const uint32_t sx = base, sw = base + X_BYTES;
  const int K = a.K, C = a.C, NR = a.H / 128;              // 128-column rounds of the hidden layers
  const int tiles = (int)((a.n + FM - 1) / FM);
  const FwdWeights wt{&mv1, &mv2, &mv3, a.e1, a.e2, a.e3, a.lstride, C, a.H, K, tiles, false};
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
    uint32_t li = 0;
    bool ok = true;
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
          if (a.off[mid] <= s) lo = mid; else hi = mid;
        }
        e = lo;
      }
      const uint4* crow = reinterpret_cast<const uint4*>(a.ctx + e * C);
      for (int g = h == 0 ? 1 : 4 * h; g < 4 * h + 4; ++g) {
        uint4 d = make_uint4(0u, 0u, 0u, 0u);
        if (valid && g <= C / 8) d = crow[g - 1];
        sts128(sx + KB_BYTES * (g >> 3) + swz(r, g & 7), d.x, d.y, d.z, d.w);
      }
      for (int l = 0; l < K; ++l, ++li) {
        const int p = l & 3;
        if (h == 0) {
          uint32_t w0, w1;
          pack_half(p, v, w0, w1);
          sts128(sx + swz(r, 0), w0, w1, 0u, 0u);
        }
        proxy_fence();
        row_arrive(&rg.xready);
        const float* bl = rg.sb[li & 1u];
        if (!(ok = row_wait(&rg.biasf[li & 1u], (li >> 1) & 1u, &rg.abort_flag))) break;
        uint32_t w[2][8];
        if (!(ok = row_wait(&rg.acc1f, li & 1u))) break;
        for (int rd = 0; rd < NR; ++rd) {                      // chunk 4 rd + h of 32 columns
          const int c = 4 * rd + h;
          fwd_hidden(lane_addr + 32u * c, bl + 32 * c, w);
          row_arrive(&rg.gready[rd]);
        }
        if (!(ok = row_wait(&rg.acc2f, li & 1u))) break;
        for (int rd = 0; rd < NR; ++rd) {
          const int c = 4 * rd + h;
          fwd_hidden(lane_addr + ACC2 + 32u * c, bl + 256 + 32 * c, w);
          row_arrive(&rg.gready[rd]);
        }
        // v_b <- v_b e^s + mu with mu_j = o_j + b3_j, s_j = 3 tanh((o_{4+j} + b3_{4+j}) / 3):
        // coordinate j by warp h = j of the quarter, handed to the others in shared memory
        if (!(ok = row_wait(&rg.acc3f, li & 1u))) break;
        uint32_t om = tmem_ld1_async(lane_addr + ACC3 + h), os = tmem_ld1_async(lane_addr + ACC3 + 4u + h);
        asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(om), "+r"(os)::"memory");
        const float s = S_MAX * tanhf((__uint_as_float(os) + bl[512 + 4 + h]) / S_MAX);
        rg.s_new[h][r] = fmaf(half_at(p, v, h), expf(s), __uint_as_float(om) + bl[512 + h]);
        rg.s_log[h][r] = s;
        __syncwarp();
        if (lane == 0) mbar_arrive(su32(&rg.cplf[q]));
        if (!(ok = row_wait(&rg.cplf[q], li & 1u))) break;
        float x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          x[j] = rg.s_new[j][r];
          ss += rg.s_log[j][r];
        }
        set_half(p, v, x);
      }
      if (!ok) break;
      if (valid && h == 0) {
        reinterpret_cast<float4*>(a.x_out + row * 8)[0] = make_float4(v[0], v[1], v[2], v[3]);
        reinterpret_cast<float4*>(a.x_out + row * 8)[1] = make_float4(v[4], v[5], v[6], v[7]);
        a.ss_out[row] = ss;
      }
    }
    if (!ok && lane == 0) atomicExch(&rg.abort_flag, 1);
  }
  fwd_end(rg, tmem, &g_flow_status);
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
  pdl_launch(k_flow_sample_fused, dim3(grid), dim3(FWD_THREADS), FUSED_SMEM, s, m1, m2, m3, a);
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
