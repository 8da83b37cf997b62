// k_resnet.cu -- the pieces of the ResNet-1D data summary of Sec. 4 around its
// convolutions: 1-D convolutions are im2col rows (channels-last activations, all taps of
// all channels per output time) times the weights on the tensor cores
// (gwx_dense_bf16 / gwx_dense_bf16_backward); these kernels build the rows (k_im2col,
// k_im2col_cf for the channels-first input strain), fold row gradients back (k_col2im),
// normalise per sample and channel group with the residual addition and the ReLU
// (k_gn_forward_s; k_gn_stats, k_gn_apply for other channel counts) and take the gradient of
// that (k_gn_backward_s, which also masks or gathers the gradient it starts from;
// k_gn_bwd_stats, k_gn_bwd_apply, k_gn_param_part / k_gn_param_finish, k_relu_mask), and pool
// (k_maxpool, k_mean_time and their backward).
#include <stdint.h>

#include <algorithm>

#include <cuda_bf16.h>

#include "gwx_internal.h"
#include "pdl.cuh"
#include "sum2.cuh"

namespace gwx {

namespace {

constexpr float GN_EPS = 1e-5f;
constexpr float GN_SCALE = 1.f / (1 << 24);   // of the sums of squares, against overflow of their total

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// Index arithmetic: every kernel runs on a grid whose y coordinate is the sample b and
// whose x threads cover one sample's elements, so the divisions below are 32-bit (the
// C-ABI keeps T C below 2^31 and B below 65536); sums are FP32 per thread over a few
// dozen terms, and FP64 or two floats across threads (GB300's FP64 rate is a small fraction of
// FP32's).

// cols[(b To + t) K + j C + c] = x[b][s t + j - p][c] (zero outside the series and for
// columns >= k C); one thread per 8 columns (C % 8 == 0, so a chunk stays in one tap).
__global__ void k_im2col(const __nv_bfloat16* x, int T, int C, int k, int s, int p, int To, int K,
                         __nv_bfloat16* __restrict__ cols) {
  pdl_enter();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int ch = K / 8;
  if (i >= To * ch) return;
  const int64_t b = blockIdx.y;
  const int t = i / ch, q = i - t * ch;
  const int col = 8 * q, j = col / C, c0 = col - j * C;
  uint4 v = make_uint4(0u, 0u, 0u, 0u);
  const int src = s * t + j - p;
  if (j < k && src >= 0 && src < T) v = *reinterpret_cast<const uint4*>(x + ((b * T + src) * C + c0));
  reinterpret_cast<uint4*>(cols + (b * To + t) * K)[q] = v;
}

// The same rows from channels-first FP32 input y [B][D][N] (the whitened strain).
__global__ void k_im2col_cf(const float* __restrict__ y, int D, int N, int k, int s, int p, int To, int K,
                            __nv_bfloat16* __restrict__ cols) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= To * K) return;
  const int64_t b = blockIdx.y;
  const int t = i / K, col = i - t * K;
  float v = 0.f;
  if (col < k * D) {
    const int j = col / D, c = col - j * D, src = s * t + j - p;
    if (src >= 0 && src < N) v = y[(b * D + c) * N + src];
  }
  cols[(b * To + t) * K + col] = __float2bfloat16_rn(v);
}

// The same, 8 columns (16 bytes) a thread (one column: 34 us for 512 windows of 2 x 2048 samples,
// 7 taps; now 11).
__global__ void k_im2col_cf8(const float* y, int D, int N, int k, int s, int p, int To, int K,
                             __nv_bfloat16* __restrict__ cols) {
  pdl_enter();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int ch = K / 8;
  if (i >= To * ch) return;
  const int64_t b = blockIdx.y;
  const int t = i / ch, q = i - t * ch;
  int j = 8 * q / D, c = 8 * q - j * D;
  float v[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const int src = s * t + j - p;
    v[e] = j < k && src >= 0 && src < N ? y[(b * D + c) * N + src] : 0.f;
    if (++c == D) c = 0, ++j;
  }
  __align__(16) __nv_bfloat162 h[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) h[e] = __floats2bfloat162_rn(v[2 * e], v[2 * e + 1]);
  reinterpret_cast<uint4*>(cols + (b * To + t) * K)[q] = *reinterpret_cast<const uint4*>(h);
}

// dx[b][t][c] = (addend) + sum over taps j with s t_out = t + p - j of dcols[b, t_out][j C + c]
__global__ void k_col2im(const float* __restrict__ dcols, int T, int C, int k, int s, int p, int To, int K,
                         const float* __restrict__ addend, float* __restrict__ dx) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= T * C) return;
  const int64_t b = blockIdx.y;
  const int t = i / C, c = i - t * C;
  const int64_t o = b * T * C + i;
  float acc = addend ? addend[o] : 0.f;
  for (int j = 0; j < k; ++j) {
    const int num = t + p - j;
    if (num < 0 || num % s) continue;
    const int to = num / s;
    if (to < To) acc += dcols[(b * To + to) * K + j * C + c];
  }
  dx[o] = acc;
}

// The same with KT taps known at compile time and four channels per thread: all taps'
// float4 loads are issued before the sums (in tap order, as above).
template <int KT>
__global__ void k_col2im4(const float* dcols, int T, int C, int s, int p, int To, int K,
                          const float* addend, float* __restrict__ dx) {
  pdl_enter();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= T * C / 4) return;
  const int64_t b = blockIdx.y;
  const int t = (4 * i) / C, c = 4 * i - t * C;
  float4 v[KT];
#pragma unroll
  for (int j = 0; j < KT; ++j) {
    const int num = t + p - j;
    const int to = num / s;
    v[j] = (num >= 0 && num - to * s == 0 && to < To)
               ? *reinterpret_cast<const float4*>(dcols + (b * To + to) * K + j * C + c)
               : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  const int64_t o = b * T * C + 4 * (int64_t)i;
  float4 acc = addend ? *reinterpret_cast<const float4*>(addend + o) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int j = 0; j < KT; ++j) {
    acc.x += v[j].x;
    acc.y += v[j].y;
    acc.z += v[j].z;
    acc.w += v[j].w;
  }
  *reinterpret_cast<float4*>(dx + o) = acc;
}

// Block sums of two FP32 per-thread partials in FP64 (warp shuffles, then the warps in
// order); the totals land in thread 0.
__device__ __forceinline__ void block_sum2(double& a, double& b2) {
  __shared__ double r[2][32];
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b2 += __shfl_down_sync(0xffffffffu, b2, o);
  }
  const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  if ((threadIdx.x & 31) == 0) {
    r[0][w] = a;
    r[1][w] = b2;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    a = 0.0;
    b2 = 0.0;
    for (int k = 0; k < nw; ++k) {
      a += r[0][k];
      b2 += r[1][k];
    }
  }
}

// Per (sample, group): mean and 1 / sqrt(var + eps) over T x C/G values.  The values are
// shifted by the group's first value before squaring, so the FP32 partial sums do not
// cancel when the mean is large against the spread.  VEC values per load (4 when C/G is a
// multiple of 4).
template <int VEC>
__global__ void __launch_bounds__(256) k_gn_stats(const float* __restrict__ z, int T, int C, int G,
                                                  float* __restrict__ ms) {
  const int b = blockIdx.x / G, g = blockIdx.x - (blockIdx.x / G) * G, cg = C / G, cv = cg / VEC;
  const float* zb = z + (int64_t)b * T * C + g * cg;
  const float k0 = __ldg(zb);
  float s1 = 0.f, s2 = 0.f;
#pragma unroll 4
  for (int e = threadIdx.x; e < T * cv; e += blockDim.x) {
    const int t = e / cv, c = (e - t * cv) * VEC;
    if constexpr (VEC == 4) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(zb + (int64_t)t * C + c));
      const float d0 = v.x - k0, d1 = v.y - k0, d2 = v.z - k0, d3 = v.w - k0;
      s1 += (d0 + d1) + (d2 + d3);
      s2 += fmaf(d0, d0, __fmul_rn(d1, d1)) + fmaf(d2, d2, __fmul_rn(d3, d3));
    } else {
      const float d = __ldg(zb + (int64_t)t * C + c) - k0;
      s1 += d;
      s2 += d * d;
    }
  }
  double a = s1, q = s2;
  block_sum2(a, q);
  if (threadIdx.x == 0) {
    const double n = (double)T * cg, m = a / n, var = fmax(q / n - m * m, 0.0);
    ms[2 * blockIdx.x] = (float)((double)k0 + m);
    ms[2 * blockIdx.x + 1] = (float)(1.0 / sqrt(var + (double)GN_EPS));
  }
}

// Per-sample group norm for C / 4 dividing 256: one block takes sample b's [T][C] slab twice,
// first for the sums and then to apply them, so that no launch and no second statistics array
// lies between; part of the second pass hits in L2.  HBM bound as long as enough loads are in
// flight: every pass first issues its rows' loads (eight, or four of several arrays) and then
// adds them (a loop of load and add kept one row in flight, 10 us a slab).  (512 windows, stem
// and two blocks, six normalisations: 337 us as a statistics and an apply kernel forward, now
// 201; ~700 us backward with the ReLU mask, the FP32 dz and its conversion as passes of their
// own, now 411.  Slabs staged in shared memory by asynchronous copies, columns split over
// blocks, read every array once but left too few threads for the runs: 194 and 504.)
// Sums: thread (run slice s, row lane l, column quad q) reads runs of 16 rows, rl = 256 / (C / 4)
// rows apart, of channels 4 q .. 4 q + 3, coalesced float4 loads; FP32 within a run (the
// contractions spelled out: the compiler's choice changes with the code around), two-float sums
// across runs (sum2.cuh; in FP64 forward 227 us, backward 510); then the lanes of each column
// quad and the quads of each group.  A block whose totals leave the range of two floats takes its
// sums again in FP64.
constexpr int GN_NT = 512;
// threads of the backward: the pooled gradient's rows hold twice the registers
constexpr int gn_bt(int src) { return src == 2 ? 256 : 512; }

// Sums of a (and q) over the threads of every group (out[2 g], out[2 g + 1], valid after the
// caller's barrier): lanes of a warp that share a column quad by shuffles, the remaining rows
// of quads in shared memory (r, NT entries), one warp per group.  True where a sum of this thread
// is not finite.
struct __align__(16) QuadSums {
  uint64_t a, q;   // as bits()
};
template <int NT, class S>
__device__ __forceinline__ bool sample_group_sums(S a, S q, int cq, int cg, int G, QuadSums* r, double* out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int o = 16; o >= cq; o >>= 1) {
    a.add_lanes(o);
    q.add_lanes(o);
  }
  const int rows = cq < 32 ? NT / 32 : NT / cq;
  if (cq >= 32) {
    r[threadIdx.x] = QuadSums{a.bits(), q.bits()};
  } else if (lane < cq) {
    r[warp * cq + lane] = QuadSums{a.bits(), q.bits()};
  }
  __syncthreads();
  const int per = cg / 4;
  bool over = false;
  for (int g = warp; g < G; g += NT / 32) {
    S x, y;
    for (int i = lane; i < rows * per; i += 32) {
      const QuadSums v = r[(i / per) * cq + g * per + i % per];
      x.add_bits(v.a);
      y.add_bits(v.q);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      x.add_lanes(o);
      y.add_lanes(o);
    }
    if (lane == 0) {
      out[2 * g] = x.value();
      out[2 * g + 1] = y.value();
    }
    over |= !x.finite() || !y.finite();
  }
  return over;
}

// 1 / sqrt(v) in FP64 from the single-precision value and two Newton steps (errors of 2^-22, 1e-13
// and FP64's rounding; the library's FP64 call is a chain of some 2000 cycles here)
__device__ __forceinline__ double inv_sqrt(double v) {
  if (!(v < 1e30)) return rsqrt(v);
  double y = (double)rsqrtf((float)v);
  y *= 1.5 - 0.5 * v * y * y;
  return y * (1.5 - 0.5 * v * y * y);
}

__device__ __forceinline__ float4 bf16x4(uint2 q) {
  const float2 lo = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.x));
  const float2 hi = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.y));
  return make_float4(lo.x, lo.y, hi.x, hi.y);
}
__device__ __forceinline__ uint2 to_bf16x4(float a, float b, float c, float d) {
  __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
  return make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
}

__global__ void __launch_bounds__(GN_NT, 2) k_gn_forward_s(const float* z, int T, int C, int G,
                                                           double inv_n, const float* gamma, const float* beta,
                                                           const float* res32, const __nv_bfloat16* res16, int relu,
                                                           __nv_bfloat16* __restrict__ out16,
                                                           float* __restrict__ out32, float* __restrict__ ms) {
  pdl_enter();
  __shared__ double sums[64];
  __shared__ float st[64];
  __shared__ QuadSums quads[GN_NT];
  const int cq = C / 4, rl = 256 / cq, cg = C / G;
  const int q4 = threadIdx.x % cq, l0 = (threadIdx.x % 256) / cq, g = (4 * q4) / cg;
  const int64_t off = (int64_t)blockIdx.x * T * C;
  const float4* z4 = reinterpret_cast<const float4*>(z + off) + q4;   // row t at t cq
  const float k0 = z[off + g * cg];
  auto collect = [&](auto zero) {   // the sums, in the arithmetic of `zero`; true: out of its range
    decltype(zero) a, q;
    for (int t0 = l0 + (threadIdx.x / 256) * 16 * rl; t0 < T; t0 += (GN_NT / 256) * 16 * rl) {
      float s1 = 0.f, s2 = 0.f;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float4 v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int t = t0 + (8 * h + i) * rl;
          v[i] = t < T ? z4[t * cq] : make_float4(k0, k0, k0, k0);   // adds zero
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float d0 = v[i].x - k0, d1 = v[i].y - k0, d2 = v[i].z - k0, d3 = v[i].w - k0;
          s1 += (d0 + d1) + (d2 + d3);
          s2 += fmaf(d0, d0, __fmul_rn(d1, d1)) + fmaf(d2, d2, __fmul_rn(d3, d3));
        }
      }
      a.add(s1);
      q.add(__fmul_rn(s2, GN_SCALE));
    }
    return sample_group_sums<GN_NT>(a, q, cq, cg, G, quads, sums);
  };
  const float kg = (int)threadIdx.x < G ? z[off + threadIdx.x * cg] : 0.f;
  const float4 gm = make_float4(gamma[4 * q4], gamma[4 * q4 + 1], gamma[4 * q4 + 2], gamma[4 * q4 + 3]);
  const float4 bt = make_float4(beta[4 * q4], beta[4 * q4 + 1], beta[4 * q4 + 2], beta[4 * q4 + 3]);
  if (__syncthreads_or(collect(Sum2()))) {
    collect(Sum64());
    __syncthreads();
  }
  if ((int)threadIdx.x < G) {
    const int i = threadIdx.x;
    const double m = sums[2 * i] * inv_n, var = fmax(sums[2 * i + 1] * (inv_n / GN_SCALE) - m * m, 0.0);
    const float mean = (float)((double)kg + m), rstd = (float)inv_sqrt(var + (double)GN_EPS);
    st[2 * i] = mean;
    st[2 * i + 1] = rstd;
    ms[2 * ((int64_t)blockIdx.x * G + i)] = mean;
    ms[2 * ((int64_t)blockIdx.x * G + i) + 1] = rstd;
  }
  __syncthreads();
  const float mean = st[2 * g], rstd = st[2 * g + 1];
  const int step = GN_NT / cq;
  for (int tb = threadIdx.x / cq; tb < T; tb += 4 * step) {
    float4 x[4], r[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int t = min(tb + k * step, T - 1);
      x[k] = ld_stream(z4 + t * cq);
      if (res32) r[k] = reinterpret_cast<const float4*>(res32 + off)[t * cq + q4];
      if (res16) r[k] = bf16x4(reinterpret_cast<const uint2*>(res16 + off)[t * cq + q4]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int t = tb + k * step;
      if (t >= T) break;
      const int64_t i = off + (int64_t)t * C + 4 * q4;
      float4 v = make_float4(fmaf((x[k].x - mean) * rstd, gm.x, bt.x), fmaf((x[k].y - mean) * rstd, gm.y, bt.y),
                             fmaf((x[k].z - mean) * rstd, gm.z, bt.z), fmaf((x[k].w - mean) * rstd, gm.w, bt.w));
      if (res32 || res16) {
        v.x += r[k].x; v.y += r[k].y; v.z += r[k].z; v.w += r[k].w;
      }
      if (relu) v = make_float4(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f), fmaxf(v.z, 0.f), fmaxf(v.w, 0.f));
      if (out16) *reinterpret_cast<uint2*>(out16 + i) = to_bf16x4(v.x, v.y, v.z, v.w);
      if (out32) *reinterpret_cast<float4*>(out32 + i) = v;
    }
  }
}

// The gradient dy the backward starts from: as given; masked by out > 0 (the ReLU after the
// normalisation); the max pool's gradient routed back to its arguments, then masked; or the
// mean over time's, dm / T, masked.  Loads and values apart, so that several rows' loads can
// be in flight.
enum : int { DY_PLAIN = 0, DY_MASK = 1, DY_POOL = 2, DY_MEAN = 3 };
struct GnSource {
  const float* dy;             // [B][T][C]; DY_POOL [B][To][C]; DY_MEAN [B][C]
  const __nv_bfloat16* out;    // [B][T][C]
  const uint8_t* arg;          // DY_POOL: [B][To][C]
  int To;
};
template <int SRC>
struct GnRow {
  float4 v0, v1;
  uchar4 a0, a1;
  uint2 o;
};

template <int SRC>
__device__ __forceinline__ void gn_load(GnRow<SRC>& r, const GnSource& s, int64_t b, int t, int c, int T, int C) {
  const int64_t i = (b * T + t) * C + c;
  if constexpr (SRC == DY_POOL) {
    // time t is argument 1 of window t/2 (even t), or 2 of window t/2, which there always is, and
    // 0 of the next (odd t, gn_load_next)
    const int64_t o = (b * s.To + t / 2) * C + c;
    r.v1 = make_float4(0.f, 0.f, 0.f, 0.f);
    r.a1 = make_uchar4(3, 3, 3, 3);
    r.v0 = *reinterpret_cast<const float4*>(s.dy + o);
    r.a0 = *reinterpret_cast<const uchar4*>(s.arg + o);
  } else if constexpr (SRC != DY_MEAN) {
    r.v0 = *reinterpret_cast<const float4*>(s.dy + i);
  }
  if constexpr (SRC != DY_PLAIN) r.o = *reinterpret_cast<const uint2*>(s.out + i);
}
// The next window's share of an odd time, behind the loads that every row has (between them, a branch a
// row, the kernel took 163 to 180 us; this order 131; both windows always 193).
__device__ __forceinline__ void gn_load_next(GnRow<DY_POOL>& r, const GnSource& s, int64_t b, int t, int c, int C) {
  const int to = t / 2 + 1;
  if ((t & 1) && to < s.To) {
    const int64_t o = (b * s.To + to) * C + c;
    r.v1 = *reinterpret_cast<const float4*>(s.dy + o);
    r.a1 = *reinterpret_cast<const uchar4*>(s.arg + o);
  }
}

template <int SRC>
__device__ __forceinline__ float4 gn_value(const GnRow<SRC>& r, int t, float4 mean_dy) {
  float4 d = r.v0;
  if constexpr (SRC == DY_MEAN) d = mean_dy;
  if constexpr (SRC == DY_POOL) {
    const int k = 1 + (t & 1);
    d = make_float4((r.a0.x == k ? r.v0.x : 0.f) + (r.a1.x == 0 ? r.v1.x : 0.f),
                    (r.a0.y == k ? r.v0.y : 0.f) + (r.a1.y == 0 ? r.v1.y : 0.f),
                    (r.a0.z == k ? r.v0.z : 0.f) + (r.a1.z == 0 ? r.v1.z : 0.f),
                    (r.a0.w == k ? r.v0.w : 0.f) + (r.a1.w == 0 ? r.v1.w : 0.f));
  }
  if constexpr (SRC != DY_PLAIN) {
    const float4 o = bf16x4(r.o);
    d = make_float4(o.x > 0.f ? d.x : 0.f, o.y > 0.f ? d.y : 0.f, o.z > 0.f ? d.z : 0.f, o.w > 0.f ? d.w : 0.f);
  }
  return d;
}

// dz = rstd (dy gamma - m1 - xhat m2) (FP32 or bfloat16), the masked dy itself (optional) and,
// per channel, this sample's sums of dy xhat and dy (part, [B][C][2] doubles), the partials
// of dgamma and dbeta that k_gn_param_finish adds.
template <int SRC, bool OUT16>
__global__ void __launch_bounds__(gn_bt(SRC), 2) k_gn_backward_s(GnSource src, const float* z, int T, int C,
                                                            int G, double inv_n, const float* ms,
                                                            const float* gamma, void* __restrict__ dz,
                                                            float* __restrict__ dsum, double* __restrict__ part) {
  pdl_enter();
  constexpr int GN_BT = gn_bt(SRC);
  __shared__ double sums[64];
  __shared__ uint64_t pr[GN_BT * 8];   // as bits()
  __shared__ float st[64];
  __shared__ QuadSums quads[GN_BT];
  constexpr int U = 4;   // rows in flight
  const int cq = C / 4, rl = 256 / cq, cg = C / G;
  const int q4 = threadIdx.x % cq, l0 = (threadIdx.x % 256) / cq, g = (4 * q4) / cg;
  const int64_t b = blockIdx.x, off = b * T * C;
  const float4* z4 = reinterpret_cast<const float4*>(z + off) + q4;   // row t at t cq
  const float mean = ms[2 * (b * G + g)], rstd = ms[2 * (b * G + g) + 1];
  const float4 gm = make_float4(gamma[4 * q4], gamma[4 * q4 + 1], gamma[4 * q4 + 2], gamma[4 * q4 + 3]);
  float4 mdy = make_float4(0.f, 0.f, 0.f, 0.f);
  if constexpr (SRC == DY_MEAN) {
    const float4 v = reinterpret_cast<const float4*>(src.dy + b * C)[q4];
    mdy = make_float4(v.x / T, v.y / T, v.z / T, v.w / T);
  }
  auto collect = [&](auto zero) {   // the sums, in the arithmetic of `zero`; true: out of its range
    using S = decltype(zero);
    S a, q, pg[4], pb[4];
    for (int t0 = l0 + (threadIdx.x / 256) * 16 * rl; t0 < T; t0 += (GN_BT / 256) * 16 * rl) {
      float s1 = 0.f, s2 = 0.f;
      float fg[4] = {0.f, 0.f, 0.f, 0.f}, fb[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
      for (int h = 0; h < 16; h += U) {
        GnRow<SRC> r[U];
        float4 x[U];
#pragma unroll
        for (int i = 0; i < U; ++i) {
          const int t = min(t0 + (h + i) * rl, T - 1);
          gn_load<SRC>(r[i], src, b, t, 4 * q4, T, C);
          x[i] = z4[t * cq];
        }
        if constexpr (SRC == DY_POOL) {
#pragma unroll
          for (int i = 0; i < U; ++i) gn_load_next(r[i], src, b, min(t0 + (h + i) * rl, T - 1), 4 * q4, C);
        }
#pragma unroll
        for (int i = 0; i < U; ++i) {
          const int t = t0 + (h + i) * rl;
          if (t >= T) break;
          const float4 d = gn_value<SRC>(r[i], t, mdy);
          const float a0 = d.x * gm.x, a1 = d.y * gm.y, a2 = d.z * gm.z, a3 = d.w * gm.w;
          const float h0 = (x[i].x - mean) * rstd, h1 = (x[i].y - mean) * rstd, h2 = (x[i].z - mean) * rstd,
                      h3 = (x[i].w - mean) * rstd;
          s1 += (a0 + a1) + (a2 + a3);
          s2 += (a0 * h0 + a1 * h1) + (a2 * h2 + a3 * h3);
          fg[0] += d.x * h0;
          fg[1] += d.y * h1;
          fg[2] += d.z * h2;
          fg[3] += d.w * h3;
          fb[0] += d.x;
          fb[1] += d.y;
          fb[2] += d.z;
          fb[3] += d.w;
        }
      }
      a.add(s1);
      q.add(s2);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        pg[m].add(fg[m]);
        pb[m].add(fb[m]);
      }
    }
    if (part) {
      // lanes of a warp that share a column quad first, then one row of quads per warp
      for (int o = 16; o >= cq; o >>= 1) {
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          pg[m].add_lanes(o);
          pb[m].add_lanes(o);
        }
      }
      const int lane = threadIdx.x & 31, at = cq >= 32 ? threadIdx.x : (threadIdx.x >> 5) * cq + lane;
      if (cq >= 32 || lane < cq) {
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          pr[at * 8 + m] = pg[m].bits();
          pr[at * 8 + 4 + m] = pb[m].bits();
        }
      }
    }
    bool over = sample_group_sums<GN_BT>(a, q, cq, cg, G, quads, sums);
    if (part) {
      // one thread per channel and sum, over the rows of quads in order
      const int rows = cq < 32 ? GN_BT / 32 : GN_BT / cq;
      for (int i = threadIdx.x; i < 2 * C; i += GN_BT) {
        const int c = i >> 1, k = (c & 3) + 4 * (i & 1);
        S t;
#pragma unroll 4
        for (int r = 0; r < rows; ++r) t.add_bits(pr[(r * cq + c / 4) * 8 + k]);
        part[b * 2 * C + i] = t.value();
        over |= !t.finite();
      }
    }
    return over;
  };
  if (__syncthreads_or(collect(Sum2()))) {
    collect(Sum64());
    __syncthreads();
  }
  if ((int)threadIdx.x < G) {
    st[2 * threadIdx.x] = (float)(sums[2 * threadIdx.x] * inv_n);
    st[2 * threadIdx.x + 1] = (float)(sums[2 * threadIdx.x + 1] * inv_n);
  }
  __syncthreads();
  const float m1 = st[2 * g], m2 = st[2 * g + 1];
  const int step = GN_BT / cq;
  for (int tb = threadIdx.x / cq; tb < T; tb += U * step) {
    GnRow<SRC> r[U];
    float4 x[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int t = min(tb + k * step, T - 1);
      gn_load<SRC>(r[k], src, b, t, 4 * q4, T, C);
      x[k] = ld_stream(z4 + t * cq);
    }
    if constexpr (SRC == DY_POOL) {
#pragma unroll
      for (int k = 0; k < U; ++k) gn_load_next(r[k], src, b, min(tb + k * step, T - 1), 4 * q4, C);
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int t = tb + k * step;
      if (t >= T) break;
      const int64_t i = off + (int64_t)t * C + 4 * q4;
      const float4 d = gn_value<SRC>(r[k], t, mdy);
      float4 o;
      o.x = rstd * (d.x * gm.x - m1 - (x[k].x - mean) * rstd * m2);
      o.y = rstd * (d.y * gm.y - m1 - (x[k].y - mean) * rstd * m2);
      o.z = rstd * (d.z * gm.z - m1 - (x[k].z - mean) * rstd * m2);
      o.w = rstd * (d.w * gm.w - m1 - (x[k].w - mean) * rstd * m2);
      if constexpr (OUT16)
        *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(dz) + i) = to_bf16x4(o.x, o.y, o.z, o.w);
      else
        *reinterpret_cast<float4*>(reinterpret_cast<float*>(dz) + i) = o;
      if (dsum) *reinterpret_cast<float4*>(dsum + i) = d;
    }
  }
}

// out = act(gamma_c (z - mean) rstd + beta_c + residual), bfloat16 or FP32 out; residual
// FP32 (res32) or bfloat16 (res16) or none.  VEC consecutive channels per thread.
template <int VEC>
__global__ void k_gn_apply(const float* __restrict__ z, int T, int C, int G, const float* __restrict__ ms,
                           const float* __restrict__ gamma, const float* __restrict__ beta,
                           const float* __restrict__ res32, const __nv_bfloat16* __restrict__ res16, int relu,
                           __nv_bfloat16* __restrict__ out16, float* __restrict__ out32) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= T * C / VEC) return;
  const int b = blockIdx.y;
  const int c = (j * VEC) % C, g = c / (C / G);
  const int64_t i = (int64_t)b * T * C + (int64_t)j * VEC;
  const float mean = ms[2 * (b * G + g)], rstd = ms[2 * (b * G + g) + 1];
  float v[VEC];
  if constexpr (VEC == 4) {
    const float4 q = *reinterpret_cast<const float4*>(z + i);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  } else {
    v[0] = z[i];
  }
#pragma unroll
  for (int u = 0; u < VEC; ++u) v[u] = fmaf((v[u] - mean) * rstd, __ldg(&gamma[c + u]), __ldg(&beta[c + u]));
  if (res32) {
    if constexpr (VEC == 4) {
      const float4 q = *reinterpret_cast<const float4*>(res32 + i);
      v[0] += q.x; v[1] += q.y; v[2] += q.z; v[3] += q.w;
    } else {
      v[0] += res32[i];
    }
  }
  if (res16) {
    if constexpr (VEC == 4) {
      const uint2 q = *reinterpret_cast<const uint2*>(res16 + i);
      const float2 lo = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.x));
      const float2 hi = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.y));
      v[0] += lo.x; v[1] += lo.y; v[2] += hi.x; v[3] += hi.y;
    } else {
      v[0] += __bfloat162float(res16[i]);
    }
  }
  if (relu) {
#pragma unroll
    for (int u = 0; u < VEC; ++u) v[u] = fmaxf(v[u], 0.f);
  }
  if constexpr (VEC == 4) {
    if (out16) {
      __nv_bfloat162 lo = __floats2bfloat162_rn(v[0], v[1]), hi = __floats2bfloat162_rn(v[2], v[3]);
      uint2 q;
      q.x = *reinterpret_cast<uint32_t*>(&lo);
      q.y = *reinterpret_cast<uint32_t*>(&hi);
      *reinterpret_cast<uint2*>(out16 + i) = q;
    }
    if (out32) *reinterpret_cast<float4*>(out32 + i) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
    if (out16) out16[i] = __float2bfloat16_rn(v[0]);
    if (out32) out32[i] = v[0];
  }
}

// dsum = dy [out > 0]
__global__ void k_relu_mask(const float* __restrict__ dy, const __nv_bfloat16* __restrict__ out, int64_t n,
                            float* __restrict__ d) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) d[i] = __bfloat162float(out[i]) > 0.f ? dy[i] : 0.f;
}

// The same, four elements per thread (n4 = n / 4 groups).
__global__ void k_relu_mask4(const float* __restrict__ dy, const __nv_bfloat16* __restrict__ out, int64_t n4,
                             float* __restrict__ d) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n4) return;
  const float4 g = __ldg(reinterpret_cast<const float4*>(dy) + i);
  const uint2 q = __ldg(reinterpret_cast<const uint2*>(out) + i);
  const float2 lo = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.x));
  const float2 hi = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.y));
  reinterpret_cast<float4*>(d)[i] = make_float4(lo.x > 0.f ? g.x : 0.f, lo.y > 0.f ? g.y : 0.f,
                                                hi.x > 0.f ? g.z : 0.f, hi.y > 0.f ? g.w : 0.f);
}

// Per (sample, group): the means of dxh = dy gamma and dxh xhat.
template <int VEC>
__global__ void __launch_bounds__(256) k_gn_bwd_stats(const float* __restrict__ dy, const float* __restrict__ z,
                                                      int T, int C, int G, const float* __restrict__ ms,
                                                      const float* __restrict__ gamma, float* __restrict__ mm) {
  const int b = blockIdx.x / G, g = blockIdx.x - (blockIdx.x / G) * G, cg = C / G, cv = cg / VEC;
  const int64_t base = (int64_t)b * T * C + g * cg;
  const float mean = ms[2 * blockIdx.x], rstd = ms[2 * blockIdx.x + 1];
  float s1 = 0.f, s2 = 0.f;
#pragma unroll 4
  for (int e = threadIdx.x; e < T * cv; e += blockDim.x) {
    const int t = e / cv, c = (e - t * cv) * VEC;
    const int64_t i = base + (int64_t)t * C + c;
    if constexpr (VEC == 4) {
      const float4 d = __ldg(reinterpret_cast<const float4*>(dy + i));
      const float4 x = __ldg(reinterpret_cast<const float4*>(z + i));
      const float4 gm = make_float4(__ldg(&gamma[g * cg + c]), __ldg(&gamma[g * cg + c + 1]),
                                    __ldg(&gamma[g * cg + c + 2]), __ldg(&gamma[g * cg + c + 3]));
      const float a0 = d.x * gm.x, a1 = d.y * gm.y, a2 = d.z * gm.z, a3 = d.w * gm.w;
      s1 += (a0 + a1) + (a2 + a3);
      s2 += (a0 * ((x.x - mean) * rstd) + a1 * ((x.y - mean) * rstd)) +
            (a2 * ((x.z - mean) * rstd) + a3 * ((x.w - mean) * rstd));
    } else {
      const float a = __ldg(dy + i) * __ldg(&gamma[g * cg + c]);
      s1 += a;
      s2 += a * ((__ldg(z + i) - mean) * rstd);
    }
  }
  double a = s1, q = s2;
  block_sum2(a, q);
  if (threadIdx.x == 0) {
    const double n = (double)T * cg;
    mm[2 * blockIdx.x] = (float)(a / n);
    mm[2 * blockIdx.x + 1] = (float)(q / n);
  }
}

// dz = rstd (dy gamma - m1 - xhat m2)
template <int VEC>
__global__ void k_gn_bwd_apply(const float* __restrict__ dy, const float* __restrict__ z, int T, int C, int G,
                               const float* __restrict__ ms, const float* __restrict__ mm,
                               const float* __restrict__ gamma, float* __restrict__ dz) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= T * C / VEC) return;
  const int b = blockIdx.y;
  const int c = (j * VEC) % C, bg = b * G + c / (C / G);
  const int64_t i = (int64_t)b * T * C + (int64_t)j * VEC;
  const float mean = ms[2 * bg], rstd = ms[2 * bg + 1], m1 = mm[2 * bg], m2 = mm[2 * bg + 1];
  if constexpr (VEC == 4) {
    const float4 d = *reinterpret_cast<const float4*>(dy + i);
    const float4 x = *reinterpret_cast<const float4*>(z + i);
    float4 o;
    o.x = rstd * (d.x * __ldg(&gamma[c]) - m1 - (x.x - mean) * rstd * m2);
    o.y = rstd * (d.y * __ldg(&gamma[c + 1]) - m1 - (x.y - mean) * rstd * m2);
    o.z = rstd * (d.z * __ldg(&gamma[c + 2]) - m1 - (x.z - mean) * rstd * m2);
    o.w = rstd * (d.w * __ldg(&gamma[c + 3]) - m1 - (x.w - mean) * rstd * m2);
    *reinterpret_cast<float4*>(dz + i) = o;
  } else {
    dz[i] = rstd * (dy[i] * gamma[c] - m1 - (z[i] - mean) * rstd * m2);
  }
}

// dgamma_c = sum dy xhat, dbeta_c = sum dy over samples and times, in two deterministic
// passes: block (channel tile of 32, row slice of about 256 rows) sums its slice (8 row
// lanes; FP32 over runs of 64 rows, FP64 across runs) into part[slice][c][2];
// k_gn_param_finish adds the slices in order.
constexpr int GN_MAX_SLICES = 1024;

int gn_slices(int64_t rows) { return (int)std::min<int64_t>(GN_MAX_SLICES, std::max<int64_t>(1, (rows + 255) / 256)); }

__global__ void __launch_bounds__(256) k_gn_param_part(const float* __restrict__ dy, const float* __restrict__ z,
                                                       int rows, int T, int C, int G,
                                                       const float* __restrict__ ms, double* __restrict__ part) {
  __shared__ double a[8][33], bb[8][33];
  const int cx = threadIdx.x & 31, ry = threadIdx.x >> 5;
  const int c = blockIdx.x * 32 + cx;
  const int per = (rows + gridDim.y - 1) / gridDim.y;
  const int r0 = blockIdx.y * per, r1 = min(rows, r0 + per);
  double sg = 0.0, sb = 0.0;
  if (c < C) {
    const int g = c / (C / G);
    int r = r0 + ry, b = r / T, t = r - b * T;
    while (r < r1) {
      float fg = 0.f, fb = 0.f;
      for (int n = 0; n < 64 && r < r1; ++n) {
        const int64_t i = (int64_t)r * C + c;
        const float d = __ldg(dy + i);
        fg += d * ((__ldg(z + i) - ms[2 * (b * G + g)]) * ms[2 * (b * G + g) + 1]);
        fb += d;
        r += 8;
        t += 8;
        while (t >= T) {
          t -= T;
          ++b;
        }
      }
      sg += fg;
      sb += fb;
    }
  }
  a[ry][cx] = sg;
  bb[ry][cx] = sb;
  __syncthreads();
  if (ry == 0 && c < C) {
    double tg = 0.0, tb = 0.0;
    for (int k = 0; k < 8; ++k) {
      tg += a[k][cx];
      tb += bb[k][cx];
    }
    part[((int64_t)blockIdx.y * C + c) * 2] = tg;
    part[((int64_t)blockIdx.y * C + c) * 2 + 1] = tb;
  }
}

// Sums of the slices: block of 2 channels x 128 slice lanes (lane l: slices l, l + 128, ...),
// the lanes of a warp by shuffles, the warps in order.  Two channels a block, so that the FP64
// additions are spread over many SMs (512 slices of 128 channels: 4 blocks of 32 took 14.7 us,
// 16 of 8 8.0, these 5.0).
constexpr int PF_C = 2, PF_NT = 256;
__global__ void __launch_bounds__(PF_NT) k_gn_param_finish(const double* part, int slices, int C,
                                                           float* __restrict__ dgamma, float* __restrict__ dbeta) {
  pdl_enter();
  __shared__ double2 r[PF_NT / 32][PF_C];
  const int c = blockIdx.x * PF_C + (threadIdx.x & (PF_C - 1));
  double tg = 0.0, tb = 0.0;
  if (c < C) {
#pragma unroll 4
    for (int s = threadIdx.x / PF_C; s < slices; s += PF_NT / PF_C) {
      const double* v = part + ((int64_t)s * C + c) * 2;   // (a caller's scratch: 8-byte aligned)
      tg += v[0];
      tb += v[1];
    }
  }
#pragma unroll
  for (int o = 16; o >= PF_C; o >>= 1) {
    tg += __shfl_xor_sync(0xffffffffu, tg, o);
    tb += __shfl_xor_sync(0xffffffffu, tb, o);
  }
  if ((threadIdx.x & 31) < PF_C) r[threadIdx.x >> 5][threadIdx.x & (PF_C - 1)] = make_double2(tg, tb);
  __syncthreads();
  if (threadIdx.x < PF_C && c < C) {
    double g = 0.0, bsum = 0.0;
#pragma unroll
    for (int y = 0; y < PF_NT / 32; ++y) {
      g += r[y][threadIdx.x].x;
      bsum += r[y][threadIdx.x].y;
    }
    dgamma[c] = (float)g;
    dbeta[c] = (float)bsum;
  }
}

// k 3, s 2, p 1 max pool over time (first maximum of a window), and its backward.
__global__ void k_maxpool(const __nv_bfloat16* __restrict__ x, int T, int C, int To, __nv_bfloat16* __restrict__ y,
                          uint8_t* __restrict__ arg) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= To * C) return;
  const int64_t b = blockIdx.y;
  const int t = i / C, c = i - t * C;
  float best = -INFINITY;
  int a = 0;
  for (int j = 0; j < 3; ++j) {
    const int src = 2 * t + j - 1;
    if (src < 0 || src >= T) continue;
    const float v = __bfloat162float(x[(b * T + src) * C + c]);
    if (v > best) {
      best = v;
      a = j;
    }
  }
  y[b * To * C + i] = __float2bfloat16_rn(best);
  arg[b * To * C + i] = (uint8_t)a;
}

// The same for eight consecutive channels per thread (C % 8 == 0, 16-byte aligned x and y,
// 8-byte aligned arg): one 16-byte load per tap (512 windows of 1024 x 64: 65 us one channel
// a thread).
__global__ void k_maxpool8(const __nv_bfloat16* x, int T, int C, int To, __nv_bfloat16* __restrict__ y,
                           uint8_t* __restrict__ arg) {
  pdl_enter();
  const int i = blockIdx.x * blockDim.x + threadIdx.x, cv = C / 8;
  if (i >= To * cv) return;
  const int64_t b = blockIdx.y;
  const int t = i / cv, c = 8 * (i - t * cv);
  uint4 v[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int src = 2 * t + j - 1;
    v[j] = src >= 0 && src < T ? *reinterpret_cast<const uint4*>(x + (b * T + src) * C + c)
                               : make_uint4(0xff80ff80u, 0xff80ff80u, 0xff80ff80u, 0xff80ff80u);   // -inf: never first
  }
  const __nv_bfloat16* e0 = reinterpret_cast<const __nv_bfloat16*>(&v[0]);
  __align__(16) __nv_bfloat16 best[8];   // stored whole below
  __align__(8) uint8_t a[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    float m = -INFINITY;
    a[k] = 0;
    best[k] = __float2bfloat16_rn(m);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const float f = __bfloat162float(e0[8 * j + k]);
      if (f > m) {
        m = f;
        best[k] = e0[8 * j + k];
        a[k] = (uint8_t)j;
      }
    }
  }
  const int64_t o = (b * To + t) * C + c;
  *reinterpret_cast<uint4*>(y + o) = *reinterpret_cast<const uint4*>(best);
  *reinterpret_cast<uint2*>(arg + o) = *reinterpret_cast<const uint2*>(a);
}

__global__ void k_maxpool_back(const float* __restrict__ dy, const uint8_t* __restrict__ arg, int T, int C, int To,
                               float* __restrict__ dx) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= T * C) return;
  const int64_t b = blockIdx.y;
  const int t = i / C, c = i - t * C;
  float acc = 0.f;
  for (int to = t / 2; to <= (t + 1) / 2; ++to) {
    if (to >= To) continue;
    const int64_t o = (b * To + to) * C + c;
    if (2 * to - 1 + (int)arg[o] == t) acc += dy[o];
  }
  dx[b * T * C + i] = acc;
}

// The same for four consecutive channels per thread (C % 4 == 0, 16-byte aligned dy, dx):
// float4 gradients, 4-byte argument groups; identical sums.
__global__ void k_maxpool_back4(const float* __restrict__ dy, const uint8_t* __restrict__ arg, int T, int C, int To,
                                float* __restrict__ dx) {
  const int i4 = blockIdx.x * blockDim.x + threadIdx.x;
  if (i4 >= T * C / 4) return;
  const int64_t b = blockIdx.y;
  const int t = (4 * i4) / C, c = 4 * i4 - t * C;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int to = t / 2; to <= (t + 1) / 2; ++to) {
    if (to >= To) continue;
    const int64_t o = (b * To + to) * C + c;
    const float4 d = __ldg(reinterpret_cast<const float4*>(dy + o));
    const uchar4 a = __ldg(reinterpret_cast<const uchar4*>(arg + o));
    const int base = 2 * to - 1;
    if (base + (int)a.x == t) acc.x += d.x;
    if (base + (int)a.y == t) acc.y += d.y;
    if (base + (int)a.z == t) acc.z += d.z;
    if (base + (int)a.w == t) acc.w += d.w;
  }
  reinterpret_cast<float4*>(dx + b * T * C)[i4] = acc;
}

__global__ void k_mean_time(const __nv_bfloat16* __restrict__ x, int64_t B, int T, int C,
                            __nv_bfloat16* __restrict__ m) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B * C) return;
  const int64_t b = i / C;
  const int c = (int)(i - b * C);
  float acc = 0.f;
#pragma unroll 16
  for (int t = 0; t < T; ++t) acc += __bfloat162float(x[(b * T + t) * C + c]);   // in order; 16 loads in flight
  m[i] = __float2bfloat16_rn(acc / T);
}

// The same, two channels a thread and 32 loads in flight (512 windows of 256 x 128: 25.4 us with one
// channel and 16 loads, now 12.7).
__global__ void k_mean_time2(const __nv_bfloat16* x, int64_t B, int T, int C,
                             __nv_bfloat16* __restrict__ m) {
  pdl_enter();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int h = C / 2;
  if (i >= B * h) return;
  const int64_t b = i / h;
  const uint32_t* p = reinterpret_cast<const uint32_t*>(x) + b * T * h + (i - b * h);
  float a0 = 0.f, a1 = 0.f;
  auto add = [&](uint32_t v) {   // a bfloat16 is the upper half of its float
    a0 += __uint_as_float(v << 16);
    a1 += __uint_as_float(v & 0xffff0000u);
  };
  int t = 0;
  for (; t + 32 <= T; t += 32) {
    uint32_t v[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = p[(t + k) * h];
#pragma unroll
    for (int k = 0; k < 32; ++k) add(v[k]);
  }
  for (; t < T; ++t) add(p[t * h]);
  reinterpret_cast<__nv_bfloat162*>(m)[i] = __floats2bfloat162_rn(a0 / T, a1 / T);
}

__global__ void k_mean_time_back(const float* __restrict__ dm, int T, int C, float* __restrict__ dx) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= T * C) return;
  const int64_t b = blockIdx.y;
  dx[b * T * C + i] = dm[b * C + i % C] / T;
}

bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }
// the per-sample statistics kernels: C / 4 divides 256, at most 32 groups of whole quads
bool per_sample_ok(int C, int G) { return C % 4 == 0 && 256 % (C / 4) == 0 && (C / G) % 4 == 0 && G <= 32; }
bool aligned8(const void* p) { return ((uintptr_t)p & 7u) == 0; }

}  // namespace

cudaError_t launch_im2col(const void* x, int64_t B, int T, int C, int k, int s, int p, int K, void* cols,
                          cudaStream_t st) {
  const int To = (T + 2 * p - k) / s + 1;
  pdl_launch(k_im2col, dim3(nblk((int64_t)To * (K / 8), 256), (unsigned)B), dim3(256), 0, st,
             reinterpret_cast<const __nv_bfloat16*>(x), T, C, k, s, p, To, K,
             reinterpret_cast<__nv_bfloat16*>(cols));
  return cudaGetLastError();
}

cudaError_t launch_im2col_cf(const float* y, int64_t B, int D, int N, int k, int s, int p, int K, void* cols,
                             cudaStream_t st) {
  const int To = (N + 2 * p - k) / s + 1;
  if (K % 8 == 0 && aligned16(cols))
    pdl_launch(k_im2col_cf8, dim3(nblk((int64_t)To * (K / 8), 256), (unsigned)B), dim3(256), 0, st, y, D, N, k, s, p,
               To, K, reinterpret_cast<__nv_bfloat16*>(cols));
  else
    k_im2col_cf<<<dim3(nblk((int64_t)To * K, 256), (unsigned)B), 256, 0, st>>>(y, D, N, k, s, p, To, K,
                                                                               reinterpret_cast<__nv_bfloat16*>(cols));
  return cudaGetLastError();
}

cudaError_t launch_col2im(const float* dcols, int64_t B, int T, int C, int k, int s, int p, int K, const float* addend,
                          float* dx, cudaStream_t st) {
  const int To = (T + 2 * p - k) / s + 1;
  const bool v4 = C % 4 == 0 && K % 4 == 0 && aligned16(dcols) && aligned16(addend) && aligned16(dx);
  const dim3 g4(nblk((int64_t)T * C / 4, 256), (unsigned)B);
  if (v4 && k == 1) {
    pdl_launch(k_col2im4<1>, g4, dim3(256), 0, st, dcols, T, C, s, p, To, K, addend, dx);
  } else if (v4 && k == 5) {
    pdl_launch(k_col2im4<5>, g4, dim3(256), 0, st, dcols, T, C, s, p, To, K, addend, dx);
  } else if (v4 && k == 7) {
    k_col2im4<7><<<g4, 256, 0, st>>>(dcols, T, C, s, p, To, K, addend, dx);
  } else {
    k_col2im<<<dim3(nblk((int64_t)T * C, 256), (unsigned)B), 256, 0, st>>>(dcols, T, C, k, s, p, To, K, addend, dx);
  }
  return cudaGetLastError();
}

cudaError_t launch_group_norm(const float* z, int64_t B, int T, int C, int G, const float* gamma, const float* beta,
                              const float* res32, const void* res16, int relu, void* out16, float* out32, float* ms,
                              cudaStream_t st) {
  const bool v4 = (C / G) % 4 == 0 && aligned16(z) && aligned16(res32) && aligned8(res16) && aligned8(out16) &&
                  aligned16(out32);
  const auto r16 = reinterpret_cast<const __nv_bfloat16*>(res16);
  const auto o16 = reinterpret_cast<__nv_bfloat16*>(out16);
  if (v4 && per_sample_ok(C, G)) {
    pdl_launch(k_gn_forward_s, dim3((unsigned)B), dim3(GN_NT), 0, st, z, T, C, G, 1.0 / ((double)T * (C / G)), gamma,
               beta, res32, r16, relu, o16, out32, ms);
  } else if (v4) {
    k_gn_stats<4><<<(unsigned)(B * G), 256, 0, st>>>(z, T, C, G, ms);
    k_gn_apply<4><<<dim3(nblk((int64_t)T * C / 4, 256), (unsigned)B), 256, 0, st>>>(z, T, C, G, ms, gamma, beta, res32,
                                                                                    r16, relu, o16, out32);
  } else {
    k_gn_stats<1><<<(unsigned)(B * G), 256, 0, st>>>(z, T, C, G, ms);
    k_gn_apply<1><<<dim3(nblk((int64_t)T * C, 256), (unsigned)B), 256, 0, st>>>(z, T, C, G, ms, gamma, beta, res32,
                                                                                r16, relu, o16, out32);
  }
  return cudaGetLastError();
}

template <int SRC, bool OUT16>
static cudaError_t launch_gn_backward(const GnSource& src, const float* z, int64_t B, int T, int C, int G,
                                      const float* ms, const float* gamma, void* dz, float* dsum, double* part,
                                      cudaStream_t st) {
  const double inv_n = 1.0 / ((double)T * (C / G));
  pdl_launch(k_gn_backward_s<SRC, OUT16>, dim3((unsigned)B), dim3(gn_bt(SRC)), 0, st, src, z, T, C, G, inv_n, ms,
             gamma, dz, dsum, part);
  return cudaGetLastError();
}

size_t group_norm_backward_scratch(int64_t B, int C, int G) {
  return (size_t)B * G * 2 * sizeof(float) + 256 + (size_t)GN_MAX_SLICES * C * 2 * sizeof(double);
}

cudaError_t launch_group_norm_backward(const float* dy, const float* z, int64_t B, int T, int C, int G,
                                       const float* ms, const float* gamma, void* scratch, float* dz, float* dgamma,
                                       float* dbeta, cudaStream_t st) {
  float* mm = reinterpret_cast<float*>(scratch);
  double* part = reinterpret_cast<double*>(reinterpret_cast<char*>(scratch) +
                                           (((size_t)B * G * 2 * sizeof(float) + 255) & ~(size_t)255));
  const bool v4 = (C / G) % 4 == 0 && aligned16(dy) && aligned16(z) && aligned16(dz);
  if (v4 && per_sample_ok(C, G)) {
    // the per-channel parameter sums come out of the statistics pass, one slice per sample
    const bool fused = B <= GN_MAX_SLICES;
    const cudaError_t e = launch_gn_backward<DY_PLAIN, false>(GnSource{dy, nullptr, nullptr, 0}, z, B, T, C, G, ms, gamma,
                                                              dz, nullptr, fused ? part : nullptr, st);
    if (e != cudaSuccess) return e;
    if (fused) {
      pdl_launch(k_gn_param_finish, dim3(nblk(C, PF_C)), dim3(PF_NT), 0, st, part, (int)B, C, dgamma, dbeta);
      return cudaGetLastError();
    }
  } else if (v4) {
    k_gn_bwd_stats<4><<<(unsigned)(B * G), 256, 0, st>>>(dy, z, T, C, G, ms, gamma, mm);
    k_gn_bwd_apply<4><<<dim3(nblk((int64_t)T * C / 4, 256), (unsigned)B), 256, 0, st>>>(dy, z, T, C, G, ms, mm, gamma,
                                                                                        dz);
  } else {
    k_gn_bwd_stats<1><<<(unsigned)(B * G), 256, 0, st>>>(dy, z, T, C, G, ms, gamma, mm);
    k_gn_bwd_apply<1><<<dim3(nblk((int64_t)T * C, 256), (unsigned)B), 256, 0, st>>>(dy, z, T, C, G, ms, mm, gamma, dz);
  }
  const int slices = gn_slices(B * T);
  k_gn_param_part<<<dim3(nblk(C, 32), slices), 256, 0, st>>>(dy, z, (int)(B * T), T, C, G, ms, part);
  pdl_launch(k_gn_param_finish, dim3(nblk(C, PF_C)), dim3(PF_NT), 0, st, part, slices, C, dgamma, dbeta);
  return cudaGetLastError();
}

bool group_norm_backward_src_ok(int C, int G) { return C % G == 0 && per_sample_ok(C, G); }

size_t group_norm_backward_src_scratch(int64_t B, int C) { return (size_t)B * C * 2 * sizeof(double); }

cudaError_t launch_group_norm_backward_src(int kind, const float* dy, const void* out, const uint8_t* arg,
                                           const float* z, int64_t B, int T, int C, int G, const float* ms,
                                           const float* gamma, void* scratch, void* dz16, float* dsum, float* dgamma,
                                           float* dbeta, cudaStream_t st) {
  const GnSource src{dy, reinterpret_cast<const __nv_bfloat16*>(out), arg, (T + 2 - 3) / 2 + 1};
  double* part = reinterpret_cast<double*>(scratch);
  cudaError_t e = cudaErrorInvalidValue;
  switch (kind) {
    case DY_PLAIN: e = launch_gn_backward<DY_PLAIN, true>(src, z, B, T, C, G, ms, gamma, dz16, dsum, part, st); break;
    case DY_MASK: e = launch_gn_backward<DY_MASK, true>(src, z, B, T, C, G, ms, gamma, dz16, dsum, part, st); break;
    case DY_POOL: e = launch_gn_backward<DY_POOL, true>(src, z, B, T, C, G, ms, gamma, dz16, dsum, part, st); break;
    case DY_MEAN: e = launch_gn_backward<DY_MEAN, true>(src, z, B, T, C, G, ms, gamma, dz16, dsum, part, st); break;
    default: break;
  }
  if (e != cudaSuccess) return e;
  pdl_launch(k_gn_param_finish, dim3(nblk(C, PF_C)), dim3(PF_NT), 0, st, part, (int)B, C, dgamma, dbeta);
  return cudaGetLastError();
}

cudaError_t launch_relu_mask(const float* dy, const void* out, int64_t n, float* d, cudaStream_t st) {
  if (n % 4 == 0 && aligned16(dy) && aligned8(out) && aligned16(d))
    k_relu_mask4<<<nblk(n / 4, 256), 256, 0, st>>>(dy, reinterpret_cast<const __nv_bfloat16*>(out), n / 4, d);
  else
    k_relu_mask<<<nblk(n, 256), 256, 0, st>>>(dy, reinterpret_cast<const __nv_bfloat16*>(out), n, d);
  return cudaGetLastError();
}

cudaError_t launch_maxpool(const void* x, int64_t B, int T, int C, void* y, uint8_t* arg, cudaStream_t st) {
  const int To = (T + 2 - 3) / 2 + 1;
  if (C % 8 == 0 && aligned16(x) && aligned16(y) && ((uintptr_t)arg & 7u) == 0) {
    pdl_launch(k_maxpool8, dim3(nblk((int64_t)To * C / 8, 256), (unsigned)B), dim3(256), 0, st,
               reinterpret_cast<const __nv_bfloat16*>(x), T, C, To, reinterpret_cast<__nv_bfloat16*>(y), arg);
    return cudaGetLastError();
  }
  k_maxpool<<<dim3(nblk((int64_t)To * C, 256), (unsigned)B), 256, 0, st>>>(
      reinterpret_cast<const __nv_bfloat16*>(x), T, C, To, reinterpret_cast<__nv_bfloat16*>(y), arg);
  return cudaGetLastError();
}

cudaError_t launch_maxpool_back(const float* dy, const uint8_t* arg, int64_t B, int T, int C, float* dx,
                                cudaStream_t st) {
  const int To = (T + 2 - 3) / 2 + 1;
  if (C % 4 == 0 && aligned16(dy) && aligned16(dx) && ((uintptr_t)arg & 3u) == 0)
    k_maxpool_back4<<<dim3(nblk((int64_t)T * C / 4, 256), (unsigned)B), 256, 0, st>>>(dy, arg, T, C, To, dx);
  else
    k_maxpool_back<<<dim3(nblk((int64_t)T * C, 256), (unsigned)B), 256, 0, st>>>(dy, arg, T, C, To, dx);
  return cudaGetLastError();
}

cudaError_t launch_mean_time(const void* x, int64_t B, int T, int C, void* m, cudaStream_t st) {
  const auto x16 = reinterpret_cast<const __nv_bfloat16*>(x);
  const auto m16 = reinterpret_cast<__nv_bfloat16*>(m);
  if (C % 2 == 0 && ((uintptr_t)x & 3u) == 0 && ((uintptr_t)m & 3u) == 0)
    pdl_launch(k_mean_time2, dim3(nblk(B * C / 2, 64)), dim3(64), 0, st, x16, B, T, C, m16);
  else
    k_mean_time<<<nblk(B * C, 64), 64, 0, st>>>(x16, B, T, C, m16);
  return cudaGetLastError();
}

cudaError_t launch_mean_time_back(const float* dm, int64_t B, int T, int C, float* dx, cudaStream_t st) {
  k_mean_time_back<<<dim3(nblk((int64_t)T * C, 256), (unsigned)B), 256, 0, st>>>(dm, T, C, dx);
  return cudaGetLastError();
}

}  // namespace gwx
