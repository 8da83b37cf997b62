// sum2.cuh -- FP32 sums that keep their rounding errors, in place of FP64 accumulation.
#pragma once

#include <stdint.h>

namespace gwx {

// A value and the rounding errors of its additions (Knuth's two-sum), about 48 bits.  Six FP32
// additions a term; an FP64 addition holds an SM's FP64 pipe for 16 cycles a warp.  Its range is
// FP32's: once a partial sum has passed 3.4e38, or a term was infinite or not a number, h is not
// finite and stays so, and whoever took the sum takes it again in FP64 (Sum64), which gives the
// value, the infinity or the not-a-number that FP64 sums give.  While h is finite nothing was lost.
struct Sum2 {
  float h = 0.f, l = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float t = __fadd_rn(h, x), z = __fsub_rn(t, h);
    l = __fadd_rn(l, __fadd_rn(__fsub_rn(h, __fsub_rn(t, z)), __fsub_rn(x, z)));
    h = t;
  }
  __device__ __forceinline__ void add(const Sum2& o) {
    add(o.h);
    l = __fadd_rn(l, o.l);
  }
  __device__ __forceinline__ void add_lanes(int o) {
    Sum2 x;
    x.h = __shfl_xor_sync(0xffffffffu, h, o);
    x.l = __shfl_xor_sync(0xffffffffu, l, o);
    add(x);
  }
  // both parts as one 64-bit word, and the sum of such a word
  __device__ __forceinline__ uint64_t bits() const {
    return (uint64_t)__float_as_uint(h) | (uint64_t)__float_as_uint(l) << 32;
  }
  __device__ __forceinline__ void add_bits(uint64_t w) {
    Sum2 x;
    x.h = __uint_as_float((uint32_t)w);
    x.l = __uint_as_float((uint32_t)(w >> 32));
    add(x);
  }
  __device__ __forceinline__ bool finite() const { return isfinite(h); }
  __device__ __forceinline__ double value() const { return (double)h + (double)l; }
  __device__ __forceinline__ float rounded() const { return __fadd_rn(h, l); }
};

// The same in FP64.
struct Sum64 {
  double v = 0.0;
  __device__ __forceinline__ void add(float x) { v += (double)x; }
  __device__ __forceinline__ void add_lanes(int o) { v += __shfl_xor_sync(0xffffffffu, v, o); }
  __device__ __forceinline__ uint64_t bits() const { return (uint64_t)__double_as_longlong(v); }
  __device__ __forceinline__ void add_bits(uint64_t w) { v += __longlong_as_double((long long)w); }
  __device__ __forceinline__ bool finite() const { return isfinite(v); }
  __device__ __forceinline__ double value() const { return v; }
  __device__ __forceinline__ float rounded() const { return (float)v; }
};

// put(the total of a warp's shares) by lane 0, if `in`: a Sum2, or out of its range a Sum64 of the n
// terms at p, `stride` apart.  (Totals rounded to FP32 without FP64 in between, whose three
// instructions by all lanes of the 32 warps of a block held the pipe for 1 us.)
template <class Put>
__device__ __forceinline__ void warp_total(Sum2 s, const float* p, int64_t n, int64_t stride, bool in, Put put) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s.add_lanes(o);   // the same h in every lane
  if (s.finite()) {
    if (lane == 0 && in) put(s);
    return;
  }
  Sum64 e;
  for (int64_t i = lane; in && i < n; i += 32) e.add(p[i * stride]);
  for (int o = 16; o > 0; o >>= 1) e.add_lanes(o);
  if (lane == 0 && in) put(e);
}

}  // namespace gwx
