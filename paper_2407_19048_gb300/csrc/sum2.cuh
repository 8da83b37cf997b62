// sum2.cuh -- FP32 sums that keep their rounding errors, in place of FP64 accumulation.
#pragma once

namespace gwx {

// A value and the rounding errors of its additions (Knuth's two-sum), about 48 bits.  Six FP32
// additions a term; an FP64 addition holds an SM's FP64 pipe for 16 cycles a warp.
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
  // (an infinite sum's error is not a number)
  __device__ __forceinline__ double value() const { return isfinite(h) ? (double)h + (double)l : (double)h; }
};

}  // namespace gwx
