// prior.cuh -- the prior draws and the whitening filter's values as device functions, for the
// kernels that compute them alone and the one that prepares a whole batch.
#pragma once

#include "common.cuh"

namespace gwx {

// Linear maps use the non-contracting intrinsics so the doubles equal a plain
// lo + (hi - lo) u evaluated with two roundings.
__device__ __forceinline__ double lin_map(double lo, double hi, double u) {
  return __dadd_rn(lo, __dmul_rn(__dsub_rn(hi, lo), u));
}

// One draw's stream: block j of draw b gives the uniforms u_2j and u_2j+1 (block 5: u_10 and
// the crop offset's word).
struct PriorStream {
  gwx_prior p;
  uint32_t k0, k1, step;

  __device__ __forceinline__ u32x4 words(int64_t b, int j) const {
    return philox4x32_10((uint32_t)b, (uint32_t)j, TAG_PRIOR, step, k0, k1);
  }
  __device__ __forceinline__ void masses(int64_t b, double& m1, double& m2) const {
    const u32x4 r = words(b, 0);
    m1 = lin_map(p.m_lo, p.m_hi, uniform52(r.x, r.y));
    m2 = lin_map(p.m_lo, p.m_hi, uniform52(r.z, r.w));
  }
  __device__ __forceinline__ void spins(int64_t b, double& c1, double& c2) const {
    const u32x4 r = words(b, 1);
    c1 = lin_map(p.chi_lo, p.chi_hi, uniform52(r.x, r.y));
    c2 = lin_map(p.chi_lo, p.chi_hi, uniform52(r.z, r.w));
  }
  __device__ __forceinline__ void dist_tc(int64_t b, double& d, double& tc) const {
    const u32x4 r = words(b, 2);
    d = lin_map(p.d_lo, p.d_hi, uniform52(r.x, r.y));
    tc = lin_map(p.tc_lo, p.tc_hi, uniform52(r.z, r.w));
  }
  __device__ __forceinline__ void phic_iota(int64_t b, double& phic, double& iota) const {
    const u32x4 r = words(b, 3);
    phic = lin_map(p.phi_lo, p.phi_hi, uniform52(r.x, r.y));
    iota = acos(__dsub_rn(1.0, __dmul_rn(2.0, uniform52(r.z, r.w))));
  }
  __device__ __forceinline__ void psi_ra(int64_t b, double& psi, double& ra) const {
    const u32x4 r = words(b, 4);
    psi = lin_map(p.psi_lo, p.psi_hi, uniform52(r.x, r.y));
    ra = __dmul_rn(6.283185307179586476925286766559, uniform52(r.z, r.w));
  }
  __device__ __forceinline__ void dec_offset(int64_t b, uint32_t span, double& dec, int64_t& off) const {
    const u32x4 r = words(b, 5);
    dec = asin(__dsub_rn(__dmul_rn(2.0, uniform52(r.x, r.y)), 1.0));
    off = (int64_t)(((uint64_t)r.z * (uint64_t)span) >> 32);
  }
};

// W_k = M_k / sqrt(S~_k fs/2) (whitening), or M_k sqrt(S~_k fs/2) with `inverse` (the
// unwhitening filter: its inverse on the band), entry i of [D][N/2 + 1]; S~ the PSD linearly
// interpolated from the grid fs/M to fs/N at the exact rational position k M / N.
__device__ __forceinline__ float whiten_filter_at(const double* __restrict__ psd, int64_t i, int64_t M, double fs,
                                                  int k_lo, int64_t N, bool inverse) {
  const int64_t F = N / 2 + 1;
  const int d = (int)(i / F);
  const int64_t k = i % F;
  if (k < k_lo || k >= N / 2) return 0.f;
  const int64_t nb = M / 2 + 1;
  const int64_t num = k * M;
  const int64_t j0 = num / N;
  const int64_t j1 = j0 + 1 < nb ? j0 + 1 : nb - 1;
  const double frac = (double)(num % N) / (double)N;
  const double* p = psd + (int64_t)d * nb;
  const double S = p[j0] + (p[j1] - p[j0]) * frac;
  return inverse ? (float)sqrt(S * fs * 0.5) : (float)(1.0 / sqrt(S * fs * 0.5));
}

}  // namespace gwx
