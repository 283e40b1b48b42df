// Evaluation of a block's far-field record (k_far_*, tdc_merge.cu) at a position: barycentric
// interpolation through its kFarM Chebyshev points, by a warp.
#pragma once

#include "tdc_common.cuh"

namespace tdc {

__device__ __forceinline__ int* far_range(double* rec) { return reinterpret_cast<int*>(rec + 5 * kFarM); }
__device__ __forceinline__ const int* far_range(const double* rec) {
  return reinterpret_cast<const int*>(rec + 5 * kFarM);
}

// Barycentric weights of the block's points for position x (relative to the block's pole
// ref): bw in lanes below kFarM, and 1 / (x - y); a point that x falls on takes all of it.
// Returns that point, or -1.
__device__ __forceinline__ int far_weights(const double* rec, double x, double& bw, double& rd) {
  const int lane = threadIdx.x & 31;
  bw = 0.0;
  rd = 0.0;
  bool hit = false;
  if (lane < kFarM) {
    const double d = x - rec[lane];
    hit = !in_range(fabs(d));
    if (!hit) {
      rd = rcp_nr(d);
      bw = rec[kFarM + lane] * rd;
    }
  }
  const unsigned h = __ballot_sync(0xffffffffu, hit);
  if (h) {
    bw = lane == __ffs(h) - 1 ? 1.0 : 0.0;
    rd = 0.0;
  }
  return __ffs(h) - 1;
}

// The interpolant's slope at point k itself.  Out of line: hardly ever called, and inside the root
// kernel it cost registers (108 -> 92 bytes of spills, roots of a bidiagonal SVD of 205 141.4 -> 139.1 us).
__device__ __noinline__ float far_slope_at(const double* rec, int k, double ff) {
  const int lane = threadIdx.x & 31;
  double t = 0.0;
  if (lane < kFarM && lane != k)
    t = rec[kFarM + lane] * (ff - rec[2 * kFarM + k]) * rcp_nr(rec[k] - rec[lane]);
  return (float)(warp_sum(t) * rcp_nr(rec[kFarM + k]));
}

// The far poles' sum p at x (relative to pole ref) and its slope, good to 2^-20 of Sf rd3: Sf
// bounds the sum of magnitudes, rd3 = 1 / (3 h) the reciprocal distance.  The slope is the sum of
// bw (p - f) / (x - y) over that of bw.  Within 2^-20 h of a point its term is a difference of
// p and f there that rounds by 2^-52 |f| or so over a distance that may be as small, and on the
// point it is 0 / 0: there the slope is taken at the point itself, sum of w_j / w_k (f_j - f_k) /
// (y_k - y_j), which differs by 2^-20 h times the second derivative, 2 / 3 of the stated error.
__device__ __forceinline__ void far_value(const double* rec, double x, double& p, float& slope, float& Sf, float& rd3) {
  const int lane = threadIdx.x & 31;
  double bw, rd, ff = 0.0;
  int k = far_weights(rec, x, bw, rd);
  Sf = 0.0f;
  if (lane < kFarM) {
    ff = rec[2 * kFarM + lane];
    Sf = (float)rec[3 * kFarM + lane];
  }
  double num = bw * ff, den = bw;
  warp_sum2(num, den);
  const double rden = rcp_nr(den);
  p = num * rden;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) Sf = fmaxf(Sf, __shfl_xor_sync(0xffffffffu, Sf, o));
  rd3 = (float)rec[5 * kFarM + 1];
  const float rdf = (float)rd;
  const unsigned near = __ballot_sync(0xffffffffu, fabsf(rdf) > 0x1.8p21f * rd3);
  if (near) k = __ffs(near) - 1;
  if (k < 0) {
    slope = ((float)bw * (float)rden) * (float)(p - ff) * rdf;  // each product within FP32's range
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) slope += __shfl_xor_sync(0xffffffffu, slope, o);
  } else {
    slope = far_slope_at(rec, k, ff);
  }
}

}  // namespace tdc
