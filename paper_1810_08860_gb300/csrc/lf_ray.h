// lf_ray.h - the FP32 arithmetic of a pixel's ray and of disk membership, shared by
// the raster, the view selection of two-level frames and the view set-up.  Every
// operation that feeds a decision is an explicit round-to-nearest intrinsic in a
// fixed order.
#pragma once
#include "lf_internal.h"

namespace lfk {

__device__ __forceinline__ float dot3_rn(float a0, float a1, float a2, float b0, float b1, float b2) {
  return __fmaf_rn(a0, b0, __fmaf_rn(a1, b1, __fmul_rn(a2, b2)));
}

// Slope of a pixel column's or row's rays: (i + 1/2 - c) / f.
__device__ __forceinline__ float ray_slope(int i, float c, float f) {
  return __fdiv_rn(__fsub_rn(__fadd_rn((float)i, 0.5f), c), f);
}

// An eye's rays by row: (ey, R1 ey + R2, R4 ey + R5, R7 ey + R8), the parts of a
// world direction d_k = R[3k] ex + (R[3k+1] ey + R[3k+2]) that a row shares.
__device__ __forceinline__ float4 ray_row(const EyeFloat& F, float ey) {
  return make_float4(ey, __fmaf_rn(F.R[1], ey, F.R[2]), __fmaf_rn(F.R[4], ey, F.R[5]), __fmaf_rn(F.R[7], ey, F.R[8]));
}

// The crossing of a pixel's ray with the capture sphere (larger root, t >= 0);
// without one the first coordinate is NaN, which no disk holds.  a = (R0, R3, R6, qc),
// o = the eye's centre relative to the sphere's (EyeFloat::ray, ::centre).
__device__ __forceinline__ void sphere_crossing(const float4& a, const float4& o, float ex, const float4& row, float* p) {
  const float d0 = __fmaf_rn(a.x, ex, row.y), d1 = __fmaf_rn(a.y, ex, row.z), d2 = __fmaf_rn(a.z, ex, row.w);
  const float qa = dot3_rn(d0, d1, d2, d0, d1, d2);
  const float qb = dot3_rn(o.x, o.y, o.z, d0, d1, d2);
  const float disc = __fsub_rn(__fmul_rn(qb, qb), __fmul_rn(qa, a.w));
  p[0] = __int_as_float(0x7fffffff);
  p[1] = p[2] = 0.0f;
  if (!(disc >= 0.0f)) return;
  const float t = __fdiv_rn(__fsub_rn(__fsqrt_rn(disc), qb), qa);
  if (!(t >= 0.0f)) return;
  p[0] = __fmaf_rn(t, d0, o.x);
  p[1] = __fmaf_rn(t, d1, o.y);
  p[2] = __fmaf_rn(t, d2, o.z);
}

// Squared distance of a crossing from a disk's centre, the membership decision's left side.
__device__ __forceinline__ float disk_d2(const float4& cc, const float* p) {
  const float dx = __fsub_rn(p[0], cc.x), dy = __fsub_rn(p[1], cc.y), dz = __fsub_rn(p[2], cc.z);
  return dot3_rn(dx, dy, dz, dx, dy, dz);
}

}  // namespace lfk
