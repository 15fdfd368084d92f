// mhd_pair.cuh -- packed FP32 pairs (f32x2: FFMA2, FADD2, FMUL2) and the
// sixth-order stencils of two x-adjacent cells, shared by the z-march kernels
// that work on cell pairs (the right-hand side / RK kernel, its adjoint point
// mode, the adjoint gather).
#pragma once
#include <cuda_runtime.h>

namespace mhd {
namespace pk {

typedef float2 f2;
__host__ __device__ __forceinline__ f2 F2(float a) { return make_float2(a, a); }
__device__ __forceinline__ f2 add(f2 a, f2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ f2 mul(f2 a, f2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { return __ffma2_rn(a, b, c); }
// a - b, one rounding
__device__ __forceinline__ f2 dif(f2 a, f2 b) { return __ffma2_rn(b, F2(-1.f), a); }
__device__ __forceinline__ f2 ld2(const float* p) { return *reinterpret_cast<const f2*>(p); }

// stencil weights divided by the spacing (D1) or its square (D2), as pairs
struct Coef {
  f2 c1, c2, c3;        // D1 weights / spacing
  f2 e0, e1, e2, e3;    // D2 weights / spacing^2
};

// ---- stencils on a box row / column at an even x position -----------------
// first and second x derivatives of the cell pair at p (p even, p - 4 .. p + 5 in the row)
__device__ __forceinline__ void dx_pair(const float* p, const Coef& c, f2& d1, f2* d2) {
  const f2 m4 = ld2(p - 4), m2 = ld2(p - 2), z0 = ld2(p), p2 = ld2(p + 2), p4 = ld2(p + 4);
  // the odd offsets straddle the loaded pairs: their sums and differences go as
  // scalars straight into place, which is shorter than assembling the pairs
  d1 = fma2(c.c1, make_float2(z0.y - m2.y, p2.x - z0.x),
            fma2(c.c2, dif(p2, m2), mul(c.c3, make_float2(p2.y - m4.y, p4.x - m2.x))));
  if (d2)
    *d2 = fma2(c.e0, z0, fma2(c.e1, make_float2(z0.y + m2.y, p2.x + z0.x),
                              fma2(c.e2, add(p2, m2), mul(c.e3, make_float2(p2.y + m4.y, p4.x + m2.x)))));
}
// first and second derivatives along a stride s (in floats) of the pair at p
__device__ __forceinline__ void ds_pair(const float* p, int s, const Coef& c, f2& d1, f2* d2) {
  const f2 z0 = ld2(p), a1 = ld2(p + s), b1 = ld2(p - s), a2 = ld2(p + 2 * s), b2 = ld2(p - 2 * s),
           a3 = ld2(p + 3 * s), b3 = ld2(p - 3 * s);
  d1 = fma2(c.c1, dif(a1, b1), fma2(c.c2, dif(a2, b2), mul(c.c3, dif(a3, b3))));
  if (d2) *d2 = fma2(c.e0, z0, fma2(c.e1, add(a1, b1), fma2(c.e2, add(a2, b2), mul(c.e3, add(a3, b3)))));
}

// The same stencils in units of their smallest weight,
//   d  = 45 (f_1 - f_-1) - 9 (f_2 - f_-2) + (f_3 - f_-3)                 (60 h D1)
//   dd = 135 (f_1 + f_-1) - 13.5 (f_2 + f_-2) + (f_3 + f_-3) - 245 f     (90 h^2 D2)
// one multiplication less each, and one set of constants for all axes; the
// scales ride on the multiply-adds that consume them.
__device__ __forceinline__ f2 comb1(f2 d1, f2 d2, f2 d3) { return fma2(F2(45.f), d1, fma2(F2(-9.f), d2, d3)); }
__device__ __forceinline__ f2 comb2(f2 c, f2 s1, f2 s2, f2 s3) {
  return fma2(F2(-245.f), c, fma2(F2(135.f), s1, fma2(F2(-13.5f), s2, s3)));
}
// first (D) and second (DD) differences in x of the pair at p, whose value is z0
template <bool D, bool DD>
__device__ __forceinline__ void ux_pair(const float* p, f2 z0, f2& d, f2& dd) {
  const f2 m4 = ld2(p - 4), m2 = ld2(p - 2), p2 = ld2(p + 2), p4 = ld2(p + 4);
  if (D)
    d = comb1(make_float2(z0.y - m2.y, p2.x - z0.x), dif(p2, m2), make_float2(p2.y - m4.y, p4.x - m2.x));
  if (DD)
    dd = comb2(z0, make_float2(z0.y + m2.y, p2.x + z0.x), add(p2, m2), make_float2(p2.y + m4.y, p4.x + m2.x));
}
// the same along a stride s (in floats)
template <bool D, bool DD>
__device__ __forceinline__ void us_pair(const float* p, int s, f2 z0, f2& d, f2& dd) {
  const f2 a1 = ld2(p + s), b1 = ld2(p - s), a2 = ld2(p + 2 * s), b2 = ld2(p - 2 * s), a3 = ld2(p + 3 * s),
           b3 = ld2(p - 3 * s);
  if (D) d = comb1(dif(a1, b1), dif(a2, b2), dif(a3, b3));
  if (DD) dd = comb2(z0, add(a1, b1), add(a2, b2), add(a3, b3));
}
__device__ __forceinline__ f2 ux1(const float* p, f2 z0) {
  f2 d, dd;
  ux_pair<true, false>(p, z0, d, dd);
  return d;
}
__device__ __forceinline__ f2 us1(const float* p, int s) {
  f2 d, dd;
  us_pair<true, false>(p, s, F2(0.f), d, dd);  // no centre value in a first difference
  return d;
}

}  // namespace pk
}  // namespace mhd
