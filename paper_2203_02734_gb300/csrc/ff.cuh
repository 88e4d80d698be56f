// ff.cuh -- pairs of floats: an unevaluated sum h + l, about 48 bits, for transforms that need more than FP32 and
// would wait for the FP64 pipe (2 operations a clock and SM against 128 in FP32).
//
// Sums are Knuth's two-sum, products Dekker's with the error term from an FMA; the low parts are added in FP32.  The
// pair is not renormalised: two-sums hold for any pair, over a transform the low part grows to some units of the
// high part's last place, and its own rounding stays near 2^-46 of the largest value.  The intrinsics keep the
// compiler from contracting a product and a sum into one FMA, which would change the error terms.  The range is
// FP32's: below about 2^-102 the low part fades out.
#pragma once
#include <cuda_runtime.h>

namespace pw {

struct ff {
  float h, l;
  ff() = default;
  __host__ __device__ constexpr ff(float x) : h(x), l(0.f) {}
  __host__ __device__ constexpr ff(double x) : h((float)x), l((float)(x - (double)(float)x)) {}
  __device__ __forceinline__ ff(float h_, float l_) : h(h_), l(l_) {}
  __device__ __forceinline__ explicit operator float() const { return h + l; }
};
struct __align__(16) ff2 {
  ff x, y;
};

namespace ffx {
__device__ __forceinline__ float err_of_sum(float a, float b, float s) {
  const float z = __fsub_rn(s, a);
  return __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z));
}
// a b + c d
__device__ __forceinline__ ff dot(ff a, ff b, ff c, ff d) {
  const float p = __fmul_rn(a.h, b.h), q = __fmul_rn(c.h, d.h), s = __fadd_rn(p, q);
  float e = __fadd_rn(err_of_sum(p, q, s), __fmaf_rn(a.h, b.h, -p));
  e = __fadd_rn(e, __fmaf_rn(c.h, d.h, -q));
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  e = __fmaf_rn(c.h, d.l, e);
  e = __fmaf_rn(c.l, d.h, e);
  return ff(s, e);
}
}  // namespace ffx

__device__ __forceinline__ ff operator-(ff a) { return ff(-a.h, -a.l); }
__device__ __forceinline__ ff operator+(ff a, ff b) {
  const float s = __fadd_rn(a.h, b.h);
  return ff(s, __fadd_rn(ffx::err_of_sum(a.h, b.h, s), __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ ff operator-(ff a, ff b) { return a + (-b); }
__device__ __forceinline__ ff operator*(ff a, ff b) {
  const float p = __fmul_rn(a.h, b.h);
  return ff(p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p))));
}

// The names that the codelets of fft.cuh use.
__device__ __forceinline__ ff fma_(ff a, ff b, ff c) { return a * b + c; }
__device__ __forceinline__ ff2 make_c(ff x, ff y) {
  ff2 v;
  v.x = x;
  v.y = y;
  return v;
}
__device__ __forceinline__ ff2 cmul(ff2 a, ff2 b) { return make_c(ffx::dot(a.x, b.x, -a.y, b.y), ffx::dot(a.x, b.y, a.y, b.x)); }

}  // namespace pw
