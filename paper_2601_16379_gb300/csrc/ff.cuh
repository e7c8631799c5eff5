// Float-float ("double-float") arithmetic for the FP64-class tensor-core path.
//
// A value is the unevaluated sum hi + lo of two floats with |lo| <= ulp(hi)/2,
// about 48 significant bits.  On this GPU the FP64 pipe runs at a small fraction
// of the FP32 rate, so the bulk transforms of the FP64-class path (the k-mesh
// DFTs of the pair tensor, Algorithm 2) run in float-float: each operation is a
// handful of FP32 instructions built on the error-free transformations
//   TwoSum  (Knuth):  s = fl(a + b),  e = (a - (s - b')) + (b - b'),  b' = s - a
//   TwoProd (FMA):    p = fl(a b),    e = fma(a, b, -p)
// (Dekker 1971; the "sloppy" addition of Bailey's double-double library, whose
// error is bounded relative to the operands rather than to the result).  The
// relative error of a multiply or add is ~2^-44, far below what the ERIs need.
#pragma once
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

namespace isdf {

struct ffloat {
  float hi, lo;
  ffloat() = default;
  __host__ __device__ __forceinline__ constexpr ffloat(float h, float l) : hi(h), lo(l) {}
  __host__ __device__ __forceinline__ ffloat(int v) : hi((float)v), lo(0.f) {}
  __host__ __device__ __forceinline__ ffloat(float v) : hi(v), lo(0.f) {}
  // from double: the float nearest to v and the float nearest to the rest
  // (on the device in integer arithmetic where v's exponent is inside the range that keeps both
  // parts normal: conversions run on the FP64 pipe, at two a clock and SM)
  __host__ __device__ __forceinline__ ffloat(double v) {
#ifdef __CUDA_ARCH__
    const uint32_t h = (uint32_t)__double2hiint(v), l = (uint32_t)__double2loint(v), e = (h >> 20) & 0x7ffu;
    if (e - 953u < 190u) {  // 2^-70 <= |v| < 2^120
      const uint32_t f = (((h & 0x7fffffffu) - (896u << 20)) << 3) | (l >> 29), rest = l & 0x1fffffffu;
      const uint32_t up = rest + (f & 1u) > 0x10000000u;  // to nearest, ties to even
      const int r = (int)rest - (int)(up << 29);
      hi = __uint_as_float((f + up) | (h & 0x80000000u));
      lo = __int2float_rn((h >> 31) ? -r : r) * __uint_as_float((e - 948u) << 23);  // r 2^(e - 1075)
      return;
    }
#endif
    hi = (float)v;
    lo = (float)(v - (double)hi);
  }
  __host__ __device__ __forceinline__ double to_double() const { return widen(hi) + widen(lo); }
  // (double)f, a normal f by its bits
  __host__ __device__ static __forceinline__ double widen(float f) {
#ifdef __CUDA_ARCH__
    const uint32_t u = __float_as_uint(f);
    if (((u >> 23) & 0xffu) - 1u < 254u)
      return __hiloint2double((int)((((u & 0x7fffffffu) >> 3) + (896u << 20)) | (u & 0x80000000u)), (int)(u << 29));
#endif
    return (double)f;
  }
};

// complex float-float (16 bytes, the size of a complex128)
struct ffcomplex {
  ffloat x, y;
};

__host__ __device__ __forceinline__ ffloat ff_fast_two_sum(float a, float b) {  // |a| >= |b| or a == 0
  const float s = a + b;
  return ffloat(s, b - (s - a));
}
__host__ __device__ __forceinline__ ffloat ff_two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  return ffloat(s, (a - (s - bb)) + (b - bb));
}

__host__ __device__ __forceinline__ ffloat operator+(ffloat a, ffloat b) {
  ffloat s = ff_two_sum(a.hi, b.hi);
  return ff_fast_two_sum(s.hi, s.lo + (a.lo + b.lo));
}
__host__ __device__ __forceinline__ ffloat operator-(ffloat a) { return ffloat(-a.hi, -a.lo); }
__host__ __device__ __forceinline__ ffloat operator-(ffloat a, ffloat b) { return a + (-b); }
__host__ __device__ __forceinline__ ffloat operator*(ffloat a, ffloat b) {
  const float p = a.hi * b.hi;
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e));
  return ff_fast_two_sum(p, e);
}
__host__ __device__ __forceinline__ ffloat& operator+=(ffloat& a, ffloat b) { return a = a + b; }
__host__ __device__ __forceinline__ ffloat& operator-=(ffloat& a, ffloat b) { return a = a - b; }
__host__ __device__ __forceinline__ ffloat& operator*=(ffloat& a, ffloat b) { return a = a * b; }
// scaling by a power of two is exact
__host__ __device__ __forceinline__ ffloat ff_ldexp(ffloat a, int e) {
  return ffloat(ldexpf(a.hi, e), ldexpf(a.lo, e));
}

__host__ __device__ __forceinline__ ffcomplex cmul(ffcomplex a, ffcomplex b) {
  return ffcomplex{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}

}  // namespace isdf
