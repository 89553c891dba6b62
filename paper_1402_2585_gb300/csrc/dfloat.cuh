// Double-float arithmetic ("df"): a value is the unevaluated sum hi + lo of
// two float32 numbers with |lo| <= ulp(hi) / 2, about 48 significant bits.
// Built from the error-free transformations TwoSum (Knuth, TAOCP vol. 2,
// 4.2.2) and TwoProd with a fused multiply-add (Dekker 1971; the FMA form is
// exact because fma(a, b, -a*b) recovers the rounding error of the product).
// The FP64 fine operator computes in this type because FP64 arithmetic on
// GB300 runs at a small fraction of the FP32 rate.  All steps use the _rn
// intrinsics so that the compiler cannot contract or reassociate them.
#pragma once

#include <cuda_runtime.h>

namespace hdcg {

// hi = RN(v), lo = RN(v - hi) of a double whose hi and lo are both normal
// floats (2^-74 <= |v| < 2^127) or zero, else false; in integer arithmetic: the
// FP64 pipe does two lanes per clock and SM, so the four FP64 conversions and
// subtractions per value bound every field conversion (a 16^4 x 16 field went
// in at 97 us; 50 us with this, the field's traffic at the copy rate is 30 us).
__device__ __forceinline__ bool split_double(double v, float& hi, float& lo) {
  const unsigned h = (unsigned)__double2hiint(v), l = (unsigned)__double2loint(v);
  const unsigned e = (h >> 20) & 0x7ffu;
  if (e - 949u > 200u) {
    hi = __uint_as_float(h);
    lo = 0.f;
    return ((h << 1) | l) == 0u;
  }
  const unsigned top = ((h & 0xfffffu) << 3) | (l >> 29);    // 23 fraction bits
  const unsigned rem = l & 0x1fffffffu;                      // the 29 below them
  const unsigned up = (rem > 0x10000000u || (rem == 0x10000000u && (top & 1u))) ? 1u : 0u;
  hi = __uint_as_float((h & 0x80000000u) | (((e - 896u) << 23 | top) + up));
  int r = (int)rem - (int)(up << 29);                        // (v - hi) 2^(1075 - e), exact
  if (h & 0x80000000u) r = -r;
  lo = __fmul_rn(__int2float_rn(r), __uint_as_float((e - 948u) << 23));   // a power of two
  return true;
}
// the double of a normal float or zero, else false
__device__ __forceinline__ bool widen_float(float f, double& d) {
  const unsigned u = __float_as_uint(f), e = (u >> 23) & 0xffu;
  if (e - 1u > 253u) {
    d = __hiloint2double((int)u, 0);
    return (u << 1) == 0u;
  }
  d = __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
  return true;
}

// a float as a double without the FP64 pipe's conversion
__device__ __forceinline__ double widen(float x) {
  double d;
  return widen_float(x, d) ? d : (double)x;
}
__device__ __forceinline__ double widen(double x) { return x; }

struct dfl {
  float hi, lo;
  dfl() = default;
  __device__ __forceinline__ dfl(float h, float l) : hi(h), lo(l) {}
  __device__ __forceinline__ dfl(int v) : hi((float)v), lo(0.f) {}
  __device__ __forceinline__ dfl(float v) : hi(v), lo(0.f) {}
  __device__ __forceinline__ dfl(double v) {
    if (!split_double(v, hi, lo)) {
      hi = __double2float_rn(v);
      lo = __double2float_rn(v - (double)hi);
    }
  }
  __device__ __forceinline__ explicit operator double() const {
    double h, l;
    if (widen_float(hi, h) && widen_float(lo, l)) return h + l;
    return (double)hi + (double)lo;
  }
};

// s + e = a + b exactly (TwoSum)
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// s + e = a + b for |a| >= |b| (FastTwoSum)
__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  e = __fsub_rn(b, __fsub_rn(s, a));
}

__device__ __forceinline__ dfl operator+(dfl a, dfl b) {
  float s, e;
  two_sum(a.hi, b.hi, s, e);
  e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
  float h, l;
  fast_two_sum(s, e, h, l);
  return dfl(h, l);
}
__device__ __forceinline__ dfl operator-(dfl a) { return dfl(-a.hi, -a.lo); }
__device__ __forceinline__ dfl operator-(dfl a, dfl b) { return a + (-b); }
__device__ __forceinline__ dfl operator*(dfl a, dfl b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);          // exact error of the product
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  float h, l;
  fast_two_sum(p, e, h, l);
  return dfl(h, l);
}
__device__ __forceinline__ dfl& operator+=(dfl& a, dfl b) { return a = a + b; }
__device__ __forceinline__ dfl& operator-=(dfl& a, dfl b) { return a = a - b; }
__device__ __forceinline__ dfl& operator*=(dfl& a, dfl b) { return a = a * b; }

// Sums of products in double-float.  A product joins a running pair (s, e) as
// in the compensated dot product of Ogita, Rump & Oishi (SIAM J. Sci. Comput.
// 26, 2005): TwoProd and TwoSum carry the leading parts exactly, the error
// terms and the hi x lo products go to e.  12 operations against 18 for a
// double-float product and a double-float sum.  Two products, then a
// renormalisation: e left to grow over more terms loses accuracy (on random
// operands six products and the sum over eight hops: 3.3e-15 with double-float
// products and sums, 4.2e-15 and more with one long compensated chain, 3.3e-15
// with dot2 and sum3 below and the hops summed in pairs).
__device__ __forceinline__ void dot_first(float& s, float& e, dfl a, dfl b) {
  s = __fmul_rn(a.hi, b.hi);
  e = __fmaf_rn(a.hi, b.hi, -s);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
}
__device__ __forceinline__ void dot_next(float& s, float& e, dfl a, dfl b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float d = __fmaf_rn(a.hi, b.hi, -p);
  d = __fmaf_rn(a.hi, b.lo, d);
  d = __fmaf_rn(a.lo, b.hi, d);
  float q;
  two_sum(s, p, s, q);
  e = __fadd_rn(__fadd_rn(d, e), q);
}
__device__ __forceinline__ dfl dot_end(float s, float e) {
  float h, l;
  fast_two_sum(s, e, h, l);
  return dfl(h, l);
}
// a b + c d
__device__ __forceinline__ dfl dot2(dfl a, dfl b, dfl c, dfl d) {
  float s, e;
  dot_first(s, e, a, b);
  dot_next(s, e, c, d);
  return dot_end(s, e);
}
// a + b + c with one renormalisation
__device__ __forceinline__ dfl sum3(dfl a, dfl b, dfl c) {
  float s, e, t, f;
  two_sum(a.hi, b.hi, s, e);
  two_sum(s, c.hi, t, f);
  return dot_end(t, __fadd_rn(__fadd_rn(__fadd_rn(a.lo, b.lo), c.lo), __fadd_rn(e, f)));
}

// a + b without the renormalisation (|lo| up to a few ulp(hi)): for summands of
// a double-float sum
__device__ __forceinline__ dfl lazy_add(dfl a, dfl b) {
  float s, e;
  two_sum(a.hi, b.hi, s, e);
  return dfl(s, __fadd_rn(e, __fadd_rn(a.lo, b.lo)));
}

// a b + c, and a b + c d
__device__ __forceinline__ float madd(float a, float b, float c) { return a * b + c; }
__device__ __forceinline__ double madd(double a, double b, double c) { return a * b + c; }
__device__ __forceinline__ dfl madd(dfl a, dfl b, dfl c) { return c + a * b; }
__device__ __forceinline__ float madd2(float a, float b, float c, float d) { return a * b + c * d; }
__device__ __forceinline__ double madd2(double a, double b, double c, double d) { return a * b + c * d; }
__device__ __forceinline__ dfl madd2(dfl a, dfl b, dfl c, dfl d) { return a * b + c * d; }

// lane shuffles of any compute type
__device__ __forceinline__ float shfl_any(float v, int src, int width) {
  return __shfl_sync(0xffffffffu, v, src, width);
}
__device__ __forceinline__ double shfl_any(double v, int src, int width) {
  return __shfl_sync(0xffffffffu, v, src, width);
}
__device__ __forceinline__ dfl shfl_any(dfl v, int src, int width) {
  return dfl(__shfl_sync(0xffffffffu, v.hi, src, width), __shfl_sync(0xffffffffu, v.lo, src, width));
}

}  // namespace hdcg
