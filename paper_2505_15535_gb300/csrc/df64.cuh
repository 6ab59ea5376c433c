// Double-float ("df64") arithmetic: a value is the unevaluated sum hi + lo of two FP32 numbers
// with |lo| <= ulp(hi)/2, giving about 48 significant bits.  Built from the error-free
// transformations of floating-point arithmetic:
//   TwoSum (Knuth): s + e = a + b exactly, any a, b;
//   Fast2Sum (Dekker): s + e = a + b exactly when |a| >= |b|;
//   TwoProd via FMA: p + e = a b exactly (e = fma(a, b, -p)).
// The _rn intrinsics keep the compiler from contracting or reassociating these sequences.
// On GB300 the FP32 pipe issues 64x the FP64 pipe's FMAs, so an FP64-accurate contraction in
// df64 (12 FP32 instructions per term of a sum of products, and 20) can outrun native FP64.
#pragma once
#include <cuda_runtime.h>

namespace nhmf {

// A running sum of products of T, as the contractions form them: set/mul start it, fma adds a
// product, get rounds it to T.
template <typename T>
struct Acc {
  T v;
  __device__ __forceinline__ void set(T a) { v = a; }
  __device__ __forceinline__ void mul(T a, T b) { v = a * b; }
  __device__ __forceinline__ void fma(T a, T b) { v = ::fma(a, b, v); }
  __device__ __forceinline__ void neg() { v = -v; }
  __device__ __forceinline__ T get() const { return v; }
};

struct __align__(8) df64 {
  float hi, lo;
  __device__ __forceinline__ df64() {}
  __device__ __forceinline__ df64(float h, float l) : hi(h), lo(l) {}
  // nearest df64 to an FP64 value: hi = fl32(d), lo = fl32(d - hi)
  __device__ __forceinline__ explicit df64(double d) {
    hi = __double2float_rn(d);
    lo = __double2float_rn(d - (double)hi);
  }
  __device__ __forceinline__ explicit df64(int i) : hi(float(i)), lo(0.f) {}
};

__device__ __forceinline__ double to_double(df64 a) { return (double)a.hi + (double)a.lo; }

__device__ __forceinline__ float two_sum(float a, float b, float& e) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return s;
}

__device__ __forceinline__ float fast_two_sum(float a, float b, float& e) {
  const float s = __fadd_rn(a, b);
  e = __fsub_rn(b, __fsub_rn(s, a));
  return s;
}

__device__ __forceinline__ df64 operator+(df64 a, df64 b) {
  float e1, e2, e3, e4;
  float s = two_sum(a.hi, b.hi, e1);
  const float t = two_sum(a.lo, b.lo, e2);
  e1 = __fadd_rn(e1, t);
  s = fast_two_sum(s, e1, e3);
  e3 = __fadd_rn(e3, e2);
  s = fast_two_sum(s, e3, e4);
  return df64(s, e4);
}

__device__ __forceinline__ df64 operator-(df64 a) { return df64(-a.hi, -a.lo); }
__device__ __forceinline__ df64 operator-(df64 a, df64 b) { return a + (-b); }

__device__ __forceinline__ df64 operator*(df64 a, df64 b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  float l;
  const float s = fast_two_sum(p, e, l);
  return df64(s, l);
}

using ::fma;  // keep the FP64/FP32 overloads visible next to the df64 one
__device__ __forceinline__ df64 fma(df64 a, df64 b, df64 c);
__device__ __forceinline__ df64& operator+=(df64& a, df64 b) {
  a = a + b;
  return a;
}

// A sum of products in double-float arithmetic without a renormalisation per term (after Ogita, Rump
// and Oishi, "Accurate sum and dot product", SIAM J. Sci. Comput. 26, 2005, algorithm Dot2): the
// high parts sum by TwoSum; its errors go to one low sum, the products' low parts to two others in
// turn (they stay small, so their roundings do), and the end adds the three with their own errors.
// 4 operations for the first term, 12 for each further one and 20 at the end (n = 4: 58) where a
// product and an accurate double-float sum took 27 a term (88).  Relative error of random sums of
// 3, 4, 5 and 12 terms in units of 1e-15: 1.86, 1.96, 2.09, 2.59; with 27 operations a term 1.97,
// 2.11, 2.24, 2.93; with a single low sum, as in Dot2 itself, 2.6 to 5.3.
template <>
struct Acc<df64> {
  float s, l, k0, k1;
  int n;  // terms so far (a compile-time value in unrolled code)
  __device__ __forceinline__ static void product(df64 a, df64 b, float& p, float& e) {
    p = __fmul_rn(a.hi, b.hi);
    e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
  }
  __device__ __forceinline__ void set(df64 a) { s = a.hi, k0 = a.lo, k1 = l = 0.f, n = 1; }
  __device__ __forceinline__ void mul(df64 a, df64 b) {
    product(a, b, s, k0);
    k1 = l = 0.f;
    n = 1;
  }
  __device__ __forceinline__ void fma(df64 a, df64 b) {
    float p, e, t;
    product(a, b, p, e);
    s = two_sum(s, p, t);
    l = n == 1 ? t : __fadd_rn(l, t);
    if (n % 2 == 0)
      k0 = __fadd_rn(k0, e);
    else
      k1 = n == 1 ? e : __fadd_rn(k1, e);
    ++n;
  }
  __device__ __forceinline__ void neg() { s = -s, l = -l, k0 = -k0, k1 = -k1; }
  __device__ __forceinline__ df64 get() const {
    float e, v, kv, x;
    if (n == 1) {
      const float h = fast_two_sum(s, k0, e);
      return df64(h, e);
    }
    const float k = two_sum(k0, k1, kv), u = two_sum(k, l, v), h = fast_two_sum(s, u, x);
    const float h2 = fast_two_sum(h, __fadd_rn(x, __fadd_rn(v, kv)), e);
    return df64(h2, e);
  }
};

__device__ __forceinline__ df64 fma(df64 a, df64 b, df64 c) {
  Acc<df64> r;
  r.set(c);
  r.fma(a, b);
  return r.get();
}

}  // namespace nhmf
