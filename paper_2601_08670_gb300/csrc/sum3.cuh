// sum3.cuh -- sums of fp32 terms held as three fp32 numbers, by error-free
// additions (Knuth's two-sum; Dekker's for ordered operands), at fp32 rate.
//
// Between two calls of sum3_settle a sum of n terms loses the rounding of n
// additions to e, which is below n^2 2^-48 of it: n^3 2^-72, against the n 2^-53
// that an fp64 accumulator may lose, so it is no less exact up to SUM3_RUN terms
// (and as many merges).  An infinite or NaN sum is s alone.
#pragma once
#include <math.h>

namespace pced {

constexpr int SUM3_RUN = 512;  // terms between two calls of sum3_settle, at most

struct Sum3 {
  float s, c, e;
};

// the additions are kept apart from contraction and reassociation
__host__ __device__ __forceinline__ float add_rn(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  volatile float y = a + b;
  return y;
#endif
}
// a + b exactly as the result + err
__host__ __device__ __forceinline__ float two_sum(float a, float b, float& err) {
  const float y = add_rn(a, b), z = add_rn(y, -a);
  err = add_rn(add_rn(a, -add_rn(y, -z)), add_rn(b, -z));
  return y;
}
// ... for |a| >= |b|
__host__ __device__ __forceinline__ float fast_two_sum(float a, float b, float& err) {
  const float y = add_rn(a, b);
  err = add_rn(b, -add_rn(y, -a));
  return y;
}

__host__ __device__ __forceinline__ void sum3_add(Sum3& p, float t) {
  float e1, e2;
  p.s = two_sum(p.s, t, e1);
  p.c = two_sum(p.c, e1, e2);
  p.e = add_rn(p.e, e2);
}
// the parts apart again, |c| at most half an ulp of s and |e| half an ulp of c
__host__ __device__ __forceinline__ void sum3_settle(Sum3& p) {
  float c, e;
  c = two_sum(p.c, p.e, e);
  if (c != c) c = e = 0.f;  // s is infinite or NaN and stays so
  p.s = two_sum(p.s, c, c);
  p.c = fast_two_sum(c, e, p.e);
}
__host__ __device__ __forceinline__ Sum3 sum3_merge(const Sum3& p, const Sum3& q) {
  Sum3 r;
  float e1, e2, e3;
  const float c = two_sum(p.c, q.c, e2);
  r.s = two_sum(p.s, q.s, e1);
  r.c = two_sum(c, e1, e3);
  r.e = add_rn(add_rn(p.e, q.e), add_rn(e2, e3));
  return r;
}
__host__ __device__ __forceinline__ double sum3_value(const Sum3& p) {
  const double lo = (double)p.c + (double)p.e;
  return lo == lo ? (double)p.s + lo : (double)p.s;
}

}  // namespace pced
