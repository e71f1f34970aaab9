// Two nodes' FP32 values per thread, for the pair kernel (lbm_step_pair.cuh).
//
// The packed instructions of sm_100 and later (add, sub, mul, fma on f32x2) carry out two
// IEEE operations per issued instruction, each half rounded exactly as the scalar
// instruction rounds it.  Nothing here contracts a product and a sum by itself: fma() is
// written where one is meant, so a node's result does not depend on which half of a pair it
// is, nor on the code around it.
#pragma once

#include <cuda_runtime.h>

namespace lbm {

struct F2 {
  float2 v;
  F2() = default;
  __device__ __forceinline__ F2(float a) : v(make_float2(a, a)) {}
  __device__ __forceinline__ explicit F2(float2 a) : v(a) {}
  __device__ __forceinline__ float operator[](int j) const { return j ? v.y : v.x; }
  __device__ __forceinline__ void set(int j, float x) { (j ? v.y : v.x) = x; }
};
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return F2(__fadd2_rn(a.v, b.v)); }
__device__ __forceinline__ F2 operator*(F2 a, F2 b) { return F2(__fmul2_rn(a.v, b.v)); }
__device__ __forceinline__ F2 operator-(F2 a, F2 b) {
  F2 r;
  asm("sub.rn.f32x2 %0, %1, %2;"
      : "=l"(reinterpret_cast<unsigned long long&>(r.v))
      : "l"(reinterpret_cast<const unsigned long long&>(a.v)), "l"(reinterpret_cast<const unsigned long long&>(b.v)));
  return r;
}
__device__ __forceinline__ F2 fma(F2 a, F2 b, F2 c) { return F2(__ffma2_rn(a.v, b.v, c.v)); }

// f applied to both nodes' values
template <class F>
__device__ __forceinline__ F2 each(const F2& a, const F& f) {
  F2 r;
  r.set(0, f(a[0]));
  r.set(1, f(a[1]));
  return r;
}

// s = fl(a + b) and its exact rounding error e = (a + b) - s (Knuth's TwoSum)
__device__ __forceinline__ F2 two_sum2(F2 a, F2 b, F2& e) {
  const F2 s = a + b;
  const F2 bb = s - a;
  e = (a - (s - bb)) + (b - bb);
  return s;
}
// balanced-tree sum of N values (the order of tree_sum in lbm_step.cuh)
template <int N>
__device__ __forceinline__ F2 tree_sum2(const F2* v) {
  if constexpr (N == 1)
    return v[0];
  else
    return tree_sum2<N / 2>(v) + tree_sum2<N - N / 2>(v + N / 2);
}

}  // namespace lbm
