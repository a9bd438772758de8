// Sums of FP64 products rounded to FP32, in FP64 or in float pairs with the same
// bits: the mass-matrix step of the BRJ block assembly (dg_precond.cu).
#pragma once

namespace dg {

template <int N, typename T>
__device__ __forceinline__ T fp64_row(const double* m, const T* x, int str) {
  double s = 0.0;
#pragma unroll
  for (int k = 0; k < N; ++k) s += m[k] * (double)x[k * str];
  return (T)s;
}
template <typename T>
__device__ __forceinline__ T fp64_scaled(double sc, T x, double add) {
  return (T)__dadd_rn(__dmul_rn(sc, (double)x), add);
}
// out of line for the values that float pairs cannot decide (PairSum): few are,
// and inlined there the assembly was no faster than without pairs
template <int N, typename T>
__device__ __noinline__ T fp64_row_call(const double* m, const T* x, int str) {
  return fp64_row<N>(m, x, str);
}
__device__ __noinline__ float fp64_scaled_call(double sc, float x, double add) {
  return fp64_scaled(sc, x, add);
}

// FP32 results of FP64 arithmetic without the FP64 pipe.  A sum of products
// m_k x_k (m_k doubles, x_k floats) is formed in float pairs (products split by
// fma, sums by Knuth's TwoSum; error below 2^-42 of the terms' magnitudes) and
// rounded; where it lies too close to a rounding boundary to tell on which side
// the FP64 sum falls, near() says so and the caller takes the FP64 form, so that
// the result is FP64's bit for bit.  The
// mass-matrix step of a P = 3 block is 49,000 FP64 multiply-adds, 25 blocks per
// element, on a pipe that retires two per clock.  Entries that cancel to
// rounding noise cannot be told and keep FP64 (6^3 elements, P = 3: 1.30 ms of
// assembly with FP64 and the former shared-memory layouts, 0.99 with both).
struct PairSum {
  float s = 0.f, c = 0.f, big = 0.f;
  __device__ __forceinline__ void add(float mh, float ml, float x) {
    const float p = __fmul_rn(mh, x);
    const float e = __fmaf_rn(ml, x, __fmaf_rn(mh, x, -p));
    const float t = __fadd_rn(s, p), b = __fsub_rn(t, s);
    const float r = __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(p, b));
    s = t;
    c = __fadd_rn(c, __fadd_rn(r, e));
    big += fabsf(p);
  }
  __device__ __forceinline__ float value() const { return __fadd_rn(s, c); }
  // the pair within 2^-42 of the terms of a boundary between two floats, or
  // out of the range where that is told apart from the value's own exponent
  // (big = 0 is the caller's)
  __device__ __forceinline__ bool near(float v) const {
    const int b = __float_as_int(v), E = b & 0x7f800000;
    const float half = __int_as_float(E - (24 << 23));  // half a unit of v
    const float left = fabsf(__fsub_rn(c, __fsub_rn(v, s)));
    return E < (60 << 23) || E > (250 << 23) || (b & 0x7fffff) == 0 ||
           !(half - left > big * 2.3e-13f);
  }
};

// one row of the mass-matrix step, m[k] = mh[k] + ml[k] to float pairs
template <int N>
__device__ __forceinline__ float pair_row(const float* mh, const float* ml, const double* m,
                                          const float* x, int str) {
  PairSum ps;
#pragma unroll
  for (int k = 0; k < N; ++k) ps.add(mh[k], ml[k], x[k * str]);
  const float v = ps.value();
  bool call = ps.near(v);
  if (ps.big == 0.f) {  // zeros (variables that do not couple), or products below 2^-150
    int any = 0;
#pragma unroll
    for (int k = 0; k < N; ++k) any |= __float_as_int(x[k * str]);
    call = (any & 0x7fffffff) != 0;
  }
  return call ? fp64_row_call<N>(m, x, str) : v;
}
// sc x + one, sc = sh + sl to a float pair
__device__ __forceinline__ float pair_scaled(float sh, float sl, double sc, float x, double one) {
  PairSum ps;
  ps.add(sh, sl, x);
  const float v = ps.value();
  const bool call = ps.big == 0.f ? x != 0.f : ps.near(v);
  return one != 0.0 || call ? fp64_scaled_call(sc, x, one) : v;
}

}  // namespace dg
