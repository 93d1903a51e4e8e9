// Sturm counts of a real symmetric tridiagonal matrix (tridiag.cu,
// project_small.cu).
#pragma once
#include <cuda_runtime.h>

#include "dfloat.cuh"

namespace lre {

// Sturm count by the three-term recurrence of the leading principal minors
// p_k = (a_k - x) p_{k-1} - b_{k-1}^2 p_{k-2} (Givens; Wilkinson, The Algebraic
// Eigenvalue Problem, Ch. 5): the number of sign changes of p_0, p_1, ... is the
// number of eigenvalues below x.  Three multiply-adds a step, where the pivot
// form above has a division on the critical path.  T is scaled to norm 1 or so
// by the caller, and every eighth step both terms are scaled by a power of two
// (exact); a zero minor counts as a sign change, as the pivot form's -pivmin.
// Where a coupling is zero T falls into two blocks and the recurrence starts over
// (p = 1): carried on after a zero minor, p and p_{k-1} would both stay 0 and
// every further row would count.  Callers set squared couplings below
// MIN_COUPLING to zero (an eigenvalue moves by 2^-60 ||T|| at most): smaller ones
// would take the eight steps between scalings below FP64's range, or FP32's.
constexpr double MIN_COUPLING = 0x1p-120;

template <typename R>
struct Minor;
template <>
struct Minor<double> {
  static __device__ __forceinline__ unsigned sign(double v) { return (unsigned)(__double2hiint(v)) >> 31; }
  static __device__ __forceinline__ bool zero(double v) {  // by the integer units: FP64 compares cost FP64 time
    return ((__double2hiint(v) & 0x7FFFFFFF) | __double2loint(v)) == 0;
  }
  // 2^-exponent of the larger of the two
  static __device__ __forceinline__ double scale(double u, double v) {
    const int a = __double2hiint(u) & 0x7FFFFFFF, b = __double2hiint(v) & 0x7FFFFFFF;
    return scale(__hiloint2double(a > b ? a : b, 0));
  }
  static __device__ __forceinline__ double scale(double m) {  // 2^-exponent(m)
    int e = (__double2hiint(m) >> 20) & 0x7FF;
    e = e < 1 ? 1 : e > 2045 ? 2045 : e;
    return __hiloint2double((2046 - e) << 20, 0);
  }
};
template <>
struct Minor<float> {
  static __device__ __forceinline__ unsigned sign(float v) { return __float_as_uint(v) >> 31; }
  static __device__ __forceinline__ bool zero(float v) { return v == 0.f; }
  static __device__ __forceinline__ float scale(float u, float v) { return scale(fmaxf(fabsf(u), fabsf(v))); }
  static __device__ __forceinline__ float scale(float m) {
    int e = (int)(__float_as_uint(m) >> 23) & 0xFF;
    e = e < 1 ? 1 : e > 253 ? 253 : e;
    return __uint_as_float((unsigned)(254 - e) << 23);
  }
};
// a: diagonal, nb2: minus the squared off-diagonal (nb2[k] couples k and k + 1).
// The entries of a whole stretch between two scalings are loaded before its steps:
// loaded one by one, their latency is on every step's path.
template <typename R>
__device__ __forceinline__ int minor_count(const R *a, const R *nb2, int n, R x) {
  R pm = (R)1, p = a[0] - x;
  unsigned sg = Minor<R>::zero(p) ? 1u : Minor<R>::sign(p);
  int cnt = (int)sg;
  auto step = [&](R ak, R bk) {
    if (Minor<R>::zero(bk)) {
      p = (R)1;
      sg = 0u;
    }
    const R t = bk * pm;
    pm = p;
    p = fma(ak - x, p, t);
    const unsigned ns = Minor<R>::zero(p) ? sg ^ 1u : Minor<R>::sign(p);
    cnt += (int)(ns ^ sg);
    sg = ns;
  };
  int k = 1;
  for (; k + 8 <= n; k += 8) {
    R ak[8], bk[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      ak[i] = a[k + i];
      bk[i] = nb2[k - 1 + i];
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) step(ak[i], bk[i]);
    const R f = Minor<R>::scale(p, pm);
    p *= f;
    pm *= f;
  }
  for (; k < n; ++k) step(a[k], nb2[k - 1]);
  return cnt;
}

// The same in double-float (FP32 pipes), |a|, |nb2|, |x| of order one.
__device__ __forceinline__ int minor_count_df(const df::D1 *a, const df::D1 *nb2, int n, df::D1 x) {
  df::D1 pm{1.f, 0.f}, p = a[0] - x;
  unsigned sg = p.h == 0.f ? 1u : Minor<float>::sign(p.h);
  int cnt = (int)sg;
  auto step = [&](df::D1 ak, df::D1 bk) {
    if (bk.h == 0.f) {
      p = {1.f, 0.f};
      sg = 0u;
    }
    const df::D1 t = bk * pm;
    pm = p;
    p = (ak - x) * p + t;
    const unsigned ns = p.h == 0.f ? sg ^ 1u : Minor<float>::sign(p.h);
    cnt += (int)(ns ^ sg);
    sg = ns;
  };
  int k = 1;
  for (; k + 4 <= n; k += 4) {
    df::D1 ak[4], bk[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      ak[i] = a[k + i];
      bk[i] = nb2[k - 1 + i];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) step(ak[i], bk[i]);
    const float f = Minor<float>::scale(p.h, pm.h);
    p = {p.h * f, p.l * f};
    pm = {pm.h * f, pm.l * f};
  }
  for (; k < n; ++k) step(a[k], nb2[k - 1]);
  return cnt;
}

}  // namespace lre
