// Double-float arithmetic on packed FP32 pairs (a complex value's real and
// imaginary part in one 64-bit register, add/mul/fma.rn.f32x2): each packed
// instruction does both parts, so a step of the Lanczos product needs half
// the FP32 instructions of the scalar form, with the same roundings.
//
// A complex double-float value is a float4 {re hi, im hi, re lo, im lo}, each
// component hi + lo to about 2^-48 relative.  Complex products are summed as
// two packed accumulators, P += (a re, a re) * (b re, b im) and
// Q += (a im, a im) * (b re, b im); the four real sums in P and Q are combined
// once at the end (df_ab: a b, df_conj_ab: conj(a) b, df_a_conjb: a conj(b)).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace lre {
namespace df {

typedef unsigned long long f2;  // two packed floats

__device__ __forceinline__ f2 pk(float x, float y) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 un(f2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
constexpr f2 kMinusOne2 = 0xBF800000BF800000ull;  // (-1, -1)
__device__ __forceinline__ f2 sub2(f2 a, f2 b) { return fma2(b, kMinusOne2, a); }  // a - b, one rounding
__device__ __forceinline__ f2 neg2(f2 a) { return a ^ 0x8000000080000000ull; }

// s + e += p + e_in: Knuth's TwoSum on the leading parts, the exact error and
// e_in into the low part
__device__ __forceinline__ void acc2(f2 &s, f2 &l, f2 p, f2 e) {
  const f2 t = add2(s, p);
  const f2 bp = sub2(t, s);
  const f2 err = add2(sub2(s, sub2(t, bp)), sub2(p, bp));
  s = t;
  l = add2(l, add2(err, e));
}
// (s, l) += m x with m one FP32 number per part and x = xh + xl: the leading
// product exactly (p and its error)
__device__ __forceinline__ void mac(f2 &s, f2 &l, f2 m, f2 xh, f2 xl) {
  const f2 p = mul2(m, xh);
  const f2 e = fma2(m, xl, fma2(m, xh, neg2(p)));
  acc2(s, l, p, e);
}
// (s, l) += (ah + al)(bh + bl), the cross terms into the low part
__device__ __forceinline__ void mac2(f2 &s, f2 &l, f2 ah, f2 al, f2 bh, f2 bl) {
  const f2 p = mul2(ah, bh);
  const f2 e = fma2(al, bh, fma2(ah, bl, fma2(ah, bh, neg2(p))));
  acc2(s, l, p, e);
}

// A complex sum of products: P over a's real parts, Q over its imaginary parts.
struct Sum {
  f2 ph = 0, pl = 0, qh = 0, ql = 0;
};
__device__ __forceinline__ f2 hi(const float4 &v) { return pk(v.x, v.y); }
__device__ __forceinline__ f2 lo(const float4 &v) { return pk(v.z, v.w); }

// a an exact complex64 value, b a double-float value
__device__ __forceinline__ void mac_c64(Sum &S, float2 a, f2 bh, f2 bl) {
  mac(S.ph, S.pl, pk(a.x, a.x), bh, bl);
  mac(S.qh, S.ql, pk(a.y, a.y), bh, bl);
}
// a and b double-float values
__device__ __forceinline__ void mac_df(Sum &S, const float4 &a, f2 bh, f2 bl) {
  mac2(S.ph, S.pl, pk(a.x, a.x), pk(a.z, a.z), bh, bl);
  mac2(S.qh, S.ql, pk(a.y, a.y), pk(a.w, a.w), bh, bl);
}

// (h, l) normalised to hi + lo
__device__ __forceinline__ float4 norm4(f2 h, f2 l) {
  const f2 t = add2(h, l);
  const f2 bp = sub2(t, h);
  const f2 e = add2(sub2(h, sub2(t, bp)), sub2(l, bp));
  const float2 a = un(t), b = un(e);
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ float4 add(const float4 &a, const float4 &b) {
  f2 h = hi(a), l = lo(a);
  acc2(h, l, hi(b), lo(b));
  return norm4(h, l);
}
__device__ __forceinline__ f2 swap_sign(f2 v, float sx, float sy) {  // (sx v.y, sy v.x), sx, sy = +-1
  const float2 a = un(v);
  return pk(sx * a.y, sy * a.x);
}
// P + (sx Q.y, sy Q.x)
__device__ __forceinline__ float4 combine(const Sum &S, float sx, float sy) {
  f2 h = S.ph, l = S.pl;
  acc2(h, l, swap_sign(S.qh, sx, sy), swap_sign(S.ql, sx, sy));
  return norm4(h, l);
}
__device__ __forceinline__ float4 df_ab(const Sum &S) { return combine(S, -1.f, 1.f); }
// conj(a) b: re = P.x + Q.y, im = P.y - Q.x
__device__ __forceinline__ float4 df_conj_ab(const Sum &S) { return combine(S, 1.f, -1.f); }

__device__ __forceinline__ float4 shfl_xor(const float4 &v, int o) {
  return make_float4(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o),
                     __shfl_xor_sync(0xffffffffu, v.z, o), __shfl_xor_sync(0xffffffffu, v.w, o));
}
__device__ __forceinline__ float4 warp_sum(float4 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = add(v, shfl_xor(v, o));
  return v;
}

// complex128 <-> double-float
__device__ __forceinline__ float4 split(double2 v) {
  const float rh = __double2float_rn(v.x), ih = __double2float_rn(v.y);
  return make_float4(rh, ih, __double2float_rn(v.x - (double)rh), __double2float_rn(v.y - (double)ih));
}
__device__ __forceinline__ double2 join(const float4 &q) {
  return make_double2((double)q.x + (double)q.z, (double)q.y + (double)q.w);
}
// a real number as a pair
__device__ __forceinline__ float2 split1(double v) {
  const float h = __double2float_rn(v);
  return make_float2(h, __double2float_rn(v - (double)h));
}

// ---- real double-float values -------------------------------------------------
struct D1 {
  float h, l;
};
__device__ __forceinline__ D1 fast_norm(float h, float l) {  // |h| >= |l|
  const float t = __fadd_rn(h, l);
  return {t, __fsub_rn(l, __fsub_rn(t, h))};
}
__device__ __forceinline__ D1 operator-(D1 a) { return {-a.h, -a.l}; }
__device__ __forceinline__ D1 operator+(D1 a, D1 b) {
  const float t = __fadd_rn(a.h, b.h), bp = __fsub_rn(t, a.h);
  const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(t, bp)), __fsub_rn(b.h, bp));
  return fast_norm(t, __fadd_rn(e, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ D1 operator-(D1 a, D1 b) { return a + (-b); }
__device__ __forceinline__ D1 operator*(D1 a, D1 b) {
  const float p = __fmul_rn(a.h, b.h);
  return fast_norm(p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p))));
}
__device__ __forceinline__ D1 d1(double v) {
  const float2 s = split1(v);
  return {s.x, s.y};
}
__device__ __forceinline__ double value(D1 a) { return (double)a.h + (double)a.l; }
// 1 / a and 1 / sqrt(a): the FP32 value and one Newton step on its residual
__device__ __forceinline__ D1 reciprocal(D1 a) {
  const float y = 1.0f / a.h;
  const D1 r = D1{1.f, 0.f} - a * D1{y, 0.f};
  return fast_norm(y, y * r.h);
}
__device__ __forceinline__ D1 inv_sqrt(D1 a) {
  const float y = rsqrtf(a.h);
  const D1 q = D1{y, 0.f} * D1{y, 0.f};
  const D1 r = D1{1.f, 0.f} - a * q;
  return fast_norm(y, 0.5f * y * r.h);
}
template <int W>
__device__ __forceinline__ D1 lane_sum(D1 v) {  // over W consecutive lanes
#pragma unroll
  for (int o = W / 2; o > 0; o >>= 1)
    v = v + D1{__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o)};
  return v;
}

}  // namespace df
}  // namespace lre
