// Step (iii) for n <= 5 (d <= 32) in one launch of one CTA.
//
// The library route (cuSOLVER Xsyevd, a walk, cublasZherk, an emit kernel) is a
// chain of launches, most of it inside the eigensolver, around a few hundred
// microseconds whatever the size.  Here the whole matrix stays in shared
// memory:
//   1. Householder reduction of mu to a real tridiagonal T = Q^dag mu Q (Golub
//      and Van Loan, Matrix Computations, Sec. 8.3), the reflectors
//      I - g u u^dag with u = x - b e_1 unnormalised, so that the reciprocal in g
//      is off the critical path (a warp of its own forms it during the product).
//      x is first scaled by a power of two to parts of order one (exact, and the
//      reflector is the same): |g| <= 1 then, whatever the column's size.  Where mu
//      has few distinct eigenvalues the columns are rounding residue of residue
//      (1e-16, 1e-32, ...), and g = 1 / |x|^2 of such an x leaves FP32's range;
//   2. every eigenvalue of T by multisection on Sturm counts, 128 / d points a
//      round (tri_minor.cuh): FP32, then double-float, then FP64 to eps ||T||;
//   3. Smolin's walk, and the spectra where they are asked for;
//   4. inverse iteration on T for the smaller of the kept and dropped sets,
//      Gram-Schmidt within clusters, the reflectors applied to those vectors, all
//      in double-float;
//   5. the kept or dropped form of the rebuild (project.cu).
// Latency bounds it: an FP64 operation's result takes about 110 cycles, and a
// reduction step was 85 of them in a row (10,000 cycles whatever d); it is now
// about 50.  Double-float operations take 40 to 80 cycles and do not queue on the
// narrow FP64 pipe, so everything after the eigenvalues, whose 2^-47 is far inside
// the complex64 result, uses them.  The eigenvalues are FP64 throughout.
// d = 16: 113 us a call with its synchronisation, against 705 us for the library
// route, which synchronises too (98 without it and with eigenvalues to 4 eps; 175
// with every step in FP64); d = 4: 39 against 400, d = 32: 261.
#include <cuda_runtime.h>

#include <cfloat>

#include "dfloat.cuh"
#include "lre_internal.cuh"
#include "tri_minor.cuh"

namespace lre {
namespace {

constexpr int PS_THREADS = 256, PS_ALL = PS_THREADS + 32;  // the last warp: reciprocals of the reduction
constexpr int PS_ROUNDS = 2;  // inverse iterations (from eigenvalues at rounding level)

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ void cfma(double2 &s, double2 a, double2 b) {  // s += a b
  s.x = fma(a.x, b.x, fma(-a.y, b.y, s.x));
  s.y = fma(a.x, b.y, fma(a.y, b.x, s.y));
}
__device__ __forceinline__ double2 conjd(double2 a) { return make_double2(a.x, -a.y); }
template <int W>
__device__ __forceinline__ double lane_sum(double v) {  // over W consecutive lanes
#pragma unroll
  for (int o = W / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// *info = 1 where T is not finite (nothing is written to the outputs then), else 0;
// info NULL: LRE_ERR_EIG_FAILED is latched in status instead.
template <int D>
__global__ void __launch_bounds__(PS_ALL) project_small(const float2 *mu, float2 *out, double *eig_mu,
                                                        double *eig_rho, int *info, int *status) {
  using df::D1;
  constexpr int LD = D + 1;                 // padded row
  constexpr int M = D / 2;                  // most vectors formed
  constexpr int TPR = PS_THREADS / D < 32 ? PS_THREADS / D : 32;  // threads per row of the reduction
  // the matrix; reflector k below its diagonal in column k, from step 4 on in
  // double-float (the same 16 bytes)
  __shared__ __align__(16) double2 A[D * LD];
  __shared__ double2 v[D], w[D], gam[D];
  __shared__ double ta[D], tb[D], nb2[D], W[D];
  __shared__ float fa[D], fb[D];
  __shared__ D1 da[D], db[D], dn[D];        // scaled T: diagonal, off-diagonal, minus its square
  __shared__ __align__(16) unsigned char lu_z[(5 * D * M * sizeof(D1)) > M * LD * sizeof(float4)
                                                  ? 5 * D * M * sizeof(D1)
                                                  : M * LD * sizeof(float4)];
  auto lu = reinterpret_cast<D1(*)[D][M]>(lu_z);     // the factors of T - l_j I ...
  auto Z = reinterpret_cast<float4(*)[LD]>(lu_z);    // ... then the vectors
  __shared__ D1 X[M][D];
  __shared__ D1 g[M];
  __shared__ double s_tn, s_lo, s_hi, s_shift, s_beta;
  __shared__ int s_kept, s_skip, s_bad;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  for (int e = tid; e < D * D; e += PS_ALL) {
    const int r = e / D, c = e % D;
    float2 x = r <= c ? mu[e] : mu[c * D + r];
    if (r > c) x.y = -x.y;
    if (r == c) x.y = 0.f;  // a Hermitian matrix has a real diagonal
    A[r * LD + c] = make_double2((double)x.x, (double)x.y);
  }
  __syncthreads();

  // ---- 1. reduction: H = I - g u u^dag, g = 1 / (b (b - conj(x_0))), H^dag x = b e_1,
  // for the scaled x (x, u, b and s_beta below; tb[k] is b scaled back)
  for (int k = 0; k + 1 < D; ++k) {
    const int m = D - 1 - k;  // length of the reflector: rows k + 1 ..
    if (warp == 0) {
      const int i = k + 1 + lane;
      double2 x = lane < m ? A[i * LD + k] : make_double2(0.0, 0.0);
      const unsigned px = __double2hiint(x.x) & 0x7FFFFFFF, py = __double2hiint(x.y) & 0x7FFFFFFF;
      const double f = Minor<double>::scale(__hiloint2double((int)__reduce_max_sync(0xffffffffu, px > py ? px : py), 0));
      x.x *= f;
      x.y *= f;
      const double sq = x.x * x.x + x.y * x.y;
      const double below = lane_sum<32>(lane > 0 ? sq : 0.0);
      if (lane == 0) {
        const double n2 = below + sq;
        const bool skip = below == 0.0 && x.y == 0.0;
        const double beta = skip ? x.x : -copysign(n2 * rsqrt(n2), x.x);
        s_skip = skip;
        s_beta = beta;
        tb[k] = beta * Minor<double>::scale(f);
        if (skip) gam[k] = make_double2(0.0, 0.0);
        x.x -= beta;
      }
      if (lane < m) {
        v[i] = x;
        A[i * LD + k] = x;
      }
    }
    __syncthreads();
    if (s_skip) {  // no reflection (uniform); s_skip is next written after a barrier
      __syncthreads();
      continue;
    }
    if (warp == PS_THREADS / 32) {
      if (lane == 0) {  // u_0 = x_0 - b, b - conj(x_0) = -conj(u_0): g = -u_0 / (b |u_0|^2)
        const double2 u0 = v[k + 1];
        const double f = -1.0 / (s_beta * (u0.x * u0.x + u0.y * u0.y));
        gam[k] = make_double2(f * u0.x, f * u0.y);
      }
    } else {  // w = B u over the trailing block B
      const int i = tid / TPR, l = tid % TPR;
      double2 s = make_double2(0.0, 0.0);
      if (i < D && i > k)
        for (int j = k + 1 + l; j < D; j += TPR) cfma(s, A[i * LD + j], v[j]);
      s.x = lane_sum<TPR>(s.x);
      s.y = lane_sum<TPR>(s.y);
      if (i < D && i > k && l == 0) w[i] = s;
    }
    __syncthreads();
    // q = g w - 1/2 |g|^2 (u^dag w) u (u^dag w is real)
    if (warp == 0) {
      const int i = k + 1 + lane;
      const double2 t = gam[k];
      const double2 a = lane < m ? w[i] : make_double2(0.0, 0.0), b = lane < m ? v[i] : make_double2(0.0, 0.0);
      const double s = lane_sum<32>(b.x * a.x + b.y * a.y);
      const double c = 0.5 * (t.x * t.x + t.y * t.y) * s;
      const double2 q = cmul(t, a);
      if (lane < m) w[i] = make_double2(q.x - c * b.x, q.y - c * b.y);
    }
    __syncthreads();
    // B -= u q^dag + q u^dag
    for (int e = tid; e < m * m; e += PS_ALL) {
      const int i = k + 1 + e / m, j = k + 1 + e % m;
      double2 s = make_double2(0.0, 0.0), r = s;
      cfma(s, v[i], conjd(w[j]));
      cfma(r, w[i], conjd(v[j]));
      A[i * LD + j].x -= s.x + r.x;
      A[i * LD + j].y -= s.y + r.y;
    }
    __syncthreads();
  }
  // ---- 2. eigenvalues of T (scaled by a power of two near 1 / ||T||)
  if (warp == 0) {
    double lo = 1e308, hi = -1e308;
    bool bad = false;
    if (lane < D) {
      const double d = A[lane * LD + lane].x;
      bad = !isfinite(d) || (lane + 1 < D && !isfinite(tb[lane]));
      const double l = lane > 0 ? fabs(tb[lane - 1]) : 0.0, r = lane + 1 < D ? fabs(tb[lane]) : 0.0;
      ta[lane] = d;
      lo = d - l - r;
      hi = d + l + r;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    const double tn = fmax(fabs(lo), fabs(hi)), pad = 2.0 * DBL_EPSILON * tn + 2.0 * DBL_MIN;
    const double sc = Minor<double>::scale(tn);
    if (lane < D) {
      const double o = lane + 1 < D ? tb[lane] * sc : 0.0;
      nb2[lane] = o * o < MIN_COUPLING ? 0.0 : -(o * o);
      W[lane] = ta[lane] * sc;  // the scaled diagonal until the values are known
      fa[lane] = (float)W[lane];
      fb[lane] = (float)nb2[lane];
      da[lane] = df::d1(W[lane]);
      db[lane] = df::d1(o);
      dn[lane] = df::d1(nb2[lane]);
    }
    bad = __any_sync(0xffffffffu, bad);
    if (lane == 0) {
      s_bad = bad;
      s_tn = tn;
      s_lo = (lo - pad) * sc;
      s_hi = (hi + pad) * sc;
    }
  }
  __syncthreads();
  if (tid == 0) {
    if (info) *info = s_bad;
    else if (s_bad) latch(status, LRE_ERR_EIG_FAILED);
  }
  if (s_bad) return;
  const double sc = Minor<double>::scale(s_tn), tn = s_tn * sc;
  {
    constexpr int P = 128 / D < 32 ? 128 / D : 32;  // points per value and round
    const int j = tid / P, l = tid % P;
    double val = 0.0;
    if constexpr (D == 2) {  // in closed form: the steps' own rounding would be most of the error
      const float2 x = mu[1];
      const double a = mu[0].x, b = mu[3].x, h = 0.5 * (a - b), xr = x.x, xi = x.y;
      const double r = sqrt(fma(h, h, fma(xr, xr, xi * xi)));
      val = 0.5 * (a + b) + (j == 0 ? -r : r);
    } else if (tid < ((D * P + 31) & ~31)) {  // whole warps
      const int jj = j < D ? j : D - 1;
      const unsigned group = P == 32 ? 0xffffffffu : ((1u << P) - 1u) << (lane / P * P);
      double lo = s_lo, hi = s_hi;  // count(lo) <= jj < count(hi)
      // points whose count is <= jj, a prefix
      auto below = [&](bool b) { return __popc(__ballot_sync(0xffffffffu, b) & group); };
      auto narrow = [&](int k, double h) {
        hi = k == P ? hi : lo + h * (k + 1);
        lo = lo + h * k;
      };
      constexpr double inv_p1 = 1.0 / (P + 1);
      int it32 = 0, it48 = 0;
      for (double wd = 1.0; wd > 1e-6; wd *= inv_p1) ++it32;
      for (double wd = 8e-6; wd > 1.2e-13; wd *= inv_p1) ++it48;
      for (int it = 0; it < it32; ++it) {
        const double h = (hi - lo) * inv_p1;
        narrow(below(minor_count<float>(fa, fb, D, (float)(lo + h * (l + 1))) <= jj), h);
      }
      const double w32 = 16.0 * 5.9604644775390625e-08 * tn;  // 16 units of FP32 rounding of T
      lo = fmax(s_lo, lo - w32);
      hi = fmin(s_hi, hi + w32);
      for (int it = 0; it < it48; ++it) {
        const double h = (hi - lo) * inv_p1;
        narrow(below(minor_count_df(da, dn, D, df::d1(lo + h * (l + 1))) <= jj), h);
      }
      const double w48 = 16.0 * 7.105427357601002e-15 * tn;  // 16 units of 2^-47
      lo = fmax(s_lo, lo - w48);
      hi = fmin(s_hi, hi + w48);
      // the ends in FP64 (two counts, P >= 2 points): back to the whole bracket if
      // the rounds before misplaced it
      {
        const bool b = minor_count<double>(W, nb2, D, l == 0 ? lo : hi) <= jj;
        const unsigned vt = __ballot_sync(0xffffffffu, b) & group;
        const unsigned first = 1u << (lane / P * P);
        if (!(vt & first) || (vt & (first << 1))) {
          lo = s_lo;
          hi = s_hi;
        }
      }
      // to one unit of rounding of ||T|| (four of them, as the Krylov checks take, showed
      // beside the error of the reduction: 2.2e-16 ||mu|| in the mean at n = 1, 4.3e-16
      // at 3, against the library eigensolver's 0.7e-16 and 2.5e-16)
      const double tol = DBL_EPSILON * tn;
      for (int it = 0; it < 64; ++it) {
        if (__all_sync(0xffffffffu, !(hi - lo > tol))) break;
        const double h = (hi - lo) * inv_p1;
        narrow(below(minor_count<double>(W, nb2, D, lo + h * (l + 1)) <= jj), h);
      }
      val = 0.5 * (lo + hi) / sc;
    }
    __syncthreads();
    if (j < D && l == 0) W[j] = val;
  }
  // the reflectors in double-float, in place
  for (int e = tid; e < D * D; e += PS_ALL) {
    const int i = e / D, k = e % D;
    if (i > k) reinterpret_cast<float4 *>(A)[i * LD + k] = df::split(A[i * LD + k]);
  }
  __syncthreads();
  // ---- 3. Smolin's walk: drop the smallest l_j while l_j + a / kept < 0
  if (tid == 0) {
    int dropped = 0, kept = D;
    double a = 0.0;
    while (kept > 0 && fma(W[dropped], (double)kept, a) < 0.0) {
      a += W[dropped];
      ++dropped;
      --kept;
    }
    s_kept = kept;
    s_shift = kept > 0 ? a / (double)kept : 0.0;
  }
  __syncthreads();
  const int kept = s_kept;
  const double shift = s_shift;
  if (tid < D) {
    const double l = W[D - 1 - tid];
    if (eig_mu) eig_mu[tid] = l;
    if (eig_rho) eig_rho[tid] = tid < kept ? l + shift : 0.0;
  }
  const bool kept_form = kept <= D - kept;
  const int m = kept_form ? kept : D - kept, off = kept_form ? D - kept : 0;
  // ---- 4. vectors: inverse iteration on the scaled T, one lane per vector
  if (warp == 0) {
    // a remainder p below double-float's rounding of T is noise, and raised to it
    // before the pivot is chosen (T changes by as little): where the blocks T falls
    // into share an eigenvalue (a projector's do), every block's vector then grows
    // alike in a solve.  With a floor of eps ||T||, or none where the coupling becomes
    // the pivot, one vector drowned the others beyond what the second round recovers.
    const float small = (float)(0x1p-47 * tn);
    if (lane < m) {
      const D1 x = df::d1(W[off + lane] * sc);
      D1 p = da[0] - x, q = db[0];
      for (int k = 0; k + 1 < D; ++k) {
        const D1 lo = db[k], dk = da[k + 1] - x, up = k + 2 < D ? db[k + 1] : D1{0.f, 0.f};
        if (fabsf(p.h) < small) p = {small, 0.f};
        const bool swap = fabsf(lo.h) > fabsf(p.h);
        const D1 r = df::reciprocal(swap ? lo : p), f = (swap ? p : lo) * r;
        lu[0][k][lane] = r;
        lu[1][k][lane] = swap ? dk : q;
        lu[2][k][lane] = swap ? up : D1{0.f, 0.f};
        lu[3][k][lane] = f;
        lu[4][k][lane] = {swap ? 1.f : 0.f, 0.f};
        p = swap ? q - f * dk : dk - f * q;
        q = swap ? -(f * up) : up;
      }
      if (fabsf(p.h) < small) p = {small, 0.f};
      lu[0][D - 1][lane] = df::reciprocal(p);
      lu[1][D - 1][lane] = lu[2][D - 1][lane] = {0.f, 0.f};
      for (int k = 0; k < D; ++k) {  // a fixed, spread-out start
        const unsigned h = (unsigned)(k * 32 + lane + 1) * 2654435761u;
        X[lane][k] = {0.5f + (float)(h >> 8) * (1.0f / 16777216.0f), 0.f};
      }
    }
    for (int it = 0; it < PS_ROUNDS; ++it) {
      if (lane < m) {
        D1 pend = X[lane][0];
        for (int k = 0; k + 1 < D; ++k) {
          const D1 nxt = X[lane][k + 1], f = lu[3][k][lane];
          const bool swap = lu[4][k][lane].h != 0.f;
          X[lane][k] = swap ? nxt : pend;
          pend = swap ? pend - f * nxt : nxt - f * pend;
        }
        X[lane][D - 1] = pend;
        D1 x1{0.f, 0.f}, x2 = x1;
        for (int k = D - 1; k >= 0; --k) {
          const D1 xk = (X[lane][k] - lu[1][k][lane] * x1 - lu[2][k][lane] * x2) * lu[0][k][lane];
          X[lane][k] = xk;
          x2 = x1;
          x1 = xk;
        }
      }
      __syncwarp();
      // unit norm (scaled by a power of two first: a solve grows by up to 1 / eps),
      // Gram-Schmidt against the cluster's earlier vectors, unit norm again
      int c0 = 0;
      for (int j = 0; j < m; ++j) {
        if (j > 0 && (W[off + j] - W[off + j - 1]) * sc > 1e-3 * tn) c0 = j;
        D1 x = lane < D ? X[j][lane] : D1{0.f, 0.f};
        float mx = fabsf(x.h);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const float f = Minor<float>::scale(mx);
        x = {x.h * f, x.l * f};
        D1 n2 = df::lane_sum<32>(x * x);
        if (n2.h > 0.f) x = x * df::inv_sqrt(n2);
        if (c0 < j) {
          for (int i = c0; i < j; ++i) {
            const D1 y = lane < D ? X[i][lane] : D1{0.f, 0.f};
            x = x - df::lane_sum<32>(x * y) * y;
          }
          n2 = df::lane_sum<32>(x * x);
          if (n2.h > 0.f) x = x * df::inv_sqrt(n2);
        }
        if (lane < D) X[j][lane] = x;
        __syncwarp();
      }
    }
  }
  __syncthreads();
  // z = H_0 H_1 .. x: the last reflector first, D lanes per vector
  if (warp < PS_THREADS / 32) {
    constexpr int VPW = 32 / D;  // vectors per warp
    const int sub = lane / D, i = lane % D;
    const float4 *U = reinterpret_cast<const float4 *>(A);
    for (int j0 = warp * VPW; j0 < ((m + VPW - 1) / VPW) * VPW; j0 += PS_THREADS / 32 * VPW) {
      const int j = j0 + sub;
      const D1 x = j < m ? X[j][i] : D1{0.f, 0.f};
      float4 z = make_float4(x.h, 0.f, x.l, 0.f);
      for (int k = D - 2; k >= 0; --k) {
        const double2 t = gam[k];
        if (t.x == 0.0 && t.y == 0.0) continue;
        const float4 u = i > k ? U[i * LD + k] : make_float4(0.f, 0.f, 0.f, 0.f);
        df::Sum S;
        df::mac_df(S, u, df::hi(z), df::lo(z));
        float4 s = df::df_conj_ab(S);
#pragma unroll
        for (int o = D / 2; o > 0; o >>= 1) s = df::add(s, df::shfl_xor(s, o));
        df::Sum C, R;
        df::mac_df(C, df::split(t), df::hi(s), df::lo(s));
        const float4 c = df::df_ab(C);
        df::mac_df(R, c, df::hi(u), df::lo(u));
        const float4 r = df::df_ab(R);
        z = df::add(z, make_float4(-r.x, -r.y, -r.z, -r.w));
      }
      if (j < m) Z[j][i] = z;
    }
    if (tid < m) {
      const double x = (kept_form ? sc : -sc) * (W[off + tid] + shift);
      g[tid] = df::d1(x > 0.0 ? x : 0.0);
    }
  }
  __syncthreads();
  // ---- 5. rebuild: the upper triangle and its mirror, of the matrix scaled as T
  // (FP32 pairs: no input's weights leave their range), scaled back at the end by
  // 2^-ex = dn1 dn2
  int ex = (__double2hiint(sc) >> 20) - 1023;
  ex = ex > 150 ? 150 : ex < -150 ? -150 : ex;  // beyond: the zero matrix
  const float up1 = __int_as_float((127 + ex / 2) << 23), up2 = __int_as_float((127 + ex - ex / 2) << 23);
  const float dn1 = __int_as_float((127 - ex / 2) << 23), dn2 = __int_as_float((127 - ex + ex / 2) << 23);
  const float2 shift_s = df::split1(shift * sc);
  for (int e = tid; e < D * D; e += PS_ALL) {
    const int r = e / D, c = e % D;
    if (r > c) continue;
    df::Sum S;
    for (int j = 0; j < m; ++j) {
      const float4 a = Z[j][r], b = Z[j][c];
      df::f2 h = 0, l = 0;
      df::mac2(h, l, df::pk(g[j].h, g[j].h), df::pk(g[j].l, g[j].l), df::hi(a), df::lo(a));
      df::mac_df(S, df::norm4(h, l), df::hi(b), df::lo(b));
    }
    float4 s = df::df_conj_ab(S);  // a conj(b) is its conjugate
    s.y = -s.y;
    s.w = -s.w;
    if (!kept_form) {
      const float2 x = mu[e];  // out may be mu: only this thread reads or writes this place and its mirror
      s = df::add(s, make_float4(x.x * up1 * up2, r == c ? 0.f : x.y * up1 * up2, 0.f, 0.f));
      if (r == c) s = df::add(s, make_float4(shift_s.x, 0.f, shift_s.y, 0.f));
    }
    const float2 o = make_float2(s.x * dn1 * dn2, r == c ? 0.f : s.y * dn1 * dn2);
    out[e] = o;
    if (r < c) out[c * D + r] = make_float2(o.x, -o.y);
  }
}

}  // namespace

lre_status project_small_run(lre_ctx *ctx, const lre_c64 *rho_in, int n, lre_c64 *rho_out, double *eig_mu,
                             double *eig_rho, cudaStream_t s) {
  const float2 *in = reinterpret_cast<const float2 *>(rho_in);
  float2 *out = reinterpret_cast<float2 *>(rho_out);
  // the call waits for its status, as after the library's solver, which the kernel writes
  // to host memory (a copy back took 5 us more); a capture cannot wait, and a replay
  // reports through lre_sync
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(s, &cap);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "projection");
  int *const st = ctx->d_status;
  int *info = nullptr;
  if (cap == cudaStreamCaptureStatusNone) {
    e = cudaHostGetDevicePointer(&info, ctx->h_info, 0);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "projection");
  }
  {
    Launch L(ctx, "project_small", s);
    switch (n) {
      case 1: project_small<2><<<1, PS_ALL, 0, s>>>(in, out, eig_mu, eig_rho, info, st); break;
      case 2: project_small<4><<<1, PS_ALL, 0, s>>>(in, out, eig_mu, eig_rho, info, st); break;
      case 3: project_small<8><<<1, PS_ALL, 0, s>>>(in, out, eig_mu, eig_rho, info, st); break;
      case 4: project_small<16><<<1, PS_ALL, 0, s>>>(in, out, eig_mu, eig_rho, info, st); break;
      case 5: project_small<32><<<1, PS_ALL, 0, s>>>(in, out, eig_mu, eig_rho, info, st); break;
      default: return LRE_ERR_UNSUPPORTED;
    }
  }
  e = cudaGetLastError();
  if (e == cudaSuccess && info) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "projection");
  if (!info || !*static_cast<volatile int *>(ctx->h_info)) return LRE_OK;
  ctx->last_error = "projection: the input's tridiagonal form is not finite";
  return LRE_ERR_EIG_FAILED;
}

}  // namespace lre
