// Step (iii) for n <= 5 (d <= 32) in one launch of one CTA.
//
// The library route (cuSOLVER Xsyevd, a walk, cublasZherk, an emit kernel) is a
// chain of launches, most of it inside the eigensolver, around a few hundred
// microseconds whatever the size.  Here the whole matrix stays in shared
// memory:
//   1. Householder reduction of mu to a real tridiagonal T = Q^dag mu Q (Golub
//      and Van Loan, Matrix Computations, Sec. 8.3; each reflector scaled so
//      that the off-diagonal comes out real);
//   2. every eigenvalue of T by multisection on Sturm counts, 128 / d points a
//      round (tri_minor.cuh), to 4 eps ||T||;
//   3. Smolin's walk, and the spectra where they are asked for;
//   4. inverse iteration on T for the smaller of the kept and dropped sets,
//      Gram-Schmidt within clusters, the reflectors applied to those vectors;
//   5. the kept or dropped form of the rebuild (project.cu).
// All in FP64: one SM does about 1.75 FP64 multiply-adds a cycle and a
// dependent one waits some 64 cycles, which is what bounds it; hence the few
// points a round and the vectors of one set only.
// d = 16: 175 us, against 705 us for the library route (d = 4: 50 against 400).
#include <cuda_runtime.h>

#include <cfloat>

#include "lre_internal.cuh"
#include "tri_minor.cuh"

namespace lre {
namespace {

constexpr int PS_THREADS = 256;
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

template <int D>
__global__ void __launch_bounds__(PS_THREADS) project_small(const float2 *mu, float2 *out, double *eig_mu,
                                                            double *eig_rho) {
  constexpr int LD = D + 1;                 // padded row
  constexpr int M = D / 2;                  // most vectors formed
  constexpr int TPR = PS_THREADS / D < 32 ? PS_THREADS / D : 32;  // threads per row of the reduction
  __shared__ double2 A[D * LD];             // the matrix; reflector k below its diagonal in column k
  __shared__ double2 v[D], w[D], tau[D];
  __shared__ double ta[D], tb[D], nb2[D], W[D];
  __shared__ float fa[D], fb[D];
  __shared__ double X[M][D];
  __shared__ double2 lu_z[(5 * D * M + 1) / 2 > M * LD ? (5 * D * M + 1) / 2 : M * LD];
  auto lu = reinterpret_cast<double(*)[D][M]>(lu_z);  // the factors of T - l_j I ...
  auto Z = reinterpret_cast<double2(*)[LD]>(lu_z);    // ... then the vectors
  __shared__ double g[M];
  __shared__ double s_tn, s_lo, s_hi, s_shift;
  __shared__ int s_kept;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  for (int e = tid; e < D * D; e += PS_THREADS) {
    const int r = e / D, c = e % D;
    float2 x = r <= c ? mu[e] : mu[c * D + r];
    if (r > c) x.y = -x.y;
    if (r == c) x.y = 0.f;  // a Hermitian matrix has a real diagonal
    A[r * LD + c] = make_double2((double)x.x, (double)x.y);
  }
  __syncthreads();

  // ---- 1. reduction
  for (int k = 0; k + 1 < D; ++k) {
    const int m = D - 1 - k;  // length of the reflector: rows k + 1 ..
    if (warp == 0) {
      const int i = k + 1 + lane;
      double2 x = lane < m ? A[i * LD + k] : make_double2(0.0, 0.0);
      const double below = lane_sum<32>(lane > 0 ? x.x * x.x + x.y * x.y : 0.0);
      const double2 x0 = make_double2(__shfl_sync(0xffffffffu, x.x, 0), __shfl_sync(0xffffffffu, x.y, 0));
      double beta = x0.x;
      double2 t = make_double2(0.0, 0.0);
      if (below != 0.0 || x0.y != 0.0) {
        beta = -copysign(sqrt(below + x0.x * x0.x + x0.y * x0.y), x0.x);
        t = make_double2((beta - x0.x) / beta, -x0.y / beta);
        const double2 den = make_double2(x0.x - beta, x0.y);  // v = x / (x0 - beta), v_0 = 1
        const double inv = 1.0 / (den.x * den.x + den.y * den.y);
        const double2 q = make_double2(den.x * inv, -den.y * inv);
        x = lane == 0 ? make_double2(1.0, 0.0) : cmul(x, q);
      } else {
        x = make_double2(lane == 0 ? 1.0 : 0.0, 0.0);
      }
      if (lane < m) {
        v[i] = x;
        A[i * LD + k] = x;
      }
      if (lane == 0) {
        tau[k] = t;
        tb[k] = beta;
      }
    }
    __syncthreads();
    const double2 t = tau[k];
    if (t.x == 0.0 && t.y == 0.0) continue;  // no reflection (uniform)
    // w = tau B v over the trailing block B
    {
      const int i = tid / TPR, l = tid % TPR;
      double2 s = make_double2(0.0, 0.0);
      if (i < D && i > k)
        for (int j = k + 1 + l; j < D; j += TPR) cfma(s, A[i * LD + j], v[j]);
      s.x = lane_sum<TPR>(s.x);
      s.y = lane_sum<TPR>(s.y);
      if (i < D && i > k && l == 0) w[i] = cmul(t, s);
    }
    __syncthreads();
    // w -= 1/2 tau (w^dag v) v
    if (warp == 0) {
      const int i = k + 1 + lane;
      const double2 a = lane < m ? w[i] : make_double2(0.0, 0.0), b = lane < m ? v[i] : make_double2(0.0, 0.0);
      double2 s = cmul(conjd(a), b);
      s.x = lane_sum<32>(s.x);
      s.y = lane_sum<32>(s.y);
      const double2 c = cmul(t, s);
      if (lane < m) {
        const double2 q = cmul(make_double2(0.5 * c.x, 0.5 * c.y), b);
        w[i] = make_double2(a.x - q.x, a.y - q.y);
      }
    }
    __syncthreads();
    // B -= v w^dag + w v^dag
    for (int e = tid; e < m * m; e += PS_THREADS) {
      const int i = k + 1 + e / m, j = k + 1 + e % m;
      double2 s = make_double2(0.0, 0.0);
      cfma(s, v[i], conjd(w[j]));
      cfma(s, w[i], conjd(v[j]));
      A[i * LD + j].x -= s.x;
      A[i * LD + j].y -= s.y;
    }
    __syncthreads();
  }
  // ---- 2. eigenvalues of T (scaled by a power of two near 1 / ||T||)
  if (warp == 0) {
    double lo = 1e308, hi = -1e308;
    if (lane < D) {
      const double d = A[lane * LD + lane].x;
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
      nb2[lane] = -(o * o);
      W[lane] = ta[lane] * sc;  // the scaled diagonal until the values are known
      fa[lane] = (float)W[lane];
      fb[lane] = (float)nb2[lane];
    }
    if (lane == 0) {
      s_tn = tn;
      s_lo = (lo - pad) * sc;
      s_hi = (hi + pad) * sc;
    }
  }
  __syncthreads();
  {
    constexpr int P = 128 / D < 32 ? 128 / D : 32;  // points per value and round
    const double sc = Minor<double>::scale(s_tn), tn = s_tn * sc;
    const int j = tid / P, l = tid % P;
    double val = 0.0;
    if (tid < ((D * P + 31) & ~31)) {  // whole warps
      const int jj = j < D ? j : D - 1;
      const unsigned group = P == 32 ? 0xffffffffu : ((1u << P) - 1u) << (lane / P * P);
      double lo = s_lo, hi = s_hi;  // count(lo) <= jj < count(hi)
      // points whose count is <= jj, a prefix
      auto below = [&](bool b) { return __popc(__ballot_sync(0xffffffffu, b) & group); };
      int it32 = 0;
      for (double wd = 1.0; wd > 1e-6; wd /= P + 1) ++it32;
      for (int it = 0; it < it32; ++it) {
        const double h = (hi - lo) / (P + 1);
        const int k = below(minor_count<float>(fa, fb, D, (float)(lo + h * (l + 1))) <= jj);
        hi = k == P ? hi : lo + h * (k + 1);
        lo = lo + h * k;
      }
      const double w32 = 16.0 * 5.9604644775390625e-08 * tn;  // 16 units of FP32 rounding of T
      lo = fmax(s_lo, lo - w32);
      hi = fmin(s_hi, hi + w32);
      // the ends in FP64 (two counts, P >= 2 points): back to the whole bracket if
      // FP32 misplaced it
      {
        const bool b = minor_count<double>(W, nb2, D, l == 0 ? lo : hi) <= jj;
        const unsigned vt = __ballot_sync(0xffffffffu, b) & group;
        const unsigned first = 1u << (lane / P * P);
        if (!(vt & first) || (vt & (first << 1))) {
          lo = s_lo;
          hi = s_hi;
        }
      }
      const double tol = 4.0 * DBL_EPSILON * tn;
      for (int it = 0; it < 64; ++it) {
        if (__all_sync(0xffffffffu, !(hi - lo > tol))) break;
        const double h = (hi - lo) / (P + 1);
        const int k = below(minor_count<double>(W, nb2, D, lo + h * (l + 1)) <= jj);
        const double nhi = k == P ? hi : lo + h * (k + 1), nlo = lo + h * k;
        hi = nhi;
        lo = nlo;
      }
      val = 0.5 * (lo + hi) / sc;
    }
    __syncthreads();
    if (j < D && l == 0) W[j] = val;
  }
  __syncthreads();
  // ---- 3. Smolin's walk: drop the smallest l_j while l_j + a / kept < 0
  if (tid == 0) {
    int dropped = 0, kept = D;
    double a = 0.0;
    while (kept > 0 && W[dropped] + a / (double)kept < 0.0) {
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
  // ---- 4. vectors: inverse iteration, one lane per vector
  if (warp == 0) {
    const double tn = s_tn, small = DBL_EPSILON * tn > DBL_MIN ? DBL_EPSILON * tn : DBL_MIN;
    if (lane < m) {
      const double x = W[off + lane];
      double p = ta[0] - x, q = D > 1 ? tb[0] : 0.0;
      for (int k = 0; k + 1 < D; ++k) {
        const double lo = tb[k], dk = ta[k + 1] - x, up = k + 2 < D ? tb[k + 1] : 0.0;
        const bool swap = fabs(lo) > fabs(p);
        double piv = swap ? lo : p;
        if (!swap && fabs(piv) < small) piv = small;
        const double r = 1.0 / piv, f = (swap ? p : lo) * r;
        lu[0][k][lane] = r;
        lu[1][k][lane] = swap ? dk : q;
        lu[2][k][lane] = swap ? up : 0.0;
        lu[3][k][lane] = f;
        lu[4][k][lane] = swap ? 1.0 : 0.0;
        p = swap ? q - f * dk : dk - f * q;
        q = swap ? -f * up : up;
      }
      if (fabs(p) < small) p = small;
      lu[0][D - 1][lane] = 1.0 / p;
      lu[1][D - 1][lane] = lu[2][D - 1][lane] = 0.0;
      for (int k = 0; k < D; ++k) {  // a fixed, spread-out start
        const unsigned h = (unsigned)(k * 32 + lane + 1) * 2654435761u;
        X[lane][k] = 0.5 + (double)(h >> 8) * (1.0 / 16777216.0);
      }
    }
    for (int it = 0; it < PS_ROUNDS; ++it) {
      if (lane < m) {
        double pend = X[lane][0];
        for (int k = 0; k + 1 < D; ++k) {
          const double nxt = X[lane][k + 1], f = lu[3][k][lane];
          const bool swap = lu[4][k][lane] != 0.0;
          X[lane][k] = swap ? nxt : pend;
          pend = swap ? pend - f * nxt : nxt - f * pend;
        }
        X[lane][D - 1] = pend;
        double x1 = 0.0, x2 = 0.0;
        for (int k = D - 1; k >= 0; --k) {
          const double xk = (X[lane][k] - lu[1][k][lane] * x1 - lu[2][k][lane] * x2) * lu[0][k][lane];
          X[lane][k] = xk;
          x2 = x1;
          x1 = xk;
        }
      }
      __syncwarp();
      // unit norm (scaled first: a solve grows by up to 1 / eps), Gram-Schmidt
      // against the cluster's earlier vectors, unit norm again
      int c0 = 0;
      for (int j = 0; j < m; ++j) {
        if (j > 0 && W[off + j] - W[off + j - 1] > 1e-3 * tn) c0 = j;
        double x = lane < D ? X[j][lane] : 0.0;
        double mx = fabs(x);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        x *= mx > 0.0 ? 1.0 / mx : 0.0;
        double n2 = lane_sum<32>(x * x);
        x *= n2 > 0.0 ? rsqrt(n2) : 0.0;
        if (c0 < j) {
          for (int i = c0; i < j; ++i) {
            const double y = lane < D ? X[i][lane] : 0.0;
            x -= lane_sum<32>(x * y) * y;
          }
          n2 = lane_sum<32>(x * x);
          x *= n2 > 0.0 ? rsqrt(n2) : 0.0;
        }
        if (lane < D) X[j][lane] = x;
        __syncwarp();
      }
    }
  }
  __syncthreads();
  // z = H_0 H_1 .. x: the last reflector first, D lanes per vector
  {
    constexpr int VPW = 32 / D;  // vectors per warp
    const int sub = lane / D, i = lane % D;
    for (int j0 = warp * VPW; j0 < ((m + VPW - 1) / VPW) * VPW; j0 += PS_THREADS / 32 * VPW) {
      const int j = j0 + sub;
      double2 z = make_double2(j < m ? X[j][i] : 0.0, 0.0);
      for (int k = D - 2; k >= 0; --k) {
        const double2 t = tau[k];
        if (t.x == 0.0 && t.y == 0.0) continue;
        const double2 vi = i > k ? A[i * LD + k] : make_double2(0.0, 0.0);
        double2 s = cmul(conjd(vi), z);
        s.x = lane_sum<D>(s.x);
        s.y = lane_sum<D>(s.y);
        const double2 c = cmul(t, s);
        z.x -= c.x * vi.x - c.y * vi.y;
        z.y -= c.x * vi.y + c.y * vi.x;
      }
      if (j < m) Z[j][i] = z;
    }
    if (tid < m) {
      const double x = (kept_form ? 1.0 : -1.0) * (W[off + tid] + shift);
      g[tid] = x > 0.0 ? x : 0.0;
    }
  }
  __syncthreads();
  // ---- 5. rebuild: the upper triangle and its mirror
  for (int e = tid; e < D * D; e += PS_THREADS) {
    const int r = e / D, c = e % D;
    if (r > c) continue;
    double2 s = make_double2(0.0, 0.0);
    if (!kept_form) {
      const float2 x = mu[e];  // out may be mu: only this thread reads or writes this place and its mirror
      s = make_double2((double)x.x, r == c ? 0.0 : (double)x.y);
      if (r == c) s.x += shift;
    }
    for (int j = 0; j < m; ++j) {
      const double2 a = Z[j][r];
      cfma(s, make_double2(g[j] * a.x, g[j] * a.y), conjd(Z[j][c]));
    }
    const float2 o = make_float2((float)s.x, r == c ? 0.f : (float)s.y);
    out[e] = o;
    if (r < c) out[c * D + r] = make_float2(o.x, -o.y);
  }
}

}  // namespace

lre_status project_small_run(lre_ctx *ctx, const lre_c64 *rho_in, int n, lre_c64 *rho_out, double *eig_mu,
                             double *eig_rho, cudaStream_t s) {
  const float2 *in = reinterpret_cast<const float2 *>(rho_in);
  float2 *out = reinterpret_cast<float2 *>(rho_out);
  {
    Launch L(ctx, "project_small", s);
    switch (n) {
      case 1: project_small<2><<<1, PS_THREADS, 0, s>>>(in, out, eig_mu, eig_rho); break;
      case 2: project_small<4><<<1, PS_THREADS, 0, s>>>(in, out, eig_mu, eig_rho); break;
      case 3: project_small<8><<<1, PS_THREADS, 0, s>>>(in, out, eig_mu, eig_rho); break;
      case 4: project_small<16><<<1, PS_THREADS, 0, s>>>(in, out, eig_mu, eig_rho); break;
      case 5: project_small<32><<<1, PS_THREADS, 0, s>>>(in, out, eig_mu, eig_rho); break;
      default: return LRE_ERR_UNSUPPORTED;
    }
  }
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? LRE_OK : cuda_fail(ctx, e, "projection");
}

}  // namespace lre
