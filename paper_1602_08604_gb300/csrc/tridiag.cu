// Symmetric tridiagonal eigenproblem kernels for the eigenvalue-first
// projection (step (iii), Sec. II): after the Hermitian matrix has been
// reduced to a real tridiagonal T (diagonal a, off-diagonal b), every
// eigenvalue comes from bisection on Sturm counts, and eigenvectors are
// computed only for the eigenvalues the projection needs, by inverse
// iteration with re-orthogonalisation inside clusters of close eigenvalues
// (the classical scheme of Wilkinson and Peters; see also Demmel, Applied
// Numerical Linear Algebra, Sec. 5.3).  FP64, but for the first rounds of the Krylov
// checks' bisection.
#include <cuda_runtime.h>

#include <cfloat>

#include "lre_internal.cuh"
#include "tri_minor.cuh"

namespace lre {

namespace {

// Number of eigenvalues of T strictly below x (Sylvester's law of inertia on
// the LDL^T factorisation of T - xI).  A pivot smaller than pivmin in
// magnitude is replaced by -pivmin, which keeps the count consistent.
__device__ __forceinline__ int64_t sturm_count(const double *a, const double *b2, int64_t n, double x,
                                               double pivmin) {
  double q = a[0] - x;
  int64_t neg = 0;
  if (fabs(q) < pivmin) q = -pivmin;
  if (q < 0.0) ++neg;
  for (int64_t k = 1; k < n; ++k) {
    q = (a[k] - x) - b2[k - 1] / q;
    if (fabs(q) < pivmin) q = -pivmin;
    if (q < 0.0) ++neg;
  }
  return neg;
}

}  // namespace

// W[j - j0] = the j-th smallest eigenvalue for j in [j0, j0 + cnt), one
// thread per eigenvalue; [lo, hi) brackets every eigenvalue (Gershgorin),
// tol is the absolute accuracy asked for.
__global__ void tri_bisect_kernel(const double *a, const double *b2, int64_t n, double lo0, double hi0, double tol,
                                  double pivmin, double *W, int64_t j0, int64_t cnt) {
  for (int64_t jj = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; jj < cnt; jj += (int64_t)gridDim.x * blockDim.x) {
    const int64_t j = j0 + jj;
    double lo = lo0, hi = hi0;  // invariant: count(lo) <= j < count(hi)
    for (int it = 0; it < 200; ++it) {
      const double mid = 0.5 * (lo + hi);
      if (hi - lo <= tol || mid <= lo || mid >= hi) break;
      if (sturm_count(a, b2, n, mid, pivmin) <= j)
        lo = mid;
      else
        hi = mid;
    }
    W[jj] = 0.5 * (lo + hi);
  }
}

namespace {

__device__ __forceinline__ double start_entry(int64_t i, int64_t j) {
  // splitmix64 of (i, j) -> uniform in [-1, 1): a fixed, well-spread start vector
  uint64_t z = (uint64_t)i * 0x9E3779B97F4A7C15ull + (uint64_t)j * 0xD1B54A32D192ED03ull + 0x632BE59BD9B4E019ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  return (double)(z >> 11) * (2.0 / 9007199254740992.0) - 1.0;
}

template <int THREADS>
__device__ double block_sum(double v, double *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
#pragma unroll
  for (int k = 0; k < THREADS / 32; ++k) s += red[k];
  return s;
}

}  // namespace

// Inverse iteration for the selected eigenvalues lam[0..m) (ascending), all
// members at once: tri_factor factors T - lam_j I = P L U for every j
// (Gaussian elimination with partial pivoting, one thread per member; U has
// two super-diagonals, its pivots stored as reciprocals so that the solves
// need no division), then TRI_ROUNDS rounds of tri_solve (every column of X
// through its own factors, in parallel) and tri_orthonormalise (one CTA per
// cluster of close eigenvalues: modified Gram-Schmidt in eigenvalue order,
// then unit norm).  X: column-major [n][m]; lu: 5 n doubles per member.
static_assert(TRI_ROUNDS >= 2, "at least two inverse-iteration rounds");

__global__ void tri_factor(const double *a, const double *b, int64_t n, const double *lam, int m, double tnorm,
                           double *lu) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= m) return;
  const double x = lam[j];
  double *ui = lu + (size_t)j * 5 * n;  // 1 / U diagonal
  double *u1 = ui + n;                  // U first super-diagonal
  double *u2 = u1 + n;                  // U second super-diagonal
  double *mul = u2 + n;                 // multipliers (row k+1 -= mul[k] * pivot row k)
  double *swp = mul + n;                // 1.0 where rows k, k+1 were exchanged
  const double small = DBL_EPSILON * tnorm > DBL_MIN ? DBL_EPSILON * tnorm : DBL_MIN;
  // the pending row holds (p, q) at columns k, k+1 (its column k+2 entry is zero)
  double p = a[0] - x, q = n > 1 ? b[0] : 0.0;
  for (int64_t k = 0; k + 1 < n; ++k) {
    const double lo = b[k];                          // row k+1, column k
    const double dk = a[k + 1] - x;                  // row k+1, column k+1
    const double up = (k + 2 < n) ? b[k + 1] : 0.0;  // row k+1, column k+2
    if (fabs(lo) > fabs(p)) {
      const double r = 1.0 / lo;
      ui[k] = r; u1[k] = dk; u2[k] = up; swp[k] = 1.0;
      const double f = p * r;
      mul[k] = f;
      p = q - f * dk;
      q = -f * up;
    } else {
      if (fabs(p) < small) p = small;
      const double r = 1.0 / p;
      ui[k] = r; u1[k] = q; u2[k] = 0.0; swp[k] = 0.0;
      const double f = lo * r;
      mul[k] = f;
      p = dk - f * q;
      q = up;
    }
  }
  if (fabs(p) < small) p = small;
  ui[n - 1] = 1.0 / p; u1[n - 1] = 0.0; u2[n - 1] = 0.0;
}

__global__ void tri_solve(const double *lu, int64_t n, int m, double *X, int first) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= m) return;
  const double *ui = lu + (size_t)j * 5 * n, *u1 = ui + n, *u2 = u1 + n, *mul = u2 + n, *swp = mul + n;
  double *v = X + (size_t)j * n;
  // forward: row exchanges and multipliers; the pending right-hand side stays
  // in a register (the start vector is generated on the fly in round one)
  double pend = first ? start_entry(0, j) : v[0];
  for (int64_t k = 0; k + 1 < n; ++k) {
    const double nxt = first ? start_entry(k + 1, j) : v[k + 1];
    if (swp[k] != 0.0) {
      v[k] = nxt;
      pend = pend - mul[k] * nxt;
    } else {
      v[k] = pend;
      pend = nxt - mul[k] * pend;
    }
  }
  v[n - 1] = pend;
  // back substitution with U
  double x1 = 0.0, x2 = 0.0;
  for (int64_t k = n - 1; k >= 0; --k) {
    const double xk = (v[k] - u1[k] * x1 - u2[k] * x2) * ui[k];
    v[k] = xk;
    x2 = x1;
    x1 = xk;
  }
}

__global__ void __launch_bounds__(TRI_THREADS) tri_orthonormalise(double *X, int64_t n, const int *cl) {
  __shared__ double red[TRI_THREADS / 32];
  const int j0 = cl[blockIdx.x], j1 = cl[blockIdx.x + 1];
  for (int j = j0; j < j1; ++j) {
    double *v = X + (size_t)j * n;
    for (int pass = 0; pass < 2; ++pass) {
      // pass 0: unit norm first (a solve grows the vector by up to 1/eps);
      // pass 1: Gram-Schmidt against the cluster's earlier vectors, unit norm
      if (pass == 1) {
        for (int k = j0; k < j; ++k) {
          const double *w = X + (size_t)k * n;
          double dot = 0.0;
          for (int64_t i = threadIdx.x; i < n; i += blockDim.x) dot += w[i] * v[i];
          dot = block_sum<TRI_THREADS>(dot, red);
          for (int64_t i = threadIdx.x; i < n; i += blockDim.x) v[i] -= dot * w[i];
          __syncthreads();
        }
      }
      double nrm = 0.0;
      for (int64_t i = threadIdx.x; i < n; i += blockDim.x) nrm += v[i] * v[i];
      nrm = block_sum<TRI_THREADS>(nrm, red);
      const double inv = nrm > 0.0 ? 1.0 / sqrt(nrm) : 0.0;
      for (int64_t i = threadIdx.x; i < n; i += blockDim.x) v[i] *= inv;
      __syncthreads();
    }
  }
}

// Cluster boundaries of the ascending selection lam[0..m): a new cluster
// starts where the gap to the previous eigenvalue exceeds gap_tol.  cl[0..k]
// (k clusters, cl[k] = m), *k_out = k.  One thread.
__global__ void tri_clusters(const double *lam, int m, double gap_tol, int *cl, int *k_out) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  int k = 0;
  cl[0] = 0;
  for (int j = 1; j < m; ++j)
    if (lam[j] - lam[j - 1] > gap_tol) cl[++k] = j;
  cl[++k] = m;
  *k_out = k;
}

// ---- the extreme eigenvalues a Krylov check needs ----------------------------

// The cb smallest and ct largest eigenvalues of T (ascending: W[0 .. cb + ct)),
// one CTA of 128 threads each: a round evaluates the count at several points over
// the bracket, both ends included.  Three rounds of 128 points run in FP32 on the
// rounded T and three in double-float, each kind ending with the bracket widened by
// its rounding; the last 12 bits (to 4 eps ||T||) are FP64 rounds, which check the
// bracket's ends and start over from [lo0, hi0] if an earlier round misplaced it.
// The FP64 pipe bounds those (three operations a step and point, 1.75 a cycle and
// SM), so they evaluate 64 points, as many as the chain of dependent operations
// hides.  Dynamic shared memory 40 n bytes.
// n = 12 projection, ten checks: 6.26 -> 2.18 ms (five FP64 rounds of 128 points, the
// entries loaded one by one, before; with 32 FP64 points a third round is needed: 3.3
// against 2.7 ms at the time).
constexpr int TRI_FP64_POINTS = 64;

__global__ void __launch_bounds__(128) tri_ends_kernel(const double *a, const double *b2, int n, double lo0, double hi0,
                                                       double tnorm, double *W, int cb, int ct) {
  extern __shared__ __align__(16) unsigned char tri_smem[];
  double *sa = reinterpret_cast<double *>(tri_smem), *sb = sa + n;
  df::D1 *da = reinterpret_cast<df::D1 *>(sb + n), *db = da + n;
  float *fa = reinterpret_cast<float *>(db + n), *fb = fa + n;
  __shared__ unsigned votes[4];
  // scale by a power of two near 1 / ||T||: exact
  const double sc = Minor<double>::scale(tnorm);
  for (int k = threadIdx.x; k < n; k += 128) {
    const double d = a[k] * sc, q = k + 1 < n ? b2[k] * sc * sc : 0.0, o = q < MIN_COUPLING ? 0.0 : -q;
    sa[k] = d;
    sb[k] = o;
    da[k] = df::d1(d);
    db[k] = df::d1(o);
    fa[k] = (float)d;
    fb[k] = (float)o;
  }
  __syncthreads();
  const int idx = blockIdx.x, j = idx < cb ? idx : n - (cb + ct) + idx;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const double L0 = lo0 * sc, H0 = hi0 * sc, tn = tnorm * sc;
  double lo = L0, hi = H0;  // count(lo) <= j < count(hi)
  // last point whose count is <= j, -1 if none
  auto last_below = [&](bool below) {
    const unsigned v = __ballot_sync(0xffffffffu, below);
    __syncthreads();
    if (lane == 0) votes[warp] = v;
    __syncthreads();
    int k = -1;
    for (int w = 0; w < 4; ++w)
      if (votes[w]) k = 32 * w + 31 - __clz(votes[w]);
    return k;
  };
  auto narrow = [&](int k, double h) {
    const int kk = k < 0 ? 0 : k > 126 ? 126 : k;
    hi = lo + h * (kk + 1);
    lo = lo + h * kk;
  };
  auto widen = [&](double by) {
    lo = fmax(L0, lo - by);
    hi = fmin(H0, hi + by);
  };
  for (int it = 0; it < 3; ++it) {
    const double h = (hi - lo) / 127.0;
    narrow(last_below(minor_count<float>(fa, fb, n, (float)(lo + h * t)) <= j), h);
  }
  widen(0x1p-20 * tn);  // 16 units of FP32 rounding of T
  for (int it = 0; it < 3; ++it) {
    const double h = (hi - lo) / 127.0;
    narrow(last_below(minor_count_df(da, db, n, df::d1(lo + h * t)) <= j), h);
  }
  widen(0x1p-41 * tn);  // the same of double-float, 2^-45
  constexpr int P = TRI_FP64_POINTS;
  const double tol = 4.0 * DBL_EPSILON * tn;
  bool restarted = false;
  for (int it = 0; it < 24 && hi - lo > tol; ++it) {
    const double h = (hi - lo) / (P - 1.0);
    const double x = t == P - 1 ? hi : lo + h * t;
    const int k = last_below(t < P && minor_count<double>(sa, sb, n, x) <= j);
    if ((k < 0 || k > P - 2) && !restarted) {
      restarted = true;
      lo = L0;
      hi = H0;
      continue;
    }
    const int kk = k < 0 ? 0 : k > P - 2 ? P - 2 : k;
    const double nlo = lo + h * kk, nhi = kk == P - 2 ? hi : lo + h * (kk + 1);
    if (!(nhi - nlo < hi - lo)) break;
    lo = nlo;
    hi = nhi;
  }
  if (t == 0) W[idx] = 0.5 * (lo + hi) / sc;
}

// log2 |v|, and LOG_ZERO for 0
constexpr double LOG_ZERO = -1e30;
__device__ __forceinline__ double log2_abs(double v) {
  const int hi = __double2hiint(v), E = (hi >> 20) & 0x7FF;
  if (E == 0) return LOG_ZERO;
  const float f = __uint_as_float(0x3F800000u | (((unsigned)hi & 0xFFFFFu) << 3) | ((unsigned)__double2loint(v) >> 29));
  return (double)(E - 1023) + (double)__log2f(f);
}

// |last component| of the unit eigenvector of T for each of the eigenvalues lam, one
// CTA each.  Column r of (T - lam)^-1 is the eigenvector to rounding where its
// diagonal entry is largest (r is then where the vector is), and its entries are
// products of leading and trailing principal minors F_k, P_k and off-diagonals:
//   u_k / u_r = F_k b_k .. b_(r-1) / F_r  (k < r),   P_(k+1) b_r .. b_(k-1) / P_(r+1)  (k > r),
// with the diagonal proportional to F_r P_(r+1) (the inverse of a Jacobi matrix,
// Gantmacher and Krein; choosing r so: Fernando, SIAM J. Matrix Anal. Appl. 18
// (1997) 1013).  Warp 0 runs the leading, warp 1 the trailing minors, three FP64
// operations a step as in minor_count; warp 2 sums the off-diagonals' logarithms;
// the rest is done in logarithms by all threads.
// Bounded by the FP64 operations a warp issues one after the other (about 105 cycles
// each, dependent or not).  Against the values in extended precision the residuals
// are right to 1e-11 relative; an inverse-iteration solve, whose vector holds its
// neighbours to eps / gap, was to 1e-4.
// n = 12 projection, nine checks: 3.60 -> 0.67 ms (n = 10, four: 1.00 -> 0.19).
__global__ void __launch_bounds__(128) tri_residual(const double *a, const double *b2, int n, const double *lam,
                                                    double tnorm, double *out) {
  extern __shared__ double tri_rs[];
  double *sa = tri_rs, *sb = sa + n, *LB = sb + n;  // diagonal, -b^2, prefix sums of log2 |b|
  double *G[2] = {LB + n, LB + n + (n + 1)};        // F_0 .. F_n; P_n .. P_0
  int *eG[2] = {reinterpret_cast<int *>(G[1] + (n + 1)), reinterpret_cast<int *>(G[1] + (n + 1)) + (n / 8 + 2)};
  __shared__ double best[4];
  __shared__ int at[4];
  __shared__ float part[4];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const double sc = Minor<double>::scale(tnorm), x = lam[blockIdx.x] * sc;
  for (int k = t; k < n; k += 128) {
    sa[k] = a[k] * sc;
    sb[k] = k + 1 < n ? -(b2[k] * sc * sc) : 0.0;
  }
  __syncthreads();
  if (warp < 2) {
    // entry i of G is scaled by 2^-eG[(i - 2) / 8]
    double *g = G[warp];
    int *e = eG[warp];
    const int s = warp ? -1 : 1, a0 = warp ? n - 1 : 0, c0 = warp ? n - 1 : -1;
    double pm = 1.0, p = sa[a0] - x;
    int E = 0;
    if (lane == 0) {
      g[0] = 1.0;
      g[1] = p;
      e[0] = 0;
    }
    auto step = [&](double ak, double bk, int k) {
      const double u = bk * pm;
      pm = p;
      p = fma(ak - x, p, u);
      if (lane == 0) g[k + 1] = p;
    };
    int k = 1;
    for (; k + 8 <= n; k += 8) {
      double ak[8], bk[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        ak[i] = sa[a0 + s * (k + i)];
        bk[i] = sb[c0 + s * (k + i)];
      }
      if (lane == 0) e[(k - 1) >> 3] = E;
#pragma unroll
      for (int i = 0; i < 8; ++i) step(ak[i], bk[i], k + i);
      const double f = Minor<double>::scale(p, pm);
      p *= f;
      pm *= f;
      E += 1023 - (__double2hiint(f) >> 20);
    }
    if (lane == 0 && k < n) e[(k - 1) >> 3] = E;
    for (; k < n; ++k) step(sa[a0 + s * k], sb[c0 + s * k], k);
  } else if (warp == 2) {
    const int c = (n + 31) / 32, k0 = lane * c < n ? lane * c : n, k1 = k0 + c < n ? k0 + c : n;
    double sum = 0.0;
    for (int k = k0; k < k1; ++k) {
      LB[k] = sum;
      if (k + 1 < n) sum += 0.5 * log2_abs(sb[k]);
    }
    double before = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double v = __shfl_up_sync(0xffffffffu, before, o);
      if (lane >= o) before += v;
    }
    before -= sum;
    for (int k = k0; k < k1; ++k) LB[k] += before;
  }
  __syncthreads();
  auto lg = [&](int w, int i) { return log2_abs(G[w][i]) + (double)eG[w][i < 2 ? 0 : (i - 2) >> 3]; };
  // lF(k) = log2 |F_k|, lP(k) = log2 |P_(k+1)|: P_(k+1) is entry n - 1 - k
  double mx = 4.0 * LOG_ZERO;
  int r = 0;
  for (int k = t; k < n; k += 128) {
    const double v = lg(0, k) + lg(1, n - 1 - k);
    if (v > mx) {
      mx = v;
      r = k;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double v = __shfl_xor_sync(0xffffffffu, mx, o);
    const int k = __shfl_xor_sync(0xffffffffu, r, o);
    if (v > mx || (v == mx && k < r)) {
      mx = v;
      r = k;
    }
  }
  if (lane == 0) {
    best[warp] = mx;
    at[warp] = r;
  }
  __syncthreads();
  for (int w = 0; w < 4; ++w)
    if (best[w] > mx || (best[w] == mx && at[w] < r)) {
      mx = best[w];
      r = at[w];
    }
  const double fr = lg(0, r) - LB[r], pr = lg(1, n - 1 - r) + LB[r];
  auto lu = [&](int k) { return k < r ? lg(0, k) - LB[k] - fr : lg(1, n - 1 - k) + LB[k] - pr; };
  float s2 = 0.f;
  for (int k = t; k < n; k += 128) s2 += exp2f((float)(2.0 * lu(k)));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
  if (lane == 0) part[warp] = s2;
  __syncthreads();
  if (t == 0) {
    const float s = part[0] + part[1] + part[2] + part[3], l = exp2f((float)lu(n - 1));
    // out of range, or T in pieces (a zero off-diagonal): not taken for converged
    const bool ok = mx > 0.5 * LOG_ZERO && LB[n - 1] > 0.25 * LOG_ZERO && s >= 0.5f && s < 3.0e38f && l < 3.0e38f;
    out[blockIdx.x] = ok ? (double)(l / sqrtf(s)) : 1.0;
  }
}

// out[k] = |last component| / norm of column k of X (n x m), one warp each.
__global__ void tri_last(const double *X, int n, int m, double *out) {
  const int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (k >= m) return;
  const double *v = X + (size_t)k * n;
  double mx = 0.0;
  for (int i = lane; i < n; i += 32) mx = fmax(mx, fabs(v[i]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  const double inv = mx > 0.0 ? 1.0 / mx : 0.0;
  double s = 0.0;
  for (int i = lane; i < n; i += 32) {
    const double t = v[i] * inv;
    s = fma(t, t, s);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) out[k] = s > 0.0 ? fabs(v[n - 1]) * inv / sqrt(s) : 1.0;
}

namespace {
__global__ void minor_counts(const double *a, const double *nb2, int n, const double *x, int m, int *out) {
  extern __shared__ __align__(16) unsigned char mc_smem[];
  df::D1 *da = reinterpret_cast<df::D1 *>(mc_smem), *db = da + n;
  float *fa = reinterpret_cast<float *>(db + n), *fb = fa + n;
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    da[k] = df::d1(a[k]);
    db[k] = df::d1(nb2[k]);
    fa[k] = (float)a[k];
    fb[k] = (float)nb2[k];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    out[3 * i] = minor_count<double>(a, nb2, n, x[i]);
    out[3 * i + 1] = minor_count_df(da, db, n, df::d1(x[i]));
    out[3 * i + 2] = minor_count<float>(fa, fb, n, (float)x[i]);
  }
}
}  // namespace

}  // namespace lre

// Test hook (not part of include/lre.h): the Sturm counts at m points of T (device
// arrays; nb2 minus the squared couplings, n <= 1024) in FP64, double-float and FP32.
extern "C" lre_status lre_debug_minor_counts(lre_ctx *ctx, const double *a, const double *nb2, int n, const double *x,
                                             int m, int *out) {
  if (!ctx || !a || !nb2 || !x || !out || n < 1 || n > 1024 || m < 1) return LRE_ERR_INVALID_ARG;
  lre::minor_counts<<<1, 128, (size_t)n * 24>>>(a, nb2, n, x, m, out);
  const cudaError_t e = cudaDeviceSynchronize();
  return e == cudaSuccess ? LRE_OK : lre::cuda_fail(ctx, e, "minor counts");
}
