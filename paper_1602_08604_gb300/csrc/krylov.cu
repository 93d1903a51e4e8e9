// Step (iii) without the O(d^3) reduction: the Smolin et al. projection of
// Sec. II needs only the eigenpairs on one side of its threshold, so they are
// computed by the Lanczos method with full reorthogonalisation on hand-written
// kernels (matrix-vector product, Gram-Schmidt projections, norms, Ritz vectors),
// and the small tridiagonal problem is solved by the bisection and
// inverse-iteration kernels of tridiag.cu.  Arithmetic: the basis as FP32 pairs,
// the product with mu, the reorthogonalisation, the Ritz vectors and the rebuild in
// double-float (about 2^-47); up to d = 4096 the step's scalars and work vector too
// (the Lanczos matrix itself in FP64), beyond in FP64.  rho is complex64: its error
// against complex128 is that rounding alone, to four digits, at every n from 1 to 12
// (1.6e-8 to 2.6e-8 in the mean over GHZ, product and low-rank estimates).
//
// Threshold.  With the eigenvalues l_1 >= ... >= l_d of mu (trace 1), the
// projection keeps l_1..l_r, shifted by s = (1 - sum_{i<=r} l_i) / r, where r
// is the largest k with l_k - (sum_{i<=k} l_i - 1)/k > 0 -- the condition
// holds exactly for k <= r, so the top eigenvalues decide r as soon as the
// first failing one is known.  From the other end, Smolin's own walk over the
// smallest eigenvalues (drop l_j while l_j + a/i < 0) decides r once the
// eigenvalue that stops it is known.  Lanczos converges at both ends of the
// spectrum at once; the first end that decides r gives the vectors to form
// (the kept set, or the dropped set for the rebuild mu + sI - sum (l_j + s)
// v v^dag), and the other end is not needed.
//
// Certification.  Ritz values are accepted when their residual
// beta_J |s_J| is below 1e-11 ||mu|| (up to d = 1024 also small against the
// distance to the next value).  Krylov spaces see each multiple
// eigenvalue once, so a value whose copy was missed could move r; a second,
// short Lanczos run from a new start vector, with the accepted vectors in its
// basis (so it works on the deflated operator), must find nothing beyond the
// threshold, else the call falls back to the tridiagonal reduction.  The
// fallback also runs when r is not decided within KRYLOV_MAX steps.
//
// Up to d = 1024 the run may go on to d steps, where T holds the whole spectrum
// and nothing is left to certify.  Up to d = 4096 the selected values are replaced
// by their Rayleigh quotients (krylov_vecs.cu), so they are as exact as a reduction's.
//
// Layout: the products read mu as complex64 (up to d = 4096 a Hermitian copy of
// the input's upper triangle); the Krylov basis Q holds one d-vector per row
// (vector t at Q + t d) in double-float.  y = mu x is the row-major product, so
// the vectors are eigenvectors of mu.  Up to d = 4096 a run of steps is one
// persistent launch (krylov_steps.cu); beyond, one launch per operation.
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <vector>

#include "dfloat.cuh"
#include "krylov.cuh"
#include "lre_internal.cuh"

namespace lre {
namespace {

constexpr int MV_CHUNK = 1024;     // x entries staged in shared memory at a time
constexpr int RED_THREADS = 256;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__global__ void kry_split(const double2 *__restrict__ x, float4 *__restrict__ xs, int64_t d) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < d; i += (int64_t)gridDim.x * blockDim.x)
    xs[i] = df::split(x[i]);
}

// ---- the Lanczos product y = mu x in double-float arithmetic on the FP32 pipes --
// mu arrives as complex64, so its entries are exact FP32 numbers; with x held
// as two FP32 parts (x = xh + xl, |x - xh - xl| about 2^-48 |x|), each real
// product m x is p = RN(m xh) plus its exact error e = fma(m, xh, -p) plus
// m xl, and the row sums are kept as unevaluated FP32 pairs (sh, sl) with
// Knuth's TwoSum on the leading part: about 2^-44 relative per term, against
// 2^-53 in FP64 -- far inside the Lanczos tolerances -- at the FP32 rate,
// where GB300's FP64 rate had made the product FP64-bound, and reading 8
// bytes per entry of mu instead of 16.  Scalar instructions: the packed ones of
// dfloat.cuh have no higher rate and cost this kernel, which holds 32 entries a lane,
// 6 % (n = 13, 832 products: 117 against 110 ms).

// (sh, sl) += m (xh + xl)
__device__ __forceinline__ void mac1(float &sh, float &sl, float m, float xh, float xl) {
  const float p = __fmul_rn(m, xh), e = __fmaf_rn(m, xh, -p);
  const float t = __fadd_rn(sh, p), bp = __fsub_rn(t, sh);
  const float err = __fadd_rn(__fsub_rn(sh, __fsub_rn(t, bp)), __fsub_rn(p, bp));
  sh = t;
  sl = __fadd_rn(sl, __fadd_rn(err, __fmaf_rn(m, xl, e)));
}

// (sh, sl) += (ah + al)(bh + bl)
__device__ __forceinline__ void mac2(float &sh, float &sl, float ah, float al, float bh, float bl) {
  const float p = __fmul_rn(ah, bh), e = __fmaf_rn(al, bh, __fmaf_rn(ah, bl, __fmaf_rn(ah, bh, -p)));
  const float t = __fadd_rn(sh, p), bp = __fsub_rn(t, sh);
  const float err = __fadd_rn(__fsub_rn(sh, __fsub_rn(t, bp)), __fsub_rn(p, bp));
  sh = t;
  sl = __fadd_rn(sl, __fadd_rn(err, e));
}

// M row-major d x d (d a multiple of MV_CHUNK), x a basis row; y also in split
// form for the reorthogonalisation.  One row per warp, x staged in shared
// memory; each lane loads its 32 entries of a chunk before their products (more
// loads in flight: 4.9 against 3.5 TB/s at d = 16384 loading one at a time), after
// the chunk of x is staged (loaded across its barriers: 110 against 97 ms).
__global__ void __launch_bounds__(256, 3) kry_matvec_df(const float2 *__restrict__ M, const float4 *__restrict__ xsplit,
                                                     double2 *__restrict__ y, float4 *__restrict__ ysplit,
                                                     int64_t d) {
  __shared__ float4 xs[MV_CHUNK];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t r = (int64_t)blockIdx.x * 8 + warp;  // d is a multiple of 8
  float rh = 0.f, rl = 0.f, ih = 0.f, il = 0.f;
  for (int64_t c0 = 0; c0 < d; c0 += MV_CHUNK) {
    const float2 *row = M + r * d + c0;
    __syncthreads();
    for (int k = threadIdx.x; k < MV_CHUNK; k += 256) xs[k] = xsplit[c0 + k];
    __syncthreads();
    float2 u[32];
#pragma unroll
    for (int q = 0; q < 32; ++q) u[q] = row[lane + 32 * q];
#pragma unroll
    for (int q = 0; q < 32; ++q) {
      const float4 x = xs[lane + 32 * q];  // {re hi, im hi, re lo, im lo}
      mac1(rh, rl, u[q].x, x.x, x.z);
      mac1(rh, rl, -u[q].y, x.y, x.w);
      mac1(ih, il, u[q].x, x.y, x.w);
      mac1(ih, il, u[q].y, x.x, x.z);
    }
  }
  const double re = warp_sum((double)rh + (double)rl), im = warp_sum((double)ih + (double)il);
  if (lane == 0) {
    y[r] = make_double2(re, im);
    ysplit[r] = df::split(make_double2(re, im));
  }
}

// h[t] = q_t^dag w for t < m (one CTA per vector), the basis rows and w in
// split form, products and sums in double-float, the partial sums added in
// FP64.
__global__ void __launch_bounds__(RED_THREADS) kry_dots(const float4 *__restrict__ Q, int m,
                                                        const float4 *__restrict__ w, double2 *__restrict__ h,
                                                        int64_t d) {
  __shared__ double sr[RED_THREADS / 32], si[RED_THREADS / 32];
  for (int t = blockIdx.x; t < m; t += gridDim.x) {
    const float4 *q = Q + (int64_t)t * d;
    float rh = 0.f, rl = 0.f, ih = 0.f, il = 0.f;
    for (int64_t i = threadIdx.x; i < d; i += blockDim.x) {
      const float4 a = q[i], b = w[i];  // conj(a) b
      mac2(rh, rl, a.x, a.z, b.x, b.z);
      mac2(rh, rl, a.y, a.w, b.y, b.w);
      mac2(ih, il, a.x, a.z, b.y, b.w);
      mac2(ih, il, -a.y, -a.w, b.x, b.z);
    }
    const double re = warp_sum((double)rh + (double)rl), im = warp_sum((double)ih + (double)il);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
      sr[warp] = re;
      si[warp] = im;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double a = 0, b = 0;
      for (int k = 0; k < RED_THREADS / 32; ++k) {
        a += sr[k];
        b += si[k];
      }
      h[t] = make_double2(a, b);
    }
    __syncthreads();
  }
}

// w -= sum_{t < m} h[t] q_t (basis rows in split form, h split into shared
// memory; dynamic shared memory m float4), and ws = the split w.  A CTA
// takes 64 entries of w; its four warp pairs sum over t = slice, slice + 4,
// ... in double-float, and the four partial sums meet in FP64.
constexpr int UPD_SLICES = 4;
__global__ void __launch_bounds__(256) kry_update(double2 *__restrict__ w, float4 *__restrict__ ws,
                                                  const float4 *__restrict__ Q, int m,
                                                  const double2 *__restrict__ h, int64_t d) {
  extern __shared__ float4 hs[];
  __shared__ double2 part[UPD_SLICES][64];
  for (int t = threadIdx.x; t < m; t += blockDim.x) hs[t] = df::split(h[t]);
  __syncthreads();
  const int e = threadIdx.x & 63, slice = threadIdx.x >> 6;
  for (int64_t i0 = (int64_t)blockIdx.x * 64; i0 < d; i0 += (int64_t)gridDim.x * 64) {
    const int64_t i = i0 + e;
    float rh = 0.f, rl = 0.f, ih = 0.f, il = 0.f;
    if (i < d) {
      for (int t = slice; t < m; t += UPD_SLICES) {
        const float4 q = Q[(int64_t)t * d + i], c = hs[t];  // q c
        mac2(rh, rl, q.x, q.z, c.x, c.z);
        mac2(rh, rl, -q.y, -q.w, c.y, c.w);
        mac2(ih, il, q.x, q.z, c.y, c.w);
        mac2(ih, il, q.y, q.w, c.x, c.z);
      }
    }
    part[slice][e] = make_double2((double)rh + (double)rl, (double)ih + (double)il);
    __syncthreads();
    if (slice == 0 && i < d) {
      double re = 0, im = 0;
#pragma unroll
      for (int k = 0; k < UPD_SLICES; ++k) {
        re += part[k][e].x;
        im += part[k][e].y;
      }
      double2 v = w[i];
      v.x -= re;
      v.y -= im;
      w[i] = v;
      ws[i] = df::split(v);
    }
    __syncthreads();
  }
}

// Sum of |w_i|^2 in one CTA per slice, added atomically into *acc (zeroed by
// the caller).
__global__ void __launch_bounds__(RED_THREADS) kry_norm2(const double2 *__restrict__ w, int64_t d, double *acc) {
  __shared__ double s[RED_THREADS / 32];
  double v = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < d; i += (int64_t)gridDim.x * blockDim.x) {
    const double2 a = w[i];
    v = fma(a.x, a.x, v);
    v = fma(a.y, a.y, v);
  }
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0;
    for (int k = 0; k < RED_THREADS / 32; ++k) t += s[k];
    atomicAdd(acc, t);
  }
}

// Close Lanczos step j: alpha[j] = Re(h1[c] + h2[c]) (c the column of q_j),
// beta[j] = ||w||, q_{j+1} = w / beta[j] (every thread recomputes the two
// scalars from device memory).  A vanishing beta (an invariant subspace) sets
// *breakdown and leaves q_{j+1} = 0.
__global__ void kry_close(const double2 *h1, const double2 *h2, int c, const double *nrm2, double tiny, double *alpha,
                          double *beta, int j, const double2 *w, float4 *qn, int64_t d, int *breakdown) {
  const double b = sqrt(*nrm2);
  const bool dead = !(b > tiny);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    alpha[j] = h1[c].x + h2[c].x;
    beta[j] = dead ? 0.0 : b;
    if (dead && *breakdown == 0) *breakdown = j + 1;  // the first vanishing step
  }
  if (!qn) return;
  const double inv = dead ? 0.0 : 1.0 / b;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < d; i += (int64_t)gridDim.x * blockDim.x) {
    const double2 v = w[i];
    qn[i] = df::split(make_double2(v.x * inv, v.y * inv));  // the basis in split form
  }
}

// A deterministic start vector (splitmix64 of the index and a seed), not yet
// normalised.
__global__ void kry_start(double2 *q, int64_t d, uint64_t seed) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < d; i += (int64_t)gridDim.x * blockDim.x) {
    uint64_t z = seed + 0x9E3779B97F4A7C15ull * (uint64_t)(i + 1);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    const double a = (double)(z >> 11) * 0x1.0p-53 - 0.5;
    const double b = (double)((z << 11) >> 11) * 0x1.0p-53 - 0.5;
    q[i] = make_double2(a, b);
  }
}

// q (a basis row, split form) = v / ||v||
__global__ void kry_scale(const double2 *v, float4 *q, int64_t d, const double *nrm2) {
  const double inv = 1.0 / sqrt(*nrm2);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < d; i += (int64_t)gridDim.x * blockDim.x) {
    const double2 a = v[i];
    q[i] = df::split(make_double2(a.x * inv, a.y * inv));
  }
}

constexpr int KRY_CHECK = 64;           // Lanczos steps between convergence checks
constexpr int KRY_VERIFY = 64;          // steps of the certification run
constexpr int64_t KRY_MAX_VECS = 1024;  // most eigenvectors formed
constexpr int64_t KRY_MAX_STEPS = 2048;
constexpr int KRY_MAX_CLUSTER = 32;     // longest run of close kept values whose vectors are formed
constexpr double KRY_RTOL = 1e-11;      // accepted residual, relative to ||mu||_2

__global__ void kry_eig_rho(const double *w_asc, int64_t r, double shift, double *out, int64_t d) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < d; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = i < r ? w_asc[r - 1 - i] + shift : 0.0;
}

struct KryBuffers {
  double2 *W, *h1, *h2;  // FP64 work vector and coefficients of the multi-launch form
  float4 *Q;             // the Krylov basis, one row per vector, double-float (about 48 bits)
  float4 *Z;             // selected Ritz vectors, rows
  const float2 *A;       // mu (d <= KRY_STEPS_MAX_D: the Hermitian copy of the input)
  float4 *Ws;            // the work vector in double-float form; persistent steps: a step's product
  float4 *Hs, *Wn;       // persistent steps: the corrections, a step's result before normalising
  void *sync;            // persistent steps: the grid barrier and what the CTAs exchange
  double *alpha, *beta, *b2, *stats, *Wr, *Xr, *lu, *last, *nrm;
  int *cl, *nclust, *breakdown;
  int64_t rows, ct_max;
  bool persistent;  // steps in one launch (krylov_steps.cu)
};

// The J x J Lanczos matrix's CB smallest and CT largest eigenvalues
// (ascending), the magnitudes of their unit eigenvectors' last components,
// beta[J-1] and ||T||.
struct RitzEnds {
  std::vector<double> w, last;
  double beta_next = 0, tnorm = 0;
};

// Convergence check.  The residual of a Ritz pair is beta_J |s_J|, s_J the last
// component of its eigenvector, which the minors at the eigenvalue (computed to
// 4 eps ||T||) give to far below the tolerance (tri_residual); the vectors that are
// used come from two rounds of inverse iteration (ritz_vectors) and are looked at again.
// Values placed less exactly will not do: an unconverged neighbour's last
// component comes through with the value's error over their gap.
lre_status ritz_values(lre_ctx *ctx, const KryBuffers &B, const double *alpha, const double *beta, int J, int CB,
                       int CT, bool want_last, cudaStream_t s, RitzEnds &out) {
  {
    Launch L(ctx, "kry_tri_prepare", s);
    tri_prepare<<<1, 256, 0, s>>>(alpha, beta, J, B.b2, B.stats);
  }
  double hst[3];
  double bnext = 0;
  cudaError_t e = cudaMemcpyAsync(hst, B.stats, sizeof(hst), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&bnext, beta + (J - 1), sizeof(double), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "Lanczos matrix bounds");
  const double tnorm = fmax(fabs(hst[0]), fabs(hst[1]));
  const double pad = 2.0 * DBL_EPSILON * tnorm + 2.0 * DBL_MIN;
  const int m = CB + CT;
  auto ends_smem = [](size_t n) { return 40 * n; };
  auto residual_smem = [](size_t n) { return 41 * n + 48; };
  const size_t smem = ends_smem(J), rsmem = residual_smem(J);
  // the limits are the functions', shared by all threads: always the largest
  e = cudaFuncSetAttribute(tri_ends_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ends_smem(KRY_MAX_STEPS));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(tri_residual, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)residual_smem(KRY_MAX_STEPS));
  if (e != cudaSuccess) return cuda_fail(ctx, e, "Ritz values");
  {
    Launch L(ctx, "kry_bisect", s);
    tri_ends_kernel<<<m, 128, smem, s>>>(alpha, B.b2, J, hst[0] - pad, hst[1] + pad, tnorm, B.Wr, CB, CT);
  }
  if (want_last) {
    Launch L(ctx, "kry_residuals", s);
    tri_residual<<<m, 128, rsmem, s>>>(alpha, B.b2, J, B.Wr, tnorm, B.last);
  }
  out.w.resize(m);
  out.last.assign(m, 0.0);
  e = cudaMemcpyAsync(out.w.data(), B.Wr, m * sizeof(double), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess && want_last)
    e = cudaMemcpyAsync(out.last.data(), B.last, m * sizeof(double), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "Ritz values");
  out.beta_next = bnext;
  out.tnorm = tnorm;
  return LRE_OK;
}

// Unit eigenvectors of the J x J Lanczos matrix for its m eigenvalues w
// (device, ascending) into Xr, and their last components on the host: inverse
// iteration, orthonormalised within clusters of values closer than 1e-6 ||T||
// (beyond that the solves' own error, eps ||T|| / gap, is below 1e-9).
lre_status ritz_vectors(lre_ctx *ctx, const KryBuffers &B, const double *alpha, const double *beta, int J,
                        const double *w, int m, double tnorm, cudaStream_t s, std::vector<double> &last) {
  int hk = 0;
  {
    Launch L(ctx, "kry_clusters", s);
    tri_clusters<<<1, 32, 0, s>>>(w, m, 1e-6 * tnorm, B.cl, B.nclust);
  }
  cudaError_t e = cudaMemcpyAsync(&hk, B.nclust, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "Ritz clusters");
  {
    // two rounds: the eigenvalues are at rounding level, and the last components
    // are looked at below
    constexpr int rounds = 2;
    Launch L(ctx, "kry_inverse_iteration", s, 2 + 2 * rounds);
    tri_factor<<<(m + 31) / 32, 32, 0, s>>>(alpha, beta, J, w, m, tnorm, B.lu);
    for (int it = 0; it < rounds; ++it) {
      tri_solve<<<(m + 31) / 32, 32, 0, s>>>(B.lu, J, m, B.Xr, it == 0);
      tri_orthonormalise<<<hk, TRI_THREADS, 0, s>>>(B.Xr, J, B.cl);
    }
    tri_last<<<(m + 3) / 4, 128, 0, s>>>(B.Xr, J, m, B.last);
  }
  last.resize(m);
  e = cudaMemcpyAsync(last.data(), B.last, m * sizeof(double), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  return e == cudaSuccess ? LRE_OK : cuda_fail(ctx, e, "Ritz vectors");
}

// Lanczos steps [j0, j1) on basis rows base + j (rows 0..base + j - 1 fixed):
// every step reorthogonalises against all earlier rows (classical
// Gram-Schmidt, twice here; krylov_steps.cu takes out the two local terms and
// then makes one full pass) and writes alpha[j], beta[j] and row base + j + 1.
lre_status lanczos_steps(lre_ctx *ctx, const KryBuffers &B, int64_t d, int64_t base, int j0, int j1, double *alpha,
                         double *beta, double tiny, cudaStream_t s) {
  if (B.persistent) {
    const KryStepBuffers K{B.A, B.Q, B.Ws, B.Wn, B.Hs, B.sync, B.breakdown, B.rows};
    return kry_steps_run(ctx, K, d, base, j0, j1, alpha, beta, tiny, s);
  }
  const int red_grid = (int)std::min<int64_t>((d + RED_THREADS - 1) / RED_THREADS, (int64_t)ctx->num_sms * 4);
  const int upd_grid = (int)((d + 63) / 64);
  for (int j = j0; j < j1; ++j) {
    const int64_t c = base + j;  // the row of q_j
    const int cols = (int)(c + 1);
    {
      Launch L(ctx, "kry_matvec", s);  // W = mu q_j and its split copy
      kry_matvec_df<<<(unsigned)(d / 8), 256, 0, s>>>(B.A, B.Q + c * d, B.W, B.Ws, d);
    }
    {
      Launch L(ctx, "kry_reorth", s, 4);
      const int dg = (int)std::min<int64_t>(cols, 2048);
      const size_t hs = (size_t)cols * sizeof(float4);
      kry_dots<<<dg, RED_THREADS, 0, s>>>(B.Q, cols, B.Ws, B.h1, d);
      kry_update<<<upd_grid, 256, hs, s>>>(B.W, B.Ws, B.Q, cols, B.h1, d);
      kry_dots<<<dg, RED_THREADS, 0, s>>>(B.Q, cols, B.Ws, B.h2, d);
      kry_update<<<upd_grid, 256, hs, s>>>(B.W, B.Ws, B.Q, cols, B.h2, d);
    }
    {
      Launch L(ctx, "kry_close", s, 2);
      cudaMemsetAsync(B.nrm, 0, sizeof(double), s);
      kry_norm2<<<red_grid, RED_THREADS, 0, s>>>(B.W, d, B.nrm);
      float4 *next = c + 1 < B.rows ? B.Q + (c + 1) * d : nullptr;
      kry_close<<<red_grid, RED_THREADS, 0, s>>>(B.h1, B.h2, (int)c, B.nrm, tiny, alpha, beta, j, B.W, next, d,
                                                 B.breakdown);
    }
  }
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? LRE_OK : cuda_fail(ctx, e, "Lanczos step");
}

// The step (from 1) whose beta vanished in the runs since the flag was zeroed, 0 if none.
// LRE_ERR_TIMEOUT where a grid barrier gave up: the run's alpha and beta are not all there.
lre_status read_breakdown(lre_ctx *ctx, const KryBuffers &B, int &brk, cudaStream_t s) {
  unsigned gave_up = 0;
  cudaError_t e = cudaMemcpyAsync(&brk, B.breakdown, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess && B.persistent)
    e = cudaMemcpyAsync(&gave_up, static_cast<unsigned *>(B.sync) + 1, sizeof(gave_up), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "Lanczos breakdown flag");
  if (!gave_up) return LRE_OK;
  ctx->last_error = "projection: a grid barrier of the Lanczos steps gave up";
  return LRE_ERR_TIMEOUT;
}

// A fresh unit start vector in row `row`, orthogonal to rows [0, row).  Its norm is
// summed by one CTA, in a fixed order, where the steps are too (krylov_steps.cu): the
// call then repeats bit for bit.
lre_status start_vector(lre_ctx *ctx, const KryBuffers &B, int64_t d, int64_t row, uint64_t seed, cudaStream_t s) {
  const int red_grid = (int)std::min<int64_t>((d + RED_THREADS - 1) / RED_THREADS, (int64_t)ctx->num_sms * 4);
  // built in the FP64 work vector, stored into the basis row in split form
  Launch L(ctx, "kry_start", s, row > 0 ? 8 : 3);
  kry_start<<<red_grid, RED_THREADS, 0, s>>>(B.W, d, seed);
  if (row > 0) {
    const int cols = (int)row;
    const size_t hs = (size_t)cols * sizeof(float4);
    kry_split<<<red_grid, RED_THREADS, 0, s>>>(B.W, B.Ws, d);
    for (int pass = 0; pass < 2; ++pass) {
      kry_dots<<<(int)std::min<int64_t>(cols, 2048), RED_THREADS, 0, s>>>(B.Q, cols, B.Ws, B.h1, d);
      kry_update<<<(unsigned)((d + 63) / 64), 256, hs, s>>>(B.W, B.Ws, B.Q, cols, B.h1, d);
    }
  }
  cudaMemsetAsync(B.nrm, 0, sizeof(double), s);
  kry_norm2<<<B.persistent ? 1 : red_grid, RED_THREADS, 0, s>>>(B.W, d, B.nrm);
  kry_scale<<<red_grid, RED_THREADS, 0, s>>>(B.W, B.Q + row * d, d, B.nrm);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? LRE_OK : cuda_fail(ctx, e, "Lanczos start vector");
}

}  // namespace

lre_status project_krylov(lre_ctx *ctx, const lre_c64 *rho_in, int64_t d, lre_c64 *rho_out, double *eig_rho,
                          cudaStream_t s, bool *fallback) {
  *fallback = true;
  // up to d = 1024 the run may go to d steps, where T holds the whole spectrum;
  // beyond, 2048 steps (and half of d) bound it
  const bool whole = d <= KRY_MAX_VECS;
  const int64_t kmax = whole ? d : std::min<int64_t>(d / 2, KRY_MAX_STEPS);
  const int64_t vecs = std::min<int64_t>(d, KRY_MAX_VECS);
  KryBuffers B{};
  B.rows = whole ? d + 1 : std::max<int64_t>(kmax + 1, KRY_MAX_VECS + KRY_VERIFY + 1);
  B.ct_max = whole ? d + 1 : vecs + 64;  // whole: 88 d^2 bytes in all, less than the reduction path's 96 d^2
  const bool copy = d <= KRY_STEPS_MAX_D;  // the steps read a Hermitian copy of the input's upper triangle
  auto u = [](size_t x) { return (x + 255) & ~(size_t)255; };
  char *p = nullptr;
  auto take = [&](size_t bytes) {
    char *q = p;
    p += u(bytes);
    return q;
  };
  float2 *herm = nullptr;
  double *alpha2 = nullptr, *beta2 = nullptr;
  auto lay_out = [&]() {
    herm = reinterpret_cast<float2 *>(take(copy ? (size_t)d * d * sizeof(float2) : 0));
    B.Q = reinterpret_cast<float4 *>(take((size_t)B.rows * d * sizeof(float4)));
    B.W = reinterpret_cast<double2 *>(take((size_t)d * sizeof(double2)));
    B.h1 = reinterpret_cast<double2 *>(take((size_t)B.rows * sizeof(double2)));
    B.h2 = reinterpret_cast<double2 *>(take((size_t)B.rows * sizeof(double2)));
    B.Z = reinterpret_cast<float4 *>(take((size_t)d * vecs * sizeof(float4)));
    B.alpha = reinterpret_cast<double *>(take((size_t)B.rows * sizeof(double)));
    B.beta = reinterpret_cast<double *>(take((size_t)B.rows * sizeof(double)));
    B.b2 = reinterpret_cast<double *>(take((size_t)B.rows * sizeof(double)));
    B.stats = reinterpret_cast<double *>(take(4 * sizeof(double)));
    B.Wr = reinterpret_cast<double *>(take((size_t)B.ct_max * sizeof(double)));
    B.Xr = reinterpret_cast<double *>(take((size_t)B.rows * B.ct_max * sizeof(double)));
    B.lu = reinterpret_cast<double *>(take((size_t)5 * B.rows * B.ct_max * sizeof(double)));
    B.last = reinterpret_cast<double *>(take((size_t)B.ct_max * sizeof(double)));
    B.nrm = reinterpret_cast<double *>(take(sizeof(double)));
    B.cl = reinterpret_cast<int *>(take((size_t)(B.ct_max + 2) * sizeof(int)));
    B.nclust = reinterpret_cast<int *>(take(sizeof(int)));
    B.breakdown = reinterpret_cast<int *>(take(sizeof(int)));
    alpha2 = reinterpret_cast<double *>(take((size_t)KRY_VERIFY * sizeof(double)));
    beta2 = reinterpret_cast<double *>(take((size_t)KRY_VERIFY * sizeof(double)));
    B.Ws = reinterpret_cast<float4 *>(take((size_t)d * sizeof(float4)));
    B.Wn = reinterpret_cast<float4 *>(take((size_t)d * sizeof(float4)));
    B.Hs = reinterpret_cast<float4 *>(take((size_t)B.rows * sizeof(float4)));
    B.sync = take(kry_sync_bytes(ctx));
  };
  lay_out();
  const size_t need = (size_t)(p - static_cast<char *>(nullptr));
  lre_status st = ensure_workspace(ctx, need);
  if (st != LRE_OK) return st;
  p = static_cast<char *>(ctx->ws);
  lay_out();
  if (!copy) herm = nullptr;
  B.A = copy ? herm : reinterpret_cast<const float2 *>(rho_in);  // the input is unchanged until the rebuild

  // the trace and the shares of the squared norm, in h1 until the first start vector
  double *const tn = reinterpret_cast<double *>(B.h1);
  std::vector<double> fro(1 + kry_norm_blocks(ctx, d));
  if ((st = kry_prepare_mu(ctx, reinterpret_cast<const float2 *>(rho_in), herm, d, tn, s)) != LRE_OK) return st;
  cudaError_t e = cudaMemsetAsync(B.breakdown, 0, sizeof(int), s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(fro.data(), tn, fro.size() * sizeof(double), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "Krylov set-up");
  double norm2 = 0.0;
  for (size_t k = 1; k < fro.size(); ++k) norm2 += fro[k];
  const double tiny = 1e-14 * sqrt(norm2);
  // the persistent steps hold squared norms in FP32 pairs, down to tiny^2: a density
  // matrix has a norm in [1/64, 1] there; anything far from that takes the FP64 work
  // vector of the multi-launch form, or the reduction where d is too small for it
  B.persistent = copy && norm2 >= 0x1p-20 && norm2 <= 0x1p60;
  if (copy && !B.persistent && d < 2048) return LRE_OK;
  const double trace = fro[0];  // Tr mu (1 up to the complex64 rounding of the diagonal)
  if ((st = start_vector(ctx, B, d, 0, 0x5EED0001ull, s)) != LRE_OK) return st;

  int ct_want = 64, cb_want = 32;
  int J = 0, step = KRY_CHECK;
  int seen = 0, seen_J = 0;  // converged leading values at the last check
  bool kept_form = true;
  int64_t r = -1, m = 0;
  double shift = 0.0;
  int sel0 = 0;  // first column (in Wr) of the selected vectors
  RitzEnds E;
  std::vector<double> last;
  while (J < kmax) {
    const int J1 = (int)std::min<int64_t>(kmax, J + step);
    if ((st = lanczos_steps(ctx, B, d, 0, J, J1, B.alpha, B.beta, tiny, s)) != LRE_OK) return st;
    J = J1;
    int brk = 0;
    if ((st = read_breakdown(ctx, B, brk, s)) != LRE_OK) return st;
    const bool broke = brk > 0 || J == d;
    if (brk > 0) J = brk;  // an invariant subspace: T_J holds exact eigenvalues
    const bool exact = J == d;  // the whole spectrum of mu
    // windows of Ritz values at each end, together at most ct_max (the
    // buffers' width) and J; all of them once they are exact and fit
    int CT = (int)std::min<int64_t>(std::min(ct_want, J), B.ct_max - 1);
    int CB = (int)std::min<int64_t>(std::min(cb_want, J - CT), B.ct_max - CT);
    if (broke && J <= B.ct_max) {
      CT = J;
      CB = 0;
    }
    if ((st = ritz_values(ctx, B, B.alpha, B.beta, J, CB, CT, !broke, s, E)) != LRE_OK) return st;
    if (broke) E.beta_next = 0.0;
    const int mm = CB + CT;
    const double anorm = fmax(fabs(E.w[0]), fabs(E.w[mm - 1]));
    // up to d = 1024, where the values are held to FP64 rounding, a residual is also small
    // against the distance to the next value: the quotient is off by its square over that
    // (a bulk spaced by 1e-12 ||mu||, the rounding of an exact state, showed 8e-14 without;
    // spacings above 1e-7 ||mu|| pass anyway)
    auto conv = [&](int k) {
      const double res = fabs(E.beta_next * E.last[k]);
      if (!(res <= KRY_RTOL * anorm)) return false;
      if (!whole) return true;
      const double below = k > 0 ? E.w[k] - E.w[k - 1] : anorm, above = k + 1 < mm ? E.w[k + 1] - E.w[k] : anorm;
      return res * res <= 2e-15 * anorm * fmin(below, above);
    };
    // top end: l_k - (S_k - Tr)/k > 0 exactly for k <= r
    int64_t r_top = -1;
    bool top_open = true;
    int conv_top = 0, guess = -1;  // converged leading values; the threshold as it looks now
    double S = 0.0, S_r = 0.0;
    for (int k = 1; k <= CT; ++k) {
      const int col = mm - k;
      if (top_open && !conv(col)) top_open = false;
      if (top_open) conv_top = k;
      S += E.w[col];
      if (E.w[col] - (S - trace) / k <= 0.0) {
        guess = k;
        if (top_open) r_top = k - 1;
        break;
      }
      if (top_open) S_r = S;
    }
    // bottom end: Smolin's walk over the smallest eigenvalues
    int64_t r_bot = -1;
    bool bot_open = CB > 0 || exact;
    const int nbot = exact ? mm : CB;
    double a = 0.0;
    int64_t kept = d;
    for (int t = 0; t < nbot && bot_open; ++t) {
      if (!conv(t)) {
        bot_open = false;
        break;
      }
      if (E.w[t] + a / (double)kept < 0.0) {
        a += E.w[t];
        --kept;
      } else {
        r_bot = kept;
        break;
      }
    }
    if (r_top >= 0 && r_bot >= 0 && r_top != r_bot) return LRE_OK;  // the two ends disagree: reduction path
    if (r_top >= 0 && r_top <= KRY_MAX_VECS && !(exact && 2 * r_top > d && r_bot >= 0)) {
      kept_form = true;
      r = r_top;
      m = r;
      shift = r > 0 ? (trace - S_r) / (double)r : 0.0;
      sel0 = mm - (int)r;
    } else if (r_bot >= 0 && d - r_bot <= KRY_MAX_VECS && (!eig_rho || exact)) {
      kept_form = false;
      r = r_bot;
      m = d - r;
      shift = r > 0 ? a / (double)r : 0.0;
      sel0 = 0;
    }
    if (r >= 0) {
      if (m == 0) break;
      if ((st = ritz_vectors(ctx, B, B.alpha, B.beta, J, B.Wr + sel0, (int)m, E.tnorm, s, last)) != LRE_OK) return st;
      bool good = true;
      for (int k = 0; k < m; ++k) good = good && fabs(E.beta_next * last[k]) <= 2.0 * KRY_RTOL * anorm;
      if (good) break;
      r = -1;  // a cluster hid a component: go on
    } else if (whole && eig_rho && r_bot >= 0 && !broke) {
      // the dropped form with every kept value wanted: they are all there after d steps
      // (d = 1024, few negative values, every other call with eig_rho: 43.7 ms in the mean
      // with the reduction after the steps so far, 20.9 so)
      step = (int)(kmax - J);
      continue;
    } else {
      if (r_top >= 0 || r_bot >= 0) return LRE_OK;  // decided, but too many vectors: reduction path
      if (broke) return LRE_OK;  // exact but undecided: reduction path
    }
    // widen an end whose values all converged without deciding; when both
    // ends are at their widest and still undecided, both sets are too large
    const bool top_full = top_open && r_top < 0 && CT == ct_want;
    const bool bot_full = bot_open && r_bot < 0 && CB == cb_want;
    const int ct_cap = (int)std::max<int64_t>(B.ct_max - 256, 64), cb_cap = 256;
    if (!whole && top_full && bot_full && ct_want >= ct_cap && cb_want >= cb_cap) return LRE_OK;  // reduction path
    if (top_full) ct_want = std::min(2 * ct_want, ct_cap);
    if (bot_full) cb_want = std::min(2 * cb_want, cb_cap);
    // the next check: a check costs ten to twenty steps, so when the leading
    // values converge at a known rate, go most of the way to the threshold
    step = KRY_CHECK;
    if (guess > conv_top && conv_top > seen && J > seen_J) {
      const double rate = (double)(conv_top - seen) / (J - seen_J);
      const int far = (int)(0.7 * (guess - conv_top) / rate) / KRY_CHECK * KRY_CHECK;
      step = std::max(KRY_CHECK, std::min(far, 4 * KRY_CHECK));
    }
    seen = conv_top;
    seen_J = J;
  }
  if (r < 0) return LRE_OK;  // undecided within the step limit: reduction path

  // the selected Ritz vectors and their values
  if (m > 0 && (st = kry_ritz_run(ctx, B.Q, J, B.Xr, (int)m, B.Z, d, s)) != LRE_OK) return st;
  // certification: Lanczos on the operator deflated by the selected vectors
  // (seeded as the first basis rows) from a new start vector; the kept form
  // needs its largest Ritz value <= tau = -shift, the dropped form its
  // smallest >= tau.  Nothing is left to certify once J = d.
  const double tau = -shift;
  const double anorm = fmax(fabs(E.w.front()), fabs(E.w.back()));
  const int L2 = J == d ? 0 : (int)std::min<int64_t>(KRY_VERIFY, d - m - 1);
  if (L2 >= 2) {
    if (m > 0) {
      e = cudaMemcpyAsync(B.Q, B.Z, (size_t)m * d * sizeof(float4), cudaMemcpyDeviceToDevice, s);
      if (e != cudaSuccess) return cuda_fail(ctx, e, "certification set-up");
    }
    if ((st = start_vector(ctx, B, d, m, 0x5EED0002ull, s)) != LRE_OK) return st;
    e = cudaMemsetAsync(B.breakdown, 0, sizeof(int), s);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "certification set-up");
    if ((st = lanczos_steps(ctx, B, d, m, 0, L2, alpha2, beta2, tiny, s)) != LRE_OK) return st;
    int brk = 0;
    if ((st = read_breakdown(ctx, B, brk, s)) != LRE_OK) return st;
    const int J2 = brk > 0 ? brk : L2;
    RitzEnds V;
    if ((st = ritz_values(ctx, B, alpha2, beta2, J2, 1, 1, false, s, V)) != LRE_OK) return st;  // smallest, largest
    // up to d = 1024 the values are held to FP64 rounding, and a copy missed within the
    // slack would show in them (by up to 1e-10, where the reduction path has 1e-14);
    // the certification's own values are good to a few 1e-15
    const double slack = (whole ? 2e-14 : 1e-10) * anorm;
    if (kept_form && V.w.back() > tau + slack) return LRE_OK;
    if (!kept_form && V.w.front() < tau - slack) return LRE_OK;
  }
  if (copy && m > 0) {  // where the steps are double-float: the selected values to FP64 rounding
    std::vector<double> q(m);
    if ((st = kry_rayleigh_run(ctx, B.A, B.Z, (int)m, d, reinterpret_cast<double2 *>(B.lu), B.last, s)) != LRE_OK)
      return st;
    e = cudaMemcpyAsync(q.data(), B.last, m * sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "Rayleigh quotients");
    std::sort(q.begin(), q.end());  // ascending as before; ties at rounding level may have changed places
    std::copy(q.begin(), q.end(), E.w.begin() + sel0);
    double sum = 0.0;
    for (double v : q) sum += v;
    if (r > 0) shift = (kept_form ? trace - sum : sum) / (double)r;
  }
  if (eig_rho && !kept_form && r > 0) {
    // J = d: the kept values by quotients of their own vectors too (from T alone they
    // are off by 2e-15 to 8e-15 ||mu||, the reduction's by 0.5e-15); clusters are
    // orthogonalised by one CTA each, so long ones are left to the reduction path
    int run = 1;
    for (int64_t k = m + 1; k < d; ++k) {
      run = E.w[k] - E.w[k - 1] > 1e-6 * E.tnorm ? 1 : run + 1;
      if (run > KRY_MAX_CLUSTER) return LRE_OK;
    }
    std::vector<double> q(r);
    float4 *const Zk = B.Z + m * d;
    if ((st = ritz_vectors(ctx, B, B.alpha, B.beta, J, B.Wr + m, (int)r, E.tnorm, s, last)) != LRE_OK) return st;
    if ((st = kry_ritz_run(ctx, B.Q, J, B.Xr, (int)r, Zk, d, s)) != LRE_OK) return st;
    if ((st = kry_rayleigh_run(ctx, B.A, Zk, (int)r, d, reinterpret_cast<double2 *>(B.lu), B.last, s)) != LRE_OK)
      return st;
    e = cudaMemcpyAsync(q.data(), B.last, r * sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "Rayleigh quotients");
    std::sort(q.begin(), q.end());
    std::copy(q.begin(), q.end(), E.w.begin() + m);
  }
  // the selected Ritz values (Wr was overwritten by the certification), then
  // for eig_rho every kept value, ascending
  std::vector<double> wsel(E.w.begin() + sel0, E.w.begin() + sel0 + m);
  if (eig_rho && !kept_form) wsel.insert(wsel.end(), E.w.begin() + m, E.w.end());  // exact: all d values
  if (!wsel.empty()) {
    e = cudaMemcpyAsync(B.Wr, wsel.data(), wsel.size() * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "selected eigenvalues");
  }
  *fallback = false;
  if ((st = kry_rebuild_run(ctx, B.Z, B.Wr, (int)m, shift, kept_form, B.A, reinterpret_cast<float2 *>(rho_out), d,
                            s)) != LRE_OK)
    return st;
  if (eig_rho) {
    Launch L(ctx, "kry_eig_rho", s);
    kry_eig_rho<<<(int)((d + 255) / 256), 256, 0, s>>>(B.Wr + (kept_form ? 0 : m), r, shift, eig_rho, d);
  }
  e = cudaGetLastError();
  return e == cudaSuccess ? LRE_OK : cuda_fail(ctx, e, "Krylov projection");
}

}  // namespace lre
