// What the Krylov projection (krylov.cu) does around the Lanczos steps: the
// Hermitian copy of mu, the Ritz vectors, and the projected matrix rebuilt from
// them, in double-float arithmetic on the FP32 pipes (dfloat.cuh): GB300's FP64
// pipe made the same sums 5-10 times slower (a rank-100 update at d = 4096 by
// cublasZherk 7.0 ms).
#include <cuda_runtime.h>

#include "dfloat.cuh"
#include "krylov.cuh"
#include "lre_internal.cuh"

namespace lre {
namespace {

// out = the Hermitian matrix of in's upper triangle (the triangle every path of
// the projection goes by; the diagonal real), 32 x 32 tiles.
__global__ void kry_hermitian(const float2 *__restrict__ in, float2 *__restrict__ out, int64_t d) {
  __shared__ float2 t[32][33];
  const int64_t r0 = (int64_t)blockIdx.y * 32, c0 = (int64_t)blockIdx.x * 32;
  if (r0 > c0) return;
  const int tx = threadIdx.x;
  for (int i = threadIdx.y; i < 32; i += 8) {
    float2 v = in[(r0 + i) * d + c0 + tx];
    if (r0 == c0 && i == tx) v.y = 0.f;
    t[i][tx] = v;
    if (r0 < c0 || i <= tx) out[(r0 + i) * d + c0 + tx] = v;
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += 8) {
    if (r0 < c0 || tx < i) {
      const float2 v = t[tx][i];
      out[(c0 + i) * d + r0 + tx] = make_float2(v.x, -v.y);
    }
  }
}

// acc[0] = the trace in FP64 (block 0), acc[1 + b] = block b's share of sum |in|^2 (a
// scale: FP32 sums per thread, once more in FP64 where those leave FP32's range); all
// in a fixed order.
__global__ void __launch_bounds__(256) kry_norm_trace(const float2 *__restrict__ in, int64_t d, double *acc) {
  __shared__ double s[8];
  auto block_sum = [&](double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0;
    for (int k = 0; k < 8; ++k) t += s[k];
    return t;
  };
  float v = 0.f;
  for (int64_t i = blockIdx.x * 256 + threadIdx.x; i < d * d; i += (int64_t)gridDim.x * 256) {
    const float2 a = in[i];
    v = fmaf(a.x, a.x, fmaf(a.y, a.y, v));
  }
  double w = (double)v;
  if (!(v > 0x1p-100f && v < 0x1p126f)) {
    w = 0.0;
    for (int64_t i = blockIdx.x * 256 + threadIdx.x; i < d * d; i += (int64_t)gridDim.x * 256) {
      const double x = in[i].x, y = in[i].y;
      w = fma(x, x, fma(y, y, w));
    }
  }
  const double t = block_sum(w);
  if (threadIdx.x == 0) acc[1 + blockIdx.x] = t;
  if (blockIdx.x == 0) {
    double tr = 0;
    for (int64_t i = threadIdx.x; i < d; i += 256) tr += (double)in[i * d + i].x;
    tr = block_sum(tr);
    if (threadIdx.x == 0) acc[0] = tr;
  }
}

// Ritz vectors Z[k] = sum_t S[t + k J] q_t (S column-major J x m, real), one row
// of d double-float entries each.  A thread sums eight vectors at one entry, so
// a basis entry is loaded once for eight products.
constexpr int RZ_K = 8, RZ_T = 32;
__global__ void __launch_bounds__(128) kry_ritz(const float4 *__restrict__ Q, int J, const double *__restrict__ S,
                                                int m, float4 *__restrict__ Z, int64_t d) {
  __shared__ float2 cs[RZ_T][RZ_K];
  const int k0 = blockIdx.y * RZ_K;
  const int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x;
  df::f2 h[RZ_K], l[RZ_K];
#pragma unroll
  for (int k = 0; k < RZ_K; ++k) h[k] = l[k] = 0;
  for (int t0 = 0; t0 < J; t0 += RZ_T) {
    __syncthreads();
    for (int e = threadIdx.x; e < RZ_T * RZ_K; e += 128) {
      const int k = e / RZ_T, t = e - k * RZ_T;
      cs[t][k] = (t0 + t < J && k0 + k < m) ? df::split1(S[t0 + t + (int64_t)(k0 + k) * J]) : make_float2(0.f, 0.f);
    }
    __syncthreads();
    if (i < d) {
      const int nt = J - t0 < RZ_T ? J - t0 : RZ_T;
#pragma unroll 4
      for (int t = 0; t < nt; ++t) {
        const float4 q = Q[(int64_t)(t0 + t) * d + i];
        const df::f2 qh = df::hi(q), ql = df::lo(q);
#pragma unroll
        for (int k = 0; k < RZ_K; ++k) {
          const float2 c = cs[t][k];
          df::mac2(h[k], l[k], df::pk(c.x, c.x), df::pk(c.y, c.y), qh, ql);
        }
      }
    }
  }
  if (i < d)
#pragma unroll
    for (int k = 0; k < RZ_K; ++k)
      if (k0 + k < m) Z[(int64_t)(k0 + k) * d + i] = df::norm4(h[k], l[k]);
}

// part[k][b] = block b's rows of z_k^dag A z_k and of z_k^dag z_k, over the upper
// triangle of the Hermitian A (a_rr |z_r|^2 + 2 Re conj(z_r) a_rc z_c).
// The double-float Lanczos leaves its values 2^-48 ||A|| or so off (the normalisation
// of a basis vector is one number for all its entries); the quotient of the finished
// vectors, whose own error enters squared, is at FP64 rounding.
// FP64 throughout up to d = 1024.  Beyond (WIDE), where that would cost as much as the
// Lanczos steps, a row's products and their sum are double-float: each row's error is
// its own, so weighted by z_r and added in FP64 they average out.  Mean error of eig_rho
// over four product-state estimates, relative to the norm, without the quotients -> now:
// d = 2048 1.2e-15 -> 0.3e-15, d = 4096 1.6e-15 -> 0.6e-15 (the FP64 coefficients and second
// Gram-Schmidt pass of one launch per operation: 0.6e-15, 1.3e-15).  d = 4096, 175
// vectors: 3.0 of 82 ms.
constexpr int RQ_ROWS = 64, RQ_FP64_D = 1024;
constexpr size_t RQ_SMEM = (size_t)KRY_STEPS_MAX_D * sizeof(float4);
template <bool WIDE>
__global__ void __launch_bounds__(256) kry_rayleigh(const float2 *__restrict__ A, const float4 *__restrict__ Z, int d,
                                                    double2 *part) {
  extern __shared__ __align__(16) unsigned char rq_smem[];
  float4 *zf = reinterpret_cast<float4 *>(rq_smem);   // WIDE
  double2 *zd = reinterpret_cast<double2 *>(rq_smem);  // else
  __shared__ double s1[8], s2[8];
  const int k = blockIdx.x, r0 = blockIdx.y * RQ_ROWS, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < d; i += 256) {
    const float4 z = Z[(int64_t)k * d + i];
    if constexpr (WIDE) zf[i] = z;
    else zd[i] = df::join(z);
  }
  __syncthreads();
  double num = 0.0, den = 0.0;
  for (int r = r0 + warp; r < r0 + RQ_ROWS && r < d; r += 8) {
    double re = 0.0, im = 0.0;  // sum_{c > r} a_rc z_c
    double2 zr;
    if constexpr (WIDE) {
      const float2 *a = A + (int64_t)r * d;
      df::Sum S;
      int c = r + 1 + lane;
      for (; c + 224 < d; c += 256) {
        float2 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = a[c + 32 * q];
#pragma unroll
        for (int q = 0; q < 8; ++q) df::mac_c64(S, v[q], df::hi(zf[c + 32 * q]), df::lo(zf[c + 32 * q]));
      }
      for (; c < d; c += 32) df::mac_c64(S, a[c], df::hi(zf[c]), df::lo(zf[c]));
      const double2 p = df::join(df::df_ab(S));
      re = p.x;
      im = p.y;
      zr = df::join(zf[r]);
    } else {
      for (int c = r + 1 + lane; c < d; c += 32) {
        const float2 a = A[(int64_t)r * d + c];
        const double ax = (double)a.x, ay = (double)a.y;
        re = fma(ax, zd[c].x, fma(-ay, zd[c].y, re));
        im = fma(ax, zd[c].y, fma(ay, zd[c].x, im));
      }
      zr = zd[r];
    }
    num = fma(2.0 * zr.x, re, fma(2.0 * zr.y, im, num));
    if (lane == 0) {
      const double q = fma(zr.x, zr.x, zr.y * zr.y);
      num = fma((double)A[(int64_t)r * d + r].x, q, num);
      den += q;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    num += __shfl_xor_sync(0xffffffffu, num, o);
    den += __shfl_xor_sync(0xffffffffu, den, o);
  }
  if (lane == 0) {
    s1[warp] = num;
    s2[warp] = den;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) {
      num += s1[w];
      den += s2[w];
    }
    part[(int64_t)k * gridDim.y + blockIdx.y] = make_double2(num, den);
  }
}

__global__ void kry_quotients(const double2 *part, int m, int nb, double *w) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= m) return;
  double num = 0.0, den = 0.0;
  for (int b = 0; b < nb; ++b) {
    num += part[(int64_t)k * nb + b].x;
    den += part[(int64_t)k * nb + b].y;
  }
  w[k] = num / den;
}

// The projected matrix from m unit vectors (rows of Z, eigenvectors of mu) and
// weights g_k >= 0:
//   kept form     out = sum_k g_k z_k z_k^dag               (g = l + s)
//   DROPPED       out = mu + s I + sum_k g_k z_k z_k^dag    (g = -(l + s))
// rounded once to complex64.  A CTA forms one 64 x 64 tile on or above the
// diagonal (sixteen outputs per thread, eight vectors staged at a time) and
// writes it and its mirror through shared memory, so the result is exactly
// Hermitian and each z is read d / 64 times.  mu and out may be the same.
constexpr int RB_K = 8;
template <bool DROPPED>
__global__ void __launch_bounds__(256) kry_rebuild(const float4 *__restrict__ Z, const double *__restrict__ w, int m,
                                                   double shift, const float2 *mu, float2 *out, int64_t d) {
  __shared__ __align__(16) unsigned char smem[64 * 65 * sizeof(float2)];
  auto As = reinterpret_cast<float4(*)[64]>(smem);  // [RB_K][64], then Bs; the output tile at the end
  auto Bs = reinterpret_cast<float4(*)[64]>(smem + RB_K * 64 * sizeof(float4));
  auto tile = reinterpret_cast<float2(*)[65]>(smem);
  static_assert(2 * RB_K * 64 * sizeof(float4) <= sizeof(smem), "the staged vectors fit");
  const int64_t bi = blockIdx.y, bj = blockIdx.x;
  if (bi > bj) return;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int64_t r0 = bi * 64, c0 = bj * 64;
  df::Sum S[4][4];
  for (int k0 = 0; k0 < m; k0 += RB_K) {
    const int nk = m - k0 < RB_K ? m - k0 : RB_K;
    __syncthreads();
    for (int e = tid; e < RB_K * 64; e += 256) {
      const int k = e >> 6, x = e & 63;
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
      if (k < nk) {
        const float4 z = Z[(int64_t)(k0 + k) * d + r0 + x];
        double g = w[k0 + k] + shift;
        if (DROPPED) g = -g;
        const float2 c = df::split1(g > 0.0 ? g : 0.0);
        df::f2 h = 0, l = 0;
        df::mac2(h, l, df::pk(c.x, c.x), df::pk(c.y, c.y), df::hi(z), df::lo(z));
        a = df::norm4(h, l);
        b = Z[(int64_t)(k0 + k) * d + c0 + x];
      }
      As[k][x] = a;
      Bs[k][x] = b;
    }
    __syncthreads();
    for (int k = 0; k < nk; ++k) {
      float4 b[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) b[q] = Bs[k][tx + 16 * q];
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const float4 a = As[k][ty + 16 * p];
#pragma unroll
        for (int q = 0; q < 4; ++q) df::mac_df(S[p][q], a, df::hi(b[q]), df::lo(b[q]));
      }
    }
  }
  const float2 sh = df::split1(shift);
  __syncthreads();
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = ty + 16 * p, c = tx + 16 * q;
      // a conj(b) = conj(conj(a) b)
      float4 v = df::df_conj_ab(S[p][q]);
      v.y = -v.y;
      v.w = -v.w;
      if (DROPPED) {
        const float2 u = mu[(r0 + r) * d + c0 + c];
        v = df::add(v, make_float4(u.x, u.y, 0.f, 0.f));
        if (r0 + r == c0 + c) v = df::add(v, make_float4(sh.x, 0.f, sh.y, 0.f));
      }
      tile[r][c] = make_float2(v.x, r0 + r == c0 + c ? 0.f : v.y);
    }
  __syncthreads();
  for (int e = tid; e < 4096; e += 256) {
    const int i = e >> 6, x = e & 63;
    if (bi < bj) {
      out[(r0 + i) * d + c0 + x] = tile[i][x];
      const float2 v = tile[x][i];
      out[(c0 + i) * d + r0 + x] = make_float2(v.x, -v.y);
    } else {
      const float2 v = tile[x][i];
      out[(r0 + i) * d + c0 + x] = i <= x ? tile[i][x] : make_float2(v.x, -v.y);
    }
  }
}

}  // namespace

int64_t kry_norm_blocks(const lre_ctx *ctx, int64_t d) {
  const int64_t g = (d * d + 2047) / 2048, cap = (int64_t)ctx->num_sms * 8;
  return g < cap ? g : cap;
}

lre_status kry_prepare_mu(lre_ctx *ctx, const float2 *in, float2 *herm, int64_t d, double *trace_norms, cudaStream_t s) {
  Launch L(ctx, "kry_prepare", s, herm ? 2 : 1);
  if (herm) {
    dim3 g((unsigned)(d / 32), (unsigned)(d / 32)), b(32, 8);
    kry_hermitian<<<g, b, 0, s>>>(in, herm, d);
    in = herm;
  }
  kry_norm_trace<<<(unsigned)kry_norm_blocks(ctx, d), 256, 0, s>>>(in, d, trace_norms);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? LRE_OK : cuda_fail(ctx, e, "Krylov set-up");
}

lre_status kry_ritz_run(lre_ctx *ctx, const float4 *Q, int J, const double *S, int m, float4 *Z, int64_t d,
                        cudaStream_t s) {
  Launch L(ctx, "kry_ritz", s);
  dim3 g((unsigned)((d + 127) / 128), (unsigned)((m + RZ_K - 1) / RZ_K));
  kry_ritz<<<g, 128, 0, s>>>(Q, J, S, m, Z, d);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? LRE_OK : cuda_fail(ctx, e, "Ritz vectors");
}

lre_status kry_rayleigh_run(lre_ctx *ctx, const float2 *A, const float4 *Z, int m, int64_t d, double2 *part, double *w,
                            cudaStream_t s) {
  if (d > KRY_STEPS_MAX_D) return LRE_ERR_UNSUPPORTED;
  const int nb = (int)((d + RQ_ROWS - 1) / RQ_ROWS);
  auto k = d > RQ_FP64_D ? kry_rayleigh<true> : kry_rayleigh<false>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RQ_SMEM);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "Rayleigh quotients");
  Launch L(ctx, "kry_rayleigh", s, 2);
  k<<<dim3((unsigned)m, (unsigned)nb), 256, (size_t)d * sizeof(float4), s>>>(A, Z, (int)d, part);
  kry_quotients<<<(m + 63) / 64, 64, 0, s>>>(part, m, nb, w);
  e = cudaGetLastError();
  return e == cudaSuccess ? LRE_OK : cuda_fail(ctx, e, "Rayleigh quotients");
}

lre_status kry_rebuild_run(lre_ctx *ctx, const float4 *Z, const double *w, int m, double shift, bool kept_form,
                           const float2 *mu, float2 *out, int64_t d, cudaStream_t s) {
  Launch L(ctx, "kry_rebuild", s);
  dim3 g((unsigned)(d / 64), (unsigned)(d / 64));
  if (kept_form) kry_rebuild<false><<<g, 256, 0, s>>>(Z, w, m, shift, mu, out, d);
  else kry_rebuild<true><<<g, 256, 0, s>>>(Z, w, m, shift, mu, out, d);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? LRE_OK : cuda_fail(ctx, e, "projection rebuild");
}

}  // namespace lre
