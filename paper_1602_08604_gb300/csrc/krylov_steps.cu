// Lanczos steps in one persistent cooperative launch (d <= KRY_STEPS_MAX_D).
//
// A step of krylov.cu's multi-launch form is eight launches, and at d <= 4096
// their gaps and tails cost more than their data: mu (8 d^2 bytes) and the
// Krylov basis sit in L2 or close to it.  Here one launch runs a whole run of
// steps with three grid-wide barriers a step.  CTA g owns the entries
// [g d / G, (g+1) d / G) of every vector:
//   product   y = mu x for the CTA's own rows (x whole in shared memory), and
//             its share of alpha = q^dag y                          -- barrier
//   dots      w' = y - alpha q - beta q_prev formed whole in shared memory by
//             every CTA, then h_t = q_t^dag w' for the basis rows t = g, g + G, ...
//                                                                   -- barrier
//   update    w'' = w' - sum_t h_t q_t on the own entries, and the own share of
//             ||w''||^2                                             -- barrier
// and the next step's x is w'' scaled by a power of two (exact), the factor
// 1 / beta applied to the product's results, while each CTA stores its own
// entries of q_next = w'' / beta.
//
// Orthogonality: a single classical Gram-Schmidt pass over the whole basis
// would leave q_t^dag w'' = -(q_t^dag q_j) alpha - (q_t^dag q_j-1) beta, which
// can grow from step to step when |alpha| > 2 beta.  Taking the two local
// terms out first makes every h_t of the full pass a small correction, so what
// is left is of second order, as after a second full pass, and the basis is
// read twice a step instead of four times.
//
// Arithmetic: packed double-float (dfloat.cuh), alpha and beta themselves in
// FP64; every CTA adds the shares in the same order, so all have the same
// scalars and a run repeats bit for bit.
// What bounds it: at d = 4096 the product's FP32 instructions (22 packed ones of
// two cycles per entry of mu: 21 us of a step's 46; with mu's next batch loaded
// during the products of the one before, 46 against 67 us a step), below that the
// barriers and dependent trips to L2 (16 us a step at d = 1024).
#include <cuda_runtime.h>

#include <algorithm>

#include "dfloat.cuh"
#include "krylov.cuh"
#include "lre_internal.cuh"
#include "sm103.cuh"

namespace lre {
namespace {

constexpr int THREADS = 512;
constexpr int WARPS = THREADS / 32;
constexpr int UNITS = 112;               // units whose per-lane partial sums fit (56 KB)
constexpr int PART = UNITS * 32;

struct StepArgs {
  const float2 *A;      // mu, row-major complex64
  float4 *Q;            // basis rows (double-float)
  float4 *Y, *W;        // [d] the product y; w'' (double-float)
  float4 *H;            // [rows] the corrections h_t
  double *alpha, *beta;
  float2 *shares;       // [2][G] the CTAs' shares of alpha and of the norm
  unsigned *bar;        // arrivals, then the abort flag; zeroed before the launch
  uint64_t wait_ns;     // bound of a barrier's wait
  unsigned stall;       // test hook: arrivals waited for that never come
  int *breakdown, *status;
  float tiny;
  int d, base, j0, j1, rows;
};

// (h, l) += (oh, ol), double-float reals
__device__ __forceinline__ void real_add(float &h, float &l, float oh, float ol) {
  const float t = __fadd_rn(h, oh), bp = __fsub_rn(t, h);
  const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(t, bp)), __fsub_rn(oh, bp));
  l = __fadd_rn(__fadd_rn(l, ol), e);
  h = t;
}
__device__ __forceinline__ void warp_real_sum(float &h, float &l) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    real_add(h, l, __shfl_xor_sync(0xffffffffu, h, o), __shfl_xor_sync(0xffffffffu, l, o));
}
// Sum over the CTA, on warp 0.  wide: threads beyond warp 0 contribute.
__device__ __forceinline__ void block_real_sum(float &h, float &l, float2 *red, bool wide) {
  if (!wide) {
    if (threadIdx.x < 32) warp_real_sum(h, l);
    return;
  }
  warp_real_sum(h, l);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = make_float2(h, l);
  __syncthreads();
  if (threadIdx.x < 32) {
    const float2 v = threadIdx.x < WARPS ? red[threadIdx.x] : make_float2(0.f, 0.f);
    h = v.x;
    l = v.y;
    warp_real_sum(h, l);
  }
}

// Barrier over all CTAs (every one resident: cooperative launch).  Bounded by
// time; false once a wait gave up anywhere.
__device__ __forceinline__ bool grid_barrier(const StepArgs &P, unsigned &target, int *s_ok) {
  target += gridDim.x + P.stall;
  __syncthreads();
  if (gridDim.x == 1) return true;
  if (threadIdx.x == 0) {
    __threadfence();  // the CTA's writes, ordered before by the barrier above
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(P.bar) : "memory");
    const uint64_t t0 = sm103::globaltimer();
    volatile unsigned *abort = P.bar + 1;
    int ok = 1;
    for (uint32_t it = 0;; ++it) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(P.bar) : "memory");
      if (v >= target) break;
      if ((it & 255u) == 255u && (*abort || sm103::globaltimer() - t0 > P.wait_ns)) {
        ok = 0;
        break;
      }
    }
    if (!ok) {
      *abort = 1;
      latch(P.status, LRE_ERR_TIMEOUT);
    }
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

// Sum of the G shares (the same on every CTA), on warp 0.
__device__ __forceinline__ void sum_shares(const float2 *p, float &h, float &l) {
  h = l = 0.f;
  for (int k = threadIdx.x; k < (int)gridDim.x; k += 32) {
    const float2 v = __ldcg(p + k);
    real_add(h, l, v.x, v.y);
  }
  warp_real_sum(h, l);
}

__device__ __forceinline__ float2 ld_mu(const float2 *p, uint64_t policy) {
  float2 v;
  asm("ld.global.nc.L2::cache_hint.v2.f32 {%0, %1}, [%2], %3;" : "=f"(v.x), "=f"(v.y) : "l"(p), "l"(policy));
  return v;
}
__device__ __forceinline__ float4 ldcg4(const float4 *p) { return __ldcg(p); }

// (h, l) += a b for double-float reals
__device__ __forceinline__ void real_mac(float &h, float &l, float ah, float al, float bh, float bl) {
  const float p = __fmul_rn(ah, bh);
  float e = __fmaf_rn(ah, bh, -p);
  e = __fmaf_rn(ah, bl, e);
  e = __fmaf_rn(al, bh, e);
  const float t = __fadd_rn(h, p), bp = __fsub_rn(t, h);
  l = __fadd_rn(l, __fadd_rn(__fadd_rn(__fsub_rn(h, __fsub_rn(t, bp)), __fsub_rn(p, bp)), e));
  h = t;
}

// v - c q with c a double-float real
__device__ __forceinline__ float4 sub_scaled(const float4 &v, float2 c, const float4 &q) {
  df::f2 h = df::hi(v), l = df::lo(v);
  df::mac2(h, l, df::pk(-c.x, -c.x), df::pk(-c.y, -c.y), df::hi(q), df::lo(q));
  return df::norm4(h, l);
}
__device__ __forceinline__ float4 scaled(const float4 &q, float2 c) {
  df::f2 h = 0, l = 0;
  df::mac2(h, l, df::pk(c.x, c.x), df::pk(c.y, c.y), df::hi(q), df::lo(q));
  return df::norm4(h, l);
}

__global__ void __launch_bounds__(THREADS, 1) kry_steps(StepArgs P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int d = P.d, G = gridDim.x, g = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int r0 = (int)((int64_t)g * d / G), r1 = (int)((int64_t)(g + 1) * d / G), nr = r1 - r0;
  const int nr_max = (d + G - 1) / G;
  float4 *xs = reinterpret_cast<float4 *>(smem_raw);  // [d] x, then w'
  float4 *hs = xs + d;                                // [rows] corrections
  float4 *part = hs + P.rows;                         // [PART] partial sums
  float4 *ys = part + PART;                           // [nr_max] own entries of y, then of w''
  float4 *qs = ys + nr_max;                           // own entries of q
  __shared__ float2 s_alpha_x, s_beta, s_inv, s_ysc;
  __shared__ float s_pow;
  __shared__ int s_ok;
  __shared__ float2 red[WARPS];
  unsigned target = 0;
  // mu passes through L2 once a step; above half of L2 (d = 4096: 134 MB) it is
  // marked evict-first, so that the basis stays (n = 12: dots and update 49k
  // against 37k cycles a step)
  const uint64_t policy = (int64_t)d * d * 8 > (64ll << 20) ? sm103::l2_evict_first() : sm103::l2_evict_normal();
  df::D1 alpha_1{0.f, 0.f}, yscale{1.f, 0.f};  // warp 0: alpha before the corrections; y = yscale (mu xs)

  // x = the basis row of the first step
  {
    const float4 *q = P.Q + (int64_t)(P.base + P.j0) * d;
    for (int i = tid; i < d; i += THREADS) xs[i] = ldcg4(q + i);
    for (int e = tid; e < nr; e += THREADS) qs[e] = ldcg4(q + r0 + e);
    if (tid == 0) {
      s_beta = df::split1(P.j0 > 0 ? P.beta[P.j0 - 1] : 0.0);
      s_ysc = make_float2(1.f, 0.f);
    }
  }
  __syncthreads();

  // Units of the product: own rows x column segments (1024 columns, shorter
  // where that leaves warps without a unit); a lane's partial sums go to shared
  // memory and are added by one warp per row: a shuffle reduction per unit
  // took as long as half a unit's products.
  int seg = d < 1024 ? d : 1024;
  while (seg > 128 && nr_max * (d / seg) < WARPS - 2) seg >>= 1;
  const int nseg = d / seg, rroom = UNITS / nseg;  // nseg <= 32
  const bool wide = nr > 32;
  for (int j = P.j0; j < P.j1; ++j) {
    const int c = P.base + j;  // the row of q_j
    // ---- product
    for (int rb = 0; rb < nr; rb += rroom) {
      const int nrow = nr - rb < rroom ? nr - rb : rroom;
      const int units = nrow * nseg;
      if (seg >= 512) {
        // batches of sixteen entries per lane; the next batch (of this unit or of the
        // warp's next one) is in flight during the products of the current one, 64 KB an SM
        const int per = seg >> 9, nb = units > warp ? ((units - warp + WARPS - 1) / WARPS) * per : 0;
        auto load = [&](int bt, float2 (&v)[16]) {
          const int u = warp + bt / per * WARPS, r = u / nseg;
          const float2 *a = P.A + (int64_t)(r0 + rb + r) * d + (u - r * nseg) * seg + (bt % per) * 512 + lane;
#pragma unroll
          for (int q = 0; q < 16; ++q) v[q] = ld_mu(a + 32 * q, policy);
        };
        float2 next[16];
        if (nb > 0) load(0, next);
        df::Sum S;
        for (int bt = 0; bt < nb; ++bt) {
          float2 v[16];
#pragma unroll
          for (int q = 0; q < 16; ++q) v[q] = next[q];
          if (bt + 1 < nb) load(bt + 1, next);
          const int u = warp + bt / per * WARPS, r = u / nseg;
          const float4 *x = xs + (u - r * nseg) * seg + (bt % per) * 512 + lane;
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            const float4 w = x[32 * q];
            df::mac_c64(S, v[q], df::hi(w), df::lo(w));
          }
          if (bt % per == per - 1) {
            part[u * 32 + lane] = df::df_ab(S);
            S = df::Sum();
          }
        }
      } else {
        for (int u = warp; u < units; u += WARPS) {
          const int r = u / nseg, sg = u - r * nseg;
          const float2 *a = P.A + (int64_t)(r0 + rb + r) * d + sg * seg + lane;
          const float4 *x = xs + sg * seg + lane;
          df::Sum S;
          for (int k = 0; k < seg; k += 64) {
            const float2 v0 = ld_mu(a + k, policy), v1 = ld_mu(a + k + 32, policy);
            const float4 w0 = x[k], w1 = x[k + 32];
            df::mac_c64(S, v0, df::hi(w0), df::lo(w0));
            df::mac_c64(S, v1, df::hi(w1), df::lo(w1));
          }
          part[u * 32 + lane] = df::df_ab(S);
        }
      }
      __syncthreads();
      for (int r = warp; r < nrow; r += WARPS) {
        float4 v = part[r * nseg * 32 + lane];
        for (int k = 1; k < nseg; ++k) v = df::add(v, part[(r * nseg + k) * 32 + lane]);
        v = scaled(df::warp_sum(v), s_ysc);
        if (lane == 0) {
          ys[rb + r] = v;
          P.Y[r0 + rb + r] = v;
        }
      }
      __syncthreads();
    }
    // share of alpha = Re(q^dag y)
    float sh = 0.f, sl = 0.f;
    for (int e = tid; e < nr; e += THREADS) {
      const float4 q = qs[e], y = ys[e];
      real_mac(sh, sl, q.x, q.z, y.x, y.z);
      real_mac(sh, sl, q.y, q.w, y.y, y.w);
    }
    block_real_sum(sh, sl, red, wide);
    const bool prev = j > 0;
    constexpr int PER = (int)(KRY_STEPS_MAX_D / THREADS), HALF = PER / 2;
    if (tid == 0) P.shares[g] = make_float2(sh, sl);
    if (!grid_barrier(P, target, &s_ok)) return;
    // ---- w' = y - alpha q - beta q_prev, whole; q = xs yscale
    if (warp == 0) {
      if (G > 1) sum_shares(P.shares, sh, sl);
      if (lane == 0) {
        alpha_1 = df::fast_norm(sh, sl);
        const df::D1 ax = alpha_1 * yscale;
        s_alpha_x = make_float2(ax.h, ax.l);
      }
    }
#pragma unroll
    for (int m0 = 0; m0 < PER; m0 += HALF) {
      float4 yv[HALF], qp[HALF];
#pragma unroll
      for (int m = 0; m < HALF; ++m) {
        const int i = tid + (m0 + m) * THREADS;
        if (i < d) {
          yv[m] = ldcg4(P.Y + i);
          if (prev) qp[m] = ldcg4(P.Q + (int64_t)(c - 1) * d + i);
        }
      }
      if (m0 == 0) __syncthreads();  // alpha
      const float2 ca = s_alpha_x, cb = s_beta;
#pragma unroll
      for (int m = 0; m < HALF; ++m) {
        const int i = tid + (m0 + m) * THREADS;
        if (i < d) {
          float4 v = sub_scaled(yv[m], ca, xs[i]);
          if (prev) v = sub_scaled(v, cb, qp[m]);
          xs[i] = v;
        }
      }
    }
    __syncthreads();
    // ---- dots: rows t = g, g + G, ... <= c, each cut into ns segments
    const int nvec = c >= g ? (c - g) / G + 1 : 0;
    if (nvec > 0) {
      int ns = 1;
      while (ns < 8 && nvec * ns < 2 * WARPS && d / (2 * ns) >= 64) ns *= 2;
      const int len = d / ns, vroom = UNITS / ns;
      for (int v0 = 0; v0 < nvec; v0 += vroom) {
        const int nv = nvec - v0 < vroom ? nvec - v0 : vroom;
        for (int u = warp; u < nv * ns; u += WARPS) {
          const int v = u / ns, sg = u - v * ns;
          const float4 *q = P.Q + (int64_t)(g + (v0 + v) * G) * d + sg * len;
          const float4 *w = xs + sg * len;
          df::Sum S;
          int k = lane;
          for (; k + 224 < len; k += 256) {
            float4 a[8];
#pragma unroll
            for (int m = 0; m < 8; ++m) a[m] = ldcg4(q + k + 32 * m);
#pragma unroll
            for (int m = 0; m < 8; ++m) {
              const float4 b = w[k + 32 * m];
              df::mac_df(S, a[m], df::hi(b), df::lo(b));
            }
          }
          for (; k + 32 < len; k += 64) {
            const float4 a0 = ldcg4(q + k), a1 = ldcg4(q + k + 32), b0 = w[k], b1 = w[k + 32];
            df::mac_df(S, a0, df::hi(b0), df::lo(b0));
            df::mac_df(S, a1, df::hi(b1), df::lo(b1));
          }
          for (; k < len; k += 32) {
            const float4 a = ldcg4(q + k), b = w[k];
            df::mac_df(S, a, df::hi(b), df::lo(b));
          }
          part[u * 32 + lane] = df::df_conj_ab(S);
        }
        __syncthreads();
        for (int v = warp; v < nv; v += WARPS) {
          float4 s = part[v * ns * 32 + lane];
          for (int k = 1; k < ns; ++k) s = df::add(s, part[(v * ns + k) * 32 + lane]);
          s = df::warp_sum(s);
          if (lane == 0) P.H[g + (v0 + v) * G] = s;
        }
        __syncthreads();
      }
    }
    if (!grid_barrier(P, target, &s_ok)) return;
    // ---- update of the own entries
    for (int t = tid; t <= c; t += THREADS) hs[t] = ldcg4(P.H + t);
    __syncthreads();
    sh = sl = 0.f;
    {
      int ew = 1;
      while (ew < nr && ew < THREADS) ew *= 2;
      const int slices = THREADS / ew, sl_ = tid / ew;
      for (int e0 = 0; e0 < nr; e0 += ew) {
        const int e = e0 + (tid & (ew - 1));
        df::Sum S;
        if (e < nr) {
          const float4 *q = P.Q + r0 + e;
          int t = sl_;
          for (; t + 7 * slices <= c; t += 8 * slices) {
            float4 b[8];
#pragma unroll
            for (int m = 0; m < 8; ++m) b[m] = ldcg4(q + (int64_t)(t + m * slices) * d);
#pragma unroll
            for (int m = 0; m < 8; ++m) df::mac_df(S, hs[t + m * slices], df::hi(b[m]), df::lo(b[m]));
          }
          for (; t + slices <= c; t += 2 * slices) {
            const float4 b0 = ldcg4(q + (int64_t)t * d), b1 = ldcg4(q + (int64_t)(t + slices) * d);
            df::mac_df(S, hs[t], df::hi(b0), df::lo(b0));
            df::mac_df(S, hs[t + slices], df::hi(b1), df::lo(b1));
          }
          for (; t <= c; t += slices) {
            const float4 b = ldcg4(q + (int64_t)t * d);
            df::mac_df(S, hs[t], df::hi(b), df::lo(b));
          }
        }
        float4 s = df::df_ab(S);
        if (slices > 1) {
          part[tid] = s;
          __syncthreads();
          for (int o = slices >> 1; o > 0; o >>= 1) {
            if (sl_ < o) {
              s = df::add(s, part[tid + o * ew]);
              part[tid] = s;
            }
            __syncthreads();
          }
        }
        if (sl_ == 0 && e < nr) {
          const float4 w = df::add(xs[r0 + e], make_float4(-s.x, -s.y, -s.z, -s.w));
          ys[e] = w;
          P.W[r0 + e] = w;
          real_mac(sh, sl, w.x, w.z, w.x, w.z);
          real_mac(sh, sl, w.y, w.w, w.y, w.w);
        }
      }
    }
    block_real_sum(sh, sl, red, wide);
    if (tid == 0) P.shares[G + g] = make_float2(sh, sl);
    if (!grid_barrier(P, target, &s_ok)) return;
    // ---- close the step
    if (warp == 0) {
      if (G > 1) sum_shares(P.shares + G, sh, sl);  // every lane has the sum
      else {
        sh = __shfl_sync(0xffffffffu, sh, 0);
        sl = __shfl_sync(0xffffffffu, sl, 0);
      }
      // what the next phase waits for in double-float (an FP64 square root and its
      // splits are twenty dependent operations of 110 cycles)
      const df::D1 b2 = df::fast_norm(sh, sl);
      const df::D1 inv0 = b2.h > 0.f ? df::inv_sqrt(b2) : df::D1{0.f, 0.f}, b = b2 * inv0;
      const bool dead = !(b.h > P.tiny);  // an invariant subspace: q_next = 0, as the host expects
      const df::D1 inv = dead ? df::D1{0.f, 0.f} : inv0;
      // xs = w'' 2^-e with beta 2^-e in [1, 2): exact, and y's factor is 2^e / beta
      int ex = dead ? 0 : (int)((__float_as_uint(b.h) >> 23) & 0xFF) - 127;
      ex = ex > 120 ? 120 : ex < -120 ? -120 : ex;
      const float up = __int_as_float((127 + ex) << 23);
      yscale = {inv.h * up, inv.l * up};
      if (lane == 0) {
        s_ysc = make_float2(yscale.h, yscale.l);
        s_pow = dead ? 0.f : __int_as_float((127 - ex) << 23);
        s_inv = make_float2(inv.h, inv.l);
        s_beta = dead ? make_float2(0.f, 0.f) : make_float2(b.h, b.l);
      }
    }
    __syncthreads();
    if (g == 0 && tid == 0) {  // the Lanczos matrix, in FP64
      const double b2 = (double)sh + (double)sl, b = b2 > 0.0 ? sqrt(b2) : 0.0;
      const bool dead = s_pow == 0.f;
      P.alpha[j] = df::value(alpha_1) + ((double)hs[c].x + (double)hs[c].z);
      P.beta[j] = dead ? 0.0 : b;
      if (dead && *P.breakdown == 0) *P.breakdown = j + 1;
    }
    const float2 inv = s_inv;
    const bool store = c + 1 < P.rows;
    for (int e = tid; e < nr; e += THREADS) {
      const float4 q = scaled(ys[e], inv);
      qs[e] = q;
      if (store) P.Q[(int64_t)(c + 1) * d + r0 + e] = q;
    }
    if (j + 1 < P.j1) {
      const float pw = s_pow;
#pragma unroll
      for (int m0 = 0; m0 < PER; m0 += HALF) {
        float4 wv[HALF];
#pragma unroll
        for (int m = 0; m < HALF; ++m)
          if (tid + (m0 + m) * THREADS < d) wv[m] = ldcg4(P.W + tid + (m0 + m) * THREADS);
#pragma unroll
        for (int m = 0; m < HALF; ++m) {
          const int i = tid + (m0 + m) * THREADS;
          if (i < d) xs[i] = make_float4(wv[m].x * pw, wv[m].y * pw, wv[m].z * pw, wv[m].w * pw);
        }
      }
    }
    __syncthreads();
  }
}

size_t steps_smem(int64_t d, int64_t rows, int G) {
  const int64_t nr = (d + G - 1) / G;
  return (size_t)(d + rows + PART + 2 * nr) * sizeof(float4);
}

}  // namespace

// Eight entries a CTA up to one CTA per SM: a step is three barriers and a dozen
// dependent trips to L2, so more CTAs pay until their share of the products is
// below that (d = 256: 3.6 ms a run on 32 CTAs, 4.0 on 16, 15.8 on one;
// d = 1024: 7.7 on 128, 9.0 on 64; d = 64: 0.8 on 8, 0.9 on one).
// Whole projections, before (the reduction path below d = 2048, one launch per
// operation above) and now: d = 64 4.9 -> 1.1 ms, 256 16 -> 4.4, 512 34 -> 7.1,
// 1024 82.7 -> 11.2 (51 vectors kept), 4096 177 -> 53 (100 kept).
int kry_steps_grid(lre_ctx *ctx, int64_t d) {
  const int64_t g = d / 8;
  return (int)std::min<int64_t>(g, ctx->num_sms);
}

size_t kry_sync_bytes(const lre_ctx *ctx) { return 4 * sizeof(unsigned) + 2 * (size_t)ctx->num_sms * sizeof(float2); }

lre_status kry_steps_run(lre_ctx *ctx, const KryStepBuffers &B, int64_t d, int64_t base, int j0, int j1,
                         double *alpha, double *beta, double tiny, cudaStream_t s) {
  StepArgs P{};
  P.A = B.A;
  P.Q = B.Q;
  P.Y = B.Y;
  P.W = B.W;
  P.H = B.H;
  const int G = kry_steps_grid(ctx, d);
  P.alpha = alpha;
  P.beta = beta;
  P.bar = static_cast<unsigned *>(B.sync);
  P.shares = reinterpret_cast<float2 *>(P.bar + 4);
  P.breakdown = B.breakdown;
  P.wait_ns = ctx->batch_wait_ns ? ctx->batch_wait_ns : sm103::kWaitNs;
  P.stall = ctx->steps_stall;
  P.status = ctx->d_status;
  P.tiny = (float)tiny;
  P.d = (int)d;
  P.base = (int)base;
  P.j0 = j0;
  P.j1 = j1;
  P.rows = (int)B.rows;
  const size_t smem = steps_smem(d, B.rows, G);
  if (d > KRY_STEPS_MAX_D || B.rows > KRY_STEPS_MAX_ROWS) return LRE_ERR_UNSUPPORTED;
  // the limit is the function's, not the context's: one value for every size, so that no
  // other thread's call lowers it between here and the launch
  const size_t most = steps_smem(KRY_STEPS_MAX_D, KRY_STEPS_MAX_ROWS, kry_steps_grid(ctx, KRY_STEPS_MAX_D));
  cudaError_t e = cudaFuncSetAttribute(kry_steps, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
  if (e == cudaSuccess) e = cudaMemsetAsync(B.sync, 0, 2 * sizeof(unsigned), s);
  if (e == cudaSuccess) {
    Launch L(ctx, "kry_matvec", s);  // named for its largest part, the products with mu
    void *args[] = {&P};
    e = cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(kry_steps), dim3(G), dim3(THREADS), args, smem, s);
  }
  return e == cudaSuccess ? LRE_OK : cuda_fail(ctx, e, "Lanczos steps");
}

}  // namespace lre

// Test hook (not part of include/lre.h): from now on each grid barrier of the Lanczos
// steps waits for arrivals that never come and gives up after wait_ms (0: as usual).
extern "C" lre_status lre_debug_steps_fault(lre_ctx *ctx, int wait_ms) {
  if (!ctx || wait_ms < 0) return LRE_ERR_INVALID_ARG;
  ctx->batch_wait_ns = (uint64_t)wait_ms * 1000000;
  ctx->steps_stall = wait_ms > 0;
  return LRE_OK;
}
