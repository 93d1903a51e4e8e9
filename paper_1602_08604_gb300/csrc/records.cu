// Shot records grouped by count tile, for the tensor-core first pass that
// builds its count tiles in shared memory straight from the records (step (i),
// Sec. III: the counts c_b(o) are only ever needed tile by tile).
//
// A tile row is 729 consecutive bases (the six lowest basis digits, al); its
// 2^(n-6) tiles are the outcome blocks oh (the outcome's bits above the six
// lowest).  tile_bucket_kernel takes one tile row per CTA and counting-sorts
// the row's 729 x N shot records into 16-bit entries (al << 6) | ol, ol = the
// outcome's six lowest bits, by bucket oh * 2 + (al >= 432) -- the tile and
// the half of its rows the first pass stages together -- with the start of
// every bucket in offs[tile row][bucket] (offsets within the tile row's
// 729 N entries; the last bucket ends at 729 N).  The order inside a bucket
// is irrelevant: the consumer only adds counts.
#include <cuda_runtime.h>

#include "lre_internal.cuh"
#include "passes.cuh"

namespace lre {

namespace {

constexpr int BUCKET_THREADS = 512;
constexpr int BUCKET_WARPS = BUCKET_THREADS / 32;
constexpr int MAX_BUCKETS = 512;  // two per tile, n <= 14: one thread per bucket
static_assert(MAX_BUCKETS <= BUCKET_THREADS, "one thread per bucket in the scan");

// One tile row per CTA (grid-stride).  Every warp counts into its own copy of
// the bucket counters (no contention between warps), a scan turns the
// per-warp counts into per-warp cursors, and the scatter pass places each
// entry through its warp's cursor.  Records are read eight at a time (shots
// a multiple of 8, rows 16-byte aligned).
__global__ void __launch_bounds__(BUCKET_THREADS) tile_bucket_kernel(const uint16_t *__restrict__ rec,
                                                                     int64_t tile_rows, int64_t shots, int n,
                                                                     uint16_t *__restrict__ out,
                                                                     int32_t *__restrict__ offs, int *status) {
  extern __shared__ int32_t wcnt[];  // [BUCKET_WARPS][nb]
  const int nb = 2 << (n - 6);
  const uint32_t d = 1u << n;
  const int warp = threadIdx.x >> 5;
  int32_t *mine = wcnt + warp * nb;
  const int64_t tv = 729 * shots / 8;  // uint4 per tile row
  const float inv_shots = 1.0f / (float)shots;
  for (int64_t tr = blockIdx.x; tr < tile_rows; tr += gridDim.x) {
    const uint4 *r4 = reinterpret_cast<const uint4 *>(rec + tr * 729 * shots);
    uint16_t *o = out + tr * 729 * shots;
    for (int b = threadIdx.x; b < BUCKET_WARPS * nb; b += blockDim.x) wcnt[b] = 0;
    __syncthreads();
    bool bad = false;
    for (int pass = 0; pass < 2; ++pass) {
      for (int64_t q0 = threadIdx.x; q0 < tv; q0 += 4 * (int64_t)blockDim.x) {
        uint4 w4[4];  // four independent 16-byte loads in flight per thread
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int64_t q = q0 + u * (int64_t)blockDim.x;
          w4[u] = q < tv ? __ldcs(r4 + q) : make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int64_t q = q0 + u * (int64_t)blockDim.x;
          if (q >= tv) continue;
          const uint32_t word[4] = {w4[u].x, w4[u].y, w4[u].z, w4[u].w};
          // basis row of these 8 records (shots is a multiple of 8): q * 8 / shots
          int al = (int)((float)(q * 8) * inv_shots);
          if ((int64_t)al * shots > q * 8) --al;
          else if ((int64_t)(al + 1) * shots <= q * 8) ++al;
          const uint32_t half = al >= 432 ? 1u : 0u;
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const uint32_t v = (word[k >> 1] >> ((k & 1) * 16)) & 0xFFFFu;
            if (v >= d) {
              bad = true;
              continue;
            }
            const uint32_t key = (v >> 6) << 1 | half;
            if (pass == 0)
              atomicAdd(&mine[key], 1);
            else
              o[atomicAdd(&mine[key], 1)] = (uint16_t)((al << 6) | (v & 63u));
          }
        }
      }
      __syncthreads();
      if (pass == 0) {
        // per bucket (one thread each): the warps' counts -> their offsets
        // inside the bucket, then an exclusive scan of the bucket totals
        // across the CTA (warp shuffles, then the warps' sums)
        int32_t tot = 0;
        const int b = threadIdx.x;
        if (b < nb)
          for (int w = 0; w < BUCKET_WARPS; ++w) {
            const int32_t c = wcnt[w * nb + b];
            wcnt[w * nb + b] = tot;
            tot += c;
          }
        int32_t incl = tot;
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int o2 = 1; o2 < 32; o2 <<= 1) {
          const int32_t t = __shfl_up_sync(0xffffffffu, incl, o2);
          if (lane >= o2) incl += t;
        }
        __shared__ int32_t wsum[BUCKET_WARPS];
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        int32_t before = 0;
        for (int w = 0; w < warp; ++w) before += wsum[w];
        const int32_t start = before + incl - tot;  // exclusive
        if (b < nb) {
          offs[tr * nb + b] = start;
          for (int w = 0; w < BUCKET_WARPS; ++w) wcnt[w * nb + b] += start;
        }
        __syncthreads();
      }
    }
    if (bad) latch(status, LRE_ERR_INVALID_ARG);
  }
}

// ---------------------------------------------------------------------------
// Records -> the sums over three qubits, without dense counts.
//
// Dense counts cost their own write (725 MB at n = 11; pure writes run at 4.0 TB/s
// here, 181 us) and the read of the first fold pass.  A CTA counts the 27 bases of
// its three lowest axis digits into shared memory instead (two 16-bit bins a word)
// and contracts them where they are: one thread per group of eight outcomes, 27 rows
// of 16 bytes, zeroed as they are read; what leaves is 64 / 216 of the counts.
// The contraction works on the packed words: lo + 65536 hi is linear, so the two
// upper qubits' butterflies and the sums over bases are single 32-bit adds, one
// accumulator set per axis of the lowest qubit (|lo|, |hi| <= 9 shots); that qubit's
// own sum and difference are taken once, at the end.
// Output int16 [3^(n-3)][2^(n-3)][64], as a three-qubit first pass stores it.
// n = 11, 1000 shots: 252 us, where the histogram and the six-qubit pass took 261 + 143
// (the second three-qubit pass adds 60); the whole estimate 516 -> 401 us.  With 104
// shots the kernel still takes about 145 us, so neither the atomics (some 105 us for
// 896 more shots) nor the stores (215 MB, 54 us) bound it alone: the phases of a CTA follow one another and
// shared memory holds two CTAs.  Measured without gain: 512 threads a CTA (277 us),
// swizzled bins with 32-byte stores (269), units without the loads ahead (291).
// ---------------------------------------------------------------------------
constexpr int RF_CELLS = 27 * 2048;  // 16-bit bins of a CTA (n = 12: twice that)

__global__ void __launch_bounds__(512) records_fold3(const uint16_t *__restrict__ rec, int64_t S, int n, int64_t groups,
                                                     int16_t *__restrict__ out, int *status) {
  extern __shared__ uint4 h4[];
  uint32_t *h = reinterpret_cast<uint32_t *>(h4);
  const int d = 1 << n, tpg = d >> 3;                         // threads per group of 27 bases
  const int G = (n == 12 ? 2 * RF_CELLS : RF_CELLS) / (27 * d);  // groups per CTA and round
  const int T = blockDim.x, t = threadIdx.x, warp = t >> 5, lane = t & 31, W = T >> 5;
  for (int i = t; i < G * 27 * tpg; i += T) h4[i] = make_uint4(0, 0, 0, 0);
  __syncthreads();
  bool bad = false;
  for (int64_t g0 = (int64_t)blockIdx.x * G; g0 < groups; g0 += (int64_t)gridDim.x * G) {
    const int ng = groups - g0 < G ? (int)(groups - g0) : G;
    // units of 512 records of a basis (two 16-byte loads per lane), dealt out over
    // the warps, the loads two units ahead of their counts
    const int nv = (int)(S >> 3), nc = (nv + 63) >> 6, units = ng * 27 * nc;
    auto fetch = [&](int u, uint4 (&q)[2]) {
      const int b = u / nc, v = (u - b * nc) * 64 + lane;
      const uint4 *r4 = reinterpret_cast<const uint4 *>(rec + (g0 * 27 + b) * S) + v;
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (u < units && v + 32 * k < nv) q[k] = __ldcs(r4 + 32 * k);
    };
    uint4 q0[2], q1[2], q2[2];
    fetch(warp, q0);
    fetch(warp + W, q1);
    for (int u = warp; u < units; u += W) {
      fetch(u + 2 * W, q2);
      const int b = u / nc, v = (u - b * nc) * 64 + lane;
      uint32_t *row = h + b * (d >> 1);
      auto add = [&](uint32_t o) {
        if (o < (uint32_t)d) atomicAdd(&row[o >> 1], 1u << ((o & 1u) << 4));
        else bad = true;
      };
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (v + 32 * k < nv) {
          add(q0[k].x & 0xFFFFu); add(q0[k].x >> 16); add(q0[k].y & 0xFFFFu); add(q0[k].y >> 16);
          add(q0[k].z & 0xFFFFu); add(q0[k].z >> 16); add(q0[k].w & 0xFFFFu); add(q0[k].w >> 16);
        }
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        q0[k] = q1[k];
        q1[k] = q2[k];
      }
    }
    __syncthreads();
    const int g = t / tpg, oh = t - g * tpg;
    if (g < ng) {
      int32_t x[3][16];
#pragma unroll
      for (int p = 0; p < 48; ++p) x[p / 16][p % 16] = 0;
      uint4 *src = h4 + (size_t)g * 27 * tpg + oh;
#pragma unroll
      for (int al = 0; al < 27; ++al) {
        const uint4 q = src[al * tpg];
        src[al * tpg] = make_uint4(0, 0, 0, 0);
        int32_t v[4] = {(int32_t)q.x, (int32_t)q.y, (int32_t)q.z, (int32_t)q.w};
        passes::wht<2>(v);
#pragma unroll
        for (int m = 0; m < 4; ++m) x[al % 3][passes::block_pauli(al / 3, m, 2)] += v[m];
      }
      uint4 *o4 = reinterpret_cast<uint4 *>(out + ((g0 + g) * tpg + oh) * 64);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          int32_t one = 0, diff[3];
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            const int32_t y = x[a][2 * k + j], lo = (int16_t)y, hi = (y - lo) >> 16;
            one += lo + hi;
            diff[a] = lo - hi;
          }
          w[2 * j] = ((uint32_t)one & 0xFFFFu) | ((uint32_t)diff[0] << 16);
          w[2 * j + 1] = ((uint32_t)diff[1] & 0xFFFFu) | ((uint32_t)diff[2] << 16);
        }
        o4[k] = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
    __syncthreads();
  }
  if (bad) latch(status, LRE_ERR_INVALID_ARG);
}

}  // namespace

lre_status tile_bucket_run(lre_ctx *ctx, const uint16_t *records, int64_t tile_rows, int64_t shots, int n,
                           uint16_t *entries, int32_t *offs, cudaStream_t s) {
  if (n < 7 || n > 14 || shots <= 0 || (int64_t)729 * shots >= (1ll << 31)) return LRE_ERR_UNSUPPORTED;
  static_assert(MAX_BUCKETS >= (2 << 8), "two buckets per tile at n = 14");
  if (tile_rows <= 0) return LRE_OK;
  if (shots % 8 != 0 || (reinterpret_cast<uintptr_t>(records) & 15) != 0) return LRE_ERR_UNSUPPORTED;
  int grid = ctx->num_sms * 2;
  if (grid > tile_rows) grid = (int)tile_rows;
  const size_t smem = (size_t)BUCKET_WARPS * (2 << (n - 6)) * sizeof(int32_t);
  Launch L(ctx, "tile_bucket", s);
  // the limit is the function's, shared by all threads: always the largest (n = 14)
  constexpr int most = BUCKET_WARPS * (2 << 8) * (int)sizeof(int32_t);
  cudaFuncSetAttribute(tile_bucket_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  tile_bucket_kernel<<<grid, BUCKET_THREADS, smem, s>>>(records, tile_rows, shots, n, entries, offs, ctx->d_status);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? LRE_OK : cuda_fail(ctx, e, "tile bucket launch");
}

// Both sides measured, whole estimate (us, this path / dense counts):
//   n = 9 to 12, rows of 16-byte multiples, int16 sums: n = 9, 1000 shots 60 / 78 (999
//     shots); n = 11, 1000 shots 401 / 486;
//   n = 8 has 243 groups of 27, 31 CTAs: 61 / 41; n = 7, 6 CTAs: 92 / 30;
//   sums past 16 bits are stored and read at twice the width: n = 12, 2000 shots 3005 /
//     2340; n = 11, 2000 shots 634 / 600;
//   rows off the 16-byte boundary load two bytes a lane: n = 11, 1003 shots 609 / 585.
namespace {
// what the kernel itself needs: its bins and sums in 16 bits, whole vector loads
bool records_fold_fits(const void *records, int n, int64_t shots) {
  return n >= 9 && n <= 12 && shots > 0 && shots <= 32767 / 27 && (shots & 7) == 0 &&
         (reinterpret_cast<uintptr_t>(records) & 15) == 0;
}
}  // namespace

bool records_fold_takes(lre_ctx *ctx, const void *records, int n, int64_t shots, size_t dense_bytes) {
  return ctx->first_variant == 1 && ctx->generic_tma && records_fold_fits(records, n, shots) &&
         dense_bytes >= (size_t)ipow(6, n - 3) * 64 * 2;
}

lre_status records_fold_run(lre_ctx *ctx, const uint16_t *records, int64_t shots, int n, void *sums, void *out,
                            cudaStream_t s) {
  if (!records_fold_fits(records, n, shots)) return LRE_ERR_UNSUPPORTED;
  const int64_t groups = ipow(3, n - 3);
  const int threads = n == 12 ? 512 : 256, per = n == 12 ? 1 : 2048 >> n;
  const size_t smem = (size_t)(n == 12 ? 2 * RF_CELLS : RF_CELLS) * 2;
  int64_t grid = (groups + per - 1) / per;
  const int64_t cap = (int64_t)ctx->num_sms * (n == 12 ? 1 : 2);
  if (grid > cap) grid = cap;
  {
    Launch L(ctx, "records_fold3", s);
    // as above
    cudaError_t e =
        cudaFuncSetAttribute(records_fold3, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * RF_CELLS * (int)sizeof(uint16_t));
    if (e == cudaSuccess) {
      records_fold3<<<(unsigned)grid, threads, smem, s>>>(records, shots, n, groups, static_cast<int16_t *>(sums),
                                                          ctx->d_status);
      e = cudaGetLastError();
    }
    if (e != cudaSuccess) return cuda_fail(ctx, e, "records fold launch");
  }
  // qubits 4..6: the six-qubit pass's output
  passes::GenParams gp;
  gp.in = sums;
  gp.out = out;
  gp.C = 64;
  gp.r = n - 3;
  gp.n = n;
  gp.n_oh = 1ll << (n - 6);
  gp.items = ipow(3, n - 6) * gp.n_oh * gp.C;
  gp.T = nullptr;
  gp.status = ctx->d_status;
  return passes::tma_pass(ctx, gp, 3, passes::T_I16, passes::T_I32, passes::M_STORE, false, s);
}

}  // namespace lre
