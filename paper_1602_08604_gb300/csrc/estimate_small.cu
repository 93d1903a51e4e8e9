// Steps (i)+(ii) for n <= 6 with uniform shots in one launch of one CTA.
//
// At these sizes (at most 46,656 counts) the pass-per-launch form is four to
// seven dependent launches of a CTA or two, and their launches and drains are
// all of its time.  Here the partial sums stay in shared memory between the
// fold passes (two qubits at a time), the last pass writes theta and leaves the
// exact integers T = S 3^(n-k) in a shared tile, and the assembly butterflies
// run on that tile; only the counts, theta and rho touch HBM.  Same integers,
// same division and same final scale as the passes (passes.cuh), so the results
// are the same bits.  One CTA: an n = 6 instance reads 187 KB, about 2 us of one
// SM's share of the bandwidth, less than a grid-wide barrier per pass would
// cost.  n = 4: 18.4 us a call as passes; 3.1 us on the device, the host's 5 us hide it.
#include <cuda_runtime.h>

#include "lre_internal.cuh"
#include "passes.cuh"
#include "sm103.cuh"

namespace lre {
namespace {

using namespace passes;

struct SmallArgs {
  const void *counts;
  double *theta;
  float2 *rho;      // or nullptr
  int64_t total;    // N 3^n
  LastScale scale;
  int *status;
  double recip[7];  // RN(1 / (N 3^k))
  int64_t dint[7];  // N 3^k
  int64_t up3[7];   // 3^(n-k)
};

__host__ __device__ constexpr int pw(int b, int e) { return e == 0 ? 1 : b * pw(b, e - 1); }
template <int N>
__host__ __device__ constexpr int es_threads() {
  return N <= 3 ? 64 : N == 4 ? 128 : N == 5 ? 256 : 512;
}
// Values after the passes over the first 2 and the first 4 qubits, as int32.
template <int N>
__host__ __device__ constexpr int es_buf_a() {
  return N > 2 ? pw(6, N - 2) * 16 : 0;
}
template <int N>
__host__ __device__ constexpr int es_buf_b() {
  return N > 4 ? pw(6, N - 4) * 256 : 0;
}
// The assembly's tile shares the first buffer.
template <int N>
__host__ __device__ constexpr int es_first_bytes() {
  const int tile = (pw(4, N) + pw(4, N) / 16 + 1) * 16, a = es_buf_a<N>() * 4;
  return ((tile > a ? tile : a) + 15) / 16 * 16;
}
template <int N>
__host__ __device__ constexpr int es_smem() {  // then the parity sums
  return es_first_bytes<N>() + es_buf_b<N>() * 4 + pw(4, N) * 4;
}

// Sums of one item of a pass over J qubits, R of them left before it: the
// layout of fold_item with C = 4^(N-R).  FIRST: counts in HBM (C = 1), a row's
// 2^J outcomes as one vector.
template <int N, int R, int J, bool FIRST, typename InT>
__device__ __forceinline__ void es_item(const InT *in, int item, int32_t (&acc)[1 << (2 * J)]) {
  constexpr int C = pw(4, N - R), NA = pw(3, J), NO = 1 << J, OH = 1 << (R - J);
  const int c = item % C, ahoh = item / C, oh = ahoh % OH, ah = ahoh / OH;
  const InT *p = in + (((ah * NA) << R) + oh * NO) * C + c;
#pragma unroll
  for (int q = 0; q < 1 << (2 * J); ++q) acc[q] = 0;
#pragma unroll
  for (int al = 0; al < NA; ++al) {
    int32_t v[NO];
    if constexpr (FIRST && J == 2) {
      ld_row_vec<NO>(p + (al << R), v);
    } else if constexpr (FIRST) {
#pragma unroll
      for (int o = 0; o < NO; ++o) v[o] = (int32_t)p[(al << R) + o];
    } else {
#pragma unroll
      for (int o = 0; o < NO; ++o) v[o] = (int32_t)p[((al << R) + o) * C];
    }
    wht<J>(v);
#pragma unroll
    for (int m = 0; m < NO; ++m) acc[block_pauli(al, m, J)] += v[m];
  }
}

template <int N, int R, int J, bool FIRST, typename InT>
__device__ __forceinline__ void es_pass(const InT *in, int32_t *out) {
  constexpr int C = pw(4, N - R), NP = 1 << (2 * J), items = pw(6, R - J) * C;
  for (int item = threadIdx.x; item < items; item += es_threads<N>()) {
    int32_t acc[NP];
    es_item<N, R, J, FIRST>(in, item, acc);
    const int o = item / C * NP * C + item % C;
#pragma unroll
    for (int q = 0; q < NP; ++q) out[o + q * C] = acc[q];
  }
  __syncthreads();
}

struct SmallTab {
  double recip[7];
  int64_t dint[7], up3[7];
  uint64_t dn[7];
  int ld[7];
};

template <int N, typename InT>
__global__ void __launch_bounds__(es_threads<N>()) estimate_small(const __grid_constant__ SmallArgs P) {
  constexpr int T = es_threads<N>();
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ SmallTab tab;
  int32_t *A = reinterpret_cast<int32_t *>(smem);
  int32_t *B = reinterpret_cast<int32_t *>(smem + es_first_bytes<N>());
  longlong2 *tile = reinterpret_cast<longlong2 *>(smem);
  const InT *counts = static_cast<const InT *>(P.counts);
  const int t = threadIdx.x;
  if (t < 7) {
    tab.recip[t] = P.recip[t];
    tab.dint[t] = P.dint[t];
    tab.up3[t] = P.up3[t];
    const int64_t d = P.dint[t] > 0 ? P.dint[t] : 1;
    tab.ld[t] = 63 - __clzll(d);
    tab.dn[t] = (uint64_t)d << (63 - tab.ld[t]);
  }
  sm103::pdl_wait();
  __syncthreads();
  sm103::pdl_trigger();
  // ---- fold
  int32_t *S = B + es_buf_b<N>();
  if constexpr (N <= 2) {
    es_pass<N, N, N, true>(counts, S);
  } else if constexpr (N <= 4) {
    es_pass<N, N, 2, true>(counts, A);
    es_pass<N, N - 2, N - 2, false>(A, S);
  } else {
    es_pass<N, N, 2, true>(counts, A);
    es_pass<N, N - 2, 2, false>(A, B);
    es_pass<N, N - 4, N - 4, false>(B, S);
  }
  // ---- theta, and T into the tile: a division is a hundred instructions, so its
  // outputs are dealt out over all threads and not left with the few that summed them
  for (int i = t; i < pw(4, N); i += T) {
    const int32_t s = S[i];
    const int k = identity_letters((uint64_t)i, N);
    if (i == 0 && s != P.total) latch(P.status, LRE_ERR_SHOTS_MISMATCH);
    P.theta[i] = div_int_rn((int64_t)s, tab.dint[k], tab.recip[k], tab.ld[k], tab.dn[k]);
    if (P.rho) tile[pad16(i)] = mk((long long)s * tab.up3[k], 0ll);
  }
  if (!P.rho) return;
  __syncthreads();
  // ---- assembly: two letters at a time, in place, then the odd one
#pragma unroll
  for (int q = 0; q + 2 <= N; q += 2) {
    const int sh = 2 * q;
    for (int it = t; it < pw(4, N) / 16; it += T) {
      const int lo = it & ((1 << sh) - 1), hi = it >> sh;
      longlong2 v[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) v[u] = tile[pad16(lo | (u << sh) | (hi << (sh + 4)))];
      m2(v);
#pragma unroll
      for (int u = 0; u < 16; ++u) tile[pad16(lo | (u << sh) | (hi << (sh + 4)))] = v[u];
    }
    __syncthreads();
  }
  if constexpr (N % 2 == 1) {
    constexpr int sh = 2 * (N - 1);
    for (int lo = t; lo < (1 << sh); lo += T) {
      longlong2 a, b, c, d;
      m_qubit(tile[pad16(lo)], tile[pad16(lo | (1 << sh))], tile[pad16(lo | (2 << sh))], tile[pad16(lo | (3 << sh))],
              a, b, c, d);
      tile[pad16(lo)] = a;
      tile[pad16(lo | (1 << sh))] = b;
      tile[pad16(lo | (2 << sh))] = c;
      tile[pad16(lo | (3 << sh))] = d;
    }
    __syncthreads();
  }
  for (int o = t; o < pw(4, N); o += T) {
    const int R = o >> N, Cc = o & ((1 << N) - 1);
    int pos = 0;
#pragma unroll
    for (int q = 0; q < N; ++q) pos |= ((((R >> q) & 1) << 1) | ((Cc >> q) & 1)) << (2 * q);
    P.rho[o] = to_c64(tile[pad16(pos)], P.scale);
  }
}

template <int N>
lre_status launch_small(lre_ctx *ctx, const SmallArgs &a, bool i16, cudaStream_t s) {
  constexpr int smem = es_smem<N>();
  auto k = i16 ? estimate_small<N, int16_t> : estimate_small<N, int32_t>;
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "small estimate");
  }
  Launch L(ctx, "estimate_small", s);
  const cudaError_t e = launch_pdl(true, k, 1, es_threads<N>(), smem, s, a);
  return e == cudaSuccess ? LRE_OK : cuda_fail(ctx, e, "small estimate launch");
}

}  // namespace

bool estimate_small_takes(const void *counts, int n, int64_t shots) {
  // int32 sums throughout; the vector loads of a row's four counts
  return n <= 6 && (reinterpret_cast<uintptr_t>(counts) & 15) == 0 &&
         (double)ipow(3, n) * (double)shots < 2147483647.0;
}

lre_status estimate_small_run(lre_ctx *ctx, const void *counts, lre_count_kind kind, int n, int64_t shots,
                              double *theta, lre_c64 *rho, cudaStream_t s) {
  SmallArgs a{};
  a.counts = counts;
  a.theta = theta;
  a.rho = reinterpret_cast<float2 *>(rho);
  a.total = shots * ipow(3, n);
  const LastScaleArgs sc = int_assembly_scale(n, shots);
  a.scale = LastScale{sc.sh, sc.sl};
  a.status = ctx->d_status;
  for (int k = 0; k <= n; ++k) {
    a.dint[k] = shots * ipow(3, k);
    a.recip[k] = 1.0 / (double)a.dint[k];
    a.up3[k] = ipow(3, n - k);
  }
  const bool i16 = kind == LRE_COUNTS_I16;
  switch (n) {
    case 1: return launch_small<1>(ctx, a, i16, s);
    case 2: return launch_small<2>(ctx, a, i16, s);
    case 3: return launch_small<3>(ctx, a, i16, s);
    case 4: return launch_small<4>(ctx, a, i16, s);
    case 5: return launch_small<5>(ctx, a, i16, s);
    case 6: return launch_small<6>(ctx, a, i16, s);
  }
  return LRE_ERR_UNSUPPORTED;
}

}  // namespace lre
