// Step (ii) of lre_estimate with uniform shots (exact integers), qubit 1 first.
//
// The butterfly's qubits commute, and a thread of the last fold pass holds all
// 4^J letter combinations of the top J qubits of one column, so it applies
// their maps to T = S 3^(n-k) in registers before storing: what it writes is a
// 2^J x 2^J matrix of columns, Hermitian because the column's coefficients are
// real, kept as its real diagonal blocks and the complex blocks above the
// diagonal -- 4^J integers, as many as T itself, with J qubits done for nothing.
// The other m = n - J qubits then run per block: six through a shared tile, the
// rest two to four at a time on square tiles, the last of them writing rho and,
// from the same tile, the conjugate transpose below the diagonal.  Against the
// passes of assemble.cu on T (which lre_assemble keeps for FP64 theta, and the
// first passes it shares) that is one pass less, no mirror pass, and blocks below
// the diagonal never formed.  Every value is an exact integer until the one
// final scale, so rho is the same bits.
//
// n = 12: the assembly 228 -> 151 us (two passes, 2.4 and 3.2 TB/s; their
// shared-memory rounds at two CTAs an SM bound them), the last fold pass, two
// qubits instead of three, 418 -> 96 us and one more one-qubit pass 70; n = 13: 973
// -> 654 us of assembly; n = 7: six launches -> three, 36 -> 23 us a call.
//
// Layout of the last fold pass's output, C = 4^m: [2^J][C] int64 diagonal
// blocks, then [2^J (2^J - 1) / 2][C] complex blocks (R, S), R < S, row by row.
// Intermediates: [block][P' 4^(m-t)][R 2^t][C 2^t] complex, t qubits done.  A
// diagonal block is Hermitian itself: of it only the tiles with
// (R mod 64) / 16 <= (C mod 64) / 16 are formed (herm_tile; 32 instead of 16
// where a pass has 32-wide tiles); the others are the mirrors of formed ones.
#include <cuda_runtime.h>

#include "lre_internal.cuh"
#include "passes.cuh"
#include "sm103.cuh"

namespace lre {
namespace {

using namespace passes;
using V = longlong2;

__device__ __forceinline__ int pair_index(int R, int S, int B) { return R * (2 * B - R - 1) / 2 + S - R - 1; }

// ---- the last fold pass ---------------------------------------------------------
template <int J, typename InT, typename AccT>
__global__ void __launch_bounds__(256) fold_final_top(GenParams P) {
  constexpr int NP = 1 << (2 * J), B = 1 << J;
  __shared__ DivTables tab;
  load_div_tables(P, tab);
  sm103::pdl_wait();
  __syncthreads();
  sm103::pdl_trigger();
  double *theta = static_cast<double *>(P.out);
  long long *diag = reinterpret_cast<long long *>(P.T);
  V *off = reinterpret_cast<V *>(diag + B * P.C);
  for (int64_t item = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; item < P.C;
       item += (int64_t)gridDim.x * blockDim.x) {
    AccT acc[NP];
    int64_t ahoh, c;
    fold_sums<J, InT, AccT, false>(P, item, acc, ahoh, c);
    long long T[NP];
    const int kc = identity_letters((uint64_t)c, P.n - J);  // identities among the column's letters
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      int kp = 0;
#pragma unroll
      for (int q = 0; q < J; ++q) kp += ((p >> (2 * q)) & 3) == 0;
      const int k = kc + kp;
      const int64_t i = p * P.C + c;
      if (i == 0 && (int64_t)acc[p] != P.total) latch(P.status, LRE_ERR_SHOTS_MISMATCH);
      // both forms are correctly rounded (fold_emit): every third output on the
      // FP64 pipe, the others on the integer ALUs
      theta[i] = p % 3 == 0 ? div_by_recip((double)acc[p], tab.denom[k], tab.recip[k])
                            : div_int_rn((int64_t)acc[p], tab.dint[k], tab.recip[k], tab.ld[k], tab.dn[k]);
      T[p] = (long long)acc[p] * tab.up3[k];
    }
    // letters I, X, Y, Z (real) -> 00 = I + Z, 11 = I - Z, 01 = X - iY
    if constexpr (J == 1) {
      diag[c] = T[0] + T[3];
      diag[P.C + c] = T[0] - T[3];
      off[c] = mk(T[1], -T[2]);
    } else {
      // digit 0 -> per letter of digit 1: real 00, real 11, complex 01
      long long h0[4], h1[4];
      V h2[4];
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        h0[p] = T[4 * p] + T[4 * p + 3];
        h1[p] = T[4 * p] - T[4 * p + 3];
        h2[p] = mk(T[4 * p + 1], -T[4 * p + 2]);
      }
      // digit 1 (the top bit of the block's row and column)
      diag[c] = h0[0] + h0[3];
      diag[2 * P.C + c] = h0[0] - h0[3];
      diag[P.C + c] = h1[0] + h1[3];
      diag[3 * P.C + c] = h1[0] - h1[3];
      off[pair_index(0, 2, 4) * P.C + c] = mk(h0[1], -h0[2]);
      off[pair_index(1, 3, 4) * P.C + c] = mk(h1[1], -h1[2]);
      V a, b, x, y;
      m_qubit(h2[0], h2[1], h2[2], h2[3], a, x, y, b);  // 00, 01, 10, 11
      off[pair_index(0, 1, 4) * P.C + c] = a;
      off[pair_index(2, 3, 4) * P.C + c] = b;
      off[pair_index(0, 3, 4) * P.C + c] = x;
      off[pair_index(1, 2, 4) * P.C + c] = mk(y.x, -y.y);  // the mirror of (2, 1)
    }
  }
}

// ---- blocks ------------------------------------------------------------------------
struct TopArgs {
  const void *in;  // the last fold pass's output, or intermediates
  void *out;       // intermediates, or rho
  int J, n, t;     // top qubits, all qubits, low qubits done before this pass
  int gsh;         // log2 of herm_tile's granularity, at least the widest tile's
  int64_t units;
  LastScale scale;
};

struct Block {
  int R, S;  // block row and column, R <= S
};
__device__ __forceinline__ Block block_of(int b, int B) {  // diagonal blocks first
  if (b < B) return {b, b};
  b -= B;
  int R = 0;
  while (b >= B - 1 - R) {
    b -= B - 1 - R;
    ++R;
  }
  return {R, R + 1 + b};
}
// Tiles of a diagonal block that are formed, by the low six bits.
__device__ __forceinline__ bool herm_tile(int64_t R, int64_t C, int gsh) {
  return ((R & 63) >> gsh) <= ((C & 63) >> gsh);
}

__device__ __forceinline__ V load_block(const void *in, int64_t C, int B, int b, int64_t i) {
  if (b < B) return mk(__ldcg(static_cast<const long long *>(in) + b * C + i), 0ll);
  return __ldcg(reinterpret_cast<const V *>(static_cast<const long long *>(in) + B * C) + (b - B) * C + i);
}

// Low qubits 0..5 of 4096 consecutive columns of a block.
template <bool LAST>
__global__ void __launch_bounds__(256) top_low6(TopArgs P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V *S = reinterpret_cast<V *>(smem_raw);
  const int B = 1 << P.J, m = P.n - P.J, tid = threadIdx.x;
  const int64_t C = 1ll << (2 * m), per = C >> 12;
  sm103::pdl_wait();
  sm103::pdl_trigger();
  for (int64_t u = blockIdx.x; u < P.units; u += gridDim.x) {
    const int b = (int)(u / per);
    const int64_t Pp = u - b * per;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const int i = tid + 256 * k;
      S[pad16(i)] = load_block(P.in, C, B, b, Pp * 4096 + i);
    }
    __syncthreads();
    if (b < B) asm_low6_rounds<true>(S);
    else asm_low6_rounds<false>(S);
    const Block bl = block_of(b, B);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const int o = tid + 256 * k, r = o >> 6, c = o & 63;
      const V v = S[pad16(low6_place(r, c))];
      if constexpr (LAST) {  // m = 6: the block is rho's
        float2 *rho = static_cast<float2 *>(P.out);
        const int64_t W = 1ll << P.n;
        rho[(bl.R * 64 + r) * W + bl.S * 64 + c] = to_c64(v, P.scale);
        if (bl.R != bl.S) {
          const V w = S[pad16(low6_place(c, r))];
          rho[(bl.S * 64 + r) * W + bl.R * 64 + c] = to_c64(mk(w.x, -w.y), P.scale);
        }
      } else if (bl.R != bl.S || herm_tile(r, c, P.gsh)) {
        static_cast<V *>(P.out)[(b * per + Pp) * 4096 + o] = v;
      }
    }
    __syncthreads();
  }
}

// Low qubits t .. t + Q - 1 of a block on square tiles: TD x TD entries of
// [R][C] times 4^Q letters = 4096 values, sixteen per thread.
template <int Q, bool LAST>
__global__ void __launch_bounds__(256) top_high(TopArgs P) {
  constexpr int TD = Q == 4 ? 4 : Q == 3 ? 8 : Q == 2 ? 16 : 32, L = TD * TD, NQ = 1 << (2 * Q);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V *S = reinterpret_cast<V *>(smem_raw);
  const int B = 1 << P.J, m = P.n - P.J, t = P.t, tid = threadIdx.x;
  const int64_t side = 1ll << t, L4 = side * side, tiles = side / TD;
  const int64_t per_b = (1ll << (2 * (m - t - Q))) * tiles * tiles;
  const int64_t C = 1ll << (2 * m), W = side << Q;
  sm103::pdl_wait();
  sm103::pdl_trigger();
  for (int64_t u = blockIdx.x; u < P.units; u += gridDim.x) {
    const int b = (int)(u / per_b);
    const int64_t x = u - b * per_b, Pp = x / (tiles * tiles), y = x - Pp * tiles * tiles;
    const int64_t R0 = y / tiles * TD, C0 = (y - y / tiles * tiles) * TD;
    const Block bl = block_of(b, B);
    if (bl.R == bl.S && !herm_tile(R0, C0, P.gsh)) continue;
    const V *src = static_cast<const V *>(P.in) + b * C + Pp * NQ * L4 + R0 * side + C0;
    // digits 0, 1 of the letters (Q = 1: digit 0), straight from memory
    V v[16];
    if constexpr (Q == 1) {
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        const int l = tid + 256 * g;
#pragma unroll
        for (int w = 0; w < 4; ++w) v[4 * g + w] = __ldcg(src + w * L4 + (l / TD) * side + (l % TD));
        V a, bb, cc, d;
        m_qubit(v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3], a, bb, cc, d);
        S[pad16(0 * L + l)] = a;
        S[pad16(1 * L + l)] = bb;
        S[pad16(2 * L + l)] = cc;
        S[pad16(3 * L + l)] = d;
      }
    } else {
      const int l = tid % L, h = tid / L;
      const V *q = src + (int64_t)(h * 16) * L4 + (l / TD) * side + (l % TD);
#pragma unroll
      for (int w = 0; w < 16; ++w) v[w] = __ldcg(q + w * L4);
      m2(v);
#pragma unroll
      for (int w = 0; w < 16; ++w) S[pad16((w | (h << 4)) * L + l)] = v[w];
    }
    __syncthreads();
    if constexpr (Q == 4) {  // digits 2, 3
      const int l = tid % L, h = tid / L;
#pragma unroll
      for (int w = 0; w < 16; ++w) v[w] = S[pad16((h | (w << 4)) * L + l)];
      m2(v);
#pragma unroll
      for (int w = 0; w < 16; ++w) S[pad16((h | (w << 4)) * L + l)] = v[w];
      __syncthreads();
    } else if constexpr (Q == 3) {  // digit 2
      const int l = tid % L, h = tid / L;
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        V a, bb, cc, d;
        const int p = 4 * h + g;
        m_qubit(S[pad16(p * L + l)], S[pad16((p | 16) * L + l)], S[pad16((p | 32) * L + l)], S[pad16((p | 48) * L + l)],
                a, bb, cc, d);
        S[pad16(p * L + l)] = a;
        S[pad16((p | 16) * L + l)] = bb;
        S[pad16((p | 32) * L + l)] = cc;
        S[pad16((p | 48) * L + l)] = d;
      }
      __syncthreads();
    }
    // letters (digit q = 2 r_q + c_q) -> rows and columns
    auto place = [&](int rJ, int cJ) {
      int p = 0;
#pragma unroll
      for (int q = 0; q < Q; ++q) p |= ((((rJ >> q) & 1) << 1) | ((cJ >> q) & 1)) << (2 * q);
      return p;
    };
    const bool mirror = bl.R != bl.S || !herm_tile(C0, R0, P.gsh);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const int e = tid + 256 * k;  // (rJ, r, cJ, c), c fastest
      const int c = e % TD, cJ = (e / TD) % (1 << Q), r = (e / (TD << Q)) % TD, rJ = e / (L << Q);
      const V o = S[pad16(place(rJ, cJ) * L + r * TD + c)];
      const int64_t R = ((int64_t)rJ << t) | (R0 + r), Cc = ((int64_t)cJ << t) | (C0 + c);
      if constexpr (LAST) {
        float2 *rho = static_cast<float2 *>(P.out);
        const int64_t N = 1ll << P.n;
        rho[(bl.R * W + R) * N + bl.S * W + Cc] = to_c64(o, P.scale);
        if (mirror) {  // the same sweep over the transposed tile
          const V z = S[pad16(place(cJ, rJ) * L + c * TD + r)];
          const int64_t Rm = ((int64_t)rJ << t) | (C0 + r), Cm = ((int64_t)cJ << t) | (R0 + c);
          rho[(bl.S * W + Rm) * N + bl.R * W + Cm] = to_c64(mk(z.x, -z.y), P.scale);
        }
      } else {
        static_cast<V *>(P.out)[b * C + Pp * W * W + R * W + Cc] = o;
      }
    }
    __syncthreads();
  }
}

template <int Q>
void launch_high(bool last, const TopArgs &a, int grid, cudaStream_t s) {
  auto k = last ? top_high<Q, true> : top_high<Q, false>;
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, ASM_TILE_SMEM);
  launch_pdl(overlaps(a.n), k, grid, 256, ASM_TILE_SMEM, s, a);
}

}  // namespace

lre_status fold_final_top_run(lre_ctx *ctx, const passes::GenParams &P, int J, int in_t, int acc_t, cudaStream_t s) {
  if (J < 1 || J > 2 || P.top7 || !P.T) return LRE_ERR_UNSUPPORTED;
  // few columns: small CTAs, so that they spread over the SMs
  const int threads = P.C <= (int64_t)ctx->num_sms * 256 ? 64 : 256;
  int64_t blocks = (P.C + threads - 1) / threads;
  const int64_t cap = (int64_t)ctx->num_sms * 64;
  if (blocks > cap) blocks = cap;
  void (*k)(GenParams) = nullptr;
  if (in_t == T_I32 && acc_t == T_I32) k = J == 1 ? fold_final_top<1, int32_t, int32_t> : fold_final_top<2, int32_t, int32_t>;
  if (in_t == T_I32 && acc_t == T_I64) k = J == 1 ? fold_final_top<1, int32_t, int64_t> : fold_final_top<2, int32_t, int64_t>;
  if (in_t == T_I64 && acc_t == T_I64) k = J == 1 ? fold_final_top<1, int64_t, int64_t> : fold_final_top<2, int64_t, int64_t>;
  if (!k) return LRE_ERR_UNSUPPORTED;
  {
    Launch L(ctx, "fold_final", s);
    launch_pdl(overlaps(P.n), k, blocks, threads, 0, s, P);
  }
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? LRE_OK : cuda_fail(ctx, e, "last fold pass launch");
}

lre_status assemble_top_run(lre_ctx *ctx, const int64_t *T, int n, int J, int64_t shots, lre_c64 *rho, void *ws,
                            cudaStream_t s) {
  const LastScaleArgs sc = int_assembly_scale(n, shots);
  const int m = n - J, B = 1 << J;
  const int64_t blocks = B * (B + 1) / 2;
  const size_t one = (((size_t)1 << (2 * n)) * sizeof(V) + 255) & ~(size_t)255;
  char *bufs[2] = {static_cast<char *>(ws), static_cast<char *>(ws) + one};
  TopArgs a{};
  a.in = T;
  a.J = J;
  a.n = n;
  a.t = 0;
  a.gsh = m == 7 ? 5 : 4;  // m = 7 ends in a pass over one qubit, on 32-wide tiles
  a.scale = LastScale{sc.sh, sc.sl};
  auto grid = [&](int64_t units) {
    const int64_t g = (int64_t)ctx->num_sms * 4;
    return (int)(units < g ? units : g);
  };
  a.units = blocks << (2 * (m - 6));
  a.out = m == 6 ? static_cast<void *>(rho) : static_cast<void *>(bufs[0]);
  {
    Launch L(ctx, "assemble_low6", s);
    auto k = m == 6 ? top_low6<true> : top_low6<false>;
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, ASM_TILE_SMEM);
    launch_pdl(overlaps(n), k, grid(a.units), 256, ASM_TILE_SMEM, s, a);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(ctx, e, "assembly launch");
  int t = 6, k = 1;
  while (t < m) {
    // up to four at a time, five as 3 + 2 and six as 3 + 3: the wider tiles move
    // whole lines
    const int left = m - t, Q = left <= 4 ? left : 3;
    const bool last = left == Q;
    a.in = a.out;
    a.out = last ? static_cast<void *>(rho) : static_cast<void *>(bufs[k & 1]);
    a.t = t;
    const int64_t tiles = (1ll << t) / (Q == 4 ? 4 : Q == 3 ? 8 : Q == 2 ? 16 : 32);
    a.units = (blocks << (2 * (m - t - Q))) * tiles * tiles;
    {
      Launch L(ctx, last ? "assemble_last" : "assemble_high", s);
      const int g = grid(a.units);
      switch (Q) {
        case 1: launch_high<1>(last, a, g, s); break;
        case 2: launch_high<2>(last, a, g, s); break;
        case 3: launch_high<3>(last, a, g, s); break;
        default: launch_high<4>(last, a, g, s); break;
      }
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(ctx, e, "assembly launch");
    t += Q;
    ++k;
  }
  return LRE_OK;
}

}  // namespace lre
