// The persistent Lanczos step kernel (krylov_steps.cu) as krylov.cu calls it.
#pragma once
#include "lre_internal.cuh"

namespace lre {

// Largest d of the persistent form: x and a step's working vector are held
// whole in shared memory (64 KB at 4096), and from there on a step's data
// outweigh its launches.
constexpr int64_t KRY_STEPS_MAX_D = 4096;
constexpr int64_t KRY_STEPS_MAX_ROWS = 2049;  // basis rows: d / 2 + 1 there

struct KryStepBuffers {
  const float2 *A;   // mu, row-major complex64
  float4 *Q;         // basis rows (double-float)
  float4 *Y, *W;     // [d] a step's product and its result before normalising
  float4 *H;         // [rows]
  void *sync;        // kry_sync_bytes
  int *breakdown;
  int64_t rows;      // basis rows there are
};

// CTAs of the persistent kernel for this d.
int kry_steps_grid(lre_ctx *ctx, int64_t d);

size_t kry_sync_bytes(const lre_ctx *ctx);

// Lanczos steps [j0, j1) on basis rows base + j (rows 0 .. base + j - 1 fixed),
// each orthogonalised against all earlier rows: alpha[j], beta[j] and row
// base + j + 1.  Enqueued on s.
lre_status kry_steps_run(lre_ctx *ctx, const KryStepBuffers &B, int64_t d, int64_t base, int j0, int j1,
                         double *alpha, double *beta, double tiny, cudaStream_t s);

// krylov_vecs.cu: herm (d x d, or NULL to leave mu as it is) = the Hermitian
// matrix of in's upper triangle; trace_norms[0] = its trace, then
// kry_norm_blocks(ctx, d) shares of its squared Frobenius norm.
int64_t kry_norm_blocks(const lre_ctx *ctx, int64_t d);
lre_status kry_prepare_mu(lre_ctx *ctx, const float2 *in, float2 *herm, int64_t d, double *trace_norms, cudaStream_t s);
// Z[k] = sum_t S[t + k J] q_t for k < m, rows of d double-float entries.
lre_status kry_ritz_run(lre_ctx *ctx, const float4 *Q, int J, const double *S, int m, float4 *Z, int64_t d,
                        cudaStream_t s);
// w[k] = the Rayleigh quotient of row k of Z to FP64 rounding (d <= KRY_STEPS_MAX_D; part: m ceil(d / 64) double2).
lre_status kry_rayleigh_run(lre_ctx *ctx, const float2 *A, const float4 *Z, int m, int64_t d, double2 *part, double *w,
                            cudaStream_t s);
// out = sum (w + shift) z z^dag (kept form) or mu + shift I - sum (w + shift) z z^dag.
lre_status kry_rebuild_run(lre_ctx *ctx, const float4 *Z, const double *w, int m, double shift, bool kept_form,
                           const float2 *mu, float2 *out, int64_t d, cudaStream_t s);

}  // namespace lre
