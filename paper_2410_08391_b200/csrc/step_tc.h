// Host interface of the tensor-core projections of the base model's single-token step for
// batches too large for the CUDA-core kernels to stay bandwidth-bound (bf16 weights).
#pragma once
#include "common.cuh"

enum StepPrepMode : int { PREP_PLAIN = 0, PREP_NORM = 1, PREP_SWIGLU = 2 };

// The operand buffer holds every activation as a sum of bf16 terms, term t of row b in row t * step_tc_rows(batch, terms) + b: value and
// remainder (16 bits), or, of up to four rows, value, remainder and the remainder's remainder (24 bits).
inline int step_tc_rows(int batch, int terms = 2) { return terms == 3 ? 4 : (batch + 7) / 8 * 8; }
inline int step_tc_operand_rows(int batch, int terms = 2) { return terms == 3 ? 16 : 2 * step_tc_rows(batch); }      // (N of the products: a multiple of 16)
bool step_tc_supported(int batch, int K, int ldw, const void* W, const void* XB);

// XB[b, :] = bf16(v_b), XB[Bp + b, :] = bf16(v_b - bf16(v_b)) (and so on) for b < batch (zero rows up to Bp), where
//   PREP_PLAIN:  v_b = x[b, 0:K]
//   PREP_NORM:   v_b = gain * x[b] / sqrt(mean(x[b]^2) + eps), x plus `add` where there is one (and their sum to `out`)
//   PREP_SWIGLU: v_b[c] = silu(x[b, gate row c]) * x[b, up row c], c < K = ffn, rows placed as in the packed w_gate/w_up
// Also clears zero_ptr[b, 0:zero_n] (row stride zero_ld) for b < batch when zero_ptr is given.
//
// With three terms the partial sums of a projection onto the residual stream x (up to 24 a row) meet in a buffer of their own, and the next
// PREP_NORM adds them to x at once: added to x one by one, each sum rounds to x, which is several times as large.
struct StepSum {            // rows of K floats
  const float* add = nullptr;
  float* out = nullptr;     // (not x: other CTAs still read it)
  float* clear = nullptr;   // where the next such projection's partial sums will meet
};
void launch_step_prep(const LaunchCtx&, int mode, const float* x, int ldx, int K, int batch, int terms, const float* gain, float eps,
                      int G, bf16* XB, float* zero_ptr, int zero_ld, int zero_n, bool overlapped = true, const StepSum& sum = StepSum());

// Y[b, n] += sum_k W[n, k] (XB[b, k] + XB[Bp + b, k] + ...) for b < batch, n < N; fp32 atomic adds.
cudaError_t launch_step_gemm_tc(const bf16* W, int ldw, int N, int K, const bf16* XB, int batch, int terms, float* Y, int ldy,
                                int n_sm, int* status, cudaStream_t st, int64_t* n_launch);
