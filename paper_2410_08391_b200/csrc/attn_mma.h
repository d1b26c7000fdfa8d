// Host interface of the warp-level tensor-core prompt attention for short sequences (same operands as attn_tc.h: head_dim 64 / 128,
// row strides and addresses of whole 16-byte pieces).
#pragma once
#include "common.cuh"

// Which form a call's prompt attention takes: 0 = launch_attn_mma, 1 or 2 = launch_attn_tc with that many query tiles per CTA
// (cu_host: [batch + 1] sequence starts; heads: query heads of the widest layer).
int attn_choose(const int* cu_host, int batch, int heads, int hd);
cudaError_t launch_attn_mma(const bf16* qkv, int ld, int nq, int nkv, int hd, const int* cu_dev, int batch, int max_len, bf16* out, int ldo,
                            cudaStream_t st, int64_t* n_launch, bool half_operands = false, bf16* out_lo = nullptr);
