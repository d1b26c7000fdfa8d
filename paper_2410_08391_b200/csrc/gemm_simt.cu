// CUDA-core GEMM  D[M,N] = A[M,K] * W[N,K]^T  with fp32 accumulation, and CUDA-core
// causal attention.  They are the fp32-mode kernels (no tensor-core type multiplies in
// fp32) and the generic path for shapes the tensor-core kernels do not take.
#include "common.cuh"

namespace {
// TS x TS tile, 256 threads, R x R outputs per thread (R = TS / 16).  A thread stages 8 consecutive k of one row of each operand; the
// next k block is on its way to registers while this one is multiplied.  Small problems are a chain of memory latencies: 32 x 32
// tiles with 64 k at a time give them four times the CTAs and a quarter of the trips.
// Every output is one chain of multiply-adds in the order of k, whatever the tile.
// fp32 mode is a chain of launches of 2 to 4 us each, so what surrounds a product is part of it there:
//   g.gain     the rows of A are RMS-normalised: products take x gain, the CTA sums its rows' squares as it reads them (all of k passes
//              through every CTA) and scales its outputs by 1 / rms
//   EPI_ROPE   tile columns 2 i and 2 i + 1 are the two halves of one rotated pair, whichever columns of W those are
//   EPI_GATED  ... are the gate and the up column of one output
// (with launches of their own for the four: 64 x 16 tokens 100.6 -> 96.1 us, 8 x 100 84.9 -> 81.8, 1 x 64 45.3 -> 44.1).
template <class T, int EPI, int TS>
__device__ __forceinline__ void gemm_simt_tile(const GemmArgs& g, const InvFreq* inv, int vec) {
  constexpr int R = TS / 16, BK = 2048 / TS, KT = BK / 8;
  __shared__ __align__(16) float As[BK][TS + 4];
  __shared__ __align__(16) float Ws[BK][TS + 4];
  __shared__ float rinv[TS];
  constexpr bool PAIRED = EPI == EPI_ROPE || EPI == EPI_GATED;
  const T* __restrict__ A = (const T*)g.A;
  const T* __restrict__ W = (const T*)g.W;
  int m0 = blockIdx.y * TS, n0 = blockIdx.x * TS;
  const T* __restrict__ A2 = (g.A2 && n0 + TS > g.split_begin) ? (const T*)g.A2 : nullptr;
  int tid = threadIdx.x;
  int tx = tid & 15, ty = tid >> 4;
  float acc[R][R] = {};
  const int lr = tid / KT, lk = (tid % KT) * 8, am = m0 + lr;
  // the row of W behind a column of the tile
  auto w_row = [&](int n) {
    if (!PAIRED || n >= g.N) return n;
    if (EPI == EPI_GATED) return map_row(n & 1 ? g.up : g.gate, n >> 1);
    const int half = g.hd >> 1, u = n >> 1, h = u / half;
    return h * g.hd + (u - h * half) + (n & 1) * half;
  };
  const int wn = w_row(n0 + lr);
  float av[8], wv[8], gv[8], ss = 0.f;
  auto load8 = [&](const T* row, bool ok, int k, float* v) {
    if (!ok || k >= g.K) {
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = 0.f;
    } else if (vec) {                        // rows of whole 16-byte pieces: K, the strides and the addresses allow it
#pragma unroll
      for (int i = 0; i < 8; i += 16 / (int)sizeof(T)) {
        const uint4 u = k + i < g.K ? *reinterpret_cast<const uint4*>(row + k + i) : make_uint4(0, 0, 0, 0);
        const T* e = reinterpret_cast<const T*>(&u);
#pragma unroll
        for (int q = 0; q < 16 / (int)sizeof(T); ++q) v[i + q] = to_f(e[q]);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = k + i < g.K ? to_f(row[k + i]) : 0.f;
    }
  };
  auto load = [&](int k0) {
    load8(A + (size_t)am * g.lda, am < g.M, k0 + lk, av);
    if (A2) {
      float a2[8];
      load8(A2 + (size_t)am * g.lda2, am < g.M, k0 + lk, a2);
#pragma unroll
      for (int i = 0; i < 8; ++i) av[i] += a2[i];
    }
    if (g.gain) {
#pragma unroll
      for (int i = 0; i < 8; ++i) gv[i] = k0 + lk + i < g.K ? g.gain[k0 + lk + i] : 0.f;
    }
  };
  load8(W + (size_t)wn * g.ldw, wn < g.N, lk, wv);
  load(0);
  for (int k0 = 0; k0 < g.K; k0 += BK) {
    if (g.gain) {
#pragma unroll
      for (int i = 0; i < 8; ++i) { ss = fmaf(av[i], av[i], ss); av[i] *= gv[i]; }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) { As[lk + i][lr] = av[i]; Ws[lk + i][lr] = wv[i]; }
    __syncthreads();
    if (k0 + BK < g.K) {
      load(k0 + BK);
      load8(W + (size_t)wn * g.ldw, wn < g.N, k0 + BK + lk, wv);
    }
#pragma unroll 16
    for (int k = 0; k < BK; ++k) {
      float a[R], w[R];
#pragma unroll
      for (int i = 0; i < R; ++i) { a[i] = As[k][ty * R + i]; w[i] = Ws[k][tx * R + i]; }
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) acc[i][j] = fmaf(a[i], w[j], acc[i][j]);
    }
    __syncthreads();
  }
  if (g.gain) {      // KT neighbouring threads have read a row
#pragma unroll
    for (int o = KT / 2; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if (tid % KT == 0) rinv[lr] = rsqrtf(ss / (float)g.K + g.eps);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < R; ++i) {
    int m = m0 + ty * R + i;
    if (m >= g.M) continue;
    if (g.gain) {
      const float r = rinv[ty * R + i];
#pragma unroll
      for (int j = 0; j < R; ++j) acc[i][j] *= r;
    }
    if (PAIRED) {
#pragma unroll
      for (int j = 0; j < R; j += 2) {
        const int n = n0 + tx * R + j;
        if (n >= g.N) continue;
        const float a = acc[i][j], b = acc[i][j + 1];
        T* row = (T*)g.C + (size_t)m * g.ldc;
        if (EPI == EPI_GATED) {
          row[n >> 1] = from_f<T>(a / (1.f + __expf(-a)) * b);
        } else {
          const int half = g.hd >> 1, u = n >> 1, h = u / half, c = u - h * half;
          float sn = 0.f, cs = 1.f;
          if (h < g.n_rot) rope_sincos(g.tok_pos[m], inv->f[c], &sn, &cs);
          row[h * g.hd + c] = from_f<T>(h < g.n_rot ? a * cs - b * sn : a);
          row[h * g.hd + c + half] = from_f<T>(h < g.n_rot ? b * cs + a * sn : b);
        }
      }
      continue;
    }
    int slot = 0;
    if (EPI == EPI_PAGED) { slot = g.paged.tok_slot[m]; if (slot < 0) continue; }
#pragma unroll
    for (int j = 0; j < R; ++j) {
      int n = n0 + tx * R + j;
      if (n >= g.N) continue;
      float v = acc[i][j];
      if (EPI == EPI_STORE) {
        ((T*)g.C)[(size_t)m * g.ldc + n] = from_f<T>(v);
      } else if (EPI == EPI_STORE32) {
        ((float*)g.C)[(size_t)m * g.ldc + n] = v;
      } else if (EPI == EPI_RESID) {
        g.X[(size_t)m * g.ldx + n] += v;
      } else {
        const PagedOut& p = g.paged;
        int s = 0;
        while (s + 1 < p.n_seg && n >= p.col0[s + 1]) ++s;
        int c = n - p.col0[s];
        int head = c / p.head_dim, dim = c - head * p.head_dim;
        if (p.bias) v += p.bias[n];
        int page = slot / PAGE_TOKENS, row = slot - page * PAGE_TOKENS;
        size_t off = (((size_t)page * p.n_kv[s] + head) * PAGE_TOKENS + row) * p.head_dim + dim;
        typedef typename KvOf<T>::type KT;     // cache element of this run dtype
        ((KT*)p.pool[s])[off] = from_f<KT>(v);
      }
    }
  }
}
template <class T, int EPI, int TS>
__global__ void __launch_bounds__(256) gemm_simt_kernel(const __grid_constant__ GemmArgs g, int vec) {
  gemm_simt_tile<T, EPI, TS>(g, nullptr, vec);
}
// The projection that leaves its heads rotated (fp32 mode; elsewhere rope_split_kernel follows the projection).
template <int TS>
__global__ void __launch_bounds__(256) gemm_rope_split_kernel(const __grid_constant__ GemmArgs g, const __grid_constant__ InvFreq inv, int vec) {
  gemm_simt_tile<float, EPI_ROPE, TS>(g, &inv, vec);
}
}  // namespace

void launch_gemm_simt(const LaunchCtx& ctx, const GemmArgs& g, int epi) {
  if (g.M == 0 || g.N == 0) return;
  // 64 x 64 tiles where they give every SM one
  const bool small = (long long)((g.N + 63) / 64) * ((g.M + 63) / 64) < 148;
  const int ts = small ? 32 : 64, per = ctx.dtype == 0 ? 4 : 8;
  const dim3 grid((g.N + ts - 1) / ts, (g.M + ts - 1) / ts);
  const int vec = g.K % per == 0 && g.lda % per == 0 && g.ldw % per == 0 && (!g.A2 || g.lda2 % per == 0) &&
                  (((uintptr_t)g.A | (uintptr_t)g.W | (uintptr_t)g.A2) & 15) == 0;
  ++*ctx.n_launch;
  // Ordinary launches.  As programmatic dependents (with this path's attention, RoPE and SwiGLU) they held SMs while they waited and
  // took longer to record: fp32 test pair, 1 x 1024 tokens 206 us a call and 700 a first one, now 144 and 572; 1 x 64 49 and 469, now
  // 45 and 438; 8 x 100 97, now 86.
#define GO(T, E) (small ? (gemm_simt_kernel<T, E, 32><<<grid, 256, 0, ctx.st>>>(g, vec)) \
                        : (gemm_simt_kernel<T, E, 64><<<grid, 256, 0, ctx.st>>>(g, vec)))
  if (epi == EPI_ROPE) {
    InvFreq inv;
    fill_inv_freq(&inv, g.hd, g.theta);
    small ? gemm_rope_split_kernel<32><<<grid, 256, 0, ctx.st>>>(g, inv, vec) : gemm_rope_split_kernel<64><<<grid, 256, 0, ctx.st>>>(g, inv, vec);
  } else if (ctx.dtype == 0) {
    if (epi == EPI_GATED) GO(float, EPI_GATED);
    else if (epi == EPI_STORE) GO(float, EPI_STORE); else if (epi == EPI_RESID) GO(float, EPI_RESID); else if (epi == EPI_STORE32) GO(float, EPI_STORE32); else GO(float, EPI_PAGED);
  } else {
    if (epi == EPI_STORE) GO(bf16, EPI_STORE); else if (epi == EPI_RESID) GO(bf16, EPI_RESID); else if (epi == EPI_STORE32) GO(bf16, EPI_STORE32); else GO(bf16, EPI_PAGED);
  }
#undef GO
}

// ---------------------------------------------------------------------------------------
// CUDA-core causal GQA attention over a ragged batch.  One CTA = 8 warps = 8 consecutive
// queries of one sequence and one q head; keys and values are staged through shared
// memory 64 at a time; online softmax in fp32 (lane = key for scores, lane = dim for PV).
// ---------------------------------------------------------------------------------------
namespace {
constexpr int AQ = 8, AKV = 64;
constexpr int ATTN_SMEM_MAX = (2 * AKV * 129 + AQ * 128) * 4;      // head_dim 128, the widest

template <class T>
__global__ void __launch_bounds__(256) attn_prefill_simt_kernel(const T* __restrict__ qkv, int ld, int nq, int nkv, int hd,
                                                                const int* __restrict__ cu, int batch, T* __restrict__ out,
                                                                int ldo, float scale) {
  extern __shared__ float smem[];
  int ldk = hd + 1;
  float* Ks = smem;                       // [AKV][hd+1]
  float* Vs = Ks + AKV * ldk;             // [AKV][hd+1]
  float* Qs = Vs + AKV * ldk;             // [AQ][hd]
  __shared__ int s_b, s_q0;
  if (threadIdx.x == 0) {
    int blk = blockIdx.x, b = 0;
    for (; b < batch; ++b) {
      int nb = (cu[b + 1] - cu[b] + AQ - 1) / AQ;
      if (blk < nb) break;
      blk -= nb;
    }
    s_b = b; s_q0 = blk * AQ;
  }
  __syncthreads();
  int b = s_b;
  if (b >= batch) return;
  int head = blockIdx.y, kvh = head / (nq / nkv);
  int base = cu[b], L = cu[b + 1] - base;
  int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int qi = s_q0 + warp;                   // query position of this warp
  bool qok = qi < L;
  if (qok)
    for (int c = lane; c < hd; c += 32) Qs[warp * hd + c] = to_f(qkv[(size_t)(base + qi) * ld + head * hd + c]) * scale;
  int koff = nq * hd + kvh * hd, voff = (nq + nkv) * hd + kvh * hd;
  float o[4] = {0.f, 0.f, 0.f, 0.f};
  float m = -INFINITY, l = 0.f;
  int kmax = min(L, s_q0 + AQ);           // keys any query of this CTA can see
  for (int k0 = 0; k0 < kmax; k0 += AKV) {
    __syncthreads();
    for (int i = threadIdx.x; i < AKV * hd; i += blockDim.x) {
      int s = i / hd, c = i - s * hd;
      int ks = k0 + s;
      float kx = 0.f, vx = 0.f;
      if (ks < kmax) {
        kx = to_f(qkv[(size_t)(base + ks) * ld + koff + c]);
        vx = to_f(qkv[(size_t)(base + ks) * ld + voff + c]);
      }
      Ks[s * ldk + c] = kx; Vs[s * ldk + c] = vx;
    }
    __syncthreads();
    if (!qok) continue;
    float sc[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      int s = lane + 32 * h, ks = k0 + s;
      float a = 0.f;
      for (int c = 0; c < hd; ++c) a = fmaf(Qs[warp * hd + c], Ks[s * ldk + c], a);
      sc[h] = (ks <= qi && ks < L) ? a : -INFINITY;
    }
    float mt = warp_max(fmaxf(sc[0], sc[1]));
    if (mt == -INFINITY) continue;
    float mn = fmaxf(m, mt);
    float alpha = __expf(m - mn);
    float p0 = __expf(sc[0] - mn), p1 = __expf(sc[1] - mn);
    l = l * alpha + warp_sum(p0 + p1);
    m = mn;
#pragma unroll
    for (int i = 0; i < 4; ++i) o[i] *= alpha;
    for (int s = 0; s < AKV; ++s) {
      float p = __shfl_sync(0xffffffffu, s < 32 ? p0 : p1, s & 31);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        int c = lane + 32 * i;
        if (c < hd) o[i] = fmaf(p, Vs[s * ldk + c], o[i]);
      }
    }
  }
  if (qok) {
    float inv = 1.f / l;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      int c = lane + 32 * i;
      if (c < hd) out[(size_t)(base + qi) * ldo + head * hd + c] = from_f<T>(o[i] * inv);
    }
  }
}
}  // namespace

void launch_attn_prefill_simt(const LaunchCtx& ctx, const void* qkv, int ld, int nq, int nkv, int hd, const int* cu_dev,
                              int batch, int total, void* out, int ldo) {
  if (total == 0) return;
  int n_blk = (total + AQ - 1) / AQ + batch;   // upper bound on sum_b ceil(L_b / AQ)
  size_t smem = (size_t)(2 * AKV * (hd + 1) + AQ * hd) * sizeof(float);
  dim3 grid(n_blk, nq);
  float scale = 1.f / sqrtf((float)hd);
  ++*ctx.n_launch;
  if (ctx.dtype == 0) {
    static bool raised[TC_MAX_DEVICES] = {};
    tc_raise_smem_limit(attn_prefill_simt_kernel<float>, ATTN_SMEM_MAX, raised);
    attn_prefill_simt_kernel<float><<<grid, 256, smem, ctx.st>>>((const float*)qkv, ld, nq, nkv, hd, cu_dev, batch, (float*)out, ldo, scale);
  } else {
    static bool raised[TC_MAX_DEVICES] = {};
    tc_raise_smem_limit(attn_prefill_simt_kernel<bf16>, ATTN_SMEM_MAX, raised);
    attn_prefill_simt_kernel<bf16><<<grid, 256, smem, ctx.st>>>((const bf16*)qkv, ld, nq, nkv, hd, cu_dev, batch, (bf16*)out, ldo, scale);
  }
}
