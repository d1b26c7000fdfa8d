// The base model's single-token step as ONE persistent cooperative kernel (batch <= 4).
//
// A step is ~170 dependent, bandwidth-bound operations of a few microseconds each; as separate
// kernels their launch and ramp-up latency is several times the time the weights need to stream
// from HBM.  Here one CTA of 16 warps per SM stays resident for the whole step.  The operations become phases:
//   per layer:  q(kv) projection (RMSNorm fused) | attention over cache pages, which takes the step's own key and value in (key-range
//               splits merged by the CTA that finishes a group's last split) | O projection + residual | gate/up + SwiGLU (RMSNorm
//               fused) | down projection + residual;   then LM head (final RMSNorm fused) + argmax.
// No grid-wide barrier stands between them: every value that crosses CTAs is one 64-bit word {fp32 value, layer tag}, and who needs
// it polls the word itself (step_waits.cuh).  With barriers, and everything that does not depend on other CTAs asked for behind them, a
// phase took 6 us on models of test size; first token of the fp32 test pair 1 x 64 45.1 -> 39.0 us, 1 x 300 61.6 -> 49.3, 4 x 250 111 -> 93.
// A word is written again, one layer on, only by who has seen values that all of its readers had a part in: every phase needs every
// output of the phase before it, and CTAs without a row (or an attention item) of a phase don't read its input.
// Weights never pass through registers on their way from HBM: every warp owns a small ring of
// shared-memory slots that it fills with bulk asynchronous copies (cp.async.bulk, completion on
// an mbarrier) of the weight rows it will need, in schedule order.  The schedule is static, so a
// warp keeps its ring full ACROSS phase boundaries: while the SMs wait for one another, or run
// attention, the first rows of the next projection are already landing.  About 190 KB per SM are
// in flight, which is what HBM latency times bandwidth asks for.
#include <math.h>

#include "common.cuh"
#include "tc_ptx.cuh"
#include "step_mega.h"
#include "step_waits.cuh"

namespace {
using namespace tcp;

constexpr int NT = 512;                 // threads per CTA, one CTA per SM
constexpr int NW = NT / 32;
constexpr int MAXG = 8;
constexpr int NSLOT = 3;                // ring slots per warp

struct GemvDesc {
  const void* W; int N, K;          // rows, row length (= leading dimension)
  int mode;                         // GEMV_STORE / GEMV_RESID / GEMV_SWIGLU
  int G, ffn;                       // SwiGLU row interleave
};

// The projection phases in schedule order: 4 per layer (q(kv), O, gate/up, down), then the LM head.
__device__ __forceinline__ GemvDesc stream_desc(const MegaParams& p, int s) {
  if (s >= 4 * p.n_layers) return GemvDesc{p.lm_head, p.vocab, p.d, GEMV_STORE, 0, 0};
  const MegaLayer& L = p.layers[s >> 2];
  switch (s & 3) {
    case 0: return GemvDesc{L.wqkv, p.generation ? L.nqkv : L.dq, p.d, GEMV_STORE, 0, 0};
    case 1: return GemvDesc{L.wo, p.d, L.dq, GEMV_RESID, 0, 0};
    case 2: return GemvDesc{L.wgu, L.ffn, p.d, GEMV_SWIGLU, L.G, L.ffn};
    default: return GemvDesc{L.wd, p.d, L.ffn, GEMV_RESID, 0, 0};
  }
}

// A warp's weight stream: chunks (pieces of rows, at most `slot_bytes` each) in the order the
// warp consumes them, over all projection phases of the step.  The producer cursor walks the
// static schedule (phase, output row, gate/up half, piece of the row) ahead of the consumer.
struct WarpStream {
  int ps;                              // producer: phase index in the schedule
  const char* base; int row_bytes, mode, G, ffn, N, cpr;   // projection of phase ps
  int n, which, part;                  // producer cursor inside phase ps
  unsigned issued, consumed;
  uint32_t ring, bars;                 // shared-memory addresses of this warp's slots and mbarriers
  int slot_bytes;
};

template <class T>
__device__ __forceinline__ void stream_load_phase(const MegaParams& p, WarpStream& ws, int gw) {
  GemvDesc g = stream_desc(p, ws.ps);
  ws.base = (const char*)g.W; ws.row_bytes = g.K * (int)sizeof(T); ws.mode = g.mode; ws.G = g.G; ws.ffn = g.ffn; ws.N = g.N;
  ws.cpr = (ws.row_bytes + ws.slot_bytes - 1) / ws.slot_bytes;
  ws.n = gw; ws.which = 0; ws.part = 0;
}

// Keep the ring full: issue copies of the next chunks of the schedule into free slots.
template <class T>
__device__ __forceinline__ void stream_fill(const MegaParams& p, WarpStream& ws, int gw, int GW, int lane) {
  const int n_stream = 4 * p.layer_end + (p.do_head ? 1 : 0);     // schedule entries of this launch end here
  while (ws.issued - ws.consumed < (unsigned)NSLOT) {
    while (ws.ps < n_stream && ws.n >= ws.N) {
      if (++ws.ps < n_stream) stream_load_phase<T>(p, ws, gw);
    }
    if (ws.ps >= n_stream) break;
    int row = ws.n;
    if (ws.mode == GEMV_SWIGLU) { RowMap m{ws.which && ws.G == 0 ? ws.ffn : 0, ws.G, ws.which, ws.ffn}; row = map_row(m, ws.n); }
    const int off = ws.part * ws.slot_bytes;
    const int bytes = min(ws.slot_bytes, ws.row_bytes - off);
    const unsigned slot = ws.issued % NSLOT;
    if (lane == 0) {
      mbar_expect_tx(ws.bars + 8u * slot, (uint32_t)bytes);
      bulk_load(ws.ring + slot * ws.slot_bytes, ws.base + (size_t)row * ws.row_bytes + off, (uint32_t)bytes, ws.bars + 8u * slot);
    }
    ++ws.issued;
    if (++ws.part == ws.cpr) {
      ws.part = 0;
      if (++ws.which == (ws.mode == GEMV_SWIGLU ? 2 : 1)) { ws.which = 0; ws.n += GW; }
    }
  }
}

// Staged activations are stored permuted so that a warp's reads are bank-conflict free: within
// every group of 256 elements, lane l's elements 8l..8l+3 sit at [4l, 4l+4) and 8l+4..8l+7 at
// [128 + 4l, 128 + 4l + 4).  (Shared-memory bandwidth, not HBM, bounds these phases otherwise.)
__device__ __forceinline__ int xs_index(int k) {
  return (k & ~255) + ((k & 4) << 5) + (((k & 255) >> 3) << 2) + (k & 3);
}
__device__ __forceinline__ int xs_stride(int K) { return (K + 255) & ~255; }

// 8 consecutive weights (16 bytes for bf16, 32 for fp32) times 8 activations, two partial sums
template <class T> __device__ __forceinline__ float dot_w8(const unsigned char* w, const float* x);
template <> __device__ __forceinline__ float dot_w8<bf16>(const unsigned char* w, const float* x) {
  const uint4 u = *reinterpret_cast<const uint4*>(w);
  const float4 x0 = *reinterpret_cast<const float4*>(x), x1 = *reinterpret_cast<const float4*>(x + 128);
  float a = __uint_as_float(u.x << 16) * x0.x;
  float b = __uint_as_float(u.x & 0xffff0000u) * x0.y;
  a = fmaf(__uint_as_float(u.y << 16), x0.z, a);
  b = fmaf(__uint_as_float(u.y & 0xffff0000u), x0.w, b);
  a = fmaf(__uint_as_float(u.z << 16), x1.x, a);
  b = fmaf(__uint_as_float(u.z & 0xffff0000u), x1.y, b);
  a = fmaf(__uint_as_float(u.w << 16), x1.z, a);
  b = fmaf(__uint_as_float(u.w & 0xffff0000u), x1.w, b);
  return a + b;
}
template <> __device__ __forceinline__ float dot_w8<float>(const unsigned char* w, const float* x) {
  const float4 w0 = *reinterpret_cast<const float4*>(w), w1 = *reinterpret_cast<const float4*>(w + 16);
  const float4 x0 = *reinterpret_cast<const float4*>(x), x1 = *reinterpret_cast<const float4*>(x + 128);
  float a = w0.x * x0.x, b = w0.y * x0.y;
  a = fmaf(w0.z, x0.z, a); b = fmaf(w0.w, x0.w, b);
  a = fmaf(w1.x, x1.x, a); b = fmaf(w1.y, x1.y, b);
  a = fmaf(w1.z, x1.z, a); b = fmaf(w1.w, x1.w, b);
  return a + b;
}

// A row of the residual stream: tagged values, or (before the first layer) the embedding of the row's token.
template <class T> struct Stream {
  const u64* x; uint32_t tag; const T* embed[4];
};
// The residual of row n of a projection on its way (lane 0, which stores the row).
template <class T, int BB>
__device__ __forceinline__ void ask_residual(const MegaParams& p, const Stream<T>& in, int n, int N, int lane, u64 (&old)[BB]) {
#pragma unroll
  for (int b = 0; b < BB; ++b) old[b] = in.x && lane == 0 && b < p.batch && n < N ? ll_load(in.x + (size_t)b * N + n) : 0ull;
}
// One projection phase for this warp: y[b, n] = sum_k W[n, k] xs[b, k] (+ residual) over the warp's rows,
// consuming the warp's chunk stream.  xs is the staged (normalised) input in shared memory and
// ring_ptr the address of the warp's first slot.  y: tagged values, or (null) the logits.
template <class T, int BB>
__device__ __forceinline__ void gemv_phase(const MegaParams& p, const GemvDesc g, WarpStream& ws, const unsigned char* ring_ptr,
                                           const float* xs, u64* y, uint32_t tag, const Stream<T>* resid, u64 (&old)[BB], int gw, int GW,
                                           int lane, unsigned long long* best, volatile int* s_abort, bool& dead) {
  const int K = g.K, row_bytes = K * (int)sizeof(T);
  const int cpr = (row_bytes + ws.slot_bytes - 1) / ws.slot_bytes;
  const int R = g.mode == GEMV_SWIGLU ? 2 : 1;
  const bool vec = (K % 8 == 0);
  const int slot_elems = ws.slot_bytes / (int)sizeof(T);
  const int KS = xs_stride(K);
  float acc[BB], accu[BB];
#pragma unroll
  for (int b = 0; b < BB; ++b) { acc[b] = 0.f; accu[b] = 0.f; }
  for (int n = gw; n < g.N; n += GW) {
    if (n != gw && resid) ask_residual<T, BB>(p, *resid, n, g.N, lane, old);      // (the first row's were asked for in front of the phase)
    bool refill = false;
    for (int which = 0; which < R; ++which) {
      for (int part = 0; part < cpr; ++part) {
        const unsigned slot = ws.consumed % NSLOT;
        const uint32_t bar = ws.bars + 8u * slot, parity = (ws.consumed / NSLOT) & 1u;
        bool got = false;
        if (!*s_abort) {
          for (unsigned it = 0; it < TRY_WAIT_LIMIT; ++it) {
            if (mbar_test(bar, parity)) { got = true; break; }
            if ((it & 1023u) == 1023u && *s_abort) break;
          }
          if (!got && !*s_abort) { *s_abort = 1; dev_flag(p.status, DEV_TIMEOUT); }
        }
        got = __all_sync(0xffffffffu, got);
        if (got) {
          const int k0 = part * slot_elems;
          const int ne = min(slot_elems, K - k0);
          const unsigned char* sp = ring_ptr + (size_t)slot * ws.slot_bytes;
          float* a = which ? accu : acc;
          if (vec) {
#pragma unroll 4
            for (int e = lane * 8; e < ne; e += 256) {   // k0 and e - 8 lane are multiples of 256
#pragma unroll
              for (int b = 0; b < BB; ++b) a[b] += dot_w8<T>(sp + (size_t)e * sizeof(T), xs + b * KS + k0 + (e - lane * 8) + lane * 4);
            }
          } else {
            const T* wp = reinterpret_cast<const T*>(sp);
            for (int e = lane; e < ne; e += 32) {
              float wv = to_f(wp[e]);
#pragma unroll
              for (int b = 0; b < BB; ++b) a[b] = fmaf(wv, xs[b * KS + xs_index(k0 + e)], a[b]);
            }
          }
        }
        ++ws.consumed;
        __syncwarp();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        // the ring is filled again behind the output, which others wait for (filled first it took 300 to 500 cycles of every phase)
        refill = got;
        if (got && !(which == R - 1 && part == cpr - 1)) stream_fill<T>(p, ws, gw, GW, lane);
      }
    }
    // all pieces of this output are in: reduce, apply, store
#pragma unroll
    for (int b = 0; b < BB; ++b) {
      float v = warp_sum(acc[b]);
      float u = R == 2 ? warp_sum(accu[b]) : 0.f;
      if (lane == 0 && b < p.batch && !*s_abort) {
        if (g.mode == GEMV_SWIGLU) v = v / (1.f + __expf(-v)) * u;
        if (resid) {
          if (!resid->x) v += resid->embed[b] ? to_f(resid->embed[b][n]) : 0.f;
          else v += ll_tag(old[b]) == resid->tag ? ll_val(old[b]) : ll_wait(resid->x + (size_t)b * g.N + n, resid->tag, dead, s_abort, p.status);
        }
        if (y) ll_store(y + (size_t)b * g.N + n, v, tag);
        else {
          p.logits[(size_t)b * g.N + n] = v;
          if (best) {   // running argmax: larger value wins, then the lower index
            unsigned bits = __float_as_uint(v);
            bits = (bits & 0x80000000u) ? ~bits : (bits | 0x80000000u);
            atomicMax(best + b, ((unsigned long long)bits << 32) | (unsigned long long)(0xFFFFFFFFu - (unsigned)n));
          }
        }
      }
      acc[b] = 0.f; accu[b] = 0.f;
    }
    if (refill) stream_fill<T>(p, ws, gw, GW, lane);
  }
}

// Stage `batch` activation rows of length K into shared memory, optionally RMS-normalised
// (one pass: the row is held in registers between the sum of squares and the scaled store).  J: elements a thread holds.
template <class T, int BB, int J>
__device__ __noinline__ void stage_rows(const MegaParams& p, const Stream<T>& in, int K, const float* gain, float* xs, float* red,
                                     volatile int* s_abort, bool& dead) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, batch = p.batch;
  const int KS = xs_stride(K);
  if (K <= J * NT) {
    float v[BB][J], g[J];
    float ss[BB];
#pragma unroll
    for (int j = 0; j < J; ++j) { const int k = tid + j * NT; g[j] = gain && k < K ? __ldg(gain + k) : 1.f; }
    constexpr int BS = J == 1 ? BB : 1;            // rows whose words are asked for together, until all have the tag
#pragma unroll
    for (int b0 = 0; b0 < BB; b0 += BS) {
      if (in.x) {
        bool ok;
        unsigned it = 0;
        do {
          ok = true;
#pragma unroll
          for (int b = b0; b < b0 + BS; ++b)
#pragma unroll
            for (int j = 0; j < J; ++j) {
              const int k = tid + j * NT;
              const u64 w = k < K && b < batch ? ll_load(in.x + (size_t)b * K + k) : (u64)in.tag << 32;
              ok = ok && ll_tag(w) == in.tag;
              v[b][j] = ll_val(w);
            }
          if (!ok && !dead && !poll_more(it, s_abort, p.status)) dead = true;
        } while (!ok && !dead);
      } else {
#pragma unroll
        for (int b = b0; b < b0 + BS; ++b)
#pragma unroll
          for (int j = 0; j < J; ++j) {
            const int k = tid + j * NT;
            v[b][j] = k < K && in.embed[b] ? to_f(in.embed[b][k]) : 0.f;
          }
      }
    }
#pragma unroll
    for (int b = 0; b < BB; ++b) {
      ss[b] = 0.f;
#pragma unroll
      for (int j = 0; j < J; ++j) ss[b] = fmaf(v[b][j], v[b][j], ss[b]);
    }
    float r[BB];
#pragma unroll
    for (int b = 0; b < BB; ++b) r[b] = 1.f;
    __syncthreads();                               // (the staging area and `red` are free: the phase before this one has been read out)
    if (gain) {
#pragma unroll
      for (int b = 0; b < BB; ++b) { float t = warp_sum(ss[b]); if (lane == 0) red[warp * BB + b] = t; }
      __syncthreads();
#pragma unroll
      for (int b = 0; b < BB; ++b) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) t += red[w * BB + b];
        r[b] = rsqrtf(t / (float)K + p.eps);
      }
    }
#pragma unroll
    for (int b = 0; b < BB; ++b)
#pragma unroll
      for (int j = 0; j < J; ++j) {
        const int k = tid + j * NT;
        if (k < K) xs[b * KS + xs_index(k)] = g[j] * v[b][j] * r[b];
      }
  } else {
    float ss[BB];
#pragma unroll
    for (int b = 0; b < BB; ++b) ss[b] = 0.f;
    __syncthreads();
    for (int k = tid; k < K; k += NT) {
#pragma unroll
      for (int b = 0; b < BB; ++b) {
        float t = 0.f;
        if (b < batch) t = in.x ? ll_wait(in.x + (size_t)b * K + k, in.tag, dead, s_abort, p.status) : (in.embed[b] ? to_f(in.embed[b][k]) : 0.f);
        ss[b] = fmaf(t, t, ss[b]);
        xs[b * KS + xs_index(k)] = t;
      }
    }
    if (gain) {
#pragma unroll
      for (int b = 0; b < BB; ++b) { float t = warp_sum(ss[b]); if (lane == 0) red[warp * BB + b] = t; }
      __syncthreads();
#pragma unroll
      for (int b = 0; b < BB; ++b) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) t += red[w * BB + b];
        const float r = rsqrtf(t / (float)K + p.eps);
        for (int k = tid; k < K; k += NT) xs[b * KS + xs_index(k)] = gain[k] * xs[b * KS + xs_index(k)] * r;      // (a thread's own elements)
      }
    }
  }
  __syncthreads();
}
template <class T, int BB>
__device__ __forceinline__ void stage_x(const MegaParams& p, const Stream<T>& in, int K, const float* gain, float* xs, float* red,
                                        volatile int* s_abort, bool& dead) {
  if (K <= NT) stage_rows<T, BB, 1>(p, in, K, gain, xs, red, s_abort, dead);      // (a model of test size: less code to fetch, all rows at once)
  else stage_rows<T, BB, 8>(p, in, K, gain, xs, red, s_abort, dead);
}

// Attention of one (sequence, kv head, key-range split) over whole cache pages: the K and V page
// (64 keys, contiguous) are copied to shared memory with independent 16-byte loads; scores with
// thread = (key, head), softmax statistics with one warp per head, value sum with thread =
// (dim, head subset).
template <class T>
__device__ __noinline__ void attn_item(const MegaParams& p, const MegaLayer& L, int b, int kvh, int sp, int n_split,
                                       const u64* q, int ldq, uint32_t tag, const float2* rope, unsigned char* sm, float* part,
                                       u64* out, volatile int* s_abort, bool& dead) {
  const int hd = p.hd, nq = L.nq, nkv = L.nkv, group = nq / nkv;
  const int row_bytes = hd * (int)sizeof(T) + 16;
  unsigned char* Ks = sm;
  unsigned char* Vs = Ks + PAGE_TOKENS * row_bytes;
  float* qs = reinterpret_cast<float*>(Vs + PAGE_TOKENS * row_bytes);
  float* ps = qs + MAXG * hd;
  float* m_run = ps + MAXG * PAGE_TOKENS;
  float* l_run = m_run + MAXG;
  float* alpha = l_run + MAXG;
  float* rn = alpha + MAXG;                            // 1 / rms of the query heads, and of the new key
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n_keys = __ldcg(p.seq_lens + b) + (p.generation ? 1 : 0);
  const int pos = n_keys - 1;
  const float scale = rsqrtf((float)hd);
  const int half = hd >> 1;
  __syncthreads();                                   // shared memory free (previous item / phase)
  typedef typename KvOf<T>::type KT;                   // cache element: fp32, or 16-bit half in bf16 mode
  const int n_pg = (n_keys + PAGE_TOKENS - 1) / PAGE_TOKENS;
  const int per = (n_pg + n_split - 1) / n_split;
  const int pg0 = sp * per, pg1 = min(n_pg, pg0 + per);
  // the step's own key and value: the item whose range ends with their page takes them into its copy of the page and into the pool
  const bool has_new = p.generation && pg0 < pg1 && pg1 == n_pg;
  // A page into shared memory (every thread; its id, or -1).  The first one is fetched in front of the wait for the queries.
  const int chunks_per_row = hd * (int)sizeof(KT) / 16;
  const int n_chunks = PAGE_TOKENS * chunks_per_row;
  auto load_page = [&](int pg) {
    const int page = pg < p.mpps ? p.block_table[(size_t)b * p.mpps + pg] : -1;
    if (page < 0 || page >= p.n_pages) {
      if (tid == 0) dev_flag(p.status, DEV_BAD_PAGE);
      return -1;
    }
    const uint4* ksrc = reinterpret_cast<const uint4*>((const KT*)L.kpool + ((size_t)page * nkv + kvh) * PAGE_TOKENS * hd);
    const uint4* vsrc = reinterpret_cast<const uint4*>((const KT*)L.vpool + ((size_t)page * nkv + kvh) * PAGE_TOKENS * hd);
    for (int i = tid; i < n_chunks; i += NT) {
      int r = i / chunks_per_row, cc = i - r * chunks_per_row;
      uint4 kx = __ldcg(ksrc + i), vx = __ldcg(vsrc + i);
      *reinterpret_cast<uint4*>(Ks + r * row_bytes + cc * 16) = kx;
      *reinterpret_cast<uint4*>(Vs + r * row_bytes + cc * 16) = vx;
    }
    return page;
  };
  int page = pg0 < pg1 ? load_page(pg0) : -1;
  float* knew = ps;                                    // (ps is free until the first page's scores) [hd] key, [hd] value
  for (int i = tid; i < group * hd; i += NT) qs[i] = ll_wait(q + (size_t)b * ldq + (size_t)kvh * group * hd + i, tag, dead, s_abort, p.status);
  if (has_new)
    for (int i = tid; i < 2 * hd; i += NT)
      knew[i] = ll_wait(q + (size_t)b * ldq + L.dq + (size_t)((i < hd ? 0 : nkv) + kvh) * hd + (i < hd ? i : i - hd), tag, dead, s_abort, p.status);
  __syncthreads();
  if (L.q_norm) {
    const int heads = group + (has_new ? 1 : 0);
    if (warp < heads) {                                // (at most 9 of the 16 warps)
      const float* x = warp < group ? qs + warp * hd : knew;
      float ss = 0.f;
      for (int c = lane; c < hd; c += 32) ss = fmaf(x[c], x[c], ss);
      ss = warp_sum(ss);
      if (lane == 0) rn[warp] = rsqrtf(ss / (float)hd + p.eps);
    }
    __syncthreads();
  }
  for (int i = tid; i < (group + (has_new ? 1 : 0)) * half; i += NT) {
    const int h = i / half, c = i - h * half;
    const bool key = h == group;
    float* x = key ? knew : qs + h * hd;
    const float cs = rope[c].x, sn = rope[c].y;
    float x1 = x[c], x2 = x[c + half];
    if (L.q_norm) { const float* gn = key ? L.k_norm : L.q_norm; x1 *= rn[h] * gn[c]; x2 *= rn[h] * gn[c + half]; }
    const float f = key ? 1.f : scale;
    x[c] = (x1 * cs - x2 * sn) * f;
    x[c + half] = (x2 * cs + x1 * sn) * f;
  }
  KT* knew_kt = reinterpret_cast<KT*>(rn + MAXG + 8);   // [2][hd], as the cache holds them
  __syncthreads();
  if (has_new && tid < 2 * hd) knew_kt[tid] = from_f<KT>(knew[tid]);
  if (tid < MAXG) { m_run[tid] = -INFINITY; l_run[tid] = 0.f; alpha[tid] = 1.f; }
  const int key = tid & 63, hh_s = tid >> 6;           // scores: thread = (key, head hh_s)
  // Value sum: NT / hd threads a dim.  They take a head each (and the one NT / hd further on), or, where there are more of them than heads,
  // every key_step-th key of a head (one thread a head went through 64 keys, 900 cycles a page, while the others waited).
  const int nhh = NT / hd, dim = tid % hd, slot_v = tid / hd;
  const bool by_keys = nhh >= 2 * group;
  const int key_step = by_keys ? nhh / group : 1, head0 = by_keys ? slot_v % group : slot_v, key0 = by_keys ? slot_v / group : 0;
  const bool sums = key0 < key_step;
  float o[MAXG];
#pragma unroll
  for (int i = 0; i < MAXG; ++i) o[i] = 0.f;
  for (int pg = pg0; pg < pg1; ++pg) {
    if (pg != pg0) {
      __syncthreads();
      page = load_page(pg);
    }
    const int nk = page >= 0 ? min(PAGE_TOKENS, n_keys - pg * PAGE_TOKENS) : 0;
    if (has_new && pg == n_pg - 1 && page >= 0) {
      __syncthreads();
      const int row = pos % PAGE_TOKENS;
      for (int i = tid; i < 2 * hd; i += NT) {
        const int c = i < hd ? i : i - hd;
        const KT x = knew_kt[i];
        reinterpret_cast<KT*>((i < hd ? Ks : Vs) + row * row_bytes)[c] = x;
        ((KT*)(i < hd ? L.kpool : L.vpool))[(((size_t)page * nkv + kvh) * PAGE_TOKENS + row) * hd + c] = x;
      }
    }
    __syncthreads();
    if (hh_s < group) {
      float sc = 0.f;
      const KT* kr = reinterpret_cast<const KT*>(Ks + key * row_bytes);
      for (int c = 0; c < hd; c += 8) {
        float kf[8];
        if (sizeof(KT) == 2) {
          uint4 u = *reinterpret_cast<const uint4*>(kr + c);
          const __half2* hp = reinterpret_cast<const __half2*>(&u);
#pragma unroll
          for (int e = 0; e < 4; ++e) { float2 t = __half22float2(hp[e]); kf[2 * e] = t.x; kf[2 * e + 1] = t.y; }
        } else {
          float4 a = *reinterpret_cast<const float4*>(kr + c), bq = *reinterpret_cast<const float4*>(kr + c + 4);
          kf[0] = a.x; kf[1] = a.y; kf[2] = a.z; kf[3] = a.w; kf[4] = bq.x; kf[5] = bq.y; kf[6] = bq.z; kf[7] = bq.w;
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) sc = fmaf(kf[e], qs[hh_s * hd + c + e], sc);
      }
      ps[hh_s * PAGE_TOKENS + key] = key < nk ? sc : -INFINITY;
    }
    __syncthreads();
    if (warp < group) {
      const int h = warp;
      float s0 = ps[h * PAGE_TOKENS + lane], s1 = ps[h * PAGE_TOKENS + 32 + lane];
      float mt = warp_max(fmaxf(s0, s1));
      float m_old = m_run[h];
      float mn = fmaxf(m_old, mt);
      float p0 = (mn == -INFINITY) ? 0.f : __expf(s0 - mn), p1 = (mn == -INFINITY) ? 0.f : __expf(s1 - mn);
      float sum = warp_sum(p0 + p1);
      ps[h * PAGE_TOKENS + lane] = p0; ps[h * PAGE_TOKENS + 32 + lane] = p1;
      if (lane == 0) {
        float a = (mn == -INFINITY) ? 1.f : __expf(m_old - mn);
        alpha[h] = a; m_run[h] = mn; l_run[h] = l_run[h] * a + sum;
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < MAXG; ++i) {
      const int h = head0 + nhh * i;
      if (i * nhh < MAXG && (i == 0 || !by_keys) && h < group && sums) {
        float acc = o[i] * alpha[h];
        const float* pr = ps + h * PAGE_TOKENS;
#pragma unroll 4
        for (int s = key0; s < nk; s += key_step) acc = fmaf(pr[s], to_f(reinterpret_cast<const KT*>(Vs + s * row_bytes)[dim]), acc);
        o[i] = acc;
      }
    }
  }
  __syncthreads();
  if (by_keys) {                                       // the parts of a sum meet in shared memory (the pages have been read)
    float* parts = reinterpret_cast<float*>(sm);       // [key_step][group][hd]
    if (sums) parts[(key0 * group + head0) * hd + dim] = o[0];
    __syncthreads();
    if (key0 == 0) for (int k = 1; k < key_step; ++k) o[0] += parts[(k * group + head0) * hd + dim];
  }
  const int ldr = hd + 2;
#pragma unroll
  for (int i = 0; i < MAXG; ++i) {
    const int h = head0 + nhh * i;
    if (i * nhh < MAXG && (i == 0 || !by_keys) && h < group && key0 == 0) {
      int qh = kvh * group + h;
      if (n_split == 1) {
        ll_store(out + (size_t)b * nq * hd + (size_t)qh * hd + dim, o[i] / l_run[h], tag);
      } else {
        float* pr = part + (((size_t)b * nq + qh) * n_split + sp) * ldr;
        pr[dim] = o[i];
        if (dim == 0) { pr[hd] = m_run[h]; pr[hd + 1] = l_run[h]; }
      }
    }
  }
}

template <class T, int BB>
__global__ void __launch_bounds__(NT, 1) step_mega_kernel(const __grid_constant__ MegaParams p) {
  extern __shared__ __align__(128) unsigned char sm_raw[];
  __shared__ float red[NW * BB];
  __shared__ int s_last;
  __shared__ int s_abort_mem;
  __shared__ __align__(8) unsigned long long s_bars[NW * NSLOT];
  __shared__ float2 rope[BB][64];      // (cos, sin) of each sequence's last position
  volatile int* s_abort = &s_abort_mem;
  // dynamic shared memory: [ x staging / attention scratch | per-warp rings ]
  float* xs = reinterpret_cast<float*>(sm_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int gw = blockIdx.x * NW + warp, GW = gridDim.x * NW;
  const int batch = p.batch;
  unsigned* counter = reinterpret_cast<unsigned*>(p.status) + 32 + p.counter_idx;
  unsigned long long* best = reinterpret_cast<unsigned long long*>(reinterpret_cast<char*>(p.status) + 64);
  if (tid == 0) {
    *s_abort = 0;
    for (int i = 0; i < NW * NSLOT; ++i) mbar_init(smem_u32(&s_bars[i]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  WarpStream ws;
  ws.ps = 4 * p.layer_begin; ws.issued = 0; ws.consumed = 0;
  ws.slot_bytes = p.slot_bytes;
  const unsigned char* ring_ptr = sm_raw + p.stage_bytes + (size_t)warp * NSLOT * p.slot_bytes;
  ws.ring = smem_u32(ring_ptr);
  ws.bars = smem_u32(&s_bars[warp * NSLOT]);
  stream_load_phase<T>(p, ws, gw);
  stream_fill<T>(p, ws, gw, GW, lane);        // the first weight rows start streaming before anything else

  if (tid < batch * (p.hd >> 1)) {     // (once, not in every layer: 2000 cycles of 64-bit arithmetic)
    const int b = tid / (p.hd >> 1), c = tid - b * (p.hd >> 1);
    float sn, cs;
    rope_sincos(__ldcg(p.seq_lens + b) + (p.generation ? 0 : -1), p.inv.f[c], &sn, &cs);
    rope[b][c] = make_float2(cs, sn);
  }
  bool dead = false;                  // this thread has given up waiting
  // the residual stream in front of the first layer
  Stream<T> first{nullptr, 0u, {nullptr, nullptr, nullptr, nullptr}};
  if (p.do_embed) {
#pragma unroll
    for (int b = 0; b < BB; ++b) {
      if (b >= batch) continue;
      const int tok = p.tokens[p.gather_idx ? p.gather_idx[b] : b];
      const bool ok = tok >= 0 && tok < p.vocab;
      if (!ok && blockIdx.x == 0 && tid == 0) dev_flag(p.status, DEV_BAD_TOKEN);
      first.embed[b] = ok ? (const T*)p.embed + (size_t)tok * p.d : nullptr;
    }
  }
  const int row0 = blockIdx.x * NW;   // the CTA's first row of a projection: without one it does not read the phase's input
  for (int i = p.layer_begin; i < p.layer_end; ++i) {
    const MegaLayer& L = p.layers[i];
    const int n_out = p.generation ? L.nqkv : L.dq;
    const uint32_t tag = (uint32_t)i + 1u;
    const Stream<T> x2{p.ll_x2, tag - 1u, {}}, x1{p.ll_x1, tag, {}}, a{p.ll_a, tag, {}}, h{p.ll_h, tag, {}};
    const Stream<T>& in = p.do_embed && i == 0 ? first : x2;
    u64 old[BB];        // the residual of the warp's first row
    // ---- q (k, v) projection
    if (row0 < n_out) {
      stage_x<T, BB>(p, in, p.d, L.attn_norm, xs, red, s_abort, dead);
      gemv_phase<T, BB>(p, stream_desc(p, 4 * i), ws, ring_ptr, xs, p.ll_q, tag, nullptr, old, gw, GW, lane, nullptr, s_abort, dead);
    }
    // ---- attention over the cache.  With split key ranges the CTA that finishes the last split of a
    // (sequence, kv head) merges that group's partial results on the spot (a counter per group tells
    // it so), which saves a merge phase of its own.
    {
      const int n_split = L.n_split, n_items = batch * L.nkv * n_split;
      const int group = L.nq / L.nkv, ldr = p.hd + 2;
      for (int it = blockIdx.x; it < n_items; it += gridDim.x) {
        const int sp = it % n_split, r = it / n_split;
        attn_item<T>(p, L, r / L.nkv, r % L.nkv, sp, n_split, p.ll_q, n_out, tag, rope[r / L.nkv], sm_raw, p.part, p.ll_a, s_abort, dead);
        if (n_split > 1) {
          __threadfence();                       // this CTA's partial results are visible before it counts itself done
          __syncthreads();
          if (tid == 0) {
            const int before = atomicAdd(p.attn_done + r, 1);
            s_last = before == n_split - 1;
            if (s_last) atomicExch(p.attn_done + r, 0);      // ready for the next layer
          }
          __syncthreads();
          if (s_last) {
            __threadfence();
            if (warp < group) {                  // one warp per q head of the group
              const int head = (r / L.nkv) * L.nq + (r % L.nkv) * group + warp;
              const float* pr = p.part + (size_t)head * n_split * ldr;
              float mm = -INFINITY;
              for (int s = lane; s < n_split; s += 32) mm = fmaxf(mm, __ldcg(pr + (size_t)s * ldr + p.hd));
              mm = warp_max(mm);
              // the loads of different splits do not depend on one another: unrolled, they are in flight together
              float ll = 0.f, o0 = 0.f, o1 = 0.f, o2 = 0.f, o3 = 0.f;
#pragma unroll 8
              for (int s = 0; s < n_split; ++s) {
                const float* rr = pr + (size_t)s * ldr;
                const float ms = __ldcg(rr + p.hd);
                const float f = (ms == -INFINITY) ? 0.f : __expf(ms - mm);
                ll = fmaf(__ldcg(rr + p.hd + 1), f, ll);
                if (lane < p.hd) o0 = fmaf(__ldcg(rr + lane), f, o0);
                if (lane + 32 < p.hd) o1 = fmaf(__ldcg(rr + lane + 32), f, o1);
                if (lane + 64 < p.hd) o2 = fmaf(__ldcg(rr + lane + 64), f, o2);
                if (lane + 96 < p.hd) o3 = fmaf(__ldcg(rr + lane + 96), f, o3);
              }
              u64* dst = p.ll_a + (size_t)head * p.hd;
              if (lane < p.hd) ll_store(dst + lane, o0 / ll, tag);
              if (lane + 32 < p.hd) ll_store(dst + lane + 32, o1 / ll, tag);
              if (lane + 64 < p.hd) ll_store(dst + lane + 64, o2 / ll, tag);
              if (lane + 96 < p.hd) ll_store(dst + lane + 96, o3 / ll, tag);
            }
          }
        }
      }
    }
    // ---- O projection + residual
    if (row0 < p.d) {
      ask_residual<T, BB>(p, in, gw, p.d, lane, old);
      stage_x<T, BB>(p, a, L.dq, nullptr, xs, red, s_abort, dead);
      gemv_phase<T, BB>(p, stream_desc(p, 4 * i + 1), ws, ring_ptr, xs, p.ll_x1, tag, &in, old, gw, GW, lane, nullptr, s_abort, dead);
    }
    // ---- gate / up + SwiGLU
    if (row0 < L.ffn) {
      stage_x<T, BB>(p, x1, p.d, L.ffn_norm, xs, red, s_abort, dead);
      gemv_phase<T, BB>(p, stream_desc(p, 4 * i + 2), ws, ring_ptr, xs, p.ll_h, tag, nullptr, old, gw, GW, lane, nullptr, s_abort, dead);
    }
    // ---- down projection + residual
    if (row0 < p.d) {
      ask_residual<T, BB>(p, x1, gw, p.d, lane, old);
      stage_x<T, BB>(p, h, L.ffn, nullptr, xs, red, s_abort, dead);
      gemv_phase<T, BB>(p, stream_desc(p, 4 * i + 3), ws, ring_ptr, xs, p.ll_x2, tag, &x1, old, gw, GW, lane, nullptr, s_abort, dead);
    }
  }
  if (p.do_head) {      // (else a later launch carries on from the residual stream in ll_x2)
    // ---- LM head (final RMSNorm fused) with running argmax
    if (row0 < p.vocab) {
      const Stream<T> x2{p.ll_x2, (uint32_t)p.n_layers, {}};
      stage_x<T, BB>(p, x2, p.d, p.final_norm, xs, red, s_abort, dead);
      u64 none[BB];
      gemv_phase<T, BB>(p, stream_desc(p, 4 * p.n_layers), ws, ring_ptr, xs, nullptr, 0u, nullptr, none, gw, GW, lane,
                        p.token_out ? best : nullptr, s_abort, dead);
    }
    // the CTA that finishes last reads the argmax
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (s_last && tid < batch) {
      __threadfence();
      if (p.token_out) {
        unsigned long long v;
        asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(best + tid) : "memory");
        p.token_out[tid] = (int)(0xFFFFFFFFu - (unsigned)(v & 0xFFFFFFFFull));
      }
      if (p.generation) p.seq_lens[tid] += 1;
    }
  }
  if (*s_abort) for (int i = 0; i < 2000; ++i) __nanosleep(1000);      // let copies in flight land before the CTA goes
}

constexpr int SMEM_LIMIT = 227 * 1024 - 3072;   // dynamic shared memory we allow ourselves per CTA

size_t stage_region_bytes(int batch, int hd, int k_max, int es) {
  int bb = batch <= 1 ? 1 : (batch == 2 ? 2 : 4);
  size_t xs = (size_t)bb * ((k_max + 255) / 256 * 256) * 4;
  size_t at = (size_t)2 * PAGE_TOKENS * (hd * es + 16) + (size_t)(MAXG * hd + MAXG * PAGE_TOKENS + 4 * MAXG + 8 + 2 * hd) * 4;
  size_t r = xs > at ? xs : at;
  return (r + 127) / 128 * 128;
}

template <class T, int BB>
cudaError_t go(MegaParams& p, size_t smem, cudaStream_t st, int n_sm) {
  auto kern = step_mega_kernel<T, BB>;
  static bool raised[TC_MAX_DEVICES] = {};
  cudaError_t e = tc_raise_smem_limit(kern, SMEM_LIMIT, raised);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorLaunchOutOfResources;
  void* args[] = {(void*)&p};
  return cudaLaunchCooperativeKernel((const void*)kern, dim3(n_sm), dim3(NT), args, smem, st);
}

}  // namespace

bool step_mega_supported(int batch, int hd, int k_max, int max_group, int es) {
  if (batch < 1 || batch > 4) return false;
  if (!(hd == 16 || hd == 32 || hd == 64 || hd == 128)) return false;
  if (max_group > MAXG) return false;
  size_t stage = stage_region_bytes(batch, hd, k_max, es);
  return stage + (size_t)NW * NSLOT * 1024 <= (size_t)SMEM_LIMIT;   // at least 1 KiB per ring slot
}

cudaError_t launch_step_mega(MegaParams p, int dtype, int k_max, int n_sm, cudaStream_t st, int64_t* n_launch) {
  const int es = dtype == 0 ? 4 : 2;
  size_t stage = stage_region_bytes(p.batch, p.hd, k_max, es);
  int slot = (int)((SMEM_LIMIT - stage) / (NW * NSLOT));
  slot = slot / 1024 * 1024;      // whole 256-element groups of either element size
  const int row = (k_max * es + 1023) / 1024 * 1024;      // no more than the longest row
  if (slot > row) slot = row;
  if (slot > 8192) slot = 8192;
  p.stage_bytes = (int)stage;
  p.slot_bytes = slot;
  size_t smem = stage + (size_t)NW * NSLOT * slot;
  ++*n_launch;
  if (dtype == 0) {
    if (p.batch <= 1) return go<float, 1>(p, smem, st, n_sm);
    if (p.batch == 2) return go<float, 2>(p, smem, st, n_sm);
    return go<float, 4>(p, smem, st, n_sm);
  }
  if (p.batch <= 1) return go<bf16, 1>(p, smem, st, n_sm);
  if (p.batch == 2) return go<bf16, 2>(p, smem, st, n_sm);
  return go<bf16, 4>(p, smem, st, n_sm);
}
