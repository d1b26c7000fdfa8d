// Single-query GQA attention of the base step over the paged half-precision cache on the warp-level
// tensor-core path (mma.sync m16n8k16, fp32 accumulation).
//
// The CUDA-core kernels of step_attn.cu spend about 300 instructions per thread and page and are bound by
// instruction issue at a third of the HBM rate.  Here the arithmetic per cached element is almost free:
//   grid (key-range split, kv head, sequence); a CTA serves the group's query heads (up to 8) and walks its
//   range of cache pages.  Warp 4 fetches pages with TMA through a tensor map over the layer's pool (64 x 64
//   boxes, 128-byte swizzle, so that the matrix loads below are free of bank conflicts) into a ring of stages;
//   warps 0-3 each take 16 of a page's 64 keys:
//   scores   S[16 x 16] = Q K^T: rows g / g + 8 of the A operand carry the half-precision value / remainder of
//            query head g (the two accumulator rows are added), K fragments by ldmatrix
//   softmax  per warp, online, on the 4 lanes that own a head's row; the rescale of what has been accumulated
//            happens only when a row maximum grows
//   values   O[16 x hd] += P V with P as value / remainder rows like Q, V fragments by transposing ldmatrix
//   The step's own key and value join the cache here, and the output leaves as the next projection's operand rows (two launches and
//   two passes less a layer: 64 x 123 keys, generation step 2147 -> 1708 us by itself).
//   The four warps' (max, sum, O) meet in shared memory after the last page; key-range splits are merged by the
//   CTA that finishes a group's last split (counter per (sequence, kv head)), as in step_attn.cu.
// Every wait is bounded (DEV_TIMEOUT, the CTA leaves); page ids are checked before they are used as coordinates.
#include <math.h>

#include "common.cuh"
#include "step_tc.h"
#include "tc_ptx.cuh"

namespace {
using namespace tcp;

constexpr int NW = 4;                       // consumer warps
constexpr int NT = (NW + 1) * 32;
constexpr int BOX_BYTES = 64 * 128;         // one 64-key x 64-dim box

template <int HD> struct MmaCfg {
  static constexpr int PAGE_BYTES = PAGE_TOKENS * HD * 2;
  static constexpr int STAGES = HD == 64 ? 5 : 3;          // most stages: two CTAs per SM
  static constexpr int PER_SM = HD == 64 ? 4 : 2;          // most CTAs per SM (registers)
  static constexpr int LDQ = HD + 8;                       // floats from head to head of the staged queries: no two heads' pieces in the same banks
  // after the ring: q [8][LDQ] fp32, then the warps' partial results [NW][8][HD + 2] fp32 (reuses the ring when it is idle)
  static constexpr int smem(int stages) { return 1024 + stages * 2 * PAGE_BYTES + 8 * LDQ * 4 + 256; }
};
// Ring stages of a launch whose CTAs walk `per_pages` pages, and how many of its CTAs an SM holds.  A short range needs no deep ring:
// with 2 or 3 stages four CTAs of head_dim 64 share an SM instead of two, and their set-up and merge overlap (64 x 59 keys: 512 CTAs
// in one wave instead of 1.7, 12.5 -> 9.9 us).
int mma_stages(int hd, int per_pages) {
  const int most = hd == 64 ? MmaCfg<64>::STAGES : MmaCfg<128>::STAGES;
  return per_pages < 2 ? 2 : (per_pages < most ? per_pages : most);
}
int mma_per_sm(int hd, int stages) {
  const int fit = (227 * 1024) / ((hd == 64 ? MmaCfg<64>::smem(stages) : MmaCfg<128>::smem(stages)) + 2048);
  const int most = hd == 64 ? MmaCfg<64>::PER_SM : MmaCfg<128>::PER_SM;
  return fit < most ? fit : most;
}

__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t* r) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm4_t(uint32_t addr, uint32_t* r) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void mma16816(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// (value, remainder) of two floats as packed halves
__device__ __forceinline__ void split2(float x, float y, uint32_t& hi, uint32_t& lo) {
  const __half2 h = __floats2half2_rn(x, y);
  const float2 f = __half22float2(h);
  const __half2 l = __floats2half2_rn(x - f.x, y - f.y);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}
// byte offset of the 16-byte piece `c` (8 dims) of key `k` inside a page stored as 64 x 64 boxes with the 128-byte swizzle
__device__ __forceinline__ uint32_t piece(int k, int c) { return (uint32_t)((c >> 3) * BOX_BYTES + k * 128 + (((c & 7) ^ (k & 7)) << 4)); }

struct MmaParams {
  const float* q; int ldq, nq, nkv;
  const int* block_table; int mpps, n_pages;
  const int* seq_lens; int extra, n_split;
  float* part; int* status;
  const float* q_gain; float eps;
  int* split_done;          // splits finished per (sequence, kv head): zero between launches
  int per_pages;            // pages per CTA
  int stages;               // of its ring
  float* out;               // output rows [batch, nq * HD], or (null) as the next projection's operand rows:
  bf16* xb; int Bp, terms;  // row b = bf16(value), row Bp + b = bf16(remainder), with three terms row 2 Bp + b what that leaves
  // Generation: q's rows go on with the step's own keys and values.  They join the cache here: the CTA whose range ends with
  // their page takes them into its copy of the page and writes them to the pool (no launch of their own: 7.7 us a layer).
  int append; const float* k_gain; kv16* kpool; kv16* vpool;
};
// element d of a head's output
__device__ __forceinline__ void emit(const MmaParams& p, int b, size_t width, int col, float v) {
  if (p.out) { p.out[(size_t)b * width + col] = v; return; }
  const bf16 h = __float2bfloat16_rn(v);
  p.xb[(size_t)b * width + col] = h;
  const float rest = v - __bfloat162float(h);
  const bf16 l = __float2bfloat16_rn(rest);
  p.xb[(size_t)(p.Bp + b) * width + col] = l;
  if (p.terms == 3) p.xb[(size_t)(2 * p.Bp + b) * width + col] = __float2bfloat16_rn(rest - __bfloat162float(l));
}

template <int HD>
__global__ void __launch_bounds__(NT, MmaCfg<HD>::PER_SM)
step_attn_mma_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                     const __grid_constant__ InvFreq inv, const MmaParams p) {
  using Cfg = MmaCfg<HD>;
  constexpr int PB = Cfg::PAGE_BYTES, LDQ = Cfg::LDQ, KS = HD / 16, NTL = HD / 8;
  extern __shared__ uint8_t sm_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(sm_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t ring = smem_u32(smem);
  const int STG = p.stages;
  float* qs = reinterpret_cast<float*>(smem + STG * 2 * PB);                     // [8][LDQ], scaled, after RoPE
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + STG * 2 * PB + 8 * LDQ * 4);   // full[STG], empty[STG]
  __shared__ int s_abort_mem;
  __shared__ float rq[8];
  __shared__ float rk;
  __shared__ float2 rope[HD / 2];                  // (cos, sin) of the last position
  __shared__ __align__(16) kv16 knew[HD];
  __shared__ __align__(16) kv16 vnew[HD];
  __shared__ int s_last;
  volatile int* abort_flag = &s_abort_mem;
  const uint32_t bar_base = smem_u32(bars);
  auto full = [&](int s) { return bar_base + 8u * s; };
  auto empty = [&](int s) { return bar_base + 8u * (STG + s); };
  const int group = p.nq / p.nkv;                  // <= 8
  const int sp = blockIdx.x, kvh = blockIdx.y, b = blockIdx.z;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int s = 0; s < STG; ++s) { mbar_init(full(s), 1); mbar_init(empty(s), NW); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid == 32) { prefetch_tensormap(&map_k); prefetch_tensormap(&map_v); }
  // Lengths, block table and cached pages do not come from the kernel before this one.  A step, and every piece of a step that waits
  // for a predictor on another stream, starts with an ordinary launch, behind which all of them are complete, and within the step a
  // layer's pages are written by this kernel only.  So the pages are on their way before the wait for the queries.
  const int n_keys = p.seq_lens[b] + p.extra;
  const int pos = n_keys - 1;
  const int n_pg = (n_keys + PAGE_TOKENS - 1) / PAGE_TOKENS;
  // every CTA walks at most `per_pages` pages, so a short sequence takes fewer CTAs instead of shorter ranges:
  // its surplus CTAs leave at once and the launch is as long as per_pages pages, not as the longest sequence's share
  // (a sequence that has grown since the launch shape was chosen, as in a replayed generation step, leaves its surplus
  // pages to the last CTA)
  const int my_splits = min(p.n_split, max(1, (n_pg + p.per_pages - 1) / p.per_pages));
  if (sp >= my_splits) return;
  const int pg0 = sp * p.per_pages, pg1 = sp == my_splits - 1 ? n_pg : pg0 + p.per_pages;
  const int n_it = max(pg1 - pg0, 0);
  const int pg_new = pos / PAGE_TOKENS, row_new = pos % PAGE_TOKENS;
  const bool has_new = p.append && sp == my_splits - 1;      // this CTA's range ends with the new key's page
  constexpr int half = HD / 2;
  for (int c = tid; c < half; c += NT) {
    float sn, cs;
    rope_sincos(pos, inv.f[c], &sn, &cs);
    rope[c] = make_float2(cs, sn);
  }
  __syncthreads();           // barriers and angles are there
  // The producer: pages [first, last) of the range into the ring, in order (warp NW, lane 0).
  bool ok = true;
  auto produce = [&](int first, int last) {
    int s = first % STG; uint32_t phase = (uint32_t)(first / STG) & 1u;
    for (int it = first; it < last; ++it) {
      if (it >= STG) ok = mbar_wait(empty(s), phase ^ 1u, abort_flag, p.status);
      if (!ok) break;
      const int pg = pg0 + it;
      const int page = pg < p.mpps ? p.block_table[(size_t)b * p.mpps + pg] : -1;
      if (page < 0 || page >= p.n_pages) {       // never used as a coordinate: the stage completes empty, consumers skip the page
        dev_flag(p.status, DEV_BAD_PAGE);
        mbar_arrive(full(s));
      } else {
        const int row0 = (page * p.nkv + kvh) * PAGE_TOKENS;
        const uint32_t dst = ring + s * 2 * PB;
        mbar_expect_tx(full(s), 2 * PB);
#pragma unroll
        for (int x = 0; x < HD / 64; ++x) {
          tma_load_2d(dst + x * BOX_BYTES, &map_k, x * 64, row0, full(s));
          tma_load_2d(dst + PB + x * BOX_BYTES, &map_v, x * 64, row0, full(s));
        }
      }
      if (++s == STG) { s = 0; phase ^= 1u; }
    }
  };
  const int n_ahead = min(n_it, STG);
  if (tid == NW * 32) produce(0, n_ahead);
  pdl_wait();
  const float* krow = p.q + (size_t)b * p.ldq + (size_t)(p.nq + kvh) * HD;
  if (has_new && p.k_gain) head_rnorm(krow, 1, HD, p.eps, &rk);
  // queries of the group: (query norm,) RoPE at the last position, scaled by 1/sqrt(hd); rows beyond the group are zero
  if (p.q_gain) head_rnorm(p.q + (size_t)b * p.ldq + (size_t)kvh * group * HD, group, HD, p.eps, rq);
  else __syncthreads();
  {
    const float scale = rsqrtf((float)HD);
    for (int i = tid; i < 8 * half; i += NT) {
      const int h = i / half, c = i - h * half;
      float r1 = 0.f, r2 = 0.f;
      if (h < group) {
        const float* qh = p.q + (size_t)b * p.ldq + (size_t)(kvh * group + h) * HD;
        const float2 cs = rope[c];
        float x1 = qh[c], x2 = qh[c + half];
        if (p.q_gain) { x1 *= rq[h] * p.q_gain[c]; x2 *= rq[h] * p.q_gain[c + half]; }
        r1 = (x1 * cs.x - x2 * cs.y) * scale;
        r2 = (x2 * cs.x + x1 * cs.y) * scale;
      }
      qs[h * LDQ + c] = r1;
      qs[h * LDQ + c + half] = r2;
    }
    if (has_new)
      for (int c = tid; c < half; c += NT) {
        const float2 cs = rope[c];
        const float* vrow = krow + (size_t)p.nkv * HD;
        float x1 = krow[c], x2 = krow[c + half];
        if (p.k_gain) { x1 *= rk * p.k_gain[c]; x2 *= rk * p.k_gain[c + half]; }
        knew[c] = from_f<kv16>(x1 * cs.x - x2 * cs.y);
        knew[c + half] = from_f<kv16>(x2 * cs.x + x1 * cs.y);
        vnew[c] = from_f<kv16>(vrow[c]);
        vnew[c + half] = from_f<kv16>(vrow[c + half]);
      }
  }
  __syncthreads();

  const int g = lane >> 2, qd = lane & 3;          // this lane's row (query head) and position in the row's quad
  float o[NTL][4];                                  // O fragments: [dims 8j..8j+7]: rows g (from P's value part), g + 8 (remainder part)
#pragma unroll
  for (int j = 0; j < NTL; ++j) { o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.f; }
  float m_run = -INFINITY, l_run = 0.f;

  if (tid == NW * 32) {
    produce(n_ahead, n_it);
    if (!ok) drain_after_abort();
  }
  if (warp < NW) {
    // ---------------- consumers: warp w takes keys 16 w .. 16 w + 15 of every page ----------------
    uint32_t qa[KS][4];                             // A fragments of Q: rows g = value part, g + 8 = remainder part
    // A head's queries are split after a multiplication by the power of two that puts its largest between 2^13 and 2^14 (`down` takes it
    // off the scores): no finite query is too large for a half, and remainders are normal halves down to 2^-16 of the largest.
    float2 qv[2 * KS];
    float mx = 0.f;
#pragma unroll
    for (int i = 0; i < 2 * KS; ++i) {
      qv[i] = *reinterpret_cast<const float2*>(qs + g * LDQ + i * 8 + 2 * qd);
      mx = fmaxf(mx, fmaxf(fabsf(qv[i].x), fabsf(qv[i].y)));
    }
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
    const int up_exp = min(253, 267 - (int)(__float_as_uint(mx) >> 23));
    const float up = __uint_as_float((uint32_t)up_exp << 23), down = __uint_as_float((uint32_t)(254 - up_exp) << 23);
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
      split2(qv[2 * ks].x * up, qv[2 * ks].y * up, qa[ks][0], qa[ks][1]);
      split2(qv[2 * ks + 1].x * up, qv[2 * ks + 1].y * up, qa[ks][2], qa[ks][3]);
    }
    const int k_lane = warp * 16 + (lane & 7);      // key row this lane addresses in matrix loads (+ 8 for the second key block)
    const int mi = lane >> 3;                        // which of the four 8 x 8 matrices of a load this lane addresses
    int s = -1; uint32_t phase = 0;
    for (int it = 0; it < n_it; ++it) {
      if (++s == STG) { s = 0; phase ^= 1u; }
      ok = mbar_wait(full(s), phase, abort_flag, p.status);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      const int pg = pg0 + it;
      const int page = pg < p.mpps ? p.block_table[(size_t)b * p.mpps + pg] : -1;
      const int nk = (page >= 0 && page < p.n_pages) ? min(PAGE_TOKENS, n_keys - pg * PAGE_TOKENS) : 0;
      if (warp * 16 < nk) {
        const uint32_t sk = ring + s * 2 * PB, sv = sk + PB;
        if (has_new && pg == pg_new && row_new >> 4 == warp) {
          // the new key and value take their row of the page: in this CTA's copy (only this warp reads it) and in the pool
          if (lane < HD / 8) {
            const uint4 uk = *reinterpret_cast<const uint4*>(knew + 8 * lane), uv = *reinterpret_cast<const uint4*>(vnew + 8 * lane);
            const uint32_t off = piece(row_new, lane);
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(sk + off), "r"(uk.x), "r"(uk.y), "r"(uk.z), "r"(uk.w) : "memory");
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(sv + off), "r"(uv.x), "r"(uv.y), "r"(uv.z), "r"(uv.w) : "memory");
            const size_t at = (((size_t)page * p.nkv + kvh) * PAGE_TOKENS + row_new) * HD + 8 * lane;
            *reinterpret_cast<uint4*>(p.kpool + at) = uk;
            *reinterpret_cast<uint4*>(p.vpool + at) = uv;
          }
          __syncwarp();
        }
        if (warp * 16 + 16 > nk) {
          // Rows at or beyond the sequence's end may hold anything, and 0 x NaN is NaN: the values of this warp's 16 become zero in the CTA's
          // copy.  (Their scores are never looked at.  Only a sequence's last page has such rows, and no copy into its stage follows.)
#pragma unroll 1
          for (int i = lane; i < (warp * 16 + 16 - nk) * (HD / 8); i += 32)
            asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(sv + piece(nk + i / (HD / 8), i % (HD / 8))), "r"(0u) : "memory");
          __syncwarp();
        }
        // ---- scores of this warp's 16 keys: two 8-key blocks
        float sc[2][4];
#pragma unroll
        for (int t = 0; t < 2; ++t) { sc[t][0] = sc[t][1] = sc[t][2] = sc[t][3] = 0.f; }
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
          uint32_t kb[4];        // matrices: (keys 0-7, dims 16ks..+7), (keys 0-7, dims +8..+15), (keys 8-15, ..), (keys 8-15, ..)
          ldsm4(sk + piece(k_lane + (mi >> 1) * 8, 2 * ks + (mi & 1)), kb);
          mma16816(sc[0], qa[ks], kb[0], kb[1]);
          mma16816(sc[1], qa[ks], kb[2], kb[3]);
        }
        // value row + remainder row of head g: this lane holds keys 2 qd, 2 qd + 1 of each 8-key block
        float sv4[4];
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          sv4[2 * t] = (sc[t][0] + sc[t][2]) * down;
          sv4[2 * t + 1] = (sc[t][1] + sc[t][3]) * down;
          const int key0 = warp * 16 + t * 8 + 2 * qd;
          if (key0 >= nk) sv4[2 * t] = -INFINITY;
          if (key0 + 1 >= nk) sv4[2 * t + 1] = -INFINITY;
        }
        float mt = fmaxf(fmaxf(sv4[0], sv4[1]), fmaxf(sv4[2], sv4[3]));
        mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 1));
        mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 2));
        if (mt > m_run) {                             // the row's maximum grows: rescale what this lane holds of the row
          const float a = (m_run == -INFINITY) ? 0.f : __expf(m_run - mt);
          l_run *= a;
#pragma unroll
          for (int j = 0; j < NTL; ++j) { o[j][0] *= a; o[j][1] *= a; o[j][2] *= a; o[j][3] *= a; }
          m_run = mt;
        }
        float pr[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) { pr[i] = (sv4[i] == -INFINITY) ? 0.f : __expf(sv4[i] - m_run); l_run += pr[i]; }
        uint32_t pa[4];          // A fragment of P: (row g, keys 2qd..) value, (row g + 8) remainder, then the second key block
        split2(pr[0], pr[1], pa[0], pa[1]);
        split2(pr[2], pr[3], pa[2], pa[3]);
        // ---- values: O[16 x HD] += P[16 x 16 keys] V[16 keys x HD]
#pragma unroll
        for (int j = 0; j < NTL; j += 2) {
          uint32_t vb[4];        // matrices: (keys 0-7, dims 8j..), (keys 8-15, dims 8j..), (keys 0-7, dims 8(j+1)..), (keys 8-15, ..)
          ldsm4_t(sv + piece(k_lane + (mi & 1) * 8, j + (mi >> 1)), vb);
          mma16816(o[j], pa, vb[0], vb[1]);
          mma16816(o[j + 1], pa, vb[2], vb[3]);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty(s));           // this warp is through with the stage
    }
  }
  // (Only now: the next projection's CTAs take a whole SM each while they wait, and over long caches they would keep it from CTAs of
  // other streams for as long as the slowest range here takes.)
  pdl_trigger();
  // every thread learns whether some wait ran out (copies may then still be landing in this CTA's shared memory)
  if (!__syncthreads_and(ok && *abort_flag == 0)) {
    drain_after_abort();
    return;
  }
  // ---- the four warps' partial results meet in shared memory (the ring is idle: every copy issued was waited for)
  constexpr int LDR = HD + 2;
  float* red = reinterpret_cast<float*>(smem);                                   // [NW][8][HD + 2]
  if (warp < NW) {
    l_run += __shfl_xor_sync(0xffffffffu, l_run, 1);
    l_run += __shfl_xor_sync(0xffffffffu, l_run, 2);
    float* r = red + (size_t)(warp * 8 + g) * LDR;
#pragma unroll
    for (int j = 0; j < NTL; ++j)
      *reinterpret_cast<float2*>(r + 8 * j + 2 * qd) = make_float2(o[j][0] + o[j][2], o[j][1] + o[j][3]);
    if (qd == 0) { r[HD] = m_run; r[HD + 1] = l_run; }
  }
  __syncthreads();
  const int ldr = HD + 2;
  for (int e = tid; e < group * HD; e += NT) {
    const int gg = e / HD, d = e - gg * HD;
    float mm = -INFINITY;
#pragma unroll
    for (int w = 0; w < NW; ++w) mm = fmaxf(mm, red[(size_t)(w * 8 + gg) * LDR + HD]);
    float v = 0.f, l = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      const float* r = red + (size_t)(w * 8 + gg) * LDR;
      const float f = (r[HD] == -INFINITY) ? 0.f : __expf(r[HD] - mm);
      v = fmaf(r[d], f, v);
      l = fmaf(r[HD + 1], f, l);
    }
    const int qh = kvh * group + gg;
    if (my_splits == 1) {
      emit(p, b, (size_t)p.nq * HD, qh * HD + d, v / l);
    } else {
      float* pr = p.part + (((size_t)b * p.nq + qh) * p.n_split + sp) * ldr;
      pr[d] = v;
      if (d == 0) { pr[HD] = mm; pr[HD + 1] = l; }
    }
  }
  // With more than one split the CTA that finishes the group's last split merges the partial results on the spot
  // (counter per (sequence, kv head), zero at launch and left zero).
  if (my_splits > 1) {
    __threadfence();                               // this CTA's partial results are visible before it counts itself done
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(p.split_done + b * p.nkv + kvh, 1) == my_splits - 1;
    __syncthreads();
    if (s_last) {
      __threadfence();
      if (tid == 0) p.split_done[b * p.nkv + kvh] = 0;
      for (int e = tid; e < group * HD; e += NT) {
        const int gg = e / HD, d = e - gg * HD;
        const int qh = kvh * group + gg;
        const float* pr = p.part + ((size_t)b * p.nq + qh) * p.n_split * ldr;
        float mm = -INFINITY;
        for (int s = 0; s < my_splits; ++s) mm = fmaxf(mm, __ldcg(pr + (size_t)s * ldr + HD));
        float ll = 0.f, v = 0.f;
        for (int s = 0; s < my_splits; ++s) {
          const float* r = pr + (size_t)s * ldr;
          const float ms = __ldcg(r + HD);
          const float f = (ms == -INFINITY) ? 0.f : __expf(ms - mm);
          ll = fmaf(__ldcg(r + HD + 1), f, ll);
          v = fmaf(__ldcg(r + d), f, v);
        }
        emit(p, b, (size_t)p.nq * HD, qh * HD + d, v / ll);
      }
    }
  }
}

// fp16 pool [rows, hd] row-major; box = 64 dims x 64 keys, 128-byte swizzle
bool make_pool_map(CUtensorMap* m, const void* pool, long long rows, int hd) {
  return tc_make_map_bf16(m, pool, rows, hd, hd, 64);      // halves are 2-byte elements like bf16 for the copy engine
}

template <int HD>
cudaError_t go_mma(const CUtensorMap& mk, const CUtensorMap& mv, const InvFreq& inv, const MmaParams& p, dim3 grid, cudaStream_t st) {
  static bool raised[TC_MAX_DEVICES] = {};
  cudaError_t e = tc_raise_smem_limit(step_attn_mma_kernel<HD>, MmaCfg<HD>::smem(MmaCfg<HD>::STAGES), raised);
  if (e != cudaSuccess) return e;
  return launch_overlapped(step_attn_mma_kernel<HD>, grid, dim3(NT), (size_t)MmaCfg<HD>::smem(p.stages), st, mk, mv, inv, p);
}

}  // namespace

// Key-range splits: at most `upper`, chosen so that the CTAs fill whole waves of the SMs' resident slots.
int step_attn_mma_splits(int batch, int nkv, int hd, int max_keys, int upper) {
  const int items = batch * nkv;
  const int n_pg = (max_keys + PAGE_TOKENS - 1) / PAGE_TOKENS;
  int best = 1; long long best_cost = -1;
  for (int n = 1; n <= upper; ++n) {
    const int per = (n_pg + n - 1) / n;
    const long long slots = 148LL * mma_per_sm(hd, mma_stages(hd, per)), waves = ((long long)items * n + slots - 1) / slots;
    const long long cost = waves * (per + 3);
    if (best_cost < 0 || cost < best_cost) { best = n; best_cost = cost; }
  }
  return best;
}

bool step_attn_mma_supported(int dtype, int nq, int nkv, int hd, const void* kpool, const void* vpool, int n_pages) {
  const int group = nq / nkv;
  return dtype == 1 && (hd == 64 || hd == 128) && group >= 1 && group <= 8 && ((uintptr_t)kpool & 15) == 0 && ((uintptr_t)vpool & 15) == 0 &&
         (long long)n_pages * nkv * PAGE_TOKENS < (1LL << 31) && tc_encode_fn() != nullptr;
}

cudaError_t launch_step_attn_mma(const LaunchCtx& ctx, const StepAttn& a, int n_split) {
  const int nq = a.nq, nkv = a.nkv, hd = a.hd, max_keys = a.max_keys;
  if (n_split > 1 && !a.split_done) return cudaErrorInvalidValue;
  const int max_pg = (max_keys + PAGE_TOKENS - 1) / PAGE_TOKENS;
  const int per_pages = (max_pg + n_split - 1) / n_split > 0 ? (max_pg + n_split - 1) / n_split : 1;
  InvFreq inv;
  fill_inv_freq(&inv, hd, a.theta);
  CUtensorMap mk, mv;
  const long long rows = (long long)a.n_pages * nkv * PAGE_TOKENS;
  if (!make_pool_map(&mk, a.kpool, rows, hd) || !make_pool_map(&mv, a.vpool, rows, hd)) return cudaErrorInvalidValue;
  MmaParams p{a.q, a.ldq, nq, nkv, a.block_table, a.mpps, a.n_pages, a.seq_lens, a.extra, n_split, a.part, ctx.status, a.q_gain, a.eps,
              a.split_done, per_pages, mma_stages(hd, per_pages), a.xb ? nullptr : a.out, a.xb, step_tc_rows(a.batch, a.terms), a.terms, a.append, a.k_gain, (kv16*)a.kpool, (kv16*)a.vpool};
  dim3 grid(n_split, nkv, a.batch);
  ++*ctx.n_launch;
  return hd == 64 ? go_mma<64>(mk, mv, inv, p, grid, ctx.st) : go_mma<128>(mk, mv, inv, p, grid, ctx.st);
}
