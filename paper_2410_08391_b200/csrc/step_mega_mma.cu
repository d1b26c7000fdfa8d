// The base model's single-token step as ONE persistent cooperative kernel for 16-bit weights (batch <= 4), with the
// multiply on the warp-level tensor cores and without grid-wide barriers.
//
// What bounds it: the step is a chain of dependent phases (5 per layer, 141 in the 1.1B shape) whose weights stream from HBM once; a
// phase's own bytes take 1-7 us, so whatever sits in series between two phases counts as much as the bytes do.  Hence:
//   - No barrier.  Every value that one CTA hands to others (projections, attention, residual stream) is stored as ONE
//     64-bit word {fp32 value, tag}, the tag being the layer; whoever needs a value polls the value itself.  That takes the
//     place of block barrier, fence (about 900 cycles), arrival, polling, block barrier and fetch.  Reuse of a buffer in the
//     next layer is safe because its writers have, through the chain of phases between, read results of all its readers.
//     The host clears the buffers in front of every step.
//   - The weights of a phase are cut by OUTPUT ROWS, one contiguous range per CTA (within one row of equal shares), and
//     travel as slots of 8 rows x up to 2048 k through one shared-memory ring per CTA (one bulk copy per row piece).  The copy
//     engine takes about 55 cycles per copy whatever its size, so pieces of 4 KB (75 bytes per cycle) feed twice as fast as
//     pieces of 2 KB; HBM's share of an SM is 23.  Two loader warps walk the static schedule of the whole step, so the ring is
//     full again before a phase's input exists, and a third asks the rows behind the ring into L2 (per line, not through the
//     copy engine, which works in order), so that HBM streams on while the ring is full (1 x 1100 keys, 1.1B shape:
//     4 % of the step).  Rows lie 4160 bytes apart: the 16-byte reads of two rows then cover all 32 banks.
//   - The 8 consumer warps cut K: warp w owns an eighth of every chunk.  A warp therefore needs only its own eighth of the
//     activations, which it fetches and converts by itself: no staging of the whole input.  The 1 / rms of RMSNorm is
//     applied to the outputs (its sum of squares falls out of the fetch), so nothing waits for it.
//   - Products are mma.sync m16n8k16 with the weights as A (read once from shared memory, no unpacking) and the activations
//     as B.  An fp32 activation enters as three bf16 terms (x = hi + mid + lo, 24 significant bits: nothing of the fp32
//     value is dropped) in three of four columns, so one 8-column instruction serves two sequences.
//   - The accumulation inside an instruction rounds towards zero: one sum over a warp's whole share of K left a step's logits
//     twice as far from 64 bits as fp32 multiply-adds do (1.1B shape 3.1e-6 against 1.5e-6, 3B shape 4.7e-6 against 2.1e-6, on
//     the same cache).  So a sum goes through few instructions: with one sequence the hi terms of successive blocks of 32 k
//     take turns in four columns, with two sequences in two; a chunk is summed apart and added in fp32.  Now 1.3e-6 .. 1.7e-6 and 1.8e-6 .. 1.9e-6, for up to 1 % of a step's time (8 heads of 128 a group: 3 %; two sequences:
//     1 .. 5 %).
//   - The cache pages of an attention item are brought into shared memory by a warp of their own, ahead of the query; the
//     step's own key and value are taken from the projection's output by the CTA whose key range ends with them (no separate
//     append phase); RoPE angles are computed once per launch.
//   - 12 warps of up to 168 registers: next to 220 KB of shared memory there is almost no L1, so every spilled register
//     is a round trip to L2.  Up to 4 heads a group nothing spills; groups of 5 to 8 heads spill 16 to 92 bytes (ptxas).
//   - The instructions of a layer's phases are fetched anew in every layer: a clock trace showed 1080 cycles a tile where its shared-memory
//     reads take 512, and more of them in proportion to the code's length.  So a group's tiles are ONE loop whose sums wait in shared
//     memory, not five straight-line copies with their sums in registers.  Generation step, 1.1B shape: 1 x 1100 keys 840 -> 807 us,
//     2 x 300 888 -> 824, 4 x 300 1109 -> 1075; on the 72 SMs of a piece, with twice the tiles a CTA, more (first token of 1 x 59 1532 -> 1363 us,
//     1 x 1024 1733 -> 1649); 3B shape 2 x 300 2242 -> 2126.  The price is a sum over columns with every chunk of a
//     tile, not one a tile (3B shape 1 x 300 1979 -> 2016, 4 x 300 2401 -> 2407); lanes that share it by rows took half of that back
//     (2000, 2374; 1.1B shape 4 x 300 1075 -> 1067; the same bits).
// Measured against the CUDA-core kernel of step_mega.cu (generation step): 1.1B shape 1 x 1100 keys 1557 -> 807 us, 4 x 300
// 2990 -> 1067 us (that kernel's multiply-adds grow with the batch); 3B shape 1 x 300 2966 -> 1787 us, 4 x 300 5578 -> 2374 us.
// The bytes of the first take 416 us.  Of the rest, per layer of 26 us: waits for inputs 0.4-0.7 us a phase, attention's exchange between
// key ranges 2.8, its wait for the queries 1.3, the tiles of O and down (4.0 us, weights 4.8 on HBM) and gate / up (3.9, 7.0).
// Every wait is bounded: on expiry DEV_TIMEOUT is recorded, no further wait is started, every CTA runs through its remaining
// phases without waiting or releasing slots, its loaders stop, and it leaves after copies in flight have had time to land.
#include <math.h>

#include "common.cuh"
#include "tc_ptx.cuh"
#include "step_mega.h"
#include "step_waits.cuh"

namespace {
using namespace tcp;

constexpr int CW = 8;                        // consumer warps: with two loader warps 3 warps per scheduler, 168 registers each
constexpr int CT = CW * 32;                  // consumer threads
constexpr int LW = 2;                        // weight loader warps
constexpr int NT = CT + 32 * (LW + 2);       // + L2 prefetch warp + cache-page loader warp: 12 warps, 168 registers each
constexpr int TR = 16;                       // weight rows of a tile
constexpr int KS = 128;                      // k elements that a warp converts at a time
// Tiles are 16 rows x up to 2048 k, in two ring slots of 8 rows (copies of 4 KB; with 2 KB copies the copy engine's cost per copy
// bounds the feed); where the accumulators and columns of four sequences leave no registers for that, 1024 k in one slot.
template <int BB> struct Geo {
  static constexpr int KC = BB == 4 ? 1024 : 2048;
  static constexpr int HR = BB == 4 ? 16 : 8;  // rows of a slot
  static constexpr int KW = KC / CW;         // k elements of a consumer warp
  static constexpr int PITCH = KC * 2 + 64;  // bytes between rows of a slot (64 mod 128: no bank conflicts)
  static constexpr int STAGE = HR * PITCH;
  static constexpr int TG = BB == 4 ? 5 : 8; // tiles whose sums a CTA holds at a time (the input is fetched anew for every group of them)
  static constexpr int AHEAD = 5;            // slots that the L2 prefetch runs ahead of the loaders (25 MB on 148 SMs)
  // k elements of a chunk of a row of K: as few chunks as possible, of about equal size, whole 64s for every consumer warp
  __device__ __forceinline__ static int chunk(int K) {
    const int n = (K + KC - 1) / KC;
    return min(KC, ((K + n - 1) / n + 64 * CW - 1) / (64 * CW) * (64 * CW));
  }
};
constexpr int MAXG = 8;                      // query heads per kv head (kernels for up to 4 and up to 8)
constexpr int XCOL = KS * 2 + 64;            // bytes between activation columns of a warp (64 mod 128)
constexpr int MAX_SLOTS = 12;
constexpr int RESID_MAX = 1024;              // residual-stream values a CTA keeps
constexpr int MAX_SPLIT = 32;
constexpr int SMEM_LIMIT = 227 * 1024;

struct Plan { int n_stage, n_kv, kv_off, scr_off; };

__device__ __forceinline__ void consumer_sync() { asm volatile("bar.sync 1, %0;" ::"n"(CT) : "memory"); }

__device__ __forceinline__ uint4 lds128(uint32_t a) {
  uint4 u;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(u.x), "=r"(u.y), "=r"(u.z), "=r"(u.w) : "r"(a));
  return u;
}

__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// A projection phase: 4 per layer (q(kv), O, gate/up, down), then the LM head.
struct Proj { const char* W; int N, K, mode, G, ffn; };
__device__ __forceinline__ Proj proj_of(const MegaParams& p, int s) {
  if (s >= 4 * p.n_layers) return Proj{(const char*)p.lm_head, p.vocab, p.d, GEMV_STORE, 0, 0};
  const MegaLayer& L = p.layers[s >> 2];
  switch (s & 3) {
    case 0: return Proj{(const char*)L.wqkv, p.generation ? L.nqkv : L.dq, p.d, GEMV_STORE, 0, 0};
    case 1: return Proj{(const char*)L.wo, p.d, L.dq, GEMV_RESID, 0, 0};
    case 2: return Proj{(const char*)L.wgu, L.ffn, p.d, GEMV_SWIGLU, L.G, L.ffn};
    default: return Proj{(const char*)L.wd, p.d, L.ffn, GEMV_RESID, 0, 0};
  }
}
// This CTA's outputs [o0, o1) of a projection with N outputs.
__device__ __forceinline__ void cta_range(int N, int& o0, int& o1) {
  o0 = (int)((long long)N * blockIdx.x / gridDim.x);
  o1 = (int)((long long)N * (blockIdx.x + 1) / gridDim.x);
}
// Key-range splits of a layer's attention: about one item per CTA, no more splits than the longest sequence has pages.
__device__ __forceinline__ int attn_splits(int batch, int nkv, int max_pages) {
  return max(1, min(min(MAX_SPLIT, max_pages), (int)gridDim.x / (batch * nkv)));
}
struct Item { int b, kvh, sp, r, pg0, pg1, n_keys; };
__device__ __forceinline__ Item item_of(const MegaParams& p, int it, int nkv, int ns, const int* s_len) {
  Item q;
  q.sp = it % ns; q.r = it / ns;
  q.b = q.r / nkv; q.kvh = q.r - q.b * nkv;
  q.n_keys = s_len[q.b] + (p.generation ? 1 : 0);
  const int n_pg = (q.n_keys + PAGE_TOKENS - 1) / PAGE_TOKENS, per = (n_pg + ns - 1) / ns;
  q.pg0 = min(n_pg, q.sp * per);
  q.pg1 = min(n_pg, q.pg0 + per);
  return q;
}

// Calls f(slot number, projection, weight row of this lane, whether the lane has one, chunk, chunk length) for every ring
// slot of the launch's schedule in the consumers' order, by a whole warp; stops when f returns false.  A tile of a SwiGLU
// projection is the 8 gate rows and the 8 up rows of 8 outputs.
template <int BB, class F>
__device__ __forceinline__ bool walk_slots(const MegaParams& p, F f) {
  constexpr int HR = Geo<BB>::HR;
  const int lane = threadIdx.x & 31, s_end = 4 * p.layer_end + (p.do_head ? 1 : 0);
  int n = 0;
  for (int s = 4 * p.layer_begin; s < s_end; ++s) {
    const Proj g = proj_of(p, s == 4 * p.layer_end ? 4 * p.n_layers : s);
    int o0, o1;
    cta_range(g.N, o0, o1);
    const bool sw = g.mode == GEMV_SWIGLU;
    const int TO = sw ? TR / 2 : TR, nt = (o1 - o0 + TO - 1) / TO, kc = Geo<BB>::chunk(g.K), nch = (g.K + kc - 1) / kc;
    for (int g0 = 0; g0 < nt; g0 += Geo<BB>::TG) {
      const int ntg = min(Geo<BB>::TG, nt - g0);
      for (int c = 0; c < nch; ++c)
        for (int hs = 0; hs < TR / HR * ntg; ++hs) {
          const int r = (hs * HR & (TR - 1)) + lane;              // row of the tile
          const int first = o0 + g0 * TO + (sw ? hs * HR / TR * TO : hs * HR);
          if (first >= o1) continue;
          const int up = r >> 3 & 1, o = sw ? first + (r & 7) : first + lane;
          const int row = sw ? map_row(RowMap{up && g.G == 0 ? g.ffn : 0, g.G, up, g.ffn}, o) : o;
          if (!f(n++, g, row, lane < HR && o < o1, c, kc)) return false;
        }
    }
  }
  return true;
}

// State of a role that walks a ring.
struct Ring {
  uint32_t base, full, empty; int n, slot; uint32_t phase; int bytes;
  __device__ __forceinline__ void next() { if (++slot == n) { slot = 0; phase ^= 1u; } }
};

// Shared by all roles of a CTA.
struct Shared {
  u64 bars[2 * MAX_SLOTS + 2 * 2 + 1];                 // ring full / empty, cache-page ring full / empty, RoPE table ready
  float ss[2][CW * 4];                         // per warp and sequence: sum of squares of its share of the input (by phase parity)
  float resid[RESID_MAX];                      // the residual stream at this CTA's outputs [row][sequence]
  float2 rope[4 * 64];                         // (cos, sin) of every sequence's position
  int len[4];                                  // cached keys per sequence
  int tok[4];                                  // token per sequence, -1 = out of range
  int kv_rows[2];                              // cached rows in a page slot, -1 = bad page
  int max_pages, abort;
  int issued;                                  // a ring slot lately asked for
  __align__(16) unsigned zeros[16];
  __align__(16) kv16 knew[128];                // the step's own key and value (of one kv head)
  __align__(16) kv16 vnew[128];
};

// What a consumer needs to know of a phase (the descriptors come from constant memory and the divisions take a while: all
// of it before the input is there).
struct Work {
  int K, N, o0, o1, mode, nt, nch, kc;
  float inv_k;
  const u64* x; const bf16* embed;             // input: tagged values, or (first layer) rows of the embedding table
  const float* gain;
  u64* y; float* logits;                       // output: tagged values, or the logits
  uint32_t tag_in, tag_out;
};
template <int BB>
__device__ __forceinline__ Work work_of(const MegaParams& p, int i, int kind, bool head) {
  const MegaLayer& L = p.layers[head ? 0 : i];
  const Proj g = proj_of(p, head ? 4 * p.n_layers : 4 * i + (kind ? kind - 1 : 0));
  Work w;
  w.K = g.K; w.N = g.N; w.mode = g.mode;
  cta_range(g.N, w.o0, w.o1);
  const int TO = g.mode == GEMV_SWIGLU ? TR / 2 : TR;
  w.nt = (w.o1 - w.o0 + TO - 1) / TO;
  w.kc = Geo<BB>::chunk(g.K);
  w.nch = (g.K + w.kc - 1) / w.kc;
  w.inv_k = 1.f / (float)g.K;
  const bool first = kind == 0 && i == 0 && !head;
  w.embed = first ? (const bf16*)p.embed : nullptr;
  w.x = kind == 2 ? p.ll_a : (kind == 4 ? p.ll_h : (kind == 3 ? p.ll_x1 : p.ll_x2));
  w.tag_in = kind == 0 || head ? (uint32_t)i : (uint32_t)i + 1u;      // x2 comes from the layer before; layer i's tag is i + 1
  w.tag_out = (uint32_t)i + 1u;
  w.gain = head ? p.final_norm : (kind == 0 ? L.attn_norm : (kind == 3 ? L.ffn_norm : nullptr));
  w.y = kind == 0 ? p.ll_q : (kind == 2 ? p.ll_x1 : (kind == 3 ? p.ll_h : p.ll_x2));
  w.logits = head ? p.logits : nullptr;
  return w;
}

// ---- projection: y[b, o] (op)= sum_k W[o, k] x[b, k] for this CTA's outputs --------------------------------------------
// xp: this warp's private shared memory (3 BB columns of XCOL bytes); red: [2][CW][TG * 16 * BB] floats.
// The loop over chunks is kept rolled: every phase runs through this code once per layer, and straight-line
// copies of it cost more in instruction fetches than the loop does.
template <int BB>
__device__ __forceinline__ void proj_phase(const MegaParams& p, const Work& g, Ring& rg, uint32_t xp, float* red0, int& par, Shared& sh, bool& dead,
                                           u64* best) {
  constexpr int NB = BB == 4 ? 2 : 1;          // 8-column groups: two sequences each
  constexpr int HR = Geo<BB>::HR, KW = Geo<BB>::KW, PITCH = Geo<BB>::PITCH, STAGE = Geo<BB>::STAGE;   // (KW: most that a warp's share can be)
  const int kws = g.kc / CW;                   // k elements of a warp's share of a chunk
  constexpr int TG = Geo<BB>::TG, RS = TG * TR * BB;
  constexpr int NJ = KW / 32;                  // 32-k blocks of a warp's share of a chunk
  constexpr int NH = KW / KS, QJ = KS / 32;    // ... handled as NH pieces of QJ blocks
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gr = lane >> 2, t = lane & 3;
  volatile int* s_abort = &sh.abort;
  const bool sw = g.mode == GEMV_SWIGLU;
  const int TO = sw ? TR / 2 : TR;
  const int nch = g.nch;
  // Columns 4 b .. 4 b + 2 of an instruction hold sequence b's hi, mid and lo terms.  With one or two sequences, the hi terms of
  // successive blocks of 32 k take turns in the columns that are left (0 and 3, and 4 and 5 beside one sequence; zeros where it
  // is another column's turn); with four, column 3 holds the lo term again and is not used.
  constexpr int TURNS = BB == 1 ? 4 : 2;
  const int cpart = BB == 1 ? gr : gr & 3, cterm = cpart == 1 || cpart == 2 ? cpart : (BB == 4 && cpart == 3 ? 2 : 0);
  const int cturn = cpart ? cpart - 2 : 0;
  const uint32_t cbase = xp + (3 * (BB == 1 ? 0 : gr >> 2) + cterm) * XCOL + t * 16, czero = smem_u32(sh.zeros) + t * 16;
  const int ss_par = par >> 1;                 // par: bit 0 = half of the partial sums, bit 1 = half of the sums of squares
  u64 xr[NH][BB][4];
  float4 gv[NH];
  int n_load = (g.nt + TG - 1) / TG * nch;     // chunks still to be asked for
  auto fetch_x = [&](int i, int c) {           // (a lane beyond the row's end holds zeros of the right tag)
    const int kl = i * KS + 4 * lane, k = kl < kws ? c * g.kc + warp * kws + kl : g.K;
#pragma unroll
    for (int b = 0; b < BB; ++b) {
#pragma unroll
      for (int e = 0; e < 4; ++e) xr[i][b][e] = (u64)g.tag_in << 32;
      if (k < g.K && b < p.batch) {
        if (!g.embed) {
          const u64* src = g.x + (size_t)b * g.K + k;
          ll_load2(src, xr[i][b][0], xr[i][b][1]);
          ll_load2(src + 2, xr[i][b][2], xr[i][b][3]);
        } else if (sh.tok[b] >= 0) {
          const uint2 u = __ldg(reinterpret_cast<const uint2*>(g.embed + (size_t)sh.tok[b] * g.K + k));
          xr[i][b][0] |= u.x << 16; xr[i][b][1] |= u.x & 0xffff0000u;
          xr[i][b][2] |= u.y << 16; xr[i][b][3] |= u.y & 0xffff0000u;
        }
      }
    }
  };
  auto fetch = [&](int c) {
    if (n_load <= 0) return;
    --n_load;
#pragma unroll
    for (int i = 0; i < NH; ++i) {
      const int kl = i * KS + 4 * lane, k = kl < kws ? c * g.kc + warp * kws + kl : g.K;
      gv[i] = (g.gain && k < g.K) ? __ldg(reinterpret_cast<const float4*>(g.gain + k)) : make_float4(1.f, 1.f, 1.f, 1.f);
      fetch_x(i, c);
    }
  };
  auto ready = [&](int i) {
    bool ok = true;
#pragma unroll
    for (int b = 0; b < BB; ++b)
#pragma unroll
      for (int e = 0; e < 4; ++e) ok = ok && ll_tag(xr[i][b][e]) == g.tag_in;
    return ok;
  };
  fetch(0);
  const int ob = threadIdx.x % BB;             // the sequence whose outputs this thread finishes
  u64 mine = 0ull;
  float ss[BB];
#pragma unroll
  for (int b = 0; b < BB; ++b) ss[b] = 0.f;
  for (int t0 = 0; t0 < g.nt; t0 += TG) {
    const int ntg = min(TG, g.nt - t0);
    float* red = red0 + (par & 1) * (CW * RS);
#pragma unroll 1
    for (int c = 0; c < nch; ++c) {
      // the chunk's activations: poll until every value carries the wanted tag
      unsigned it = 0;
      while (!dead) {
        bool ok = true;
#pragma unroll
        for (int i = 0; i < NH; ++i) ok = ok && ready(i);
        if (__all_sync(0xffffffffu, ok)) break;
        // One lane waits for one of the missing values before the warp asks for all of them again: every SM wants the same
        // few lines, and whole warps that poll them hold up the stores that everybody is waiting for.
        const int who = __ffs(__ballot_sync(0xffffffffu, !ok)) - 1;
        if (lane == who) {
          int k = c * g.kc + warp * kws + 4 * lane, b = 0;
#pragma unroll
          for (int i = 0; i < NH; ++i)
#pragma unroll
            for (int bb = 0; bb < BB; ++bb)
              if (ll_tag(xr[i][bb][0]) != g.tag_in || ll_tag(xr[i][bb][1]) != g.tag_in || ll_tag(xr[i][bb][2]) != g.tag_in ||
                  ll_tag(xr[i][bb][3]) != g.tag_in) { k = c * g.kc + warp * kws + i * KS + 4 * lane; b = bb; }
          u64 q0, q1, q2, q3;
          do {
            if (!poll_more(it, s_abort, p.status)) { dead = true; break; }
            const u64* src = g.x + (size_t)b * g.K + k;
            ll_load2(src, q0, q1);
            ll_load2(src + 2, q2, q3);
          } while (ll_tag(q0) != g.tag_in || ll_tag(q1) != g.tag_in || ll_tag(q2) != g.tag_in || ll_tag(q3) != g.tag_in);
        }
        dead = __any_sync(0xffffffffu, dead);
#pragma unroll
        for (int i = 0; i < NH; ++i)
          if (!ready(i)) fetch_x(i, c);
      }
      auto column = [&](int nb, int j) {
        return lds128(BB == 4 || cterm || cturn == (j & (TURNS - 1)) ? cbase + 6 * nb * XCOL + j * 64 : czero);
      };
      uint4 bq[NJ];
#pragma unroll
      for (int i = 0; i < NH; ++i) {
#pragma unroll
        for (int b = 0; b < BB; ++b) {
          const float v0 = ll_val(xr[i][b][0]), v1 = ll_val(xr[i][b][1]), v2 = ll_val(xr[i][b][2]), v3 = ll_val(xr[i][b][3]);
          if (t0 == 0) ss[b] += fmaf(v0, v0, v1 * v1) + fmaf(v2, v2, v3 * v3);
          float e[4] = {v0 * gv[i].x, v1 * gv[i].y, v2 * gv[i].z, v3 * gv[i].w};
#pragma unroll
          for (int part = 0; part < 3; ++part) {
            const __nv_bfloat162 h0 = __floats2bfloat162_rn(e[0], e[1]), h1 = __floats2bfloat162_rn(e[2], e[3]);
            asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(xp + (3 * b + part) * XCOL + lane * 8),
                         "r"(*reinterpret_cast<const uint32_t*>(&h0)), "r"(*reinterpret_cast<const uint32_t*>(&h1)) : "memory");
            const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
            e[0] -= f0.x; e[1] -= f0.y; e[2] -= f1.x; e[3] -= f1.y;
          }
        }
        __syncwarp();
        if (NB == 1) {                         // (two groups of columns are read again for every tile: no registers for them)
#pragma unroll
          for (int j = 0; j < QJ; ++j) bq[i * QJ + j] = column(0, j);
          __syncwarp();                        // every lane has read the columns
        }
      }
      fetch(c + 1 < nch ? c + 1 : 0);
      const int kw = min(kws, g.K - c * g.kc - warp * kws);      // of them within the row
      // One copy of a tile's code for all of them (see the head of the file)
#pragma unroll 1
      for (int ti = 0; ti < ntg; ++ti) {
        // the tile's two slots: rows 0-7 and 8-15 (SwiGLU: the gate rows and the up rows); a last tile may have the first only
        const bool two = HR < TR && (sw || g.o0 + (t0 + ti) * TR + HR < g.o1);
        const uint32_t off = gr * PITCH + warp * (kws * 2) + t * 16;
        const uint32_t a = rg.base + rg.slot * STAGE + off, bar_a = rg.empty + 8u * rg.slot;
        if (!dead) dead = !quick_wait(rg.full + 8u * rg.slot, rg.phase, s_abort, p.status);
        rg.next();
        const uint32_t b = HR == TR ? a + 8 * PITCH : (two ? rg.base + rg.slot * STAGE + off : a), bar_b = rg.empty + 8u * rg.slot;
        if (two) {
          if (!dead) dead = !quick_wait(rg.full + 8u * rg.slot, rg.phase, s_abort, p.status);
          rg.next();
        }
        __syncwarp();
        float part[NB][4];                     // the tile's share of the chunk
#pragma unroll
        for (int nb = 0; nb < NB; ++nb)
#pragma unroll
          for (int e = 0; e < 4; ++e) part[nb][e] = 0.f;
        if (kw > 0) {
#pragma unroll
          for (int jh = 0; jh < NJ; jh += 2) {
            if (jh * 32 >= kws) break;
            uint4 ua[2], ub[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) { ua[j] = lds128(a + (jh + j) * 64); ub[j] = lds128(b + (jh + j) * 64); }
            if (kw < kws) {                    // k beyond the rows' end
#pragma unroll
              for (int j = 0; j < 2; ++j)
                if ((jh + j) * 32 + t * 8 >= kw) { ua[j] = make_uint4(0, 0, 0, 0); ub[j] = ua[j]; }
            }
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
              for (int nb = 0; nb < NB; ++nb) {
                const uint4 bb = NB == 1 ? bq[jh + j] : column(nb, jh + j);
                mma16816(part[nb], ua[j].x, ub[j].x, ua[j].y, ub[j].y, bb.x, bb.y);
                mma16816(part[nb], ua[j].z, ub[j].z, ua[j].w, ub[j].w, bb.z, bb.w);
              }
          }
        }
        __syncwarp();
        if (lane == 0 && !dead) { mbar_arrive(bar_a); if (two) mbar_arrive(bar_b); }
        // hi + mid + lo columns; the chunks of K add up in this warp's part of `red`
#pragma unroll
        for (int nb = 0; nb < NB; ++nb) {
          const bool pair = BB < 4 || !(t & 1);
          const float v0 = part[nb][0] + (pair ? part[nb][1] : 0.f), v1 = part[nb][2] + (pair ? part[nb][3] : 0.f);
          // an even lane of the quad goes on with row gr, an odd one with row gr + 8
          const float out = t & 1 ? v0 : v1;
          float v = t & 1 ? v1 : v0;
          v += __shfl_xor_sync(0xffffffffu, out, 1);
          if (BB == 1) v += __shfl_xor_sync(0xffffffffu, v, 2);
          const int bs = BB == 1 ? 0 : nb * 2 + (t >> 1);
          if (BB == 1 ? t < 2 : bs < BB) {
            float* d = red + warp * RS + (ti * TR + gr + 8 * (t & 1)) * BB + bs;
            if (c > 0) v += *d;
            *d = v;
          }
        }
      }
      dead = __any_sync(0xffffffffu, dead);    // (also: every lane has read this chunk's columns)
    }
    // ---- the group's outputs: the sum over the warps' k ranges
    if (t0 == 0 && g.gain) {
#pragma unroll
      for (int b = 0; b < BB; ++b) {
        const float s = warp_sum(ss[b]);
        if (lane == 0) sh.ss[ss_par][warp * BB + b] = s;
      }
    }
    consumer_sync();
    const int n_vals = ntg * TO * BB;          // (output, sequence) pairs of the group, the sequence running fastest
    const int o_base = g.o0 + t0 * TO;
    float r = 1.f;
    if (g.gain) {
      float s = 0.f;
#pragma unroll
      for (int w = 0; w < CW; ++w) s += sh.ss[ss_par][w * BB + ob];
      r = rsqrtf(s * g.inv_k + p.eps);
    }
    for (int i = threadIdx.x; i < n_vals; i += CT) {
      const int orow = i / BB, o = o_base + orow;
      if (o >= g.o1 || ob >= p.batch) break;
      const int src = sw ? ((orow >> 3) * TR + (orow & 7)) * BB + ob : i;
      float v = 0.f, u = 0.f;
#pragma unroll
      for (int w = 0; w < CW; ++w) v += red[w * RS + src];
      v *= r;
      if (sw) {
#pragma unroll
        for (int w = 0; w < CW; ++w) u += red[w * RS + src + 8 * BB];
        u *= r;
        v = v / (1.f + __expf(-v)) * u;
      }
      if (g.mode == GEMV_RESID) {              // (O and down have the same outputs: this thread's value both times)
        v += sh.resid[t0 * TO * BB + i];
        sh.resid[t0 * TO * BB + i] = v;
      }
      if (!g.logits) ll_store(g.y + (size_t)ob * g.N + o, v, g.tag_out);
      else {
        g.logits[(size_t)ob * g.N + o] = v;
        if (best) {       // running argmax: larger value wins, then the lower index
          unsigned bits = __float_as_uint(v);
          bits = (bits & 0x80000000u) ? ~bits : (bits | 0x80000000u);
          const u64 key = ((u64)bits << 32) | (u64)(0xFFFFFFFFu - (unsigned)o);
          mine = mine > key ? mine : key;
        }
      }
    }
    par ^= 1;      // the next group (or phase) leaves its partial sums in the other half: one block barrier per group is enough
  }
  if (g.gain) par ^= 2;
  if (best) {
#pragma unroll
    for (int d = 16; d >= BB; d >>= 1) {
      const u64 other = __shfl_xor_sync(0xffffffffu, mine, d);
      mine = mine > other ? mine : other;
    }
    if (lane < BB && lane < p.batch && mine) atomicMax(best + lane, mine);   // CT and 32 are multiples of BB: lane l serves sequence l
  }
}

// ---- attention over the cache -------------------------------------------------------------------------------------------
// A CTA's item = (sequence, kv head, range of pages).  Consumer warp w owns keys 8 w .. 8 w + 7 of every page for all query
// heads of the group: for the scores 8 lanes share a key, for the value sum a lane owns HD / 32 dimensions.  The warps'
// results are merged in shared memory; where the key range is split, every CTA of the group hands its partial result
// (maximum, sum, values) to the others as tagged values and merges its own share of the group's outputs.
template <int HD, int GQ>
__device__ __forceinline__ void attn_phase(const MegaParams& p, const MegaLayer& L, uint32_t tag, Ring& rg, unsigned char* scr, Shared& sh, bool& dead) {
  constexpr int DV = HD / 32, HALF = HD / 2, LDR = HD + 2;
  constexpr int KEYS = PAGE_TOKENS / CW;       // keys of a page per warp
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int group = L.nq / L.nkv, n_out = p.generation ? L.nqkv : L.dq;
  const int ns = attn_splits(p.batch, L.nkv, sh.max_pages), n_items = p.batch * L.nkv * ns;
  volatile int* s_abort = &sh.abort;
  float* qs = reinterpret_cast<float*>(scr);               // [GQ][HD], scaled; zero beyond the group
  float* mo = qs + GQ * HD;                                // [CW][group][HD]
  float* mm = mo + CW * group * HD;                        // [CW][group]
  float* ml = mm + CW * group;
  const float scale = rsqrtf((float)HD);
  for (int i = group * HD + tid; i < GQ * HD; i += CT) qs[i] = 0.f;
  for (int it = blockIdx.x; it < n_items; it += gridDim.x) {
    const Item im = item_of(p, it, L.nkv, ns, sh.len);
    const int pos = im.n_keys - 1, pg_new = pos / PAGE_TOKENS;
    const bool has_new = p.generation && pg_new >= im.pg0 && pg_new < im.pg1;
    const u64* q = p.ll_q + (size_t)im.b * n_out + (size_t)im.kvh * group * HD;
    const u64* kin = p.ll_q + (size_t)im.b * n_out + L.dq + (size_t)im.kvh * HD;
    // of a split key range: this CTA's share [i0, i1) of the group's outputs, `width` lanes (splits) per output
    const int wlog = 32 - __clz(ns - 1 | 1), width = 1 << wlog, per_warp = 32 >> wlog, sub = lane >> wlog, sq = lane & (width - 1);
    const int i0 = group * HD * im.sp / ns, i1 = group * HD * (im.sp + 1) / ns;
    if (it != (int)blockIdx.x) consumer_sync();            // the previous item's scratch is free
    // A warp per head: query heads (normalised where the model has it, rotated, scaled), the step's own key and value.
    for (int hh = warp; hh < CW + 2; hh += CW) {
      const bool is_q = hh < group, is_k = has_new && hh == CW, is_v = has_new && hh == CW + 1;
      if (!is_q && !is_k && !is_v) continue;
      const u64* src = is_q ? q + hh * HD : (is_k ? kin : kin + (size_t)L.nkv * HD);
      float x1[HALF / 32], x2[HALF / 32];
#pragma unroll
      for (int j = 0; j < HALF / 32; ++j) {
        const int c = j * 32 + lane;
        x1[j] = ll_wait(src + c, tag, dead, s_abort, p.status);
        x2[j] = ll_wait(src + c + HALF, tag, dead, s_abort, p.status);
      }
      dead = __any_sync(0xffffffffu, dead);
      const float* gain = is_q ? L.q_norm : (is_k ? L.k_norm : nullptr);
      if (gain) {
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < HALF / 32; ++j) s = fmaf(x1[j], x1[j], fmaf(x2[j], x2[j], s));
        const float r = rsqrtf(warp_sum(s) / (float)HD + p.eps);
#pragma unroll
        for (int j = 0; j < HALF / 32; ++j) { x1[j] *= r * gain[j * 32 + lane]; x2[j] *= r * gain[j * 32 + lane + HALF]; }
      }
      const int page = pg_new < p.mpps && !is_q ? p.block_table[(size_t)im.b * p.mpps + pg_new] : -1;
      const bool page_ok = page >= 0 && page < p.n_pages;
      const size_t off = (((size_t)page * L.nkv + im.kvh) * PAGE_TOKENS + pos % PAGE_TOKENS) * HD;
#pragma unroll
      for (int j = 0; j < HALF / 32; ++j) {
        const int c = j * 32 + lane;
        const float2 cs = sh.rope[im.b * HALF + c];
        const float y1 = is_v ? x1[j] : x1[j] * cs.x - x2[j] * cs.y, y2 = is_v ? x2[j] : x2[j] * cs.x + x1[j] * cs.y;
        if (is_q) {
          qs[hh * HD + c] = y1 * scale;
          qs[hh * HD + c + HALF] = y2 * scale;
        } else {                                           // into the cache, and to this CTA's own attention
          const kv16 k1 = from_f<kv16>(y1), k2 = from_f<kv16>(y2);
          kv16* own = is_k ? sh.knew : sh.vnew;
          own[c] = k1; own[c + HALF] = k2;
          if (page_ok) {
            kv16* pool = (kv16*)(is_k ? L.kpool : L.vpool) + off;
            pool[c] = k1; pool[c + HALF] = k2;
          }
        }
      }
    }
    consumer_sync();
    float m[GQ], l[GQ], o[GQ][DV];
#pragma unroll
    for (int h = 0; h < GQ; ++h) {
      m[h] = -INFINITY; l[h] = 0.f;
#pragma unroll
      for (int d = 0; d < DV; ++d) o[h][d] = 0.f;
    }
    const uint32_t knew = smem_u32(sh.knew), vnew = smem_u32(sh.vnew);
    for (int pg = im.pg0; pg < im.pg1; ++pg) {
      if (!dead) dead = !quick_wait(rg.full + 8u * rg.slot, rg.phase, s_abort, p.status);
      __syncwarp();
      const int nk = *reinterpret_cast<volatile int*>(&sh.kv_rows[rg.slot]) < 0 ? 0 : min(PAGE_TOKENS, im.n_keys - pg * PAGE_TOKENS);
      const int new_row = has_new && pg == pg_new ? pos - pg * PAGE_TOKENS : -1;
      const uint32_t ks = rg.base + rg.slot * rg.bytes, vs = ks + PAGE_TOKENS * HD * 2;
      if (warp * KEYS < nk) {
        const int part = lane & 7;
        float kf[KEYS / 4][HD / 8];
#pragma unroll
        for (int kb = 0; kb < KEYS / 4; ++kb) {
          const int row = warp * KEYS + kb * 4 + (lane >> 3);
          const uint32_t kr = row == new_row ? knew : ks + row * HD * 2;
#pragma unroll
          for (int j = 0; j < HD / 64; ++j) {
            const uint4 u = lds128(kr + j * 128 + part * 16);
            const uint32_t ww[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) { kf[kb][8 * j + 2 * e] = kv_lo(ww[e]); kf[kb][8 * j + 2 * e + 1] = kv_hi(ww[e]); }
          }
        }
        float pv[GQ][KEYS / 4];                            // (heads beyond the group have a zero query and are not stored)
#pragma unroll
        for (int h = 0; h < GQ; ++h) {
#pragma unroll
          for (int kb = 0; kb < KEYS / 4; ++kb) pv[h][kb] = 0.f;
#pragma unroll
          for (int j = 0; j < HD / 32; ++j) {
            const float4 a = *reinterpret_cast<const float4*>(qs + h * HD + (j >> 1) * 64 + part * 8 + (j & 1) * 4);
#pragma unroll
            for (int kb = 0; kb < KEYS / 4; ++kb) {
              pv[h][kb] = fmaf(kf[kb][4 * j], a.x, pv[h][kb]); pv[h][kb] = fmaf(kf[kb][4 * j + 1], a.y, pv[h][kb]);
              pv[h][kb] = fmaf(kf[kb][4 * j + 2], a.z, pv[h][kb]); pv[h][kb] = fmaf(kf[kb][4 * j + 3], a.w, pv[h][kb]);
            }
          }
        }
#pragma unroll
        for (int d = 1; d <= 4; d <<= 1)
#pragma unroll
          for (int h = 0; h < GQ; ++h)
#pragma unroll
            for (int kb = 0; kb < KEYS / 4; ++kb) pv[h][kb] += __shfl_xor_sync(0xffffffffu, pv[h][kb], d);
        float mt[GQ], sum[GQ];
#pragma unroll
        for (int h = 0; h < GQ; ++h) {
          mt[h] = -INFINITY;
#pragma unroll
          for (int kb = 0; kb < KEYS / 4; ++kb) {
            if (warp * KEYS + kb * 4 + (lane >> 3) >= nk) pv[h][kb] = -INFINITY;
            mt[h] = fmaxf(mt[h], pv[h][kb]);
          }
        }
#pragma unroll
        for (int d = 8; d <= 16; d <<= 1)
#pragma unroll
          for (int h = 0; h < GQ; ++h) mt[h] = fmaxf(mt[h], __shfl_xor_sync(0xffffffffu, mt[h], d));
#pragma unroll
        for (int h = 0; h < GQ; ++h) {
          const float mn = fmaxf(m[h], mt[h]), mb = mn == -INFINITY ? 0.f : mn, al = __expf(m[h] - mb);
          sum[h] = 0.f;
#pragma unroll
          for (int kb = 0; kb < KEYS / 4; ++kb) { pv[h][kb] = __expf(pv[h][kb] - mb); sum[h] += pv[h][kb]; }
          l[h] *= al;
          m[h] = mn;
#pragma unroll
          for (int d = 0; d < DV; ++d) o[h][d] *= al;
        }
#pragma unroll
        for (int d = 8; d <= 16; d <<= 1)
#pragma unroll
          for (int h = 0; h < GQ; ++h) sum[h] += __shfl_xor_sync(0xffffffffu, sum[h], d);
#pragma unroll
        for (int h = 0; h < GQ; ++h) l[h] += sum[h];
#pragma unroll
        for (int j = 0; j < KEYS; ++j) {
          const int r = warp * KEYS + j;
          const uint32_t vr = (r == new_row ? vnew : vs + r * HD * 2) + lane * (DV * 2);
          float vf[DV];
#pragma unroll
          for (int d = 0; d < DV; d += 2) {
            uint32_t u;
            asm volatile("ld.shared.b32 %0, [%1];" : "=r"(u) : "r"(vr + d * 2));
            u = r < nk ? u : 0u;                           // rows beyond the sequence may hold anything
            vf[d] = kv_lo(u); vf[d + 1] = kv_hi(u);
          }
#pragma unroll
          for (int h = 0; h < GQ; ++h) {
            const float w = __shfl_sync(0xffffffffu, pv[h][j >> 2], 8 * (j & 3));
#pragma unroll
            for (int d = 0; d < DV; ++d) o[h][d] = fmaf(w, vf[d], o[h][d]);
          }
        }
      }
      __syncwarp();
      if (lane == 0 && !dead) mbar_arrive(rg.empty + 8u * rg.slot);
      rg.next();
    }
    // merge the warps
#pragma unroll
    for (int h = 0; h < GQ; ++h) {
      if (h < group) {
#pragma unroll
        for (int d = 0; d < DV; ++d) mo[(warp * group + h) * HD + lane * DV + d] = o[h][d];
        if (lane == 0) { mm[warp * group + h] = m[h]; ml[warp * group + h] = l[h]; }
      }
    }
    dead = __any_sync(0xffffffffu, dead);
    consumer_sync();
    u64* part = p.ll_part + (size_t)im.r * ns * group * LDR;
    u64* out = p.ll_a + (size_t)im.b * L.dq + (size_t)im.kvh * group * HD;
    for (int i = tid; i < group * HD; i += CT) {
      const int h = i / HD, d = i - h * HD;
      float M = -INFINITY, s = 0.f, v = 0.f;
#pragma unroll
      for (int w = 0; w < CW; ++w) M = fmaxf(M, mm[w * group + h]);
#pragma unroll
      for (int w = 0; w < CW; ++w) {
        const float mw = mm[w * group + h];
        const float f = mw == -INFINITY ? 0.f : __expf(mw - M);
        s = fmaf(ml[w * group + h], f, s);
        v = fmaf(mo[(w * group + h) * HD + d], f, v);
      }
      if (ns == 1) ll_store(out + i, v / s, tag);
      else {
        u64* pr = part + ((size_t)im.sp * group + h) * LDR;
        ll_store(pr + d, v, tag);
        if (d == 0) { ll_store(pr + HD, M, tag); ll_store(pr + HD + 1, s, tag); }
      }
    }
    if (ns == 1) continue;
    for (int ib = i0 + warp * per_warp; ib < i1; ib += CW * per_warp) {
      const int i = ib + sub;
      const bool mine = i < i1 && sq < ns;
      float M = -INFINITY, s = 0.f, v = 0.f;
      if (mine) {
        const int h = i / HD;
        const u64* pr = part + ((size_t)sq * group + h) * LDR;
        u64 a = ll_load(pr + HD), b = ll_load(pr + HD + 1), c = ll_load(pr + (i - h * HD));
        unsigned n = 0;
        while ((ll_tag(a) != tag || ll_tag(b) != tag || ll_tag(c) != tag) && !dead) {
          if (!poll_more(n, s_abort, p.status)) dead = true;
          a = ll_load(pr + HD); b = ll_load(pr + HD + 1); c = ll_load(pr + (i - h * HD));
        }
        M = ll_val(a); s = ll_val(b); v = ll_val(c);
      }
      __syncwarp();
      float mt = M;
      for (int d = width >> 1; d; d >>= 1) mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, d));
      const float f = M == -INFINITY ? 0.f : __expf(M - mt);
      s *= f; v *= f;
      for (int d = width >> 1; d; d >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, d);
        v += __shfl_xor_sync(0xffffffffu, v, d);
      }
      if (mine && sq == 0) ll_store(out + i, v / s, tag);
    }
    dead = __any_sync(0xffffffffu, dead);
  }
}

template <int BB, int HD, int GQ>
__global__ void __launch_bounds__(NT, 1) step_mega_mma_kernel(const __grid_constant__ MegaParams p, const __grid_constant__ Plan pl) {
  constexpr int HR = Geo<BB>::HR, PITCH = Geo<BB>::PITCH, STAGE = Geo<BB>::STAGE;
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ Shared sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int batch = p.batch;
  const uint32_t bars = smem_u32(sh.bars);
  volatile int* s_abort = &sh.abort;
  Ring wr{smem_u32(sm), bars, bars + 8u * pl.n_stage, pl.n_stage, 0, 0u, STAGE};
  Ring kr{smem_u32(sm) + pl.kv_off, bars + 16u * pl.n_stage, bars + 16u * pl.n_stage + 8u * pl.n_kv, pl.n_kv, 0, 0u, 2 * PAGE_TOKENS * HD * 2};
  const uint32_t rope_bar = bars + 16u * pl.n_stage + 16u * pl.n_kv;
  if (tid < 16) sh.zeros[tid] = 0u;
  if (tid == 0) {
    sh.abort = 0; sh.issued = 0;
    for (int i = 0; i < pl.n_stage; ++i) { mbar_init(wr.full + 8u * i, 1); mbar_init(wr.empty + 8u * i, CW); }
    for (int i = 0; i < pl.n_kv; ++i) { mbar_init(kr.full + 8u * i, 1); mbar_init(kr.empty + 8u * i, CW); sh.kv_rows[i] = -1; }
    mbar_init(rope_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    int mp = 1;
    for (int b = 0; b < batch; ++b) {
      const int n = __ldcg(p.seq_lens + b);
      sh.len[b] = n;
      mp = max(mp, (n + (p.generation ? 1 : 0) + PAGE_TOKENS - 1) / PAGE_TOKENS);
    }
    sh.max_pages = mp;
  }
  if (p.do_embed && tid >= 32 && tid < 32 + batch) {
    const int b = tid - 32, tok = p.tokens[p.gather_idx ? p.gather_idx[b] : b];
    const bool ok = tok >= 0 && tok < p.vocab;
    if (!ok && blockIdx.x == 0) dev_flag(p.status, DEV_BAD_TOKEN);
    sh.tok[b] = ok ? tok : -1;
  }
  __syncthreads();

  if (warp >= CW && warp < CW + LW) {
    // ---------------- weight loaders: slots of the whole schedule, in the order the consumers use them ----------------
    const bool ok = walk_slots<BB>(p, [&](int n, const Proj& g, int row, bool valid, int c, int kc) {
      if (n % LW != warp - CW) { wr.next(); return true; }
      const uint32_t bytes = (uint32_t)min(kc, g.K - c * kc) * 2u;
      const int nv = __popc(__ballot_sync(0xffffffffu, valid));
      if (!lazy_wait(wr.empty + 8u * wr.slot, wr.phase ^ 1u, s_abort, p.status)) return false;
      if (lane == 0) { mbar_expect_tx(wr.full + 8u * wr.slot, nv * bytes); *reinterpret_cast<volatile int*>(&sh.issued) = n; }
      __syncwarp();
      if (valid) bulk_load(wr.base + wr.slot * STAGE + lane * PITCH, g.W + (size_t)row * g.K * 2 + (size_t)c * kc * 2, bytes, wr.full + 8u * wr.slot);
      wr.next();
      return true;
    });
    if (!ok) drain_after_abort();
    return;
  }
  if (warp == CW + LW) {
    // ---------------- L2 prefetch: HBM keeps streaming while the ring is full or its depth does not cover the latency ----------
    walk_slots<BB>(p, [&](int n, const Proj& g, int row, bool valid, int c, int kc) {
      int tries = 0;                             // (a hint only: gives up when the loaders do not move for some milliseconds)
      while (n > *reinterpret_cast<volatile int*>(&sh.issued) + Geo<BB>::AHEAD) {
        if (*s_abort || ++tries > 100000) return false;
        __nanosleep(100);
      }
      const char* src = g.W + (size_t)row * g.K * 2 + (size_t)c * kc * 2;
      const int bytes = min(kc, g.K - c * kc) * 2;
#pragma unroll 1
      for (int r = 0; r < HR; ++r) {
        const char* q = (const char*)__shfl_sync(0xffffffffu, (u64)src, r);
        if (!__shfl_sync(0xffffffffu, (int)valid, r)) break;
        for (int off = lane * 128; off < bytes; off += 4096) asm volatile("prefetch.global.L2 [%0];" ::"l"(q + off) : "memory");
      }
      return true;
    });
    return;
  }
  if (warp == CW + LW + 1) {
    // ---------------- RoPE table, then the cache-page loader ----------------
    for (int i = lane; i < batch * (HD / 2); i += 32) {
      const int b = i / (HD / 2);
      float sn, cs;
      rope_sincos(sh.len[b] + (p.generation ? 0 : -1), p.inv.f[i - b * (HD / 2)], &sn, &cs);
      sh.rope[i] = make_float2(cs, sn);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(rope_bar);
    bool ok = true;
    for (int i = p.layer_begin; i < p.layer_end && ok; ++i) {
      const MegaLayer& L = p.layers[i];
      const int ns = attn_splits(batch, L.nkv, sh.max_pages), n_items = batch * L.nkv * ns;
      for (int it = blockIdx.x; it < n_items && ok; it += gridDim.x) {
        const Item im = item_of(p, it, L.nkv, ns, sh.len);
        for (int pg = im.pg0; pg < im.pg1; ++pg, kr.next()) {
          const int page = pg < p.mpps ? p.block_table[(size_t)im.b * p.mpps + pg] : -1;
          const bool page_ok = page >= 0 && page < p.n_pages;
          const int rows = page_ok ? min(PAGE_TOKENS, sh.len[im.b] - pg * PAGE_TOKENS) : -1;
          ok = lazy_wait(kr.empty + 8u * kr.slot, kr.phase ^ 1u, s_abort, p.status);
          if (!ok) break;
          if (lane == 0) {
            if (!page_ok) dev_flag(p.status, DEV_BAD_PAGE);
            *reinterpret_cast<volatile int*>(&sh.kv_rows[kr.slot]) = rows;
            const uint32_t bar = kr.full + 8u * kr.slot, dst = kr.base + kr.slot * kr.bytes;
            if (rows > 0) {
              const size_t off = ((size_t)page * L.nkv + im.kvh) * PAGE_TOKENS * HD;
              mbar_expect_tx(bar, 2u * rows * HD * 2);
              bulk_load(dst, (const kv16*)L.kpool + off, rows * HD * 2, bar);
              bulk_load(dst + PAGE_TOKENS * HD * 2, (const kv16*)L.vpool + off, rows * HD * 2, bar);
            } else {
              mbar_arrive(bar);
            }
          }
        }
      }
    }
    if (!ok) drain_after_abort();
    return;
  }

  // ---------------- consumers ----------------
  unsigned* counter = reinterpret_cast<unsigned*>(p.status) + 32 + p.counter_idx;
  u64* best = reinterpret_cast<u64*>(reinterpret_cast<char*>(p.status) + 64);
  // scratch: [ activation columns per warp | partial sums, twice | attention ]
  unsigned char* scr = sm + pl.scr_off;
  const uint32_t xp = smem_u32(scr) + warp * (3 * BB * XCOL);
  float* red = reinterpret_cast<float*>(scr + CW * 3 * BB * XCOL);
  unsigned char* attn_scr = scr + CW * 3 * BB * XCOL + 2 * CW * Geo<BB>::TG * TR * BB * 4;
  bool dead = false;
  int par = 0;
  {
    // the residual stream at this CTA's outputs: the embedding, or what the launch before left
    int o0, o1;
    cta_range(p.d, o0, o1);
    for (int i = tid; i < (o1 - o0) * BB; i += CT) {
      const int b = i % BB, o = o0 + i / BB;
      float v = 0.f;
      if (b < batch) {
        if (p.layer_begin > 0) v = ll_val(ll_load(p.ll_x2 + (size_t)b * p.d + o));
        else if (sh.tok[b] >= 0) v = to_f(((const bf16*)p.embed)[(size_t)sh.tok[b] * p.d + o]);
      }
      sh.resid[i] = v;
    }
    consumer_sync();
  }
  // five phases a layer (q(kv), attention, O, gate/up, down), then the LM head
  const int n_ph = 5 * (p.layer_end - p.layer_begin) + (p.do_head ? 1 : 0);
#pragma unroll 1
  for (int ph = 0, i = p.layer_begin, kind = 0; ph < n_ph; ++ph) {
    if (kind == 1) {
      if (i == p.layer_begin && !dead) dead = !quick_wait(rope_bar, 0, s_abort, p.status);
      dead = __any_sync(0xffffffffu, dead);
      attn_phase<HD, GQ>(p, p.layers[i], (uint32_t)i + 1u, kr, attn_scr, sh, dead);
    } else {
      const bool head = i == p.layer_end;
      proj_phase<BB>(p, work_of<BB>(p, i, kind, head), wr, xp, red, par, sh, dead, head && p.token_out ? best : nullptr);
    }
    if (p.trace && blockIdx.x == 0 && tid == 0) p.trace[ph] = clock64();
    if (++kind == 5) { kind = 0; ++i; }
  }
  if (*s_abort) { drain_after_abort(); return; }
  if (!p.do_head) return;             // a later launch carries on from the residual stream in ll_x2
  // the CTA that finishes last writes the tokens and moves the lengths on: every other CTA has read them long ago
  consumer_sync();
  if (tid == 0) {
    __threadfence();
    if (atomicAdd(counter, 1u) == gridDim.x - 1) {
      __threadfence();
      for (int b = 0; b < batch; ++b) {
        if (p.token_out) {
          u64 v;
          asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(best + b) : "memory");
          p.token_out[b] = (int)(0xFFFFFFFFu - (unsigned)(v & 0xFFFFFFFFull));
        }
        if (p.generation) p.seq_lens[b] += 1;
      }
    }
  }
}

constexpr size_t SMEM_ROOM = SMEM_LIMIT - sizeof(Shared) - 256;      // dynamic shared memory of a CTA

// Shared-memory plan: scratch and page slots first, the weight ring takes what is left (at least 3 slots).  A second page slot, which lets
// a page's load overlap the arithmetic on the one before, is not worth the weight slots of a tile: where tiles take two slots (up to
// two sequences), fewer than four would be left beside it and head_dim is 128, there is one.  Generation step, 3B shape, with two page
// slots and 3 weight slots / with one and 4: 1 x 300 keys 2000 / 1787 us, 1 x 4090 2133 / 2025, 2 x 300 2111 / 1899, 2 x 4000 2380 / 2360; eight
// heads of 128 a group, 8 layers of 4096, 1 x 300 726 / 632, 1 x 4000 751 / 663.  (Four sequences of head_dim 128, and two with more
// than 4 heads a group, have room for one page slot and three weight slots only.)
bool make_plan(int batch, int hd, int max_group, Plan* pl, size_t* bytes) {
  const int bb = batch <= 1 ? 1 : (batch == 2 ? 2 : 4);
  const size_t proj = (size_t)CW * 3 * bb * XCOL + (size_t)2 * CW * (bb == 4 ? Geo<4>::TG : Geo<1>::TG) * TR * bb * 4;
  const size_t attn = (size_t)((max_group <= 4 ? 4 : MAXG) + CW * max_group) * hd * 4 + (size_t)2 * CW * max_group * 4;
  const size_t scr = (proj + attn + 127) / 128 * 128;
  const int STAGE = bb == 4 ? Geo<4>::STAGE : Geo<1>::STAGE;
  for (int n_kv = 2; n_kv >= 1; --n_kv) {
    const size_t kv = (size_t)n_kv * 2 * PAGE_TOKENS * hd * 2;
    if (scr + kv + (n_kv > 1 && bb < 4 ? 4 : 3) * (size_t)STAGE > SMEM_ROOM) continue;
    int n = (int)((SMEM_ROOM - scr - kv) / STAGE);
    if (n > MAX_SLOTS) n = MAX_SLOTS;
    pl->n_stage = n; pl->n_kv = n_kv; pl->kv_off = n * STAGE; pl->scr_off = pl->kv_off + (int)kv;
    *bytes = (size_t)pl->scr_off + scr;
    return true;
  }
  return false;
}

template <int BB, int HD, int GQ>
cudaError_t go(MegaParams& p, Plan& pl, size_t smem, cudaStream_t st, int n_sm) {
  auto kern = step_mega_mma_kernel<BB, HD, GQ>;
  static bool raised[TC_MAX_DEVICES] = {};
  cudaError_t e = tc_raise_smem_limit(kern, SMEM_ROOM, raised);
  if (e != cudaSuccess) return e;
  void* args[] = {(void*)&p, (void*)&pl};
  return cudaLaunchCooperativeKernel((const void*)kern, dim3(n_sm), dim3(NT), args, smem, st);
}
template <int HD, int GQ>
cudaError_t go_batch(MegaParams& p, Plan& pl, size_t smem, cudaStream_t st, int n_sm) {
  if (p.batch <= 1) return go<1, HD, GQ>(p, pl, smem, st, n_sm);
  if (p.batch == 2) return go<2, HD, GQ>(p, pl, smem, st, n_sm);
  return go<4, HD, GQ>(p, pl, smem, st, n_sm);
}

}  // namespace

// head_dim 64 / 128 (the layout of the attention phase), rows of whole 16-byte pieces (checked by the caller for every layer),
// a CTA's share of the residual stream in its array (n_sm: the smallest grid of the call).
bool step_mega_mma_supported(int batch, int hd, int max_group, int d, int n_sm) {
  Plan pl;
  size_t bytes;
  return batch >= 1 && batch <= 4 && (hd == 64 || hd == 128) && max_group <= MAXG && (d / n_sm + 1) * 4 <= RESID_MAX &&
         make_plan(batch, hd, max_group, &pl, &bytes);
}

cudaError_t launch_step_mega_mma(MegaParams p, int max_group, int n_sm, cudaStream_t st, int64_t* n_launch) {
  Plan pl;
  size_t smem;
  if (!make_plan(p.batch, p.hd, max_group, &pl, &smem)) return cudaErrorInvalidValue;
  ++*n_launch;
  if (p.hd == 64) return max_group <= 4 ? go_batch<64, 4>(p, pl, smem, st, n_sm) : go_batch<64, 8>(p, pl, smem, st, n_sm);
  return max_group <= 4 ? go_batch<128, 4>(p, pl, smem, st, n_sm) : go_batch<128, 8>(p, pl, smem, st, n_sm);
}
