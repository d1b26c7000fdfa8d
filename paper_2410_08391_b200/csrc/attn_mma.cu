// Causal grouped-query attention over a ragged batch on the warp-level tensor cores (mma.sync), for short sequences.
//
// What bounds the other kernel (attn_tc.cu) there: a CTA of it takes a whole SM (512 tensor-memory columns, 160 KB of shared memory)
// for one pair of 128-query tiles and one head, and spends about 6 us on set-up, the first loads, one softmax chain and the
// store, whatever the length.  64 prompts of 59 tokens and 20 heads are 1280 such CTAs in 8.6 waves.  Here a CTA is 4 warps with 64 queries of one
// head, 40 KB of shared memory (head_dim 64) and needs no tensor memory, so that four share an SM and their latencies overlap:
//   - K and V tiles of 64 keys come in by 16-byte asynchronous copies, two stages; rows beyond the sequence are zero-filled.
//   - a warp owns 16 queries; scores, probabilities and output stay in its registers (the accumulator layout of one product is
//     the operand layout of the next); online softmax on the quads that share a row; the running sum is fp32, of unrounded values.
//   - the output leaves through the query tile's shared memory as whole 16-byte pieces.
// Where sequences are long the other kernel's tensor rate wins (this one reaches half of it): attn_choose() draws the line.
#include <math.h>

#include <vector>

#include "attn_mma.h"

namespace {

constexpr int BQ = 64, BKV = 64, NT = 128;

template <int HD> struct Cfg {
  static constexpr int ROW = HD * 2, TILE = 64 * ROW;      // bytes of a row, of a 64-row tile
  static constexpr int SMEM = TILE + 2 * 2 * TILE;         // queries, two stages of keys and values
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t* r) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm4_t(uint32_t addr, uint32_t* r) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
template <bool F16>
__device__ __forceinline__ void mma16816(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
  if (F16)
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
  else
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
template <bool F16> __device__ __forceinline__ uint32_t pack2(float x, float y) {
  if (F16) { const __half2 h = __floats2half2_rn(x, y); return *reinterpret_cast<const uint32_t*>(&h); }
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// byte offset of 16-byte piece c of row r in a tile: pieces are swizzled by the row within groups of eight
template <int HD> __device__ __forceinline__ uint32_t piece(int r, int c) { return (uint32_t)(r * Cfg<HD>::ROW + ((c ^ (r & 7)) << 4)); }

struct Params {
  const bf16* qkv; int ld;
  const int* cu; int nq, nkv;
  bf16* out; bf16* out_lo; int ldo;
  float scale_log2e;
};

// 64 rows of HD elements, rows first .. first + 63 of the sequence at column col, by all threads; rows >= n_rows are zeros
template <int HD>
__device__ __forceinline__ void load_tile(uint32_t dst, const bf16* seq, int ld, int col, int first, int n_rows) {
  constexpr int PER = HD / 8;                              // pieces per row
#pragma unroll
  for (int i = 0; i < 64 * PER / NT; ++i) {
    const int e = i * NT + threadIdx.x, r = e / PER, c = e % PER, row = first + r;
    const bool in = row < n_rows;
    const bf16* src = seq + (size_t)(in ? row : 0) * ld + col + c * 8;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + piece<HD>(r, c)), "l"(src), "r"(in ? 16 : 0) : "memory");
  }
}

// grid (query head, sequence, query tile counted from the sequence's last): the CTAs with the most keys start first
template <int HD, bool F16>
__global__ void __launch_bounds__(NT, HD == 64 ? 4 : 2) attn_mma_kernel(const Params p) {
  constexpr int KS = HD / 16, NTL = HD / 8, TILE = Cfg<HD>::TILE;
  extern __shared__ __align__(128) unsigned char sm[];
  pdl_wait();
  const int head = blockIdx.x, b = blockIdx.y;
  const int base = p.cu[b], L = p.cu[b + 1] - base;
  const int n_tiles = (L + BQ - 1) / BQ, qt = n_tiles - 1 - (int)blockIdx.z;
  if (qt < 0) return;
  const int kvh = head / (p.nq / p.nkv);
  const bf16* seq = p.qkv + (size_t)base * p.ld;
  const int kcol = (p.nq + kvh) * HD, vcol = (p.nq + p.nkv + kvh) * HD;
  const uint32_t sq = smem_addr(sm), skv = sq + TILE;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, qd = lane & 3, mi = lane >> 3;
  const int q0 = qt * BQ;
  load_tile<HD>(sq, seq, p.ld, head * HD, q0, L);
  load_tile<HD>(skv, seq, p.ld, kcol, 0, L);
  asm volatile("cp.async.commit_group;" ::: "memory");
  load_tile<HD>(skv + TILE, seq, p.ld, vcol, 0, L);
  asm volatile("cp.async.commit_group;" ::: "memory");
  uint32_t qa[KS][4];
  float o[NTL][4];
#pragma unroll
  for (int j = 0; j < NTL; ++j) { o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.f; }
  float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
  const int row0 = q0 + warp * 16 + g;                     // this lane's rows: row0, row0 + 8
  for (int kt = 0; kt <= qt; ++kt) {
    const uint32_t sk = skv + (kt & 1) * 2 * TILE, sv = sk + TILE;
    if (kt < qt) {                                         // the next tile's keys and values (their stage was left before the last barrier)
      const uint32_t nk = skv + ((kt + 1) & 1) * 2 * TILE;
      load_tile<HD>(nk, seq, p.ld, kcol, (kt + 1) * BKV, L);
      asm volatile("cp.async.commit_group;" ::: "memory");
      load_tile<HD>(nk + TILE, seq, p.ld, vcol, (kt + 1) * BKV, L);
      asm volatile("cp.async.commit_group;" ::: "memory");
      asm volatile("cp.async.wait_group 3;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    }
    __syncthreads();
    if (kt == 0) {
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) ldsm4(sq + piece<HD>(warp * 16 + (lane & 15), 2 * ks + (lane >> 4)), qa[ks]);
    }
    // ---- scores of 16 queries x 64 keys
    float s[8][4];
#pragma unroll
    for (int t = 0; t < 8; ++t) { s[t][0] = s[t][1] = s[t][2] = s[t][3] = 0.f; }
#pragma unroll
    for (int ks = 0; ks < KS; ++ks)
#pragma unroll
      for (int t = 0; t < 8; t += 2) {
        uint32_t kb[4];          // (keys 8t.., dims 16ks..), (.., dims + 8), (keys 8(t+1).., dims 16ks..), (.., dims + 8)
        ldsm4(sk + piece<HD>(t * 8 + (mi >> 1) * 8 + (lane & 7), 2 * ks + (mi & 1)), kb);
        mma16816<F16>(s[t], qa[ks], kb[0], kb[1]);
        mma16816<F16>(s[t + 1], qa[ks], kb[2], kb[3]);
      }
    if (kt == qt) {                                        // only the last key tile reaches the diagonal
#pragma unroll
      for (int t = 0; t < 8; ++t)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (kt * BKV + t * 8 + 2 * qd + (e & 1) > row0 + (e >> 1) * 8) s[t][e] = -INFINITY;
    }
    float mt[2] = {m[0], m[1]};
#pragma unroll
    for (int t = 0; t < 8; ++t) { mt[0] = fmaxf(mt[0], fmaxf(s[t][0], s[t][1])); mt[1] = fmaxf(mt[1], fmaxf(s[t][2], s[t][3])); }
    float mc[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      mt[h] = fmaxf(mt[h], __shfl_xor_sync(0xffffffffu, mt[h], 1));
      mt[h] = fmaxf(mt[h], __shfl_xor_sync(0xffffffffu, mt[h], 2));
      mc[h] = mt[h] == -INFINITY ? 0.f : mt[h] * p.scale_log2e;
      const float a = m[h] == -INFINITY ? 0.f : ex2(m[h] * p.scale_log2e - mc[h]);
      m[h] = mt[h];
      l[h] *= a;
#pragma unroll
      for (int j = 0; j < NTL; ++j) { o[j][2 * h] *= a; o[j][2 * h + 1] *= a; }
    }
    uint32_t pa[4][4];           // P as the A operand: 16 keys per k step
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      float e[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) e[i] = ex2(fmaf(s[t][i], p.scale_log2e, -mc[i >> 1]));
      l[0] += e[0] + e[1]; l[1] += e[2] + e[3];
      pa[t >> 1][(t & 1) * 2] = pack2<F16>(e[0], e[1]);
      pa[t >> 1][(t & 1) * 2 + 1] = pack2<F16>(e[2], e[3]);
    }
    if (kt < qt) asm volatile("cp.async.wait_group 2;" ::: "memory");
    else asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    // ---- O += P V
#pragma unroll
    for (int ks = 0; ks < 4; ++ks)
#pragma unroll
      for (int j = 0; j < NTL; j += 2) {
        uint32_t vb[4];          // (keys 16ks.., dims 8j..), (keys + 8, dims 8j..), (keys 16ks.., dims 8(j+1)..), (keys + 8, ..)
        ldsm4_t(sv + piece<HD>(ks * 16 + (mi & 1) * 8 + (lane & 7), j + (mi >> 1)), vb);
        mma16816<F16>(o[j], pa[ks], vb[0], vb[1]);
        mma16816<F16>(o[j + 1], pa[ks], vb[2], vb[3]);
      }
    __syncthreads();             // this stage is free
  }
  pdl_trigger();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    l[h] += __shfl_xor_sync(0xffffffffu, l[h], 1);
    l[h] += __shfl_xor_sync(0xffffffffu, l[h], 2);
    l[h] = 1.f / l[h];
  }
  // ---- out: a warp's 16 rows through its own rows of the query tile
  const int n_out = p.out_lo ? 2 : 1;
  for (int pass = 0; pass < n_out; ++pass) {
    __syncwarp();
#pragma unroll
    for (int j = 0; j < NTL; ++j)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float x = o[j][2 * h] * l[h], y = o[j][2 * h + 1] * l[h];
        if (pass) { x -= __bfloat162float(__float2bfloat16_rn(x)); y -= __bfloat162float(__float2bfloat16_rn(y)); }
        const int r = warp * 16 + g + 8 * h;
        asm volatile("st.shared.b32 [%0], %1;" ::"r"(sq + piece<HD>(r, j) + 4 * qd), "r"(pack2<false>(x, y)) : "memory");
      }
    __syncwarp();
    bf16* dst = (pass ? p.out_lo : p.out) + (size_t)base * p.ldo + (size_t)head * HD;
    constexpr int PER = HD / 8;
#pragma unroll
    for (int i = 0; i < 16 * PER / 32; ++i) {
      const int e = i * 32 + lane, r = e / PER, c = e % PER, row = q0 + warp * 16 + r;
      if (row < L) {
        uint4 u;
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(u.x), "=r"(u.y), "=r"(u.z), "=r"(u.w) : "r"(sq + piece<HD>(warp * 16 + r, c)));
        *reinterpret_cast<uint4*>(dst + (size_t)row * p.ldo + c * 8) = u;
      }
    }
  }
}

template <int HD, bool F16>
cudaError_t go(const Params& p, dim3 grid, cudaStream_t st) {
  static bool raised[TC_MAX_DEVICES] = {};
  cudaError_t e = tc_raise_smem_limit(attn_mma_kernel<HD, F16>, Cfg<HD>::SMEM, raised);
  if (e != cudaSuccess) return e;
  return launch_overlapped(attn_mma_kernel<HD, F16>, grid, dim3(NT), Cfg<HD>::SMEM, st, p);
}

// Time of CTAs with k key tiles, count[k] of them, a + b k each, on 148 SMs that take one at a time, longest first
double one_per_sm(const std::vector<int>& count, double a, double b) {
  double total = 0, longest = 0, second = 0;
  long long seen = 0;
  for (int k = (int)count.size() - 1; k >= 0; --k) {
    if (!count[k]) continue;
    const double t = a + b * k;
    total += t * count[k];
    longest = longest > t ? longest : t;
    if (seen < 148 && seen + count[k] >= 148) second += t;        // the 148th and the 149th share an SM
    if (seen < 149 && seen + count[k] >= 149) second += t;
    seen += count[k];
  }
  if (seen < 149) second = 0;
  const double spread = total / 148;
  return longest > spread ? (longest > second ? longest : second) : (spread > second ? spread : second);
}

}  // namespace

// Microseconds of the three forms, fitted to 226 launches (1 to 64 sequences of 16 to 4096 tokens, 12 to 32 heads, both head widths):
// taken by this rule they are 0.6 % above the best of the three (geometric mean); the rule before (attn_tc.cu only, one tile per CTA where
// the pairs would not fill the SMs) 29 %.  64 x 59 tokens, 20 heads: 47.9 -> 11.5 us; 8 x 256: 15.3 -> 11.6; 1 x 59: 5.9 -> 3.3; the other
// way round at 1 x 1024: 15.2 against 25.4 here.
int attn_choose(const int* cu_host, int batch, int heads, int hd) {
  std::vector<int> one, two;
  double ctas = 0, units = 0;
  int most = 0;
  auto add = [&](std::vector<int>& v, int k) { if ((int)v.size() <= k) v.resize(k + 1, 0); v[k] += heads; };
  for (int b = 0; b < batch; ++b) {
    const int len = cu_host[b + 1] - cu_host[b], n = (len + 127) / 128, t = (len + BQ - 1) / BQ;
    for (int k = 1; k <= n; ++k) add(one, k);
    for (int k = 2; k < n + 2; k += 2) add(two, k < n ? k : n);
    ctas += (double)heads * t;
    units += (double)heads * t * (t + 1) / 2;
    most = most > t ? most : t;
  }
  const bool w = hd == 128;
  const double t1 = 1.5 + one_per_sm(one, w ? 4.8 : 3.7, w ? 1.6 : 1.25), t2 = 1.5 + one_per_sm(two, w ? 5.6 : 3.4, w ? 2.0 : 1.95);
  // several CTAs share an SM: the longest chain (slower beside others), or the work of all
  const double chain = ((w ? 2.9 : 2.3) + (w ? 1.5 : 1.15) * most) * (ctas > 148 ? 1.45 : 1.0);
  const double all = 2.0 + (w ? 5.0e-3 : 2.5e-3) * ctas + (w ? 7.4e-3 : 3.6e-3) * units, t0 = chain > all ? chain : all;
  return t0 <= t1 && t0 <= t2 ? 0 : (t1 < t2 ? 1 : 2);
}

cudaError_t launch_attn_mma(const bf16* qkv, int ld, int nq, int nkv, int hd, const int* cu_dev, int batch, int max_len, bf16* out, int ldo,
                            cudaStream_t st, int64_t* n_launch, bool half_operands, bf16* out_lo) {
  Params p{qkv, ld, cu_dev, nq, nkv, out, out_lo, ldo, (1.f / sqrtf((float)hd)) * 1.4426950408889634f};
  const dim3 grid(nq, batch, (max_len + BQ - 1) / BQ);
  ++*n_launch;
  if (half_operands) return hd == 64 ? go<64, true>(p, grid, st) : go<128, true>(p, grid, st);
  return hd == 64 ? go<64, false>(p, grid, st) : go<128, false>(p, grid, st);
}
