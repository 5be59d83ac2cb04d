// Decode attention over the packed cache (Eq. 3) and the inspection kernels.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <chrono>
#include <math_constants.h>
#include <type_traits>

#include "pq_common.cuh"

namespace pq {

// ---- reading codes of (token, block) from a token-block held in global or shared memory ----
__device__ inline uint32_t get_l1(const uint8_t* tb, const Layout& L, int tok, int blk) {
  return *reinterpret_cast<const uint32_t*>(tb + tok * L.b1 + blk * 4);
}
__device__ inline uint32_t get_l2(const uint8_t* tb, const Layout& L, int tok, int blk) {
  return tb[L.o2 + tok * L.b2 + blk];
}
__device__ inline uint32_t get_l3(const uint8_t* tb, const Layout& L, int tok, int blk) {
  return (tb[L.o3 + tok * L.b3 + (blk >> 1)] >> (4 * (blk & 1))) & 0xFu;
}
__device__ inline uint32_t get_l4(const uint8_t* tb, const Layout& L, int tok, int blk) {
  return (tb[L.o4 + tok * L.b4 + (blk >> 2)] >> (2 * (blk & 3))) & 0x3u;
}
__device__ inline float get_radius(const uint8_t* tb, const Layout& L, int tok, int blk) {
  return __half2float(reinterpret_cast<const __half*>(tb + L.orad + tok * L.br)[blk]);
}

// DeQuant of one block in the rotated basis (Algorithm 1, DeQuant, without the final S^T):
// from the level-4 radius down, child 2j = parent * cos(theta), child 2j+1 = parent * sin(theta).
__device__ inline void decode_block(const uint8_t* tb, const Layout& L, int tok, int blk, const float* cen_cos,
                                    const float* cen_sin, float* y) {
  const uint32_t l1 = get_l1(tb, L, tok, blk), l2 = get_l2(tb, L, tok, blk);
  const uint32_t l3 = get_l3(tb, L, tok, blk), l4 = get_l4(tb, L, tok, blk);
  const float r = get_radius(tb, L, tok, blk);
  float r3[2], r2[4], r1[8];
  r3[0] = r * cen_cos[24 + l4];
  r3[1] = r * cen_sin[24 + l4];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const uint32_t c = (l3 >> (2 * j)) & 3u;
    r2[2 * j] = r3[j] * cen_cos[20 + c];
    r2[2 * j + 1] = r3[j] * cen_sin[20 + c];
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t c = (l2 >> (2 * j)) & 3u;
    r1[2 * j] = r2[j] * cen_cos[16 + c];
    r1[2 * j + 1] = r2[j] * cen_sin[16 + c];
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint32_t c = (l1 >> (4 * j)) & 15u;
    y[2 * j] = r1[j] * cen_cos[c];
    y[2 * j + 1] = r1[j] * cen_sin[c];
  }
}

// One rotated coordinate of one token.
__device__ inline float decode_coord(const uint8_t* tb, const Layout& L, int tok, int coord, const float* cen_cos,
                                     const float* cen_sin) {
  const int blk = coord >> 4, i = coord & 15;
  const uint32_t c1 = (get_l1(tb, L, tok, blk) >> (4 * (i >> 1))) & 15u;
  const uint32_t c2 = (get_l2(tb, L, tok, blk) >> (2 * (i >> 2))) & 3u;
  const uint32_t c3 = (get_l3(tb, L, tok, blk) >> (2 * (i >> 3))) & 3u;
  const uint32_t c4 = get_l4(tb, L, tok, blk);
  float v = get_radius(tb, L, tok, blk);
  v *= (i & 8) ? cen_sin[24 + c4] : cen_cos[24 + c4];
  v *= (i & 4) ? cen_sin[20 + c3] : cen_cos[20 + c3];
  v *= (i & 2) ? cen_sin[16 + c2] : cen_cos[16 + c2];
  v *= (i & 1) ? cen_sin[c1] : cen_cos[c1];
  return v;
}

// ---- workspace -----------------------------------------------------------------------------
constexpr int kFastMaxGridHost = 160;  // upper bound on the persistent kernel's grid (one CTA per SM)

struct Workspace {   // of the persistent head_dim-128 kernel; nothing else needs scratch, and none of it needs clearing
  uint32_t* elected;  // [B][Hkv]: the epoch of the last call whose parts of the unit were combined
  uint32_t* flags;    // [slot]: the epoch of the last call whose partial result is in the slot
  float* ml;          // [slot][head in group][2]   slot = first slot of the unit + part
  float* o;           // [slot][head in group][d]
  int64_t bytes;
};

// `units` with `rows` (query, head) rows each.
__host__ inline Workspace carve_workspace(void* base, int d, int64_t units, int64_t rows) {
  Workspace w;
  auto align = [](int64_t x) { return (x + 255) & ~(int64_t)255; };
  int64_t off = 0;
  uint8_t* p = reinterpret_cast<uint8_t*>(base);
  const int64_t n_slots = (d == 128 && units <= 2048) ? units + kFastMaxGridHost : 0;
  w.elected = reinterpret_cast<uint32_t*>(p + off);
  off = align(off + units * 4);
  w.flags = reinterpret_cast<uint32_t*>(p + off);
  off = align(off + n_slots * 4);
  w.ml = reinterpret_cast<float*>(p + off);
  off = align(off + n_slots * rows * 2 * 4);
  w.o = reinterpret_cast<float*>(p + off);
  off = align(off + n_slots * rows * d * 4);
  w.bytes = off;
  return w;
}

// How rows_attention_kernel cuts the n_q * g rows of a kv head: blocks of equal size of at most 32 rows, whole groups of four.
struct RowCut {
  int blocks, rows;
};
__host__ inline RowCut cut_rows(int64_t all_rows) {
  const int64_t groups = (all_rows + 3) / 4, blocks = (groups + 7) / 8;
  RowCut c;
  c.rows = (int)(4 * ((groups + blocks - 1) / blocks));
  c.blocks = (int)((all_rows + c.rows - 1) / c.rows);
  if (c.blocks == 1) c.rows = (int)all_rows;
  return c;
}

struct DecodeArgs {
  int d, n_q_heads, n_kv_heads, batch, capacity, io_dtype;
  int n_q;  // queries per sequence (1: decode).  `batch` counts (sequence, query) pairs: q and out are
            // [batch][n_q_heads][d] with pair p = sequence * n_q + query; `lens` and the cache are per sequence.
  const __half* qrot;  // of prefill_tc_kernel and rows_attention_kernel: the rotated queries [batch][n_q_heads][value | residual][128]
  int n_splits;        // of prefill_tc_kernel: ranges of a sequence's blocks, each with a part of its own in
  float* part_out;     // [split][batch][n_q_heads][128] (rotated basis) and
  float* part_lse;     // [split][batch][n_q_heads] (natural log)
  int rows_per_block, n_row_blocks;   // of rows_attention_kernel: its cut of a kv head's n_q * group rows and, with qrot, where
  int2* unit_parts;                   // it says which slots a unit's parts are in (first, number)
  float scale;
  uint32_t epoch;  // differs from call to call (top bit set): tags the parts' flags of the persistent kernel
  uint32_t debug;  // test hooks.  bit 0: the first bounded wait of CTA 0 of the persistent kernel reports failure;
                   // bit 1: the MMA thread of CTA (0, 0, 0) of the tcgen05 multi-query kernel reports its wait for the
                   // third decoded block (the last one of a shorter sequence) as failed
  const float* S;
  const Tables* tables;
  const void* q;
  const uint8_t* cache;
  const int32_t* lens;
  void* out;
  float* lse;  // optional [batch][n_q_heads]: natural log of the softmax denominator (for merging partial attentions);
               // with it, a sequence of length 0 is not an error (zeros and -inf)
  int32_t* status;
  Workspace ws;
  Paging pg;  // where the cache's token-blocks live
  // Sequence of (sequence, query) pair p, and the cached tokens its query sees: query j of the n_q last positions of
  // a sequence attends to the tokens before and at its own position (Section 4: the i-th query sees i tokens).
  __device__ __forceinline__ int seq_of(int p) const { return n_q == 1 ? p : p / n_q; }
  __device__ __forceinline__ int visible_len(int p) const {
    if (n_q == 1) return lens[p];
    const int b = p / n_q, v = lens[b] - (n_q - 1 - (p - b * n_q));
    return v > 0 ? v : 0;
  }
};

}  // namespace pq
#include "pq_decode_fast.cuh"
#include "pq_rows.cuh"
#include "pq_rotate.cuh"
#include "pq_prefill.cuh"
#include "pq_prefill_tc.cuh"
#include "pq_split_attention.cuh"
namespace pq {

// The packed cache for split_attention_kernel.  A tile is part of a token-block: five pieces, one per plane, each a multiple
// of 16 bytes long and 16-byte aligned in the cache and in the buffer.
template <int D, bool kWithPairs = false>
struct PackedSplit {
  static constexpr bool kEarlyTables = true, kPairs = kWithPairs;   // see kPairTokens
  static constexpr int kTabMax = 32, kDim = D;
  // the planes of a token-block (make_layout for this head_dim)
  static constexpr int kNb = D / 16, kB1 = 4 * kNb, kB2 = kNb, kB3 = kNb >= 2 ? kNb / 2 : 1, kB4 = kNb >= 4 ? kNb / 4 : 1, kBr = 2 * kNb;
  static constexpr int kRow = kB1 + kB2 + kB3 + kB4 + kBr, kBlockBytes = kTokenBlock * kRow;
  SplitCommon c;
  int n_q;
  int64_t head_bytes;
  const Tables* tables;
  const uint8_t* cache;
  const int32_t* lens;
  Paging pg;

  // Tokens of a tile, as size_split chooses them (packed rows are short): a constant, so that the planes of a staged tile are at
  // constant distances.
  template <int kU>
  __host__ __device__ static constexpr int tile_tokens() { return D <= kU ? 32 : 16; }
  static int tile_bytes(int n) { return n * kRow; }
  __device__ __forceinline__ int len(int pair) const {
    const int b = pair / n_q, v = lens[b] - (n_q - 1 - (pair - b * n_q));
    return v > 0 ? v : 0;
  }
  __device__ __forceinline__ void fill_tables(float2* tab, int tid) const {
    if (tid < PQ_N_CENTROIDS) tab[tid] = make_float2(tables->cen_cos[tid], tables->cen_sin[tid]);
  }
  __device__ __forceinline__ void fill_pairs(float4* pairs, int tid, int n_threads) const {
#pragma unroll 4
    for (int i = tid; i < 256 * 8; i += n_threads) {
      const int a = i >> 3 & 15, b = i >> 7;
      pairs[i] = make_float4(tables->cen_cos[a], tables->cen_sin[a], tables->cen_cos[b], tables->cen_sin[b]);
    }
  }
  __device__ __forceinline__ int shift(int, int, int, int) const { return 0; }
  __device__ __forceinline__ void stage(uint8_t* buf, int pair, int hk, int kv, int t0, int, int lane) const {
    Layout L;
    L.block_bytes = kBlockBytes;
    L.head_bytes = head_bytes;
    const uint8_t* src = cache + kv_block_pair_offset(L, pg, c.n_kv_heads, pair / n_q, hk, t0 / kTokenBlock, c.status) +
                         (int64_t)kv * kBlockBytes;
    const int tok = t0 % kTokenBlock, tile = c.tile;   // a multiple of 16 at these row lengths
    // byte i of the tile: plane by plane, [tile][bytes per token] each
#pragma unroll 1
    for (int i = 16 * lane; i < tile * kRow; i += 512) {
      int at = tok * kB1 + i;
      if (i >= tile * kB1) at = kTokenBlock * kB1 + tok * kB2 + i - tile * kB1;
      if (i >= tile * (kB1 + kB2)) at = kTokenBlock * (kB1 + kB2) + tok * kB3 + i - tile * (kB1 + kB2);
      if (i >= tile * (kB1 + kB2 + kB3)) at = kTokenBlock * (kB1 + kB2 + kB3) + tok * kB4 + i - tile * (kB1 + kB2 + kB3);
      if (i >= tile * (kB1 + kB2 + kB3 + kB4))
        at = kTokenBlock * (kB1 + kB2 + kB3 + kB4) + tok * kBr + i - tile * (kB1 + kB2 + kB3 + kB4);
      split_cp16(buf + i, src + at);
    }
  }
  // kU = 16: a block; kU = 8: half of one (the angles above it are the block's)
  template <int kU>
  __device__ __forceinline__ void decode(const uint8_t* buf, int, int t, int unit, const float2* tab, const float4* pairs, float* y) const {
    constexpr int tile = tile_tokens<kU>();
    const int blk = kU == 16 ? unit : unit >> 1;
    const uint8_t* p2 = buf + tile * kB1;
    const uint8_t* p3 = p2 + tile * kB2;
    const uint8_t* p4 = p3 + tile * kB3;
    const __half* pr = reinterpret_cast<const __half*>(p4 + tile * kB4);
    uint32_t l2 = p2[t * kB2 + blk], l3 = p3[t * kB3 + (blk >> 1)] >> (4 * (blk & 1));
    const uint32_t l4 = p4[t * kB4 + (blk >> 2)] >> (2 * (blk & 3));
    const float r = __half2float(pr[t * kNb + blk]);
    const float2 e4 = tab[24 + (l4 & 3u)];
    float r1[kU / 2];
    uint32_t l1;
    if (kU == 16) {
      l1 = *reinterpret_cast<const uint32_t*>(buf + t * kB1 + 4 * blk);
      const float r3[2] = {r * e4.x, r * e4.y};
      float r2[4];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float2 e = tab[20 + ((l3 >> (2 * j)) & 3u)];
        r2[2 * j] = r3[j] * e.x;
        r2[2 * j + 1] = r3[j] * e.y;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 e = tab[16 + ((l2 >> (2 * j)) & 3u)];
        r1[(2 * j) % (kU / 2)] = r2[j] * e.x;
        r1[(2 * j + 1) % (kU / 2)] = r2[j] * e.y;
      }
    } else {
      const int hi = unit & 1;
      l1 = *reinterpret_cast<const uint16_t*>(buf + t * kB1 + 4 * blk + 2 * hi);
      l2 >>= 4 * hi;
      l3 >>= 2 * hi;
      const float r3 = r * (hi ? e4.y : e4.x);
      const float2 e3 = tab[20 + (l3 & 3u)];
      const float r2[2] = {r3 * e3.x, r3 * e3.y};
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float2 e = tab[16 + ((l2 >> (2 * j)) & 3u)];
        r1[2 * j] = r2[j] * e.x;
        r1[2 * j + 1] = r2[j] * e.y;
      }
    }
    if (kPairs) {
#pragma unroll
      for (int j = 0; j < kU / 4; ++j) {   // byte j of the codes: 128 bytes per entry of the table
        const uint32_t row = (j == 0 ? l1 << 7 : l1 >> (8 * j - 7)) & 0x7F80u;
        const float4 e = *reinterpret_cast<const float4*>(reinterpret_cast<const uint8_t*>(pairs) + row);
        y[4 * j] = r1[2 * j] * e.x;
        y[4 * j + 1] = r1[2 * j] * e.y;
        y[4 * j + 2] = r1[2 * j + 1] * e.z;
        y[4 * j + 3] = r1[2 * j + 1] * e.w;
      }
    } else {
#pragma unroll
      for (int j = 0; j < kU / 2; ++j) {
        const float2 e = tab[(l1 >> (4 * j)) & 15u];
        y[2 * j] = r1[j] * e.x;
        y[2 * j + 1] = r1[j] * e.y;
      }
    }
  }
};

// Pairs of level-1 codes in a table of their own (32 KB, filled by every block before its first tile) where the loop over the tokens is what
// takes the time: head_dim 64 from so many tokens of a block on.  16/8 heads, without and with them: one sequence of 4096 tokens (256
// a block) 9.35 and 9.19 us, four of 4096 (1024) 13.9 and 13.6; four of 1500 (375) 9.24 and 9.22, of 700 (175) 7.16 and 7.38, one of 300
// 5.91 and 6.08.  At head_dim 32 nothing is gained at 4096 tokens (10.27 and 10.20 us), at 128 the kernel has short contexts only.
constexpr int kPairTokens = 256;
template <int D, bool kWithPairs = false>
static PackedSplit<D, kWithPairs> packed_split(const SplitCommon& c, int n_q, const Tables* tables, const uint8_t* cache, const int32_t* lens,
                                               const Paging& pg) {
  PackedSplit<D, kWithPairs> p;
  p.c = c; p.n_q = n_q; p.tables = tables; p.cache = cache; p.lens = lens; p.pg = pg;
  p.head_bytes = make_layout(D, pg.page_tokens).head_bytes;
  return p;
}

// ---- partial attentions: merge, and exact attention over an uncompressed window -----------------
// out = sum_p w_p out_p with w_p = exp(lse_p - lse) and lse = log sum_p exp(lse_p): the attention over the union of
// the token sets behind the parts (token shards on several GPUs; the packed cache and a 16-bit tail).
// A thread takes kV neighbouring elements of a row (4: 16-byte loads), every part's loads independent of the others'.
template <int kV>
__global__ void __launch_bounds__(256) merge_attention_kernel(int d, int64_t n_rows, int n_parts, const void* parts_out, int parts_dtype,
                                                              const float* parts_lse, void* out, int out_dtype, float* lse_out,
                                                              int32_t* status) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");   // the parts come from the kernels before this one
  const int64_t idx = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * kV;
  if (idx >= n_rows * d) return;
  const int64_t row = idx / d;
  float mx = -CUDART_INF_F;
#pragma unroll 8
  for (int p = 0; p < n_parts; ++p) mx = fmaxf(mx, parts_lse[(int64_t)p * n_rows + row]);
  float acc[kV], wsum = 0.f;
#pragma unroll
  for (int e = 0; e < kV; ++e) acc[e] = 0.f;
  if (mx > -CUDART_INF_F) {
#pragma unroll 4
    for (int p = 0; p < n_parts; ++p) {   // part order: the result does not depend on the launch
      const float l = parts_lse[(int64_t)p * n_rows + row];
      const int64_t i = (int64_t)p * n_rows * d + idx;
      float v[kV];
      if (parts_dtype == PQ_DTYPE_BF16) {
        if (kV == 4) {
          const uint2 w = *reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(parts_out) + i);
          v[0] = __uint_as_float(w.x << 16);
          v[1 % kV] = __uint_as_float(w.x & 0xFFFF0000u);
          v[2 % kV] = __uint_as_float(w.y << 16);
          v[3 % kV] = __uint_as_float(w.y & 0xFFFF0000u);
        } else {
          v[0] = __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(parts_out)[i]);
        }
      } else if (kV == 4) {
        const float4 w = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(parts_out) + i);
        v[0] = w.x; v[1 % kV] = w.y; v[2 % kV] = w.z; v[3 % kV] = w.w;
      } else {
        v[0] = reinterpret_cast<const float*>(parts_out)[i];
      }
      if (l == -CUDART_INF_F) continue;   // a part without tokens (its output may hold anything)
      const float w = __expf(l - mx);
#pragma unroll
      for (int e = 0; e < kV; ++e) acc[e] = fmaf(w, v[e], acc[e]);
      wsum += w;
    }
#pragma unroll
    for (int e = 0; e < kV; ++e) acc[e] /= wsum;
  } else if (idx == row * d) {
    set_status(status, PQ_ERR_EMPTY);
  }
  if (out_dtype == PQ_DTYPE_BF16) {
    __nv_bfloat16 o[kV];
#pragma unroll
    for (int e = 0; e < kV; ++e) o[e] = __float2bfloat16(acc[e]);
    if (kV == 4) *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(out) + idx) = *reinterpret_cast<const uint2*>(o);
    else reinterpret_cast<__nv_bfloat16*>(out)[idx] = o[0];
  } else if (kV == 4) {
    *reinterpret_cast<float4*>(reinterpret_cast<float*>(out) + idx) = make_float4(acc[0], acc[1 % kV], acc[2 % kV], acc[3 % kV]);
  } else {
    reinterpret_cast<float*>(out)[idx] = acc[0];
  }
  if (lse_out != nullptr && idx == row * d) lse_out[row] = mx > -CUDART_INF_F ? mx + __logf(wsum) : -CUDART_INF_F;
}

static int32_t launch_merge(int d, int64_t n_rows, int n_parts, const void* parts_out, int parts_dtype, const float* parts_lse, void* out,
                            int out_dtype, float* lse_out, int32_t* status, cudaStream_t stream) {
  const bool wide = d % 4 == 0 && (((uintptr_t)parts_out | (uintptr_t)out) & 15) == 0;
  const dim3 grid((unsigned)((n_rows * d / (wide ? 4 : 1) + 255) / 256));
  return launch_dependent(wide ? merge_attention_kernel<4> : merge_attention_kernel<1>, grid, 256, 0, stream, d, n_rows, n_parts, parts_out,
                          parts_dtype, parts_lse, out, out_dtype, lse_out, status);
}

// Exact softmax attention (Eq. 2) of one query per sequence over an uncompressed window of keys and values (the
// tokens a serving loop keeps in 16 bits, Section 5.3's protocol for generated tokens), whatever the head dim, the rows' type and the group;
// bf16 rows of 128 with up to four heads go to tail_mma_kernel.  One CTA per (kv head,
// sequence, split of the window's tokens); a CTA writes the partial attention of its tokens (part blockIdx.z of the
// output), to be merged by merge_attention_kernel.  Steps of kTailStage tokens (half as many for a float32 window): the
// key and value rows are copied to shared memory with coalesced 16-byte cp.async (all of a step's loads in flight at
// once), then scores by a thread per token (key rows 16 bytes apart modulo 128: conflict-free 16-byte reads), running
// maximum and denominator per head, then a thread per coordinate accumulates P . V.  Bound by the latency of its few steps, so the
// next step's keys are requested as soon as the scores are done and its values as soon as P . V is (batch 8, window of 1024,
// 32/8 heads, 8 splits, 33 MB: 17.5 -> 15.3 us).  Not launched as a programmatic dependent: behind the persistent decode kernel that
// took 7 us longer.
constexpr int kTailThreads = 128, kTailStage = 64;
static_assert(2 * kTailStage <= kTailThreads, "two threads per staged token");
constexpr int kTailSmemMax = 80 * 1024;
__host__ __device__ inline int tail_stage_tokens(int kv_dtype) { return kv_dtype == PQ_DTYPE_BF16 ? kTailStage : kTailStage / 2; }
__host__ __device__ inline size_t tail_smem_bytes(int d, int g, int kv_dtype) {
  const int T = tail_stage_tokens(kv_dtype), row = d * (kv_dtype == PQ_DTYPE_BF16 ? 2 : 4);
  const int h = 4 * ((g + 3) / 4);
  return (size_t)4 * (h * d + h * kTailStage + 3 * kMaxGroup + 4) + (size_t)T * (row + 16) + (size_t)T * row;
}
struct TailArgs {
  int d, n_q_heads, n_kv_heads, io_dtype, kv_dtype, capacity, batch;
  float scale;
  const void* q;
  const void* k;
  const void* v;
  const int32_t* lens;
  void* out;
  float* lse;
  int32_t* status;
};
__device__ __forceinline__ float tail_elem(const void* p, int dtype, int64_t i) {
  return dtype == PQ_DTYPE_BF16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p)[i])
                                : reinterpret_cast<const float*>(p)[i];
}
// kHG = groups of four query heads per kv head (heads past the group read q' = 0 and are not stored).
template <int kHG>
__device__ __forceinline__ void tail_attention(const TailArgs& a, float* tsm) {
  constexpr int kH = 4 * kHG;
  const int d = a.d, g = a.n_q_heads / a.n_kv_heads, hk = blockIdx.x, b = blockIdx.y, tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  float* qs = tsm;                       // [d][kH]: q' = q * scale * log2(e), the heads of a coordinate side by side
  float* sc = qs + kH * d;               // [kTailStage][kH]: scores, then probabilities, of a step
  float* m_sm = sc + kH * kTailStage;    // [kH] running maximum (log2 domain)
  float* l_sm = m_sm + kMaxGroup;        // [kH] running denominator
  float* corr_sm = l_sm + kMaxGroup;     // [kH]
  const int esz = a.kv_dtype == PQ_DTYPE_BF16 ? 2 : 4, row_bytes = d * esz, krow = row_bytes + 16;
  const int T = tail_stage_tokens(a.kv_dtype);
  uint8_t* ks = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(corr_sm + kMaxGroup) + 15) & ~(uintptr_t)15);   // [T][krow]
  uint8_t* vs = ks + (size_t)T * krow;                                                                          // [T][row_bytes]
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  for (int i = tid; i < kH * d; i += kTailThreads) {
    const int c = i / kH, h = i - c * kH;
    qs[i] = h < g ? tail_elem(a.q, a.io_dtype, ((int64_t)b * a.n_q_heads + hk * g + h) * d + c) * a.scale * 1.4426950408889634f : 0.f;
  }
  if (tid < kH) {
    m_sm[tid] = -CUDART_INF_F;
    l_sm[tid] = 0.f;
  }
  int len_all = a.lens[b];
  len_all = len_all < 0 ? 0 : (len_all > a.capacity ? a.capacity : len_all);
  const int per = (len_all + (int)gridDim.z - 1) / (int)gridDim.z;
  const int t_begin = min(len_all, (int)blockIdx.z * per), len = min(len_all, t_begin + per) - t_begin;
  const int64_t part_rows = (int64_t)blockIdx.z * a.batch * a.n_q_heads;   // this split's part of out and lse
  float acc[kH];
#pragma unroll
  for (int h = 0; h < kH; ++h) acc[h] = 0.f;
  const uint32_t ks_s = (uint32_t)__cvta_generic_to_shared(ks), vs_s = (uint32_t)__cvta_generic_to_shared(vs);
  const int gr_shift = 31 - __clz(row_bytes >> 4);   // 16-byte pieces of a row: a power of two
  const int64_t row_stride = (int64_t)a.n_kv_heads * row_bytes;
  const int64_t base = (((int64_t)b * a.capacity + t_begin) * a.n_kv_heads + hk) * row_bytes;
  auto request = [&](uint32_t dst, int stride, const void* src, int c0) {   // the rows of step c0 as one group of copies
    const int n = min(T, len - c0);
    for (int i = tid; i < (n << gr_shift); i += kTailThreads) {
      const int t = i >> gr_shift, piece = i - (t << gr_shift);
      pf_cp16(dst + t * stride + 16 * piece, reinterpret_cast<const uint8_t*>(src) + base + (c0 + t) * row_stride + 16 * piece);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  request(ks_s, krow, a.k, 0);
  request(vs_s, row_bytes, a.v, 0);
  for (int c0 = 0; c0 < len; c0 += T) {
    const int n = min(T, len - c0);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();   // the keys have landed (first step: q', m, l are set)
    {   // scores: two threads per token, each over half of the coordinates (a stage holds at most 64 tokens)
      const int t = tid >> 1, i0 = (tid & 1) * (d >> 1);
      const uint8_t* row = ks + t * krow;
      float s[kH];
#pragma unroll
      for (int h = 0; h < kH; ++h) s[h] = 0.f;
#pragma unroll 2
      for (int i = i0; i < i0 + (d >> 1) && t < n; i += 8) {   // d is a multiple of 16
        float kv[8];
        if (a.kv_dtype == PQ_DTYPE_BF16) {
          const uint4 raw = *reinterpret_cast<const uint4*>(row + 2 * i);
          const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            kv[2 * e] = __uint_as_float(w[e] << 16);
            kv[2 * e + 1] = __uint_as_float(w[e] & 0xFFFF0000u);
          }
        } else {
          const float4 lo = *reinterpret_cast<const float4*>(row + 4 * i);
          const float4 hi = *reinterpret_cast<const float4*>(row + 4 * i + 16);
          kv[0] = lo.x; kv[1] = lo.y; kv[2] = lo.z; kv[3] = lo.w; kv[4] = hi.x; kv[5] = hi.y; kv[6] = hi.z; kv[7] = hi.w;
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
#pragma unroll
          for (int hg = 0; hg < kHG; ++hg) {   // one 16-byte broadcast read gives q' of four heads
            const float4 q4 = *reinterpret_cast<const float4*>(qs + (i + e) * kH + 4 * hg);
            s[4 * hg] = fmaf(q4.x, kv[e], s[4 * hg]);
            s[4 * hg + 1] = fmaf(q4.y, kv[e], s[4 * hg + 1]);
            s[4 * hg + 2] = fmaf(q4.z, kv[e], s[4 * hg + 2]);
            s[4 * hg + 3] = fmaf(q4.w, kv[e], s[4 * hg + 3]);
          }
        }
      }
#pragma unroll
      for (int h = 0; h < kH; ++h) s[h] += __shfl_xor_sync(0xffffffffu, s[h], 1);
      if (t < n && (tid & 1) == 0) {
#pragma unroll
        for (int hg = 0; hg < kHG; ++hg)
          *reinterpret_cast<float4*>(sc + t * kH + 4 * hg) = make_float4(s[4 * hg], s[4 * hg + 1], s[4 * hg + 2], s[4 * hg + 3]);
      }
    }
    __syncthreads();   // the keys are used
    request(ks_s, krow, a.k, c0 + T);   // no copies, but a group, past the last step
    for (int h = warp; h < g; h += kTailThreads / 32) {   // a warp per head: maximum, probabilities, their sum
      float mx = -CUDART_INF_F;
      for (int t = lane; t < n; t += 32) mx = fmaxf(mx, sc[t * kH + h]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      const float m_new = fmaxf(m_sm[h], mx);
      float sum = 0.f;
      for (int t = lane; t < n; t += 32) {
        const float p = exp2f(sc[t * kH + h] - m_new);
        sc[t * kH + h] = p;
        sum += p;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      if (lane == 0) {
        const float corr = exp2f(m_sm[h] - m_new);   // 0 on the first step
        corr_sm[h] = corr;
        l_sm[h] = l_sm[h] * corr + sum;
        m_sm[h] = m_new;
      }
    }
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();   // the probabilities are complete, the values have landed
    if (tid < d) {
#pragma unroll
      for (int h = 0; h < kH; ++h) acc[h] *= h < g ? corr_sm[h] : 0.f;
#pragma unroll 8
      for (int t = 0; t < n; ++t) {
        const float vv = a.kv_dtype == PQ_DTYPE_BF16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(vs + t * row_bytes)[tid])
                                                     : reinterpret_cast<const float*>(vs + t * row_bytes)[tid];
#pragma unroll
        for (int hg = 0; hg < kHG; ++hg) {
          const float4 p4 = *reinterpret_cast<const float4*>(sc + t * kH + 4 * hg);
          acc[4 * hg] = fmaf(p4.x, vv, acc[4 * hg]);
          acc[4 * hg + 1] = fmaf(p4.y, vv, acc[4 * hg + 1]);
          acc[4 * hg + 2] = fmaf(p4.z, vv, acc[4 * hg + 2]);
          acc[4 * hg + 3] = fmaf(p4.w, vv, acc[4 * hg + 3]);
        }
      }
    }
    __syncthreads();   // the values and probabilities are used
    request(vs_s, row_bytes, a.v, c0 + T);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  if (tid < d) {
#pragma unroll
    for (int h = 0; h < kH; ++h)
      if (h < g) {
        const float o = len > 0 ? acc[h] / l_sm[h] : 0.f;
        const int64_t oi = (part_rows + (int64_t)b * a.n_q_heads + hk * g + h) * d + tid;
        if (a.io_dtype == PQ_DTYPE_BF16) reinterpret_cast<__nv_bfloat16*>(a.out)[oi] = __float2bfloat16(o);
        else reinterpret_cast<float*>(a.out)[oi] = o;
      }
  }
  if (tid < g) {
    const int64_t li = part_rows + (int64_t)b * a.n_q_heads + hk * g + tid;
    if (a.lse != nullptr) a.lse[li] = len > 0 ? (m_sm[tid] + log2f(l_sm[tid])) * 0.693147180559945309f : -CUDART_INF_F;
    else if (len <= 0) set_status(a.status, PQ_ERR_EMPTY);
  }
}
template <int kHG>
__global__ void __launch_bounds__(kTailThreads) tail_attention_kernel(const __grid_constant__ TailArgs a) {
  extern __shared__ __align__(16) float tsm[];
  tail_attention<kHG>(a, tsm);
}

}  // namespace pq
#include "pq_tail_mma.cuh"
namespace pq {

// ---- inspection kernels ----------------------------------------------------------------------
__global__ void unpack_codes_kernel(int d, int n_kv_heads, const uint8_t* cache, int batch, Paging pg,
                                    int n_tokens, uint8_t* codes, __half* radii) {
  const Layout L = make_layout(d, pg.page_tokens);
  const int64_t n = (int64_t)batch * n_kv_heads * 2 * n_tokens;
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  const int tok = (int)(v % n_tokens);
  const int kv = (int)((v / n_tokens) & 1);
  const int h = (int)((v / (2 * (int64_t)n_tokens)) % n_kv_heads);
  const int b = (int)(v / (2 * (int64_t)n_tokens * n_kv_heads));
  const int64_t off = block_offset(L, pg, n_kv_heads, b, h, kv, tok);
  if (off < 0) return;  // a page outside the pool: the outputs of this token keep what they held
  const uint8_t* tb = cache + off;
  const int t = tok % kTokenBlock;
  const int n_codes = 15 * L.nb;
  uint8_t* out = codes + v * n_codes;
  for (int blk = 0; blk < L.nb; ++blk) {
    const uint32_t l1 = get_l1(tb, L, t, blk), l2 = get_l2(tb, L, t, blk);
    const uint32_t l3 = get_l3(tb, L, t, blk), l4 = get_l4(tb, L, t, blk);
    for (int j = 0; j < 8; ++j) out[blk * 8 + j] = (l1 >> (4 * j)) & 15u;
    for (int j = 0; j < 4; ++j) out[8 * L.nb + blk * 4 + j] = (l2 >> (2 * j)) & 3u;
    for (int j = 0; j < 2; ++j) out[12 * L.nb + blk * 2 + j] = (l3 >> (2 * j)) & 3u;
    out[14 * L.nb + blk] = l4;
    radii[v * L.nb + blk] = reinterpret_cast<const __half*>(tb + L.orad + t * L.br)[blk];
  }
}

__global__ void dequant_kernel(int d, int n_kv_heads, const float* S, const Tables* tables, const uint8_t* cache,
                               Paging pg, int n_tokens, float* x_hat) {
  extern __shared__ float ysm[];
  __shared__ float cc[32], cs[32];
  const Layout L = make_layout(d, pg.page_tokens);
  const int64_t v = blockIdx.x;
  const int j = threadIdx.x;
  for (int i = j; i < PQ_N_CENTROIDS; i += blockDim.x) {
    cc[i] = tables->cen_cos[i];
    cs[i] = tables->cen_sin[i];
  }
  __syncthreads();
  const int tok = (int)(v % n_tokens);
  const int kv = (int)((v / n_tokens) & 1);
  const int h = (int)((v / (2 * (int64_t)n_tokens)) % n_kv_heads);
  const int b = (int)(v / (2 * (int64_t)n_tokens * n_kv_heads));
  const int64_t off = block_offset(L, pg, n_kv_heads, b, h, kv, tok);
  if (off < 0) return;  // uniform over the CTA
  const uint8_t* tb = cache + off;
  if (d == 128) {
    // the fp16 arithmetic of the attention kernel's value path: u = rn(r * U), x = rn(u * t1)
    const int t = tok % kTokenBlock, blk = j >> 4, i = j & 15;
    const uint32_t c1 = (get_l1(tb, L, t, blk) >> (4 * (i >> 1))) & 15u;
    const uint32_t c2 = (get_l2(tb, L, t, blk) >> (2 * (i >> 2))) & 3u;
    const uint32_t c3 = (get_l3(tb, L, t, blk) >> (2 * (i >> 3))) & 3u;
    const uint32_t c4 = get_l4(tb, L, t, blk);
    const uint32_t up = tables->u_tab[i >> 2][c2 | (c3 << 2) | (c4 << 4)].x;
    const __half2 uh = *reinterpret_cast<const __half2*>(&up);
    const __half r = reinterpret_cast<const __half*>(tb + L.orad + t * L.br)[blk];
    const __half u = __hmul(r, (i & 2) ? __high2half(uh) : __low2half(uh));
    const __half2 t1 = *reinterpret_cast<const __half2*>(&tables->l1_hi[c1]);  // (cos, sin) of the centroid
    ysm[j] = __half2float(__hmul(u, (i & 1) ? __high2half(t1) : __low2half(t1)));
  } else {
    ysm[j] = decode_coord(tb, L, tok % kTokenBlock, j, cc, cs);
  }
  __syncthreads();
  float acc = 0.f;
  for (int k = 0; k < d; ++k) acc = fmaf(ysm[k], S[(int64_t)j * d + k], acc);
  x_hat[v * d + j] = acc;
}

}  // namespace pq

namespace pq {

// The flags in the (uninitialised, possibly shared) scratch are tagged with a per-call number.  It starts at a value drawn from
// the clock and the address space of this process, advances by an odd constant and always has its top bit set, so it
// cannot equal a small integer that another kernel left in the same bytes.
static uint32_t next_epoch() {
  static std::atomic<uint32_t> call_epoch{[] {
    uint64_t x = (uint64_t)std::chrono::steady_clock::now().time_since_epoch().count() ^ (uint64_t)(uintptr_t)&next_epoch;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return (uint32_t)(x ^ (x >> 31));
  }()};
  return call_epoch.fetch_add(0x9E3779B1u, std::memory_order_relaxed) | 0x80000000u;
}

// A persistent kernel (one CTA per SM) as a programmatic dependent: it may be set up while the kernel before it in the stream
// finishes (it waits inside).
static int32_t launch_persistent(void (*kernel)(DecodeArgs), const DecodeArgs& a, int n_sm, int threads, int smem, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_sm < kFastMaxGrid ? n_sm : kFastMaxGrid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, a);
  if (e != cudaSuccess) {
    note_cuda_error(e);
    cudaGetLastError();
    return PQ_ERR_CUDA;
  }
  return launch_status();
}

template <int kHG, bool kAround>
static int32_t launch_rows_as(const DecodeArgs& a, bool paged, cudaStream_t stream) {
  static DeviceMemo configured[2];
  void (*kernel)(DecodeArgs) = paged ? rows_attention_kernel<kHG, kAround, true> : rows_attention_kernel<kHG, kAround, false>;
  const int n_sm = configure_for_device(kernel, kRowSmTotal, configured[paged ? 1 : 0]);
  return n_sm == 0 ? PQ_ERR_CUDA : launch_persistent(kernel, a, n_sm, kRowThreads, kRowSmTotal, stream);
}
// Groups of four rows that the instance for a row block of `rows` rows is built for.
static int rows_groups(int rows) { return rows <= 8 ? 2 : rows <= 24 ? (rows + 3) / 4 : 8; }
static int32_t launch_rows_attention(DecodeArgs a, const RowCut& cut, int n_seq, bool paged, cudaStream_t stream) {
  a.rows_per_block = cut.rows;
  a.n_row_blocks = cut.blocks;
  const int64_t units = (int64_t)n_seq * a.n_kv_heads * cut.blocks;
  a.ws = carve_workspace(a.ws.elected, 128, units, cut.rows);
  a.epoch = next_epoch();
  // Several queries: their rotation, and the merge of the parts with the rotation back, are kernels before and after, whose set-up
  // overlaps this one's.  Inside, a part's rotation of 20 rows takes 7 us and the last part of a unit 12 us for the merge and the
  // rotation back, and a block that works on two units pays twice (five drafted tokens in four sequences of up to 8192 tokens, encode
  // included: 73.9 -> 58.4 us).  One query has at most eight rows, and its workspace may be the static scratch, which has no room for
  // rotated queries.
  if (a.n_q == 1) return launch_rows_as<2, false>(a, paged, stream);
  const int64_t all_rows = (int64_t)a.batch * a.n_q_heads;
  uint8_t* behind = reinterpret_cast<uint8_t*>(a.ws.elected) + a.ws.bytes;
  __half* qrot = reinterpret_cast<__half*>(behind);
  a.qrot = qrot;
  a.unit_parts = reinterpret_cast<int2*>(qrot + all_rows * 256);
  int32_t st = launch_rotate(a.S, a.q, a.io_dtype, all_rows, a.scale * 1.4426950408889634f, qrot, stream);
  if (st != PQ_OK) return st;
  switch (rows_groups(cut.rows)) {
    case 2: st = launch_rows_as<2, true>(a, paged, stream); break;
    case 3: st = launch_rows_as<3, true>(a, paged, stream); break;
    case 4: st = launch_rows_as<4, true>(a, paged, stream); break;
    case 5: st = launch_rows_as<5, true>(a, paged, stream); break;
    case 6: st = launch_rows_as<6, true>(a, paged, stream); break;
    default: st = launch_rows_as<8, true>(a, paged, stream); break;
  }
  return st != PQ_OK ? st : launch_merge_rows(a, stream);
}

// ---- which kernel takes a head_dim-128 call ------------------------------------------------------
// Four kernels compute the same attention; which is fastest depends on the rows per kv head (queries x heads of the group), on
// the number of (kv head, sequence) units and on the length.  Each is estimated in us by a formula fitted to measurements on
// B200 (SM clock 1.9 GHz; 1 to 64 queries, 1 to 32 sequences of 150 to 65536 tokens, 32/8, 28/4, 16/2, 8/8 and 8/1 heads: 3376
// calls, up to four kernels each, and the tcgen05 kernel with 1 to 16 ranges in 18 of them), and the shortest estimate wins; over those calls
// the choice is 0.13 % slower than the best one on average, 20 % at worst (0.5 % and 34 % before the last fit):
//   * cluster kernel, a unit per (query, kv head, sequence): start and end, then per token of a block and wave;
//   * persistent kernel, a unit per (query, kv head, sequence) too: start and end, then 242 SM cycles per 16-token tile (248 with
//     more than four heads), more where a block has several units, and the merge of a unit's parts;
//   * rows kernel, up to 32 rows decoded together: one query 294 + 52 groups cycles per tile and 3.4 us per group of four rows, whose
//     rotations are inside; several queries 261 + 56 groups, start, end and per row the rotations before and after, which are kernels
//     of their own;
//   * tcgen05 kernel, up to 256 rows per decoded block, from 32 rows on: 1.2 us per 64-token block of a pair of CTAs; rotating the
//     queries before and merging and rotating back after grow with the rows and the parts; never below 19.3 us, and 2.7 us more below
//     192 rows.
enum AttentionKernel { kClusterKernel, kPersistentKernel, kRowsKernel, kTensorKernel };
struct AttentionPlan {
  AttentionKernel kernel, persistent;   // `persistent`: what takes the call if the cluster kernel must not
  int n_splits;
};
constexpr int kMaxSplits = 16;
// Whether the persistent and the tcgen05 kernel's maps of shared memory hold on the current device: they count on the place where
// dynamic shared memory starts.
static bool window_as_mapped() {
  static DeviceMemo reserved;   // bytes + 1
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return false;
  int known = reserved[dev].load(std::memory_order_relaxed);
  if (known == 0) {
    int bytes = 0;
    if (cudaDeviceGetAttribute(&bytes, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    reserved[dev].store(known = bytes + 1, std::memory_order_relaxed);
  }
  return known - 1 == (int)kWindowBase;
}
// Whether a kernel takes a call at all.
static bool kernel_takes(AttentionKernel kernel, int64_t batch, int n_q, int n_kv_heads, int g) {
  if (kernel == kPersistentKernel) return batch * n_q * n_kv_heads <= kFastMaxUnits && window_as_mapped();
  if (kernel == kRowsKernel) return batch * n_kv_heads * cut_rows((int64_t)n_q * g).blocks <= kFastMaxUnits;
  return true;
}
// Room for the parts of split tcgen05 calls in the workspace of pq_workspace_bytes: a call whose parts would not fit is split
// less.  (148 SMs with 128 rows each, twice over, bound what a useful split can need.)
__host__ inline int64_t part_rows_room(int64_t pairs, int64_t n_q_heads) {
  return std::max(pairs * n_q_heads, std::min<int64_t>(kMaxSplits * pairs * n_q_heads, 2 * 160 * 128));
}
// `load`: of the cluster kernel (plan_split).  `tensor`: the tcgen05 kernel may be taken.
static AttentionPlan plan_attention(int64_t batch, int n_q, int n_kv_heads, int g, int max_len, int n_sm, const SplitLoad& load, bool tensor) {
  const double kNever = 1e30;
  const int64_t pairs = batch * n_q, rows = (int64_t)n_q * g, stages = ((int64_t)max_len + kStageTokens - 1) / kStageTokens;
  const double tiles = std::ceil(max_len / 16.0), sm_hz = n_sm * 1900.0;   // cycles per us of the device
  // of a persistent schedule (list_segments): units of a block beyond its first one, log2 of the parts of a unit
  auto more_units = [&](int64_t units) -> double {
    const double range = units * (stages + kSegmentCost) / (double)n_sm - (kSegmentCost + 1.5);
    return range <= 0.0 ? 0.0 : 1.0 + std::floor(range / (stages + kSegmentCost));
  };
  auto log_parts = [&](int64_t units) { return std::log2(std::min((double)stages, std::max(1.0, (double)n_sm / units))); };
  double est[4] = {kNever, kNever, kNever, kNever};
  AttentionPlan plan = {kClusterKernel, kClusterKernel, 1};
  est[kClusterKernel] = g <= 2   ? 6.9 + 0.0140 * load.waves * load.tokens + 7.5 * (load.waves - 1)
                        : g <= 4 ? 9.4 + 0.0223 * load.waves * load.tokens + 7.9 * (load.waves - 1)
                                 : 14.5 + 0.0408 * load.waves * load.tokens + 13.5 * (load.waves - 1);
  if (kernel_takes(kPersistentKernel, batch, n_q, n_kv_heads, g)) {
    const int64_t units = pairs * n_kv_heads;
    const double full = std::max(0.0, units / (double)n_sm - 1.0);
    est[kPersistentKernel] = g <= 4 ? 17.0 + units * tiles * 242.0 / sm_hz + 4.0 * more_units(units) + 4.4 * full + 0.7 * log_parts(units) / units
                                    : 22.0 + units * tiles * 248.0 / sm_hz + 5.1 * more_units(units) + 11.0 * full + 2.75 * log_parts(units) / units;
  }
  if (kernel_takes(kRowsKernel, batch, n_q, n_kv_heads, g)) {
    const RowCut cut = cut_rows(rows);
    const int64_t units = batch * n_kv_heads * cut.blocks;
    if (n_q == 1) {
      const int groups = (cut.rows + 3) / 4;
      est[kRowsKernel] = 19.1 + units * tiles * (294.0 + 52.0 * groups) / sm_hz + groups * (3.4 + 1.5 * more_units(units) + 0.94 * log_parts(units) / units);
    } else {
      const int groups = rows_groups(cut.rows);
      const double full = std::max(0.0, units / (double)n_sm - 1.0), all_rows = (double)pairs * n_kv_heads * g;
      est[kRowsKernel] = 13.7 + units * tiles * (261.0 + 56.3 * groups) / sm_hz + groups * (0.71 + 0.24 * more_units(units)) + 3.2 * log_parts(units) / units -
                         1.3 * full + 3.66e-3 * all_rows + 3.33e-3 * std::min(all_rows, 2368.0);
    }
  }
  if (tensor) {
    const int qb_rows = kPtRows / g;
    const int64_t q_blocks = (n_q + qb_rows - 1) / qb_rows, blocks = ((int64_t)max_len + kTokenBlock - 1) / kTokenBlock;
    const int64_t all_rows = pairs * n_kv_heads * g, room = part_rows_room(pairs, (int64_t)n_kv_heads * g) / all_rows;
    for (int s = 1; s <= kMaxSplits && s <= blocks && (s == 1 || (s <= room && batch * s <= 65535)); ++s) {
      const int64_t clusters = (q_blocks + 1) / 2 * n_kv_heads * batch * s, at_once = n_sm / 2;   // two query blocks each
      const double waves = (double)((clusters + at_once - 1) / at_once), work = waves * ((blocks + s - 1) / s);
      const double t = 13.9 + 1.2 * work + 0.79 * std::min(work, 4.0) + 10.2 * (waves - 1.0) + 2.7e-3 * std::min<int64_t>(all_rows, 2368) +
                       1.3e-3 * all_rows + 0.165e-3 * s * all_rows;
      if (t < est[kTensorKernel]) {
        est[kTensorKernel] = t;
        plan.n_splits = s;
      }
    }
    est[kTensorKernel] = std::max(19.3, est[kTensorKernel]) + (all_rows < 192 ? 2.7 : 0.0);
  }
  for (AttentionKernel k : {kPersistentKernel, kRowsKernel, kTensorKernel})
    if (est[k] < est[plan.kernel]) plan.kernel = k;
  plan.persistent = est[kPersistentKernel] <= est[kRowsKernel] ? kPersistentKernel : kRowsKernel;
  if (est[plan.persistent] == kNever) plan.persistent = kClusterKernel;   // too many units for either
  return plan;
}

static int32_t launch_prefill_tc(DecodeArgs a, int batch, int n_q, int n_splits, cudaStream_t stream) {
  static DeviceMemo configured;
  if (configure_for_device(prefill_tc_kernel, kPtSmTotal, configured) == 0) return PQ_ERR_CUDA;
  const int qb_rows = kPtRows / (a.n_q_heads / a.n_kv_heads), q_blocks = (n_q + qb_rows - 1) / qb_rows;
  a.debug = take_debug_wait_failure(4) ? 2u : 0u;
  a.n_splits = n_splits;
  const int64_t all_rows = (int64_t)a.batch * a.n_q_heads;   // the workspace: rotated queries, parts, their log-sum-exps
  __half* qrot = reinterpret_cast<__half*>(a.ws.elected);
  a.qrot = qrot;
  a.part_out = reinterpret_cast<float*>(qrot + all_rows * 256);
  a.part_lse = a.part_out + n_splits * all_rows * 128;
  const int32_t st = launch_rotate(a.S, a.q, a.io_dtype, all_rows, a.scale * 1.4426950408889634f, qrot, stream);
  if (st != PQ_OK) return st;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((q_blocks + 1) & ~1, a.n_kv_heads, batch * n_splits);
  cfg.blockDim = dim3(kPtThreads);
  cfg.dynamicSmemBytes = kPtSmTotal;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // set up while the kernel before it finishes (it waits inside)
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, prefill_tc_kernel, a, (int)n_q);
  if (e != cudaSuccess) {
    note_cuda_error(e);
    cudaGetLastError();
    return PQ_ERR_CUDA;
  }
  const int32_t main_st = launch_status();
  if (main_st != PQ_OK) return main_st;
  return launch_unrotate(a.S, a.part_out, a.part_lse, n_splits, all_rows, a.out, a.io_dtype, a.status, stream);
}

}  // namespace pq

extern "C" {

int64_t pq_workspace_bytes(int32_t head_dim, int32_t batch, int32_t n_q_heads, int32_t n_kv_heads, int32_t max_len) {
  if (!(head_dim == 16 || head_dim == 32 || head_dim == 64 || head_dim == 128)) return PQ_ERR_UNSUPPORTED;
  if (batch <= 0 || n_q_heads <= 0 || n_kv_heads <= 0 || max_len <= 0 || n_q_heads % n_kv_heads) return PQ_ERR_INVALID_ARG;
  // `batch` may be sequences or (sequence, query) pairs: enough for any way the rows of the pairs are cut into units.  A cut into
  // units of at most 32 rows has no more rows than pairs * (group + 3), and 160 more slots.
  const int64_t units = (int64_t)batch * n_kv_heads, g = n_q_heads / n_kv_heads;
  const int64_t one = pq::carve_workspace(nullptr, head_dim, units, g).bytes;
  if (head_dim != 128) return one;
  const int64_t rows = units * (g + 3) + 32 * pq::kFastMaxGridHost;
  // ... and, for several queries, the rotated queries and a record per unit
  const int64_t cut = 6 * 256 + units * 4 + (units + pq::kFastMaxGridHost) * 4 + rows * (2 + 128) * 4 + (int64_t)batch * n_q_heads * 512 + units * 8;
  const int64_t parts = 1024 + (int64_t)batch * n_q_heads * 512 + pq::part_rows_room(batch, n_q_heads) * (1 + 128) * 4;
  return std::max(std::max(cut, one), parts);
}

static int32_t launch_attention(int32_t head_dim, int32_t n_q_heads, int32_t n_kv_heads, const float* S_dev,
                                const void* tables_dev, const void* q_dev, int32_t io_dtype, const void* cache_dev,
                                const int32_t* cache_lens_dev, int32_t batch, int32_t n_q, int32_t capacity, const pq::Paging& pg,
                                int32_t max_len, float scale, void* out_dev, void* workspace_dev, int32_t* status_dev,
                                void* stream, float* lse_dev = nullptr) {
  pq::NvtxRange nvtx_range("pq attention");
  if (!(head_dim == 16 || head_dim == 32 || head_dim == 64 || head_dim == 128)) return PQ_ERR_UNSUPPORTED;
  if (!S_dev || !tables_dev || !q_dev || !cache_dev || !cache_lens_dev || !out_dev || !workspace_dev || !status_dev)
    return PQ_ERR_INVALID_ARG;
  if (batch <= 0 || n_q <= 0 || n_q_heads <= 0 || n_kv_heads <= 0 || capacity <= 0 || max_len <= 0) return PQ_ERR_INVALID_ARG;
  if (n_q_heads % n_kv_heads) return PQ_ERR_INVALID_ARG;
  if (n_q_heads / n_kv_heads > pq::kMaxGroup) return PQ_ERR_UNSUPPORTED;
  if (io_dtype != PQ_DTYPE_F32 && io_dtype != PQ_DTYPE_BF16) return PQ_ERR_UNSUPPORTED;
  const uintptr_t bits = (uintptr_t)S_dev | (uintptr_t)tables_dev | (uintptr_t)q_dev | (uintptr_t)cache_dev |
                         (uintptr_t)out_dev | (uintptr_t)workspace_dev;
  if (bits & 15) return PQ_ERR_ALIGNMENT;
  const int64_t pairs = (int64_t)batch * n_q;  // (sequence, query) pairs: the kernels' batch
  if (pairs > 65535 || n_kv_heads > 65535) return PQ_ERR_UNSUPPORTED;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  pq::DecodeArgs a;
  a.d = head_dim; a.n_q_heads = n_q_heads; a.n_kv_heads = n_kv_heads; a.batch = (int)pairs; a.n_q = n_q; a.capacity = capacity;
  a.io_dtype = io_dtype; a.scale = scale; a.S = S_dev; a.tables = reinterpret_cast<const pq::Tables*>(tables_dev);
  a.q = q_dev; a.cache = reinterpret_cast<const uint8_t*>(cache_dev); a.lens = cache_lens_dev; a.out = out_dev;
  a.status = status_dev;
  a.lse = lse_dev;
  a.pg = pg;
  a.ws = pq::carve_workspace(workspace_dev, head_dim, pairs * n_kv_heads, n_q_heads / n_kv_heads);
  a.rows_per_block = a.n_row_blocks = 0; a.n_splits = 1; a.part_out = a.part_lse = nullptr; a.qrot = nullptr; a.unit_parts = nullptr; a.epoch = a.debug = 0u;
  const int g = n_q_heads / n_kv_heads;
  if (lse_dev != nullptr && n_q != 1) return PQ_ERR_UNSUPPORTED;
  pq::SplitCommon c;
  c.d = head_dim; c.n_q_heads = n_q_heads; c.n_kv_heads = n_kv_heads; c.io_dtype = io_dtype; c.scale = scale;
  c.S = S_dev; c.q = q_dev; c.out = out_dev; c.lse = lse_dev; c.status = status_dev;
  if (head_dim == 128) {
    const bool paged = pg.table != nullptr;
    static pq::DeviceMemo sm_count;
    const int n_sm = pq::sm_count_of_device(sm_count);
    if (n_sm == 0) return PQ_ERR_CUDA;
    if (n_q * g >= pq::kPfRows && pq::take_debug_wait_failure(3)) {
      // the register-fragment kernel: decode each block of the cache once for 64 (query, head) rows; only reached here (it is
      // slower than the tcgen05 kernel at every size)
      static pq::DeviceMemo configured_pf;
      if (pq::configure_for_device(pq::prefill_attention_kernel, pq::kPfTotal, configured_pf) == 0) return PQ_ERR_CUDA;
      const int qb_rows = pq::kPfRows / g;
      dim3 grid((n_q + qb_rows - 1) / qb_rows, n_kv_heads, batch);
      pq::prefill_attention_kernel<<<grid, pq::kPfThreads, pq::kPfTotal, st>>>(a, n_q);
      return pq::launch_status();
    }
    pq::PackedSplit<128> split = pq::packed_split<128>(c, n_q, a.tables, a.cache, cache_lens_dev, pg);
    pq::size_split(split);
    pq::SplitLoad load = {};
    if (pq::plan_split(split, pairs, max_len, &load) == 0) return PQ_ERR_CUDA;
    const bool tensor = lse_dev == nullptr && pq::window_as_mapped() && !pq::take_debug_wait_failure(10);
    pq::AttentionPlan plan = pq::plan_attention(batch, n_q, n_kv_heads, g, max_len, n_sm, load, tensor && n_q * g >= 32);
    if (const int named = pq::take_debug_hook(6, 9)) {   // test hook: the kernel is named
      plan.kernel = named == 6 ? pq::kClusterKernel : named == 7 ? pq::kPersistentKernel : named == 8 ? pq::kRowsKernel : pq::kTensorKernel;
      if (!pq::kernel_takes(plan.kernel, batch, n_q, n_kv_heads, g) || (plan.kernel == pq::kTensorKernel && !tensor))
        return PQ_ERR_UNSUPPORTED;
    }
    const bool forced = n_q * g <= 32 && pq::take_debug_wait_failure(5), fail_wait = n_q * g <= 32 && pq::take_debug_wait_failure(2);
    pq::AttentionKernel kernel = plan.kernel;
    if ((forced || fail_wait) && kernel == pq::kClusterKernel) kernel = plan.persistent;
    if (kernel == pq::kTensorKernel) return pq::launch_prefill_tc(a, batch, n_q, plan.n_splits, st);
    a.debug = fail_wait ? 1u : 0u;
    if (kernel == pq::kRowsKernel) return pq::launch_rows_attention(a, pq::cut_rows((int64_t)n_q * g), batch, paged, st);
    if (kernel == pq::kPersistentKernel) {
      a.epoch = pq::next_epoch();
      static pq::DeviceMemo configured[4];
      void (*fast)(pq::DecodeArgs) =
          g <= 4 ? (paged ? pq::decode_attention_fast_kernel<1, true> : pq::decode_attention_fast_kernel<1, false>)
                 : (paged ? pq::decode_attention_fast_kernel<2, true> : pq::decode_attention_fast_kernel<2, false>);
      if (pq::configure_for_device(fast, pq::kFsTotal, configured[(g > 4 ? 2 : 0) + (paged ? 1 : 0)]) == 0) return PQ_ERR_CUDA;
      return pq::launch_persistent(fast, a, n_sm, pq::kFastThreads, pq::kFsTotal, st);
    }
  }
  switch (head_dim) {
    case 16: return pq::dispatch_split_attention(pq::packed_split<16>(c, n_q, a.tables, a.cache, cache_lens_dev, pg), pairs, max_len, st);
    case 32: return pq::dispatch_split_attention(pq::packed_split<32>(c, n_q, a.tables, a.cache, cache_lens_dev, pg), pairs, max_len, st);
    case 64: {
      auto split = pq::packed_split<64>(c, n_q, a.tables, a.cache, cache_lens_dev, pg);
      pq::size_split(split);
      pq::SplitLoad load = {};
      if (pq::plan_split(split, pairs, max_len, &load) == 0) return PQ_ERR_CUDA;
      if (load.waves * load.tokens < pq::kPairTokens) return pq::dispatch_split_attention(split, pairs, max_len, st);
      return pq::dispatch_split_attention(pq::packed_split<64, true>(c, n_q, a.tables, a.cache, cache_lens_dev, pg), pairs, max_len, st);
    }
    default: return pq::dispatch_split_attention(pq::packed_split<128>(c, n_q, a.tables, a.cache, cache_lens_dev, pg), pairs, max_len, st);
  }
}

int32_t pq_decode_attention(int32_t head_dim, int32_t n_q_heads, int32_t n_kv_heads, const float* S_dev,
                            const void* tables_dev, const void* q_dev, int32_t io_dtype, const void* cache_dev,
                            const int32_t* cache_lens_dev, int32_t batch, int32_t capacity, int32_t max_len,
                            float scale, void* out_dev, void* workspace_dev, int32_t* status_dev, void* stream) {
  return launch_attention(head_dim, n_q_heads, n_kv_heads, S_dev, tables_dev, q_dev, io_dtype, cache_dev, cache_lens_dev,
                          batch, 1, capacity, pq::contiguous_paging(capacity, batch), max_len, scale, out_dev, workspace_dev,
                          status_dev, stream);
}

int32_t pq_decode_attention_paged(int32_t head_dim, int32_t n_q_heads, int32_t n_kv_heads, const float* S_dev,
                                  const void* tables_dev, const void* q_dev, int32_t io_dtype, const void* cache_dev,
                                  const int32_t* cache_lens_dev, int32_t batch, const pq_paging* paging, int32_t max_len,
                                  float scale, void* out_dev, void* workspace_dev, int32_t* status_dev, void* stream) {
  pq::Paging pg;
  const int32_t st = pq::paging_from(paging, head_dim, &pg);
  if (st != PQ_OK) return st;
  return launch_attention(head_dim, n_q_heads, n_kv_heads, S_dev, tables_dev, q_dev, io_dtype, cache_dev, cache_lens_dev,
                          batch, 1, pg.page_tokens * pg.pages_per_seq, pg, max_len, scale, out_dev, workspace_dev, status_dev,
                          stream);
}

int32_t pq_multi_query_attention(int32_t head_dim, int32_t n_q_heads, int32_t n_kv_heads, const float* S_dev,
                                 const void* tables_dev, const void* q_dev, int32_t io_dtype, const void* cache_dev,
                                 const int32_t* cache_lens_dev, int32_t batch, int32_t n_q, int32_t capacity,
                                 int32_t max_len, float scale, void* out_dev, void* workspace_dev, int32_t* status_dev,
                                 void* stream) {
  return launch_attention(head_dim, n_q_heads, n_kv_heads, S_dev, tables_dev, q_dev, io_dtype, cache_dev, cache_lens_dev,
                          batch, n_q, capacity, pq::contiguous_paging(capacity, batch), max_len, scale, out_dev, workspace_dev,
                          status_dev, stream);
}

int32_t pq_multi_query_attention_paged(int32_t head_dim, int32_t n_q_heads, int32_t n_kv_heads, const float* S_dev,
                                       const void* tables_dev, const void* q_dev, int32_t io_dtype, const void* cache_dev,
                                       const int32_t* cache_lens_dev, int32_t batch, int32_t n_q, const pq_paging* paging,
                                       int32_t max_len, float scale, void* out_dev, void* workspace_dev,
                                       int32_t* status_dev, void* stream) {
  pq::Paging pg;
  const int32_t st = pq::paging_from(paging, head_dim, &pg);
  if (st != PQ_OK) return st;
  return launch_attention(head_dim, n_q_heads, n_kv_heads, S_dev, tables_dev, q_dev, io_dtype, cache_dev, cache_lens_dev,
                          batch, n_q, pg.page_tokens * pg.pages_per_seq, pg, max_len, scale, out_dev, workspace_dev, status_dev,
                          stream);
}

int32_t pq_decode_attention_lse(int32_t head_dim, int32_t n_q_heads, int32_t n_kv_heads, const float* S_dev,
                                const void* tables_dev, const void* q_dev, int32_t io_dtype, const void* cache_dev,
                                const int32_t* cache_lens_dev, int32_t batch, int32_t capacity, const pq_paging* paging,
                                int32_t max_len, float scale, void* out_dev, float* lse_dev, void* workspace_dev,
                                int32_t* status_dev, void* stream) {
  if (lse_dev == nullptr || ((uintptr_t)lse_dev & 3)) return lse_dev == nullptr ? PQ_ERR_INVALID_ARG : PQ_ERR_ALIGNMENT;
  pq::Paging pg = pq::contiguous_paging(capacity, batch);
  if (paging != nullptr) {
    const int32_t st = pq::paging_from(paging, head_dim, &pg);
    if (st != PQ_OK) return st;
    capacity = pg.page_tokens * pg.pages_per_seq;
  }
  return launch_attention(head_dim, n_q_heads, n_kv_heads, S_dev, tables_dev, q_dev, io_dtype, cache_dev, cache_lens_dev,
                          batch, 1, capacity, pg, max_len, scale, out_dev, workspace_dev, status_dev, stream, lse_dev);
}

int32_t pq_merge_attention(int32_t head_dim, int32_t n_q_heads, int32_t batch, int32_t n_parts, const void* parts_out_dev,
                           int32_t parts_dtype, const float* parts_lse_dev, void* out_dev, int32_t out_dtype,
                           float* lse_out_dev, int32_t* status_dev, void* stream) {
  if (head_dim <= 0 || n_q_heads <= 0 || batch <= 0 || n_parts <= 0 || n_parts > 1024) return PQ_ERR_INVALID_ARG;
  if (!parts_out_dev || !parts_lse_dev || !out_dev || !status_dev) return PQ_ERR_INVALID_ARG;
  if ((parts_dtype != PQ_DTYPE_F32 && parts_dtype != PQ_DTYPE_BF16) || (out_dtype != PQ_DTYPE_F32 && out_dtype != PQ_DTYPE_BF16))
    return PQ_ERR_UNSUPPORTED;
  const int64_t n_rows = (int64_t)batch * n_q_heads, n = n_rows * head_dim;
  if (n * n_parts >= (1ll << 40)) return PQ_ERR_UNSUPPORTED;
  return pq::launch_merge(head_dim, n_rows, n_parts, parts_out_dev, parts_dtype, parts_lse_dev, out_dev, out_dtype, lse_out_dev, status_dev,
                          reinterpret_cast<cudaStream_t>(stream));
}

int32_t pq_tail_attention(int32_t head_dim, int32_t n_q_heads, int32_t n_kv_heads, const void* q_dev, int32_t io_dtype,
                          const void* k_tail_dev, const void* v_tail_dev, int32_t kv_dtype, const int32_t* tail_lens_dev,
                          int32_t batch, int32_t tail_capacity, int32_t n_splits, float scale, void* out_dev, float* lse_dev,
                          int32_t* status_dev, void* stream) {
  if (n_splits < 1 || n_splits > 1024 || (n_splits > 1 && lse_dev == nullptr)) return PQ_ERR_INVALID_ARG;
  if (((uintptr_t)k_tail_dev | (uintptr_t)v_tail_dev) & 15) return PQ_ERR_ALIGNMENT;
  if (!(head_dim == 16 || head_dim == 32 || head_dim == 64 || head_dim == 128)) return PQ_ERR_UNSUPPORTED;
  if (!q_dev || !k_tail_dev || !v_tail_dev || !tail_lens_dev || !out_dev || !status_dev) return PQ_ERR_INVALID_ARG;
  if (batch <= 0 || batch > 65535 || n_q_heads <= 0 || n_kv_heads <= 0 || tail_capacity <= 0 || n_q_heads % n_kv_heads)
    return PQ_ERR_INVALID_ARG;
  if (n_q_heads / n_kv_heads > pq::kMaxGroup) return PQ_ERR_UNSUPPORTED;
  if ((io_dtype != PQ_DTYPE_F32 && io_dtype != PQ_DTYPE_BF16) || (kv_dtype != PQ_DTYPE_F32 && kv_dtype != PQ_DTYPE_BF16))
    return PQ_ERR_UNSUPPORTED;
  pq::TailArgs a;
  a.d = head_dim; a.n_q_heads = n_q_heads; a.n_kv_heads = n_kv_heads; a.io_dtype = io_dtype; a.kv_dtype = kv_dtype;
  a.capacity = tail_capacity; a.batch = batch; a.scale = scale; a.q = q_dev; a.k = k_tail_dev; a.v = v_tail_dev; a.lens = tail_lens_dev;
  a.out = out_dev; a.lse = lse_dev; a.status = status_dev;
  const int g = n_q_heads / n_kv_heads;
  const size_t smem = pq::tail_smem_bytes(head_dim, g, kv_dtype);
  static pq::DeviceMemo configured1, configured2;
  if (smem > (size_t)pq::kTailSmemMax) return PQ_ERR_UNSUPPORTED;
  if (pq::configure_for_device(pq::tail_attention_kernel<1>, pq::kTailSmemMax, configured1) == 0) return PQ_ERR_CUDA;
  if (pq::configure_for_device(pq::tail_attention_kernel<2>, pq::kTailSmemMax, configured2) == 0) return PQ_ERR_CUDA;
  dim3 grid(n_kv_heads, batch, n_splits);
  if (head_dim == 128 && g <= 4 && kv_dtype == PQ_DTYPE_BF16) {
    static pq::DeviceMemo configured_mma;
    const int need = std::max((int)smem, pq::kTmSmTotal);   // a block may fall back on tail_attention
    if (pq::configure_for_device(pq::tail_mma_kernel, pq::kTailSmemMax, configured_mma) == 0) return PQ_ERR_CUDA;
    pq::tail_mma_kernel<<<grid, pq::kTailThreads, need, reinterpret_cast<cudaStream_t>(stream)>>>(a);
  } else if (g <= 4) pq::tail_attention_kernel<1><<<grid, pq::kTailThreads, smem, reinterpret_cast<cudaStream_t>(stream)>>>(a);
  else pq::tail_attention_kernel<2><<<grid, pq::kTailThreads, smem, reinterpret_cast<cudaStream_t>(stream)>>>(a);
  return pq::launch_status();
}

// ---- decode attention on the library's own scratch ---------------------------------------------
// Scratch for callers that cannot allocate: lives in every GPU context that loads the library.
// In host code the name below is only a handle; the device address comes from
// cudaGetSymbolAddress, once per device, and is what the kernels receive.
static __device__ __align__(256) unsigned char g_static_scratch[PQ_STATIC_SCRATCH_BYTES];

int64_t pq_static_scratch_bytes(void) { return PQ_STATIC_SCRATCH_BYTES; }

int32_t pq_decode_attention_static(int32_t head_dim, int32_t n_q_heads, int32_t n_kv_heads, const float* S_dev,
                                   const void* tables_dev, const void* q_dev, int32_t io_dtype,
                                   const void* cache_dev, const int32_t* cache_lens_dev, int32_t batch,
                                   int32_t capacity, int32_t max_len, float scale, void* out_dev,
                                   int32_t* status_dev, void* stream) {
  if (const int64_t st = pq_workspace_bytes(head_dim, batch, n_q_heads, n_kv_heads, max_len); st < 0) return (int32_t)st;
  const int64_t need = pq::carve_workspace(nullptr, head_dim, (int64_t)batch * n_kv_heads, n_q_heads / n_kv_heads).bytes;
  if (need > PQ_STATIC_SCRATCH_BYTES) return PQ_ERR_SCRATCH;
  static std::atomic<void*> scratch_of_device[pq::kMaxDevices];
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= pq::kMaxDevices) {
    pq::note_cuda_error(e == cudaSuccess ? cudaErrorInvalidDevice : e);
    return PQ_ERR_CUDA;
  }
  void* scratch = scratch_of_device[dev].load(std::memory_order_acquire);
  if (scratch == nullptr) {  // first call on this device (which is current): resolve the symbol
    e = cudaGetSymbolAddress(&scratch, g_static_scratch);
    if (e != cudaSuccess || scratch == nullptr) {
      pq::note_cuda_error(e == cudaSuccess ? cudaErrorInvalidSymbol : e);
      return PQ_ERR_CUDA;
    }
    scratch_of_device[dev].store(scratch, std::memory_order_release);
  }
  return pq_decode_attention(head_dim, n_q_heads, n_kv_heads, S_dev, tables_dev, q_dev, io_dtype, cache_dev,
                             cache_lens_dev, batch, capacity, max_len, scale, out_dev, scratch, status_dev, stream);
}

static int32_t unpack_entry(int32_t head_dim, int32_t n_kv_heads, const void* cache_dev, int32_t batch, int32_t capacity,
                            const pq::Paging& pg, int32_t n_tokens, uint8_t* codes_dev, void* radii_dev, void* stream) {
  if (!(head_dim == 16 || head_dim == 32 || head_dim == 64 || head_dim == 128)) return PQ_ERR_UNSUPPORTED;
  if (!cache_dev || !codes_dev || !radii_dev || batch <= 0 || n_kv_heads <= 0 || n_tokens <= 0 || n_tokens > capacity)
    return PQ_ERR_INVALID_ARG;
  const int64_t n = (int64_t)batch * n_kv_heads * 2 * n_tokens;
  pq::unpack_codes_kernel<<<(unsigned)((n + 127) / 128), 128, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      head_dim, n_kv_heads, reinterpret_cast<const uint8_t*>(cache_dev), batch, pg, n_tokens, codes_dev,
      reinterpret_cast<__half*>(radii_dev));
  return pq::launch_status();
}

int32_t pq_unpack_codes(int32_t head_dim, int32_t n_kv_heads, const void* cache_dev, int32_t batch, int32_t capacity,
                        int32_t n_tokens, uint8_t* codes_dev, void* radii_dev, void* stream) {
  return unpack_entry(head_dim, n_kv_heads, cache_dev, batch, capacity, pq::contiguous_paging(capacity, batch), n_tokens,
                      codes_dev, radii_dev, stream);
}

int32_t pq_unpack_codes_paged(int32_t head_dim, int32_t n_kv_heads, const void* cache_dev, int32_t batch,
                              const pq_paging* paging, int32_t n_tokens, uint8_t* codes_dev, void* radii_dev, void* stream) {
  pq::Paging pg;
  const int32_t st = pq::paging_from(paging, head_dim, &pg);
  if (st != PQ_OK) return st;
  return unpack_entry(head_dim, n_kv_heads, cache_dev, batch, pg.page_tokens * pg.pages_per_seq, pg, n_tokens, codes_dev,
                      radii_dev, stream);
}

static int32_t dequant_entry(int32_t head_dim, int32_t n_kv_heads, const float* S_dev, const void* tables_dev,
                             const void* cache_dev, int32_t batch, int32_t capacity, const pq::Paging& pg, int32_t n_tokens,
                             float* x_hat_dev, void* stream) {
  if (!(head_dim == 16 || head_dim == 32 || head_dim == 64 || head_dim == 128)) return PQ_ERR_UNSUPPORTED;
  if (!S_dev || !tables_dev || !cache_dev || !x_hat_dev || batch <= 0 || n_kv_heads <= 0 || n_tokens <= 0 ||
      n_tokens > capacity)
    return PQ_ERR_INVALID_ARG;
  const int64_t n = (int64_t)batch * n_kv_heads * 2 * n_tokens;
  if (n >= (1ll << 31)) return PQ_ERR_UNSUPPORTED;
  pq::dequant_kernel<<<(unsigned)n, head_dim, head_dim * sizeof(float), reinterpret_cast<cudaStream_t>(stream)>>>(
      head_dim, n_kv_heads, S_dev, reinterpret_cast<const pq::Tables*>(tables_dev),
      reinterpret_cast<const uint8_t*>(cache_dev), pg, n_tokens, x_hat_dev);
  return pq::launch_status();
}

int32_t pq_dequant_kv(int32_t head_dim, int32_t n_kv_heads, const float* S_dev, const void* tables_dev,
                      const void* cache_dev, int32_t batch, int32_t capacity, int32_t n_tokens, float* x_hat_dev,
                      void* stream) {
  return dequant_entry(head_dim, n_kv_heads, S_dev, tables_dev, cache_dev, batch, capacity,
                       pq::contiguous_paging(capacity, batch), n_tokens, x_hat_dev, stream);
}

int32_t pq_dequant_kv_paged(int32_t head_dim, int32_t n_kv_heads, const float* S_dev, const void* tables_dev,
                            const void* cache_dev, int32_t batch, const pq_paging* paging, int32_t n_tokens,
                            float* x_hat_dev, void* stream) {
  pq::Paging pg;
  const int32_t st = pq::paging_from(paging, head_dim, &pg);
  if (st != PQ_OK) return st;
  return dequant_entry(head_dim, n_kv_heads, S_dev, tables_dev, cache_dev, batch, pg.page_tokens * pg.pages_per_seq, pg,
                       n_tokens, x_hat_dev, stream);
}

}  // extern "C"
