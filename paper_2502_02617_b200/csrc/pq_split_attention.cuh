// Decode attention in float32 over any packed layout (included by pq_decode.cu and pq_general.cu): one cluster of
// thread blocks per (kv head, sequence), every warp of the cluster an independent stream of small token tiles.
//
// A lane owns kU consecutive coordinates of the head (its "unit") for the whole call: its share of the rotated queries and
// of the output accumulators stay in registers, and d / kU neighbouring lanes work on one token.  Per token of a tile a lane
// decodes its unit of the key (one 8-byte (cos, sin) lookup per angle, two multiplications), multiplies it into the
// group's query heads (packed float32 multiply-adds), the lanes of the token sum their partial scores, and the decoded
// unit of the value is accumulated with p = 2^(score - m).  m moves lazily: only when a score exceeds it by more than 8
// (log2 units) are the accumulators rescaled.  Units lie side by side in the packed rows, so neighbouring lanes read
// neighbouring bytes.  Tiles of 16 tokens (32 at head_dim 16) go round the warps of the cluster, so a short context
// spreads over all of them; each warp copies its own tiles (16-byte cp.async, three ahead), and nothing in the loop
// waits for another warp.
// The warps of a block merge in shared memory, the blocks of the cluster through distributed shared memory, and each
// block un-rotates d / C coordinates of the output: one launch, no scratch in global memory.
// Bound by instruction issue (angle decode) for long sequences and by the chain of phases for short ones, hence: S is copied
// to shared memory (head dims up to 128) before the kernel ahead in the stream has finished, every block rotates the
// whole query by itself instead of meeting the others first, and the merge has one cluster barrier.
// Measured (32/8 heads; two launches and a workspace before): one sequence of 1000 tokens, head_dim 128 19.8 -> 10.7 us; eight of
// 4096, head_dim 64 111 -> 32 us; the general layout with three bits and seven levels, eight of 4096, 5330 -> 95 us.
// Level 1 of the packed layout, head_dim 64: one 16-byte lookup per byte of codes instead of two of 8 bytes, and planes of a staged
// tile at constant distances: 8 sequences of up to 4096 tokens at head_dim 64, four steps with their appends 127.2 -> 123.4 us.
// kU = 16 for up to four query heads per kv head, 8 for up to eight (the registers of q' and of the accumulators).
#pragma once
#include <cstdint>

namespace pq {

// Warps of a block.  With four or eight query heads q' and the accumulators take 128 registers and the loop is bound by the
// latency of a warp's own chain: two warps per scheduler with 255 registers (31.6 us for 64 units of 2048 tokens at
// head_dim 128, four heads; three warps with 168 and a few spills 39 us, four with half units 32.3 us).  With one or two
// heads four warps per scheduler fit (19.0 us against 20.0 with three and 22.6 with two; head_dim 64, two heads).
__host__ __device__ constexpr int split_warps(int kh) { return kh <= 2 ? 16 : 8; }
constexpr int kSplitStages = 4;            // tiles in flight per warp
constexpr int kSplitSmemMax = 216 * 1024;
constexpr int kSplitPairBytes = 256 * 8 * 16;   // (cos, sin) of both level-1 codes of a byte, eight copies for conflict-free 16-byte reads
constexpr int kUnitStride = 20;            // floats between the 16-coordinate groups of q' in shared memory

// What the kernel needs beside the layout.
struct SplitCommon {
  int d, n_q_heads, n_kv_heads, io_dtype;
  int tile, stage_bytes;   // tokens of a tile, bytes of its staged keys (or values): set by dispatch_split_attention
  float scale;
  const float* S;
  const void* q;
  void* out;
  float* lse;  // may be null; with it an empty sequence is not an error
  int32_t* status;
};

__host__ __device__ constexpr int split_heads(int g) { return g <= 1 ? 1 : g <= 2 ? 2 : g <= 4 ? 4 : 8; }   // heads a block is built for
__host__ __device__ constexpr int split_unit(int kh) { return kh == 8 ? 8 : 16; }
__host__ __device__ inline int split_lanes(int d, int kh) { return d < split_unit(kh) ? 1 : d / split_unit(kh); }   // per token
__host__ __device__ inline int split_pad(int d) { return d < 16 ? 16 : d; }
// Dynamic shared memory: q', the query and partial sums of q', (m, l) of the warps, the block's output, m and l and the merged output, then the
// tiles in flight, whose place the warps' outputs take at the end.
__host__ __device__ inline int split_fixed_bytes(int d, int kh) {
  const int dp = split_pad(d);
  return (4 * (kh * dp / 16 * kUnitStride + 3 * kh * dp + 34 * split_warps(kh) * kh + 2 * kh) + 15) & ~15;
}
__host__ __device__ inline int split_s_bytes(int d) { return d <= 128 ? (d * d * 4 + 15) & ~15 : 0; }   // S, where it fits
__host__ __device__ inline int split_smem_bytes(int d, int kh, int stage_bytes, bool pairs) {
  const int ring = split_warps(kh) * kSplitStages * 2 * stage_bytes, merge = split_warps(kh) * kh * split_pad(d) * 4;
  return (pairs ? kSplitPairBytes : 0) + split_fixed_bytes(d, kh) + split_s_bytes(d) + (ring > merge ? ring : merge);
}

__device__ __forceinline__ uint32_t cluster_map(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ float cluster_ld(uint32_t addr) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ float4 cluster_ld4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}
__device__ __forceinline__ void split_cp16(uint8_t* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void split_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void split_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(kPending) : "memory");
}
__device__ __forceinline__ float split_exp2(float x) {   // relative error 2^-22, 2^-inf = 0
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Sum of v[0 .. kN) over the lanes that own the same unit (lanes L, L + kLanes, ...): halving exchanges while the count
// is even, so that such a lane ends with kN / (32 / kLanes) of the sums, from (L / kLanes) * that on; *from is the index
// of the first.  The order of the additions is fixed.
template <int kN, int kLanes>
__device__ __forceinline__ void unit_lane_sums(float* v, int lane, int* from, int* count) {
  int n = kN, at = 0;
#pragma unroll
  for (int mask = 16; mask >= kLanes; mask >>= 1) {
    if (n > 1) {
      const bool up = lane & mask;
      n >>= 1;
#pragma unroll
      for (int i = 0; i < kN / 2; ++i)
        if (i < n) v[i] = (up ? v[i + n] : v[i]) + __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + n], mask);
      at += up ? n : 0;
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], mask);
    }
  }
  *from = at;
  *count = n;
}

// Layout policies (template parameter P, passed by value) provide
//   SplitCommon c;
//   int tile_bytes(n)                 bytes of n staged tokens of keys (or values)
//   int len(pair)                     tokens the pair's query sees
//   kTabMax, fill_tables(tab, tid)    the (cos, sin) table; kEarlyTables: filled before the kernel ahead in the stream has
//                                     finished (it may not write them)
//   kPairs, fill_pairs(pairs, tid, n) with kPairs also a table of pairs of level-1 codes (kSplitPairBytes)
//   kDim                              head_dim where it is a compile-time constant, else 0
//   void stage(buf, pair, hk, kv, t0, n, lane)  issue a warp's copies of the keys (kv = 0) or values (1) of tokens
//                                     t0 .. t0 + n - 1 (n = tile size, or less in the last tile)
//   int shift(pair, hk, kv, t0)       where in the buffer the tile that starts at token t0 begins
//   void decode<kU>(buf, at, t, unit, tab, pairs, y)   the coordinates of a unit of token t of the tile at buf + at
template <class P, int kH>
__global__ void __launch_bounds__(32 * split_warps(kH), 1) split_attention_kernel(const __grid_constant__ P p) {
  constexpr int kU = split_unit(kH), kSplitWarps = split_warps(kH), kSplitThreads = 32 * kSplitWarps;
  extern __shared__ __align__(16) uint8_t split_smem[];
  __shared__ float2 tab[P::kTabMax];   // at a fixed address: a lookup's offset needs no addition
  const SplitCommon& c = p.c;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int C = gridDim.x, rank = blockIdx.x, hk = blockIdx.y, pair = blockIdx.z;   // the cluster spans the x dimension
  const int d = P::kDim ? P::kDim : c.d, dp = split_pad(d), grp = c.n_q_heads / c.n_kv_heads;
  const int lanes = split_lanes(d, kH), T = c.tile, qs = dp / 16 * kUnitStride;
  float4* pairs = reinterpret_cast<float4*>(split_smem);   // [256][8] where the layout has them
  float* qg = reinterpret_cast<float*>(split_smem + (P::kPairs ? kSplitPairBytes : 0));   // [kH][dp / 16][kUnitStride]
  float* q_in = qg + kH * qs;                         // [kH][dp]
  float* o_sm = q_in + kH * dp;                       // [kH][dp] this block's output (relative to m_sm)
  float* y_sm = o_sm + kH * dp;                       // [kH][dp] merged output
  float* rot_sm = y_sm + kH * dp;                     // [kSplitThreads * kH] partial sums of q'
  float* wm_sm = rot_sm + kSplitThreads * kH;         // [warps][kH]
  float* wl_sm = wm_sm + kSplitWarps * kH;            // [warps][kH]
  float* m_sm = wl_sm + kSplitWarps * kH;             // [kH]
  float* l_sm = m_sm + kH;                            // [kH]
  float* S_sm = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(qg) + split_fixed_bytes(d, kH));   // [d][d], or nothing
  uint8_t* ring = reinterpret_cast<uint8_t*>(S_sm) + split_s_bytes(d);
  float* w_out = reinterpret_cast<float*>(ring);      // [warps][kH][dp], after the loop
  uint8_t* mine = ring + warp * (kSplitStages * 2 * c.stage_bytes);

  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const bool s_staged = d <= 128 && d >= 4 && (reinterpret_cast<uintptr_t>(c.S) & 15) == 0;
  if (s_staged) {
#pragma unroll 2
    for (int i = 4 * tid; i < d * d; i += 4 * kSplitThreads) split_cp16(reinterpret_cast<uint8_t*>(S_sm + i), c.S + i);
  }
  split_commit();
  if (P::kEarlyTables) p.fill_tables(tab, tid);
  if constexpr (P::kPairs) p.fill_pairs(pairs, tid, kSplitThreads);
  asm volatile("griddepcontrol.wait;" ::: "memory");   // lengths, cache and queries may come from the kernel before this one
  const int64_t q0 = ((int64_t)pair * c.n_q_heads + hk * grp) * d;
  const int len = p.len(pair);
  for (int i = tid; i < kH * dp; i += kSplitThreads) {
    const int h = i / dp, k = i - h * dp;
    float v = 0.f;
    if (h < grp && k < d)
      v = c.io_dtype == PQ_DTYPE_BF16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(c.q)[q0 + h * d + k])
                                      : reinterpret_cast<const float*>(c.q)[q0 + h * d + k];
    q_in[i] = v;
    if (d < 16) qg[h * qs + k] = 0.f;   // coordinates past d
  }
  // tiles of this warp: worker, worker + workers, ...; consecutive tiles go to different blocks first.  Where there are
  // fewer tiles than warps, `share` warps take a tile together, each every share-th pass over it.
  const int n_tiles = (len + T - 1) / T, per_pass = 32 / lanes;   // tokens side by side in a warp
  int share = 1;
  while (2 * share * n_tiles <= C * kSplitWarps && 2 * share * per_pass <= T) share *= 2;
  const int worker = (warp * C + rank) / share, sub = (warp * C + rank) - worker * share, workers = C * kSplitWarps / share;
  auto stage = [&](int i) {
    const int tile = worker + i * workers;
    if (tile < n_tiles && worker < workers) {
      uint8_t* buf = mine + (i % kSplitStages) * 2 * c.stage_bytes;
      p.stage(buf, pair, hk, 0, tile * T, min(T, len - tile * T), lane);
      p.stage(buf + c.stage_bytes, pair, hk, 1, tile * T, min(T, len - tile * T), lane);
    }
    split_commit();
  };
#pragma unroll 1
  for (int i = 0; i < kSplitStages - 1; ++i) stage(i);
  if (!P::kEarlyTables) p.fill_tables(tab, tid);

  // ---- q' = q S * scale * log2(e): thread = column tid % d of one of `parts` slices of the sum
  split_wait<kSplitStages - 1>();   // S has landed (the tiles are younger)
  __syncthreads();
  const int parts = max(1, kSplitThreads / d), rot_j = tid % d, rot_k = tid / d;   // threads past parts * d idle
  const int slice = ((d + parts - 1) / parts + 3) & ~3, k_end = min(d, (rot_k + 1) * slice);
  if (rot_k < parts) {
    float acc[kH];
#pragma unroll
    for (int h = 0; h < kH; ++h) acc[h] = 0.f;
    if (s_staged) {
#pragma unroll 1
      for (int k = rot_k * slice; k < k_end; k += 4) {
        float s[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) s[e] = S_sm[(k + e) * d + rot_j];
#pragma unroll
        for (int h = 0; h < kH; ++h) {
          const float4 q4 = *reinterpret_cast<const float4*>(q_in + h * dp + k);
          acc[h] = fmaf(q4.w, s[3], fmaf(q4.z, s[2], fmaf(q4.y, s[1], fmaf(q4.x, s[0], acc[h]))));
        }
      }
    } else {
#pragma unroll 8
      for (int k = rot_k * slice; k < k_end; ++k) {
        const float s = __ldg(c.S + (int64_t)k * d + rot_j);
#pragma unroll
        for (int h = 0; h < kH; ++h) acc[h] = fmaf(q_in[h * dp + k], s, acc[h]);
      }
    }
#pragma unroll
    for (int h = 0; h < kH; ++h) rot_sm[(rot_k * kH + h) * d + rot_j] = acc[h];
  }
  __syncthreads();
#pragma unroll 1
  for (int i = tid; i < kH * d; i += kSplitThreads) {
    float v = rot_sm[i];
#pragma unroll 2
    for (int r = 1; r < parts; ++r) v += rot_sm[r * kH * d + i];
    const int h = i / d, j = i - h * d;
    qg[h * qs + (j >> 4) * kUnitStride + (j & 15)] = v * (c.scale * 1.4426950408889634f);
  }
  __syncthreads();

  // ---- the stream of this warp
  pairs += lane & 7;   // this lane's copy
  const int unit = lane & (lanes - 1);   // this lane's unit
  uint64_t q2[kH][kU / 2], acc[kH][kU / 2];
  float m_run[kH], l_run[kH];   // running reference of every head (the same in all lanes), this lane's share of the denominator
#pragma unroll
  for (int h = 0; h < kH; ++h) {
    m_run[h] = -CUDART_INF_F;
    l_run[h] = 0.f;
    const float* src = qg + h * qs + (unit * kU >> 4) * kUnitStride + (unit * kU & 15);
#pragma unroll
    for (int i = 0; i < kU / 4; ++i) {
      const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(src + 4 * i);
      q2[h][2 * i] = w.x;
      q2[h][2 * i + 1] = w.y;
    }
#pragma unroll
    for (int i = 0; i < kU / 2; ++i) acc[h][i] = 0ull;
  }
  int n_mine = 0;
#pragma unroll 1
  for (int tile = worker; tile < n_tiles && worker < workers; tile += workers, ++n_mine) {
    split_wait<kSplitStages - 2>();
    __syncwarp();
    const uint8_t* kbuf = mine + (n_mine % kSplitStages) * 2 * c.stage_bytes;
    const uint8_t* vbuf = kbuf + c.stage_bytes;
    const int t0 = tile * T, n = min(T, len - t0);
    const int at_k = p.shift(pair, hk, 0, t0), at_v = p.shift(pair, hk, 1, t0);
#pragma unroll 1
    for (int tb = sub * per_pass; tb < n; tb += share * per_pass) {
      const int tt = tb + lane / lanes, t = min(tt, n - 1);   // past the end: the last token again, with weight 0
      float y[kU];
      p.template decode<kU>(kbuf, at_k, t, unit, tab, pairs, y);
      float s[kH];
#pragma unroll
      for (int h = 0; h < kH; ++h) {
        uint64_t s2 = 0ull;
#pragma unroll
        for (int i = 0; i < kU / 2; ++i) s2 = f2_fma(f2_pack(y[2 * i], y[2 * i + 1]), q2[h][i], s2);
        float a, b;
        f2_unpack(s2, a, b);
        s[h] = a + b;
      }
      for (int m = 1; m < lanes; m <<= 1)
#pragma unroll
        for (int h = 0; h < kH; ++h) s[h] += __shfl_xor_sync(0xffffffffu, s[h], m);
      bool over = false;
#pragma unroll
      for (int h = 0; h < kH; ++h) {
        if (tt >= n) s[h] = -CUDART_INF_F;
        over = over || s[h] > m_run[h] + 8.f;
      }
      if (__any_sync(0xffffffffu, over)) {
#pragma unroll
        for (int h = 0; h < kH; ++h) {
          float mx = s[h];
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
          const float m_new = fmaxf(m_run[h], mx);   // finite: the tile has a token
          const float k = split_exp2(m_run[h] - m_new);   // 0 at first
          m_run[h] = m_new;
          l_run[h] *= k;
          const uint64_t kk = f2_pack(k, k);
#pragma unroll
          for (int i = 0; i < kU / 2; ++i) acc[h][i] = f2_mul(acc[h][i], kk);
        }
      }
      p.template decode<kU>(vbuf, at_v, t, unit, tab, pairs, y);
#pragma unroll
      for (int h = 0; h < kH; ++h) {
        const float e = split_exp2(s[h] - m_run[h]);
        l_run[h] += e;
        const uint64_t ee = f2_pack(e, e);
#pragma unroll
        for (int i = 0; i < kU / 2; ++i) acc[h][i] = f2_fma(ee, f2_pack(y[2 * i], y[2 * i + 1]), acc[h][i]);
      }
    }
    __syncwarp();
    stage(n_mine + kSplitStages - 1);
  }
  // ---- merge the warps: bring every warp to the block's reference, then add
  float mb[kH];
#pragma unroll
  for (int h = 0; h < kH; ++h)
    for (int m = lanes; m < 32; m <<= 1) l_run[h] += __shfl_xor_sync(0xffffffffu, l_run[h], m);
  if (lane == 0) {
#pragma unroll
    for (int h = 0; h < kH; ++h) {
      wm_sm[warp * kH + h] = m_run[h];
      wl_sm[warp * kH + h] = l_run[h];
    }
  }
  split_wait<0>();
  __syncthreads();   // the ring is free
  {
    float o[kH * kU];
#pragma unroll
    for (int h = 0; h < kH; ++h) {
      mb[h] = -CUDART_INF_F;
#pragma unroll
      for (int w = 0; w < kSplitWarps; ++w) mb[h] = fmaxf(mb[h], wm_sm[w * kH + h]);
      const float k = m_run[h] == -CUDART_INF_F ? 0.f : split_exp2(m_run[h] - mb[h]);
#pragma unroll
      for (int i = 0; i < kU / 2; ++i) {
        f2_unpack(acc[h][i], o[h * kU + 2 * i], o[h * kU + 2 * i + 1]);
        o[h * kU + 2 * i] *= k;
        o[h * kU + 2 * i + 1] *= k;
      }
    }
    int from, count;
    switch (lanes) {
      case 1: unit_lane_sums<kH * kU, 1>(o, lane, &from, &count); break;
      case 2: unit_lane_sums<kH * kU, 2>(o, lane, &from, &count); break;
      case 4: unit_lane_sums<kH * kU, 4>(o, lane, &from, &count); break;
      case 8: unit_lane_sums<kH * kU, 8>(o, lane, &from, &count); break;
      case 16: unit_lane_sums<kH * kU, 16>(o, lane, &from, &count); break;
      default: from = 0; count = kH * kU; break;
    }
#pragma unroll
    for (int i = 0; i < kH * kU; ++i)
      if (i < count) {   // value from + i: head / coordinate of the unit
        const int e = from + i;
        w_out[(warp * kH + e / kU) * dp + unit * kU + e % kU] = o[i];
      }
  }
  __syncthreads();
  for (int i = tid; i < kH * dp; i += kSplitThreads) {
    float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int w = 0; w < kSplitWarps; ++w) v[w & 3] += w_out[w * kH * dp + i];
    o_sm[i] = (v[0] + v[1]) + (v[2] + v[3]);
  }
  if (warp == 0) {
#pragma unroll
    for (int h = 0; h < kH; ++h) {
      float l = 0.f;
      if (lane < kSplitWarps) {
        const float m = wm_sm[lane * kH + h];
        l = m == -CUDART_INF_F ? 0.f : wl_sm[lane * kH + h] * split_exp2(m - mb[h]);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
      if (lane == 0) {
        m_sm[h] = mb[h];
        l_sm[h] = l;
      }
    }
  }
  // ---- merge the blocks: every block reads all partial outputs (in rank order) and un-rotates d / C coordinates
  const int nc = d / C, j0 = rank * nc;
  if (C > 1) {
    cluster_arrive();
    cluster_wait();
  } else {
    __syncthreads();
  }
  for (int i = tid; i < kH * dp / 4; i += kSplitThreads) {
    const int h = 4 * i / dp;
    const uint32_t m_a = (uint32_t)__cvta_generic_to_shared(m_sm + h), l_a = (uint32_t)__cvta_generic_to_shared(l_sm + h);
    const uint32_t o_a = (uint32_t)__cvta_generic_to_shared(o_sm + 4 * i);
    float M = -CUDART_INF_F, L = 0.f;
    float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int r0 = 0; r0 < C; r0 += 8) {   // eight ranks at a time: their remote loads are all in flight together
      float m[8], l[8];
      float4 o[8];
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const uint32_t from = r0 + r < C ? r0 + r : r0;
        m[r] = cluster_ld(cluster_map(m_a, from));
        l[r] = cluster_ld(cluster_map(l_a, from));
        o[r] = cluster_ld4(cluster_map(o_a, from));
      }
      float m8 = M;
#pragma unroll
      for (int r = 0; r < 8; ++r) m8 = fmaxf(m8, m[r]);
      if (m8 == -CUDART_INF_F) continue;
      const float k = split_exp2(M - m8);   // 0 at first
      L *= k;
      y.x *= k; y.y *= k; y.z *= k; y.w *= k;
      M = m8;
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const float w = r0 + r < C ? split_exp2(m[r] - M) : 0.f;   // 0 for a block without tokens
        L = fmaf(l[r], w, L);
        y.x = fmaf(o[r].x, w, y.x);
        y.y = fmaf(o[r].y, w, y.y);
        y.z = fmaf(o[r].z, w, y.z);
        y.w = fmaf(o[r].w, w, y.w);
      }
    }
    const float inv = len > 0 ? 1.f / L : 0.f;
    *reinterpret_cast<float4*>(y_sm + 4 * i) = make_float4(y.x * inv, y.y * inv, y.z * inv, y.w * inv);
    if (c.lse != nullptr && rank == 0 && 4 * i == h * dp && h < grp)   // scores are in the log2 domain
      c.lse[(int64_t)pair * c.n_q_heads + hk * grp + h] = len > 0 ? (M + log2f(L)) * 0.693147180559945309f : -CUDART_INF_F;
  }
  if (rank == 0 && tid == 0 && len <= 0 && c.lse == nullptr) set_status(c.status, PQ_ERR_EMPTY);
  __syncthreads();
  if (C > 1) cluster_arrive();   // this block has read the others' shared memory; waited for before it gives up its own
  // x_hat_j = sum_k y_k S[j][k]: a warp per row of S
#pragma unroll 1
  for (int jj = warp; jj < nc; jj += kSplitWarps) {
    const float* row = (s_staged ? S_sm : c.S) + (j0 + jj) * d;
    float sum[kH];
#pragma unroll
    for (int h = 0; h < kH; ++h) sum[h] = 0.f;
#pragma unroll 4
    for (int k = lane; k < d; k += 32) {
      const float s = row[k];
#pragma unroll
      for (int h = 0; h < kH; ++h) sum[h] = fmaf(y_sm[h * dp + k], s, sum[h]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int h = 0; h < kH; ++h) sum[h] += __shfl_xor_sync(0xffffffffu, sum[h], o);
    float mine_h = sum[0];   // lane h stores head h
#pragma unroll
    for (int h = 1; h < kH; ++h) mine_h = lane == h ? sum[h] : mine_h;
    if (lane < grp) {
      const int64_t idx = q0 + lane * d + j0 + jj;
      if (c.io_dtype == PQ_DTYPE_BF16) reinterpret_cast<__nv_bfloat16*>(c.out)[idx] = __float2bfloat16(mine_h);
      else reinterpret_cast<float*>(c.out)[idx] = mine_h;
    }
  }
  if (C > 1) cluster_wait();
}

// Clusters of 2^log2c blocks that the device holds at once, one block per SM: a cluster lies inside a GPC, whose SMs need not be
// a multiple of its size (measured: 148 SMs hold 33 clusters of four, 15 of eight, 7 of sixteen).  The runtime is asked once per
// kernel, device and amount of shared memory; `memo` keeps (bytes + 1) << 32 | answer.
constexpr int kClusterSizes = 5;
using ClusterMemo = std::atomic<int64_t>[kMaxDevices][kClusterSizes];
template <typename Kernel>
inline int clusters_at_once(Kernel kernel, int threads, int smem, int log2c, int n_sm, ClusterMemo& memo) {
  if (log2c == 0) return n_sm;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return n_sm >> log2c;
  const int64_t known = memo[dev][log2c].load(std::memory_order_relaxed);
  if (known >> 32 == smem + 1) return (int)(known & 0x7fffffff);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1 << log2c, (unsigned)n_sm);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1u << log2c;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
    cudaGetLastError();
    n = 0;
  }
  n = n < (n_sm >> log2c) ? n : n_sm >> log2c;
  memo[dev][log2c].store((int64_t)(smem + 1) << 32 | n, std::memory_order_relaxed);
  return n;
}

// Blocks per cluster: a power of two that divides d, four tiles per block or more, at most 16 (above the portable limit of 8: for
// a few units of a long context).  The choice is the one with the shortest estimated time: waves of clusters that
// are resident together times (tokens of a block plus what its set-up and merge cost, as long as 25000 / d tokens).  room(i):
// clusters of 2^i blocks at once.
struct SplitLoad {
  int64_t waves, tokens;   // of the choice: waves of clusters, tokens of a block in each
};
template <class Room>
inline int split_cluster_size(int d, int tile, int64_t units, int max_len, Room room, SplitLoad* load) {
  int best = 1;
  int64_t best_cost = INT64_MAX;
  for (int i = 0, C = 1; i < kClusterSizes && C <= d; ++i, C *= 2) {
    if (C > 1 && (int64_t)(C / 2) * tile * 4 >= max_len) break;   // half as many blocks already have no more than four tiles each
    const int at_once = room(i);
    if (at_once <= 0) continue;
    const int64_t waves = (units + at_once - 1) / at_once;
    const int64_t cost = waves * ((max_len + C - 1) / C + 25000 / d);
    if (cost < best_cost) {
      best_cost = cost;
      best = C;
      *load = {waves, (max_len + C - 1) / C};
    }
  }
  return best;
}

// The kernel's cluster size for a call, 0 with the CUDA error noted; P sized by size_split.
template <class P, int kH>
int plan_split_as(const P& p, int64_t pairs, int max_len, SplitLoad* load) {
  static DeviceMemo configured;
  static ClusterMemo memo;
  auto kernel = split_attention_kernel<P, kH>;
  const int n_sm = configure_for_device(kernel, kSplitSmemMax, configured, true);
  if (n_sm == 0) return 0;
  const int smem = split_smem_bytes(p.c.d, kH, p.c.stage_bytes, P::kPairs);
  return split_cluster_size(p.c.d, p.c.tile, pairs * p.c.n_kv_heads, max_len,
                            [&](int i) { return clusters_at_once(kernel, 32 * split_warps(kH), smem, i, n_sm, memo); }, load);
}

template <class P, int kH>
int32_t launch_split_attention(const P& p, int64_t pairs, int max_len, cudaStream_t stream) {
  auto kernel = split_attention_kernel<P, kH>;
  const int smem = split_smem_bytes(p.c.d, kH, p.c.stage_bytes, P::kPairs);
  if (smem > kSplitSmemMax) return PQ_ERR_UNSUPPORTED;
  SplitLoad load;
  const int C = plan_split_as<P, kH>(p, pairs, max_len, &load);
  if (C == 0) return PQ_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(C, p.c.n_kv_heads, (unsigned)pairs);
  cfg.blockDim = dim3(32 * split_warps(kH));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // set up while the kernel before it finishes (it waits inside)
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = C;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = C > 1 ? 2 : 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, p);
  if (e != cudaSuccess) {
    note_cuda_error(e);
    cudaGetLastError();
    return PQ_ERR_CUDA;
  }
  return launch_status();
}

// Tiles of 16 tokens (32 where a lane takes a whole token), fewer where long rows would take more than 200 KB of shared memory.
template <class P>
void size_split(P& p) {
  const int kh = split_heads(p.c.n_q_heads / p.c.n_kv_heads), lanes = split_lanes(p.c.d, kh);
  int T = lanes == 1 ? 32 : 16;
  while (T > 32 / lanes && split_smem_bytes(p.c.d, kh, p.tile_bytes(T), P::kPairs) > 200 * 1024) T /= 2;
  p.c.tile = T;
  p.c.stage_bytes = p.tile_bytes(T);
  if constexpr (P::kDim != 0) p.c.tile = kh == 8 ? P::template tile_tokens<8>() : P::template tile_tokens<16>();   // the same
}
// The instantiation for the group size.
template <class P>
int plan_split(const P& p, int64_t pairs, int max_len, SplitLoad* load) {
  switch (split_heads(p.c.n_q_heads / p.c.n_kv_heads)) {
    case 1: return plan_split_as<P, 1>(p, pairs, max_len, load);
    case 2: return plan_split_as<P, 2>(p, pairs, max_len, load);
    case 4: return plan_split_as<P, 4>(p, pairs, max_len, load);
    default: return plan_split_as<P, 8>(p, pairs, max_len, load);
  }
}
template <class P>
int32_t dispatch_split_attention(P p, int64_t pairs, int max_len, cudaStream_t stream) {
  size_split(p);
  switch (split_heads(p.c.n_q_heads / p.c.n_kv_heads)) {
    case 1: return launch_split_attention<P, 1>(p, pairs, max_len, stream);
    case 2: return launch_split_attention<P, 2>(p, pairs, max_len, stream);
    case 4: return launch_split_attention<P, 4>(p, pairs, max_len, stream);
    default: return launch_split_attention<P, 8>(p, pairs, max_len, stream);
  }
}

}  // namespace pq
