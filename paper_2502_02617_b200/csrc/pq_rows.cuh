// Attention of a few queries per sequence (drafted tokens, short chunks) and of one query with more than four heads per kv
// head, head_dim 128 (included by pq_decode.cu): the persistent kernel of pq_decode_fast.cuh with up to 32 (query, head) rows
// per decoded key and value.
//
// A unit is (sequence, kv head, row block); a row block is 4 kHG rows, row r = query r / g, head r % g of the kv head's
// group, each with its own causal limit.  Tiles are decoded exactly as in the persistent kernel, then the score and value
// MMAs run once per group of four rows on the same fragments.  Decoding is three quarters of a four-row tile, so 20 rows
// cost far less than five calls: it is bound by instruction issue, like the persistent kernel.
// Eight warps with up to 255 registers (16 accumulators per group of rows, all in registers) instead of sixteen with 128; the
// query fragments stay in shared memory (one conflict-free 8-byte read per MMA pair).  All four ring slots belong to the one
// group of eight warps, so copies run three stages ahead.
// Measured (32/8 heads, 4 sequences of 8192 tokens; one decode per query before): 2 queries 52 -> 44 us, 5 107 -> 66, 8 162 -> 84.
#pragma once

namespace pq {

constexpr int kRowWarps = 8, kRowThreads = kRowWarps * 32;
constexpr int kRowMax = 32;                                // rows of a row block
constexpr int kRowSmQ = kSmSegs + 768;                     // q' fragments [row group][k-step][lane], 8 bytes
constexpr int kRowSmRing = (kRowSmQ + 8 * 8 * 32 * 8 + 127) / 128 * 128;
// S, rows 528 bytes apart (a thread per row reads it without bank conflicts), lies where the ring is: before the first copies
// of a segment for the rotation of the query, and after the merge for the last part's un-rotation; behind it its heads' rows in float32
// (one query per sequence; several are rotated by kernels of their own).  Both products are rolled loops over shared memory:
// straight-line code that runs once per segment takes longer to fetch than to run.
constexpr int kRowSStride = 132, kRowQIn = 128 * kRowSStride * 4;
constexpr int kRowMergeMl = kRowWarps * 16 * kMrgStride * 4;   // in the merge buffer, behind 16 rows of every warp: (m, l)
constexpr int kRowMergeBytes = kRowMergeMl + kRowWarps * kRowMax * 8;
constexpr int kRowRingBytes = kRowQIn + 16 * 512 > kRowMergeBytes ? kRowQIn + 16 * 512 : kRowMergeBytes;
constexpr int kRowSmTotal = kRowSmRing + kRowRingBytes + kSmAlign;
constexpr int kRowSmInfo = kSmSegs + 448;                  // int2 [kRowMax]: the row's index in q and out, tokens it sees
constexpr int kRowSmBarS = kSmSegs + 752;                  // mbarrier of the copies of S (the segments take 384 bytes)
static_assert(kStages * kStageBytes <= kRowRingBytes, "ring");
static_assert(kFastMaxSegs * sizeof(Segment) <= 448 && 448 + kRowMax * 8 <= 752 && kRowSmInfo % 8 == 0, "behind the segments");
static_assert(kRowSmTotal <= 227 * 1024, "shared memory of one CTA");

// One warp: copy S into the ring's place (nothing in it is in use any more; a barrier has ordered what was).  Every copy is waited
// for with wait_S before the block reuses the place or ends.
__device__ __forceinline__ void fetch_S(const float* S, uint32_t ring, uint32_t bar, int lane) {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (lane == 0) mbar_expect_tx(bar, 128 * 512);
  __syncwarp();
#pragma unroll 1
  for (int r = lane; r < 128; r += 32) bulk_load(ring + r * kRowSStride * 4, S + r * 128, 512, bar);
}

// Waits for copy `phase` of S.  Bounded, but a wait that gave up elsewhere does not cut it short: the copy is the block's own,
// and it must not be in flight when its place is reused or the block ends.
__device__ __forceinline__ void wait_S(uint32_t bar, uint32_t phase, volatile int* abort_flag) {
  for (int i = 0; i < kSpinLimit; ++i) {
    if (mbar_try_wait(bar, phase)) return;
    if (i > 64) __nanosleep(64);
  }
  *abort_flag = 1;
}

// The last part of a unit: merge the `ns` partials of its rows in slot order, normalise, rotate back by S^T and store.
// `y_sm`: kRowMax * 128 floats, `stat`: 2 * kRowMax; S_sm: see fetch_S (the caller has started it; waited for on `bar`, `phase`).
__device__ __forceinline__ void combine_rows(const DecodeArgs& a, const int2* info, int n_rows, int slot0, int ns, float* y_sm,
                                             float* stat, const float* S_sm, uint32_t bar, uint32_t phase, volatile int* abort_flag) {
  const int tid = threadIdx.x, R = a.rows_per_block;
  {   // eight lanes per row: common reference and denominator
    const int r = tid >> 3, l8 = tid & 7;
    const float2* mlp = reinterpret_cast<const float2*>(a.ws.ml) + (int64_t)slot0 * R + min(r, n_rows - 1);
    float M = -CUDART_INF_F, L = 0.f;
#pragma unroll 2
    for (int s = l8; s < ns; s += 8) {
      const float2 ml = __ldcg(mlp + (int64_t)s * R);
      const float m_new = fmaxf(M, ml.x);
      if (m_new > -CUDART_INF_F) L = L * fast_exp2(M - m_new) + ml.y * fast_exp2(ml.x - m_new);
      M = m_new;
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      const float m2 = __shfl_xor_sync(0xffffffffu, M, o), l2 = __shfl_xor_sync(0xffffffffu, L, o), m_new = fmaxf(M, m2);
      if (m_new > -CUDART_INF_F) L = L * fast_exp2(M - m_new) + l2 * fast_exp2(m2 - m_new);
      M = m_new;
    }
    if (l8 == 0 && r < n_rows) {
      stat[2 * r] = M;
      stat[2 * r + 1] = L > 0.f ? 1.f / L : 0.f;
      if (a.lse != nullptr)   // scores are in the log2 domain
        a.lse[info[r].x] = L > 0.f ? (M + log2f(L)) * 0.693147180559945309f : -CUDART_INF_F;
      else if (info[r].y <= 0) set_status(a.status, PQ_ERR_EMPTY);   // a query that sees no token
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int i = tid; i < n_rows * 32; i += kRowThreads) {   // four coordinates of a row
    const int r = i >> 5;
    const float4* op = reinterpret_cast<const float4*>(a.ws.o + ((int64_t)slot0 * R + r) * 128) + (i & 31);
    const float2* mlp = reinterpret_cast<const float2*>(a.ws.ml) + (int64_t)slot0 * R + r;
    const float M = stat[2 * r], k = stat[2 * r + 1];
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int s = 0; s < ns; ++s) {
      const float4 v = __ldcg(op + (int64_t)s * R * 32);
      const float m = __ldcg(mlp + (int64_t)s * R).x;
      const float w = m == -CUDART_INF_F ? 0.f : fast_exp2(m - M);
      acc.x = fmaf(v.x, w, acc.x);
      acc.y = fmaf(v.y, w, acc.y);
      acc.z = fmaf(v.z, w, acc.z);
      acc.w = fmaf(v.w, w, acc.w);
    }
    *reinterpret_cast<float4*>(y_sm + 4 * i) = make_float4(acc.x * k, acc.y * k, acc.z * k, acc.w * k);
  }
  wait_S(bar, phase, abort_flag);
  __syncthreads();
  // x_hat_i = sum_j y_hat_j S[i][j]: a thread takes output coordinate i of four of the (at most eight) rows
  const int i_out = tid & 127, r0 = (tid >> 7) * 4;
  const float* srow = S_sm + i_out * kRowSStride;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
  for (int j = 0; j < 128; j += 4) {
    const float4 s = *reinterpret_cast<const float4*>(srow + j);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float4 y = *reinterpret_cast<const float4*>(y_sm + (r0 + r) * 128 + j);   // rows past n_rows are not stored
      acc[r] = fmaf(y.w, s.w, fmaf(y.z, s.z, fmaf(y.y, s.y, fmaf(y.x, s.x, acc[r]))));
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
    if (r0 + r < n_rows) {
      const int64_t idx = (int64_t)info[r0 + r].x * 128 + i_out;
      if (a.io_dtype == PQ_DTYPE_BF16) reinterpret_cast<__nv_bfloat16*>(a.out)[idx] = __float2bfloat16(acc[r]);
      else reinterpret_cast<float*>(a.out)[idx] = acc[r];
    }
}

// kAround: the rotations are kernels of their own, before and after (several queries, see launch_rows_attention).  Otherwise one query per
// sequence: the rows are the heads of a group, one row block of at most eight.
template <int kHG, bool kAround, bool kPaged>
__global__ void __launch_bounds__(kRowThreads, 1) rows_attention_kernel(DecodeArgs a) {
  static_assert(kAround || kHG == 2, "one query has at most eight rows");
  extern __shared__ __align__(128) uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((kSmAlign - (smem_u32(smem_raw) & (kSmAlign - 1))) & (kSmAlign - 1));
  const int g_heads = a.n_q_heads / a.n_kv_heads, all_rows = a.n_q * g_heads, R = a.rows_per_block, nrb = a.n_row_blocks;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t sm_base = smem_u32(smem);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kSmFlags);
  int* is_last = reinterpret_cast<int*>(smem + kSmFlags) + 1;
  int* n_segs = reinterpret_cast<int*>(smem + kSmFlags) + 2;
  int* first_rank = reinterpret_cast<int*>(smem + kSmFlags) + 3;
  Segment* segs = reinterpret_cast<Segment*>(smem + kSmSegs);
  const int64_t head_bytes = make_layout(128, a.pg.page_tokens).head_bytes;
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(sm_base + kSmBar + 8 * s, 1);                          // full: producer + tx bytes
      mbar_init(sm_base + kSmBar + 8 * (kStages + s), kRowWarps);      // empty: one arrive per warp
    }
    mbar_init(sm_base + kRowSmBarS, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // a programmatic dependent of the kernel before it, like the persistent kernel
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __syncthreads();   // the barriers are initialised
  if (warp == 0 && !kAround) fetch_S(a.S, sm_base + kRowSmRing, sm_base + kRowSmBarS, lane);   // a constant of the caller, like the tables
  build_fast_tables<kRowThreads>(smem, a.tables);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __syncthreads();
  const uint32_t ring = sm_base + kRowSmRing, bar_S = sm_base + kRowSmBarS;
  const float* S_sm = reinterpret_cast<const float*>(smem + kRowSmRing);
  uint32_t n_S = 0;   // copies of S waited for so far

  const int n_units = a.batch / a.n_q * a.n_kv_heads * nrb;
  // rows of a unit's block, tokens its last row sees (query j sees the tokens t < len - (n_q - 1 - j))
  auto unit_rows = [&](int rb) -> int { return min(R, all_rows - rb * R); };
  auto unit_len = [&](int seq, int rb) -> int {
    const int v = a.lens[seq] - (a.n_q - 1 - (rb * R + unit_rows(rb) - 1) / g_heads);
    return v > 0 ? v : 0;
  };
  auto stages_of = [&](int u) -> int {
    const int len_u = u < n_units ? unit_len(u / (a.n_kv_heads * nrb), u % nrb) : 0;
    return (len_u + kStageTokens - 1) / kStageTokens;
  };
  auto empty_unit = [&](int u) {   // no row sees a token: zeros, and the status says so
    if constexpr (kAround) {
      a.unit_parts[u] = make_int2(0, 0);
    } else {
#pragma unroll 1
      for (int e = 0; e < g_heads * 128; ++e) {   // u: sequence and kv head
        const int64_t idx = (int64_t)u * g_heads * 128 + e;
        if (a.io_dtype == PQ_DTYPE_BF16) reinterpret_cast<__nv_bfloat16*>(a.out)[idx] = __float2bfloat16(0.f);
        else reinterpret_cast<float*>(a.out)[idx] = 0.f;
        if (a.lse != nullptr && (e & 127) == 0) a.lse[idx >> 7] = -CUDART_INF_F;
      }
      if (a.lse == nullptr) set_status(a.status, PQ_ERR_EMPTY);
    }
  };

  const int g = lane >> 2, c = lane & 3;
  const uint32_t rep = (lane & 15) * 8;
  const uint32_t ua = sm_base + kSmU + rep, t1a = sm_base + kSmT1p + rep;
  const int tk_k = (warp & 3) * 16 + g, tk_v = (warp & 3) * 16 + c;   // see decode_attention_fast_kernel
  const uint32_t ok_l1 = tk_k * 32 + c * 8, ok_r = kORad + tk_k * 16 + c * 4;
  const uint32_t ok_c2 = kO2 + tk_k * 8 + c * 2, ok_c3 = kO3 + tk_k * 4 + c, ok_c4 = kO4 + tk_k * 2;
  const uint32_t ov_l1 = tk_v * 32 + g * 4, ov_r = kORad + tk_v * 16 + g * 2;
  const uint32_t ov_c2 = kO2 + tk_v * 8 + g, ov_c3 = kO3 + tk_v * 4 + (lane >> 3), ov_c4 = kO4 + tk_v * 2;
  const uint32_t qf = sm_base + kRowSmQ + lane * 8;
  int gl0 = 0;   // stages streamed so far

  int my_units = list_segments<kRowThreads>(0, n_units, smem + kRowSmQ, segs, n_segs, first_rank, stages_of, empty_unit);
  for (int batch_no = 0; batch_no * kFastMaxSegs < my_units; ++batch_no) {
    if (batch_no > 0)
      my_units = list_segments<kRowThreads>(batch_no, n_units, smem + kRowSmQ, segs, n_segs, first_rank, stages_of, empty_unit);
    const int my_segs = min(kFastMaxSegs, my_units - batch_no * kFastMaxSegs);
    for (int sg = 0; sg < my_segs; ++sg) {
      const int u = segs[sg].unit, st0 = segs[sg].st0, st1 = segs[sg].st1;
      const int n_parts = segs[sg].n_parts, unit_slot = segs[sg].slot0, part = segs[sg].part;
      const int seq = u / (a.n_kv_heads * nrb), rb = u % nrb, hk = (u / nrb) % a.n_kv_heads;
      const int row0 = rb * R, n_rows = unit_rows(rb), len = unit_len(seq, rb);
      const int nblk_total = (len + kTokenBlock - 1) / kTokenBlock;
      const uint8_t* head_base = a.cache + ((int64_t)seq * a.n_kv_heads + hk) * head_bytes;  // of a contiguous cache

      const int n_li = st1 - st0;
      int issued = 0;
      auto issue_copy = [&](int li) {
        const int gl = gl0 + li, s = gl % kStages;
        if (gl >= kStages && !mbar_wait(sm_base + kSmBar + 8 * (kStages + s), (gl / kStages - 1) & 1, abort_flag)) return;
        const int st = st0 + li;
        const uint32_t bytes = min(2, nblk_total - 2 * st) * 2 * kBlockBytes128;
        mbar_expect_tx(sm_base + kSmBar + 8 * s, bytes);
        const uint8_t* src = head_base + (int64_t)st * kStageBytes;
        if (kPaged) {
          Layout Lp;  // the two fields the offset needs
          Lp.block_bytes = kBlockBytes128;
          Lp.head_bytes = head_bytes;
          src = a.cache + kv_block_pair_offset(Lp, a.pg, a.n_kv_heads, seq, hk, 2 * st, a.status);
        }
        bulk_load(ring + s * kStageBytes, src, bytes, sm_base + kSmBar + 8 * s);
        issued = li + 1;
      };
      auto first_copies = [&]() {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        for (int li = 0; li < min(kStages - 1, n_li); ++li) issue_copy(li);
      };
      if (kAround) {
        if (tid == 0) first_copies();
      } else if (warp == 0 && batch_no + sg > 0) {
        fetch_S(a.S, ring, bar_S, lane);
      }
      int2* info = reinterpret_cast<int2*>(smem + kRowSmInfo);
      if (warp == 1) {
        const int row = row0 + min(lane, n_rows - 1), j = row / g_heads;
        info[lane] = make_int2((seq * a.n_q + j) * a.n_q_heads + hk * g_heads + (row - j * g_heads),
                               lane < n_rows ? a.lens[seq] - (a.n_q - 1 - j) : 0);
      }
      // q' = (q S) * scale * log2(e) of the rows as fp16 value + residual in fragment order: the fragment of
      // (row group, k-step ks, lane) holds, for column n = lane / 4 (row n / 2 of the group; value or residual), coordinates
      // 0, 2 | 1, 3 of sub-block ks & 3 of block 2 (lane & 3) + ks / 4.  Read as it is where it was formed before.
      if constexpr (kAround) {
        __syncthreads();   // info
        static_assert(kRowThreads == 8 * 32, "a thread per fragment of a row group");
        const int ks = tid >> 5, at = (lane >> 2 & 1) * 128 + (2 * (lane & 3) + (ks >> 2)) * 16 + (ks & 3) * 4;
        uint2 frag[kHG];
#pragma unroll
        for (int hg = 0; hg < kHG; ++hg)   // rows past the last repeat it
          frag[hg] = __ldcg(reinterpret_cast<const uint2*>(a.qrot + (int64_t)info[4 * hg + (lane >> 3)].x * 256 + at));
#pragma unroll
        for (int hg = 0; hg < kHG; ++hg) *reinterpret_cast<uint2*>(smem + kRowSmQ + hg * 2048 + tid * 8) = frag[hg];
        __syncthreads();
      } else {
        float* q_in = reinterpret_cast<float*>(smem + kRowSmRing + kRowQIn);
        constexpr int kMine = 4;                                            // rows of a thread
        const int j = tid & 127, r_mine = (tid >> 7) * kMine;               // its rotated coordinate
        const int blk = j >> 4, ks = (blk & 1) * 4 + ((j >> 2) & 3);
        uint8_t* dst = smem + kRowSmQ + ks * 256 + (blk >> 1) * 8 + (j & 1) * 4 + ((j >> 1) & 1) * 2;
        __syncthreads();
        if (tid < 8 * 16) {   // eight elements of a row (rows past the last repeat it)
          const int64_t at = (int64_t)info[tid >> 4].x * 128 + 8 * (tid & 15);
          float4 lo, hi;
          if (a.io_dtype == PQ_DTYPE_BF16) {
            const uint4 w = *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(a.q) + at);
            lo = make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xFFFF0000u), __uint_as_float(w.y << 16),
                             __uint_as_float(w.y & 0xFFFF0000u));
            hi = make_float4(__uint_as_float(w.z << 16), __uint_as_float(w.z & 0xFFFF0000u), __uint_as_float(w.w << 16),
                             __uint_as_float(w.w & 0xFFFF0000u));
          } else {
            lo = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(a.q) + at);
            hi = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(a.q) + at + 4);
          }
          *reinterpret_cast<float4*>(q_in + 8 * tid) = lo;
          *reinterpret_cast<float4*>(q_in + 8 * tid + 4) = hi;
        }
        wait_S(bar_S, n_S++ & 1, abort_flag);
        __syncthreads();
        float acc[kMine];
#pragma unroll
        for (int r = 0; r < kMine; ++r) acc[r] = 0.f;
#pragma unroll 4
        for (int k = 0; k < 128; k += 4) {
          float s_col[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) s_col[e] = S_sm[(k + e) * kRowSStride + j];
#pragma unroll
          for (int r = 0; r < kMine; ++r) {
            const float4 q4 = *reinterpret_cast<const float4*>(q_in + (r_mine + r) * 128 + k);
            acc[r] = fmaf(q4.w, s_col[3], fmaf(q4.z, s_col[2], fmaf(q4.y, s_col[1], fmaf(q4.x, s_col[0], acc[r]))));
          }
        }
#pragma unroll
        for (int r = 0; r < kMine; ++r) {
          const int row = r_mine + r;
          const float v = acc[r] * (a.scale * 1.4426950408889634f);
          const __half qh = __float2half_rn(v);
          __half* at = reinterpret_cast<__half*>(dst + (row >> 2) * 2048 + 2 * (row & 3) * 32);
          at[0] = qh;
          at[16] = __float2half_rn(v - __half2float(qh));
        }
        __syncthreads();   // S has been used: the ring takes its place
      }
      if (tid == 0 && !kAround) first_copies();
      float o_acc[kHG][4][4];
      float m_run[kHG], l_run[kHG];   // of row c + 4 hg, as in the persistent kernel
      int limit[kHG];                 // tokens the row sees
#pragma unroll
      for (int hg = 0; hg < kHG; ++hg) {
#pragma unroll
        for (int i = 0; i < 4; ++i) o_acc[hg][i][0] = o_acc[hg][i][1] = o_acc[hg][i][2] = o_acc[hg][i][3] = 0.f;
        m_run[hg] = -CUDART_INF_F;
        l_run[hg] = 0.f;
        limit[hg] = info[c + 4 * hg].y;
      }
#pragma unroll 1
      for (int li = 0; li < n_li; ++li) {
        const int gl = gl0 + li, s = gl % kStages, st = st0 + li;
        if (tid == 0 && li + kStages - 1 < n_li) issue_copy(li + kStages - 1);
        __syncwarp();
        if (!mbar_wait(sm_base + kSmBar + 8 * s, (gl / kStages) & 1, abort_flag)) break;
        if ((a.debug & 1u) && unit_slot == 0 && part == 0 && li == 0 && warp == 0) {   // test hook: see the persistent kernel
          *abort_flag = 1;
          break;
        }
        const int tile_tok0 = st * kStageTokens + warp * 16;
        if (tile_tok0 < len) {
          const uint32_t kblk = sm_base + kRowSmRing + s * kStageBytes + (warp >> 2) * 2 * kBlockBytes128;
          const uint32_t vblk = kblk + kBlockBytes128;
          // scores: the residual operand's MMA first, into the same accumulators (small terms first)
          float sc[kHG][4];
#pragma unroll
          for (int hg = 0; hg < kHG; ++hg)
#pragma unroll
            for (int i = 0; i < 4; ++i) sc[hg][i] = 0.f;
          {
            const uint2 l1A = lds64i<0>(kblk + ok_l1), l1B = lds64i<8 * 32>(kblk + ok_l1);
            const uint32_t rrA = lds32i<0>(kblk + ok_r), rrB = lds32i<8 * 16>(kblk + ok_r);
            const uint32_t c2A = lds16i<0>(kblk + ok_c2), c2B = lds16i<8 * 8>(kblk + ok_c2);
            const uint32_t c3A = lds8i<0>(kblk + ok_c3), c3B = lds8i<8 * 4>(kblk + ok_c3);
            const uint32_t c4A = lds16i<0>(kblk + ok_c4) >> (4 * c), c4B = lds16i<8 * 2>(kblk + ok_c4) >> (4 * c);
#define PQ_KSTEP(H, S)                                                                                      \
  {                                                                                                         \
    __half2 xhA, yhA, xlA, ylA, xhB, yhB, xlB, ylB;                                                         \
    sub_block_hilo<S>(bA, t1a, xhA, yhA, xlA, ylA);                                                         \
    sub_block_hilo<S>(bB, t1a, xhB, yhB, xlB, ylB);                                                         \
    uint2 qv[kHG];                                                                                          \
    _Pragma("unroll") for (int hg = 0; hg < kHG; ++hg) qv[hg] = lds64(qf + hg * 2048 + (4 * (H) + (S)) * 256); \
    _Pragma("unroll") for (int hg = 0; hg < kHG; ++hg)                                                      \
        mma_16816(sc[hg], as_u32(xlA), as_u32(xlB), as_u32(ylA), as_u32(ylB), qv[hg].x, qv[hg].y);          \
    _Pragma("unroll") for (int hg = 0; hg < kHG; ++hg)                                                      \
        mma_16816(sc[hg], as_u32(xhA), as_u32(xhB), as_u32(yhA), as_u32(yhB), qv[hg].x, qv[hg].y);          \
  }
            {
              const BlockRef bA = make_block_ref(l1A.x, c2A, c3A, c4A & 3u, __low2half2(as_h2(rrA)), ua);
              const BlockRef bB = make_block_ref(l1B.x, c2B, c3B, c4B & 3u, __low2half2(as_h2(rrB)), ua);
              PQ_KSTEP(0, 0) PQ_KSTEP(0, 1) PQ_KSTEP(0, 2) PQ_KSTEP(0, 3)
            }
            {
              const BlockRef bA = make_block_ref(l1A.y, c2A >> 8, c3A >> 4, (c4A >> 2) & 3u, __high2half2(as_h2(rrA)), ua);
              const BlockRef bB = make_block_ref(l1B.y, c2B >> 8, c3B >> 4, (c4B >> 2) & 3u, __high2half2(as_h2(rrB)), ua);
              PQ_KSTEP(1, 0) PQ_KSTEP(1, 1) PQ_KSTEP(1, 2) PQ_KSTEP(1, 3)
            }
#undef PQ_KSTEP
          }
          // online softmax, lazily updated reference (see the persistent kernel); a row may see nothing of the tile, or
          // nothing at all yet: its reference is then -inf and its p are 2^-inf = 0
          const int t0 = tile_tok0 + g;
          bool over = false;
#pragma unroll
          for (int hg = 0; hg < kHG; ++hg) {
            sc[hg][0] = t0 < limit[hg] ? sc[hg][0] + sc[hg][1] : -CUDART_INF_F;
            sc[hg][1] = t0 + 8 < limit[hg] ? sc[hg][2] + sc[hg][3] : -CUDART_INF_F;
            over = over || fmaxf(sc[hg][0], sc[hg][1]) > m_run[hg] + kLazyMax;
          }
          if (__any_sync(0xffffffffu, over)) {
#pragma unroll
            for (int hg = 0; hg < kHG; ++hg) {
              float mx = fmaxf(sc[hg][0], sc[hg][1]);
              mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
              mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
              mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
              const float m_new = fmaxf(m_run[hg], mx);
              const float corr = m_run[hg] == -CUDART_INF_F ? 0.f : fast_exp2(m_run[hg] - m_new);
              l_run[hg] *= corr;
              m_run[hg] = m_new;
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                o_acc[hg][i][0] *= corr;
                o_acc[hg][i][1] *= corr;
                o_acc[hg][i][2] *= corr;
                o_acc[hg][i][3] *= corr;
              }
            }
          }
          uint32_t pb[kHG][2][2];   // B operand of the value MMAs, as in the persistent kernel
#pragma unroll
          for (int hg = 0; hg < kHG; ++hg) {
            const float m = m_run[hg] == -CUDART_INF_F ? 0.f : m_run[hg];
            const float p0 = fast_exp2(sc[hg][0] - m), p1 = fast_exp2(sc[hg][1] - m);
            l_run[hg] += p0 + p1;
            const uint32_t ph = as_u32(__floats2half2_rn(p0, p1));
            const int srcA = c * 4 + (g >> 1);
            const uint32_t uA = __shfl_sync(0xffffffffu, ph, srcA), uB = __shfl_sync(0xffffffffu, ph, srcA + 16);
            const uint32_t sel_lo = (g & 1) ? 0x1044u : 0x4410u, sel_hi = (g & 1) ? 0x3244u : 0x4432u;
            pb[hg][0][0] = __byte_perm(uA, 0u, sel_lo);
            pb[hg][0][1] = __byte_perm(uB, 0u, sel_lo);
            pb[hg][1][0] = __byte_perm(uA, 0u, sel_hi);
            pb[hg][1][1] = __byte_perm(uB, 0u, sel_hi);
          }
          {
            BlockRef bv[4];
#define PQ_VLOAD(J)                                                                                          \
  {                                                                                                          \
    const uint32_t l1 = lds32i<4 * (J) * 32>(vblk + ov_l1);                                                  \
    uint32_t rr = lds16i<4 * (J) * 16>(vblk + ov_r);                                                         \
    const uint32_t c2 = lds8i<4 * (J) * 8>(vblk + ov_c2);                                                    \
    const uint32_t c3 = lds8i<4 * (J) * 4>(vblk + ov_c3) >> (4 * (g & 1));                                   \
    const uint32_t c4 = lds16i<4 * (J) * 2>(vblk + ov_c4) >> (2 * g);                                        \
    if (tile_tok0 + c + 4 * (J) >= len) rr = 0u; /* stale bytes past the sequence end stay out of the sums */ \
    bv[J] = make_block_ref(l1, c2, c3, c4 & 3u, as_h2(rr | (rr << 16)), ua);                                 \
  }
            PQ_VLOAD(0) PQ_VLOAD(1) PQ_VLOAD(2) PQ_VLOAD(3)
#undef PQ_VLOAD
#define PQ_VSTEP(S)                                                                                        \
  {                                                                                                        \
    __half2 x0, y0, x1, y1, x2, y2, x3, y3;                                                                \
    sub_block_h2<S>(bv[0], t1a, x0, y0);                                                                   \
    sub_block_h2<S>(bv[1], t1a, x1, y1);                                                                   \
    sub_block_h2<S>(bv[2], t1a, x2, y2);                                                                   \
    sub_block_h2<S>(bv[3], t1a, x3, y3);                                                                   \
    _Pragma("unroll") for (int hg = 0; hg < kHG; ++hg)                                                     \
        mma_16816(o_acc[hg][S], as_u32(x0), as_u32(y0), as_u32(x1), as_u32(y1), pb[hg][0][0], pb[hg][0][1]); \
    _Pragma("unroll") for (int hg = 0; hg < kHG; ++hg)                                                     \
        mma_16816(o_acc[hg][S], as_u32(x2), as_u32(y2), as_u32(x3), as_u32(y3), pb[hg][1][0], pb[hg][1][1]); \
  }
            PQ_VSTEP(0) PQ_VSTEP(1) PQ_VSTEP(2) PQ_VSTEP(3)
#undef PQ_VSTEP
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(sm_base + kSmBar + 8 * (kStages + s));
      }
      gl0 += n_li;
      __syncthreads();
      if (*abort_flag) {   // gave up: let the copies still in flight land (bounded) before the ring is reused
        if (tid == 0)
          for (int li = max(0, issued - kStages); li < issued; ++li) {
            const int gl = gl0 - n_li + li;
            for (int i = 0; i < kSpinLimit && !mbar_try_wait(sm_base + kSmBar + 8 * (gl % kStages), (gl / kStages) & 1); ++i)
              __nanosleep(64);
          }
        __syncthreads();
      }

      // ---- merge the warps (fixed order), 16 rows at a time; write this part's partial; the last part combines the unit
      float* mrg_o = reinterpret_cast<float*>(smem + kRowSmRing);                 // [warps][16 rows][kMrgStride]
      float* mrg_ml = reinterpret_cast<float*>(smem + kRowSmRing + kRowMergeMl);  // [warps][kRowMax][2]
#pragma unroll
      for (int hg = 0; hg < kHG; ++hg) {
        l_run[hg] += __shfl_xor_sync(0xffffffffu, l_run[hg], 4);
        l_run[hg] += __shfl_xor_sync(0xffffffffu, l_run[hg], 8);
        l_run[hg] += __shfl_xor_sync(0xffffffffu, l_run[hg], 16);
        if (g == 0) *reinterpret_cast<float2*>(mrg_ml + (warp * kRowMax + c + 4 * hg) * 2) = make_float2(m_run[hg], l_run[hg]);
      }
      __syncthreads();
      const int slot = unit_slot + part;
#pragma unroll
      for (int h0 = 0; h0 < kHG; h0 += 4) {
        if (4 * h0 >= n_rows) break;
        if (h0 > 0) __syncthreads();
#pragma unroll
        for (int hg = h0; hg < h0 + 4 && hg < kHG; ++hg) {
          float M = -CUDART_INF_F;
#pragma unroll
          for (int w = 0; w < kRowWarps; ++w) M = fmaxf(M, mrg_ml[(w * kRowMax + c + 4 * hg) * 2]);
          const float wgt = m_run[hg] == -CUDART_INF_F ? 0.f : fast_exp2(m_run[hg] - M);
          float* o0 = mrg_o + (warp * 16 + c + 4 * (hg - h0)) * kMrgStride + g;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            o0[(4 * i) * 8] = o_acc[hg][i][0] * wgt;
            o0[(4 * i + 2) * 8] = o_acc[hg][i][1] * wgt;
            o0[(4 * i + 1) * 8] = o_acc[hg][i][2] * wgt;
            o0[(4 * i + 3) * 8] = o_acc[hg][i][3] * wgt;
          }
        }
        __syncthreads();
        const int n_here = min(16, n_rows - 4 * h0);
#pragma unroll 1
        for (int i = tid; i < n_here * 128; i += kRowThreads) {
          const int r = i >> 7, j = i & 127;
          float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int w = 0; w < kRowWarps; ++w) acc[w & 3] += mrg_o[(w * 16 + r) * kMrgStride + (j & 15) * 8 + (j >> 4)];
          __stcg(a.ws.o + ((int64_t)slot * R + 4 * h0 + r) * 128 + j, (acc[0] + acc[1]) + (acc[2] + acc[3]));
        }
      }
      if (tid < n_rows) {
        float M = -CUDART_INF_F, l = 0.f;
#pragma unroll
        for (int w = 0; w < kRowWarps; ++w) M = fmaxf(M, mrg_ml[(w * kRowMax + tid) * 2]);
#pragma unroll
        for (int w = 0; w < kRowWarps; ++w) {
          const float2 ml = *reinterpret_cast<const float2*>(mrg_ml + (w * kRowMax + tid) * 2);
          l += ml.x == -CUDART_INF_F ? 0.f : ml.y * fast_exp2(ml.x - M);
        }
        __stcg(reinterpret_cast<float2*>(a.ws.ml) + (int64_t)slot * R + tid, make_float2(M, l));
      }
      if constexpr (kAround) {   // merge_rows_kernel does the rest
        if (part == 0 && tid == 0) a.unit_parts[u] = make_int2(unit_slot, n_parts);
      } else {
        __syncthreads();
        if (warp == 0) elect_combiner(a, u, unit_slot, part, n_parts, lane, is_last);
        __syncthreads();
        if (*is_last) {
          if (warp == 0) fetch_S(a.S, ring, bar_S, lane);
          combine_rows(a, info, n_rows, unit_slot, n_parts, reinterpret_cast<float*>(smem + kRowSmQ),
                       reinterpret_cast<float*>(smem + kRowSmRing + kRowQIn), S_sm, bar_S, n_S++ & 1, abort_flag);
          if (tid == 0 && n_parts > 1) *reinterpret_cast<volatile uint32_t*>(a.ws.elected + u) = 0u;
        }
      }
      __syncthreads();  // the ring is free again for the next unit
    }
  }
  // A block whose range of the work lies between two units has no segment: the copy of S that it started ahead of the split lands
  // before the block ends.
  if (n_S == 0 && !kAround) wait_S(bar_S, 0u, abort_flag);
  if (tid == 0 && *abort_flag) set_status(a.status, PQ_ERR_TIMEOUT);
}

}  // namespace pq
