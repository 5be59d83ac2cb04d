// Multi-query attention over the packed cache on the 5th-generation tensor cores, head_dim 128 (included by
// pq_decode.cu).  Same computation as pq_prefill.cuh -- the last n_q positions of a sequence attend causally to the
// cached tokens (Eq. 2 / Eq. 3) -- for chunks that fill 128 rows = (128 / g) queries x the g query heads of a kv head.
//
// Two CTAs of sixteen warps form a cluster; each owns 128 rows of one (kv head, sequence), and both loop together over a range of
// the 64-token blocks the queries may see, on one 256-row MMA (see prefill_tc_kernel).  Where rows and sequences leave SMs idle
// the blocks are cut into several ranges, whose parts merge_unrotate_kernel (pq_rotate.cuh) merges; rotate_rows_kernel rotates the
// queries before.  In a CTA
//   * warps 4-14 ("decoders") DeQuant the packed blocks, which bulk copies bring in four ahead (Algorithm 1 by the table lookups of
//     the decode kernel on its replicated, conflict-free tables: fp16 with error-free residuals) and write the tensor-core
//     operands into shared memory as 128-byte-swizzled tiles of 64-coordinate rows: per coordinate half the fp16 values of the
//     tokens followed by their fp16 residuals (K-major: the contraction runs over the coordinates), and V_hat as fp16 values
//     [token][64 coordinates] (MN-major: the contraction runs over the tokens); four stages, so they run ahead of the MMAs.
//     The lookups deliver coordinates (4s, 4s+2 | 4s+1, 4s+3); K_hat keeps that order and Q' is stored in the same one (the
//     contraction does not care), V_hat is put back in natural order by two byte permutes per sub-block;
//   * warp 15 issues the MMAs: S = Q'lo K_hi^T + Q'hi K_lo^T + Q'hi K_hi^T (N = 64, eight k-steps per term) into one of four
//     64-column accumulators in tensor memory, up to three blocks ahead of the softmax, and O += P_j V_hat (N = 128, four
//     k-steps) into a 128-column accumulator.  The A operands live in tensor memory too (Q' hi and lo, written once; P_j,
//     written by the row owners), the B operands are read from shared memory by the tensor core itself;
//   * warps 0-3 ("row owners": tensor-memory lane = row = thread) read the scores with tcgen05.ld, apply the causal mask and the
//     online softmax in the log2 domain without any shuffle (a thread owns its whole row), and write P_j in fp16 over the
//     first columns of the accumulator the scores came from, as the A operand of the value MMA.  The running maximum is
//     updated lazily: only when a score exceeds it by more than 8 is the output accumulator rescaled (tcgen05.ld / multiply /
//     tcgen05.st by the row's owner, after the previous value MMA has completed); otherwise p <= 2^8 stays well inside fp16.
// All hand-offs are mbarriers (packed block full / free, decoded stage full, scores full, P full, value MMA done = stage free);
// every wait is bounded, and a wait that gives up makes every role leave its loop, after which the pair drains its copies
// and MMAs, releases tensor memory and records PQ_ERR_TIMEOUT.
// Measured (32/8 heads, 64 queries, 8 sequences of 32768 tokens): 757 us with the rotations inside, per-lane tables, the score
// terms in two accumulators and MMAs issued from one thread's registers (60 cycles each); 710 with the rotations outside; 582 now:
// 1.1 us per block of a pair.  Decoding and MMAs share the bound: 420 us with the tables left unread and no softmax, 558 without the
// softmax, 469 without the decoding.  Score MMAs of two blocks with N = 128 (24 per two blocks instead of 48) took 675: such an MMA
// runs for 110 cycles, one with N = 64 for 40.  Keys and values in one piece of decoding: 599.
#pragma once

#include "pq_tc_common.cuh"

namespace pq {


constexpr int kPtThreads = 512;   // warps 0-3 row owners, 4-14 decoders, 15 the MMA issuer (registers are allocated per four warps)
constexpr int kPtDecoderWarps = 11;
constexpr int kPtRows = 128;
// Decoded blocks in flight.  Per CTA: the keys of 32 tokens -- for each of the two halves of the coordinates the fp16 values of
// the tokens (128-byte rows) followed by their residuals, one B operand of 64 rows -- and 64 coordinates of the values of 64 tokens.
constexpr int kPtStages = 4;
constexpr int kPtKLo = 32 * 128, kPtKHalf = 2 * kPtKLo, kPtKTile = 2 * kPtKHalf, kPtStage = kPtKTile + 64 * 128;
constexpr int kPtRawBytes = 2 * kBlockBytes128;     // a packed K block and V block
constexpr int kPtRawBufs = 4;                       // of them in flight
constexpr int kPtScores = 4;                        // score accumulators: the score MMAs run ahead of the softmax
constexpr int kPtGroups = 16;                       // warp-sized pieces of a block's decoding
// Shared memory, as offsets in the CTA's shared window (whose addresses carry the CTA's rank in the cluster above): dynamic shared
// memory starts behind what the system keeps (1 KB; where it is not, the kernel is not taken: window_as_mapped), the
// decode tables (those of the decode kernel: 96 KB, replicated for conflict-free lookups) on a 32 KB boundary, so that a
// table address is the OR of disjoint bit fields.
constexpr uint32_t kPtBase = kWindowBase;
constexpr uint32_t kPtRaw = kPtBase;
constexpr uint32_t kPtTab = 32768, kPtT1 = kPtTab + kSmT1p, kPtU = kPtTab + kSmU;
constexpr uint32_t kPtKv = kPtTab + kSmBar;         // the stages; also Q' at the start and O at the end
constexpr uint32_t kPtBar = kPtKv + kPtStages * kPtStage;
constexpr uint32_t kPtBarKv = kPtBar, kPtBarPv = kPtBarKv + 8 * kPtStages, kPtBarRawFull = kPtBarPv + 8 * kPtStages,
                   kPtBarRawEmpty = kPtBarRawFull + 8 * kPtRawBufs, kPtBarS = kPtBarRawEmpty + 8 * kPtRawBufs, kPtBarP = kPtBarS + 8 * kPtScores,
                   kPtBarDrain = kPtBarP + 8 * kPtScores;
constexpr uint32_t kPtMisc = kPtBarDrain + 16;      // tensor-memory base, abort flag
constexpr int kPtSmTotal = (int)(kPtMisc + 16 - kPtBase);
constexpr int kPtOStride = 132;                     // floats per row of the output staging
constexpr int kPtQStride = 136;                     // halves per row of the Q' staging (rows 16 bytes apart mod 128)
// tensor-memory columns: four score accumulators of 64 tokens (P_j, two fp16 per column, later takes the first 32 columns of
// the accumulator it came from), the output accumulator, Q' hi and lo
constexpr uint32_t kPtTmS = 0, kPtTmO = 256, kPtTmQhi = 384, kPtTmQlo = 448;
static_assert(kPtSmTotal <= 227 * 1024, "shared memory of one CTA");
static_assert(kPtRaw + kPtRawBufs * kPtRawBytes <= kPtTab, "the packed blocks fit below the tables");
static_assert(128 * kPtOStride * 4 <= kPtStages * kPtStage, "float32 output staging fits in the stages");
static_assert(2 * 128 * kPtQStride * 2 <= kPtStages * kPtStage, "Q' staging fits in the stages");
static_assert(kPtKv % 1024 == 0 && kPtStage % 1024 == 0, "swizzled tiles start on 1024-byte boundaries");

__device__ __forceinline__ void pt_sts128(uint32_t addr, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
__device__ __forceinline__ uint32_t pt_mapa(uint32_t addr, uint32_t cta_rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(cta_rank));
  return r;
}
__device__ __forceinline__ void pt_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Arrival on a barrier of the even CTA of the pair (`bar` = its shared::cluster address, from mapa).  What the arriving
// warp wrote before is read by its own SM's tensor core (operands in shared memory after fence.proxy.async, P in
// tensor memory after tcgen05.wait::st), which the even CTA's MMA triggers after it has seen the arrival.
__device__ __forceinline__ void pt_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}

// (a0, a1) + (b0, b1) as one packed float32 instruction
__device__ __forceinline__ void pt_add2(float a0, float a1, float b0, float b1, float& c0, float& c1) {
  asm("{\n\t.reg .b64 a, b, c;\n\t"
      "mov.b64 a, {%2, %3};\n\t"
      "mov.b64 b, {%4, %5};\n\t"
      "add.rn.f32x2 c, a, b;\n\t"
      "mov.b64 {%0, %1}, c;\n\t}"
      : "=f"(c0), "=f"(c1)
      : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}

// c += both halves of p, in float32
__device__ __forceinline__ void pt_add_halves(float& c, uint32_t p) {
  asm("{\n\t.reg .b16 lo, hi;\n\t"
      "mov.b32 {lo, hi}, %1;\n\t"
      "add.rn.f32.f16 %0, lo, %0;\n\t"
      "add.rn.f32.f16 %0, hi, %0;\n\t}"
      : "+f"(c)
      : "r"(p));
}

// The CTAs of two consecutive query blocks of one (kv head, sequence) form a cluster and run ONE 256-row MMA per
// step (cta_group::2, issued by a thread of the even CTA): every CTA keeps its own 128 rows of Q', S, P and O in its own
// tensor memory and supplies half of each B operand from its own shared memory -- the keys of 32 of the block's 64
// tokens, the values of 64 of the 128 coordinates -- so a CTA decodes half a block per block and no decoded data
// crosses between the CTAs.  The even CTA's barriers collect the arrivals of both CTAs' decoder and row-owner warps;
// its commits are multicast to both CTAs' barriers.  An odd count of query blocks is completed by a CTA without rows.
__global__ void __launch_bounds__(kPtThreads, 1) prefill_tc_kernel(DecodeArgs a, int n_q) {
  extern __shared__ __align__(1024) uint8_t pt_smem_raw[];
  uint8_t* smem = pt_smem_raw - kPtBase;
  const uint32_t sb = tc_smem_u32(pt_smem_raw) - kPtBase;   // the window: rank << 24
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // known to be uniform
  const int g = a.n_q_heads / a.n_kv_heads;
  const int qb_rows = kPtRows / g;                      // queries of a CTA
  const int n_splits = a.n_splits, split = blockIdx.z % n_splits;   // a pair takes one of n_splits ranges of the blocks
  const int q0 = blockIdx.x * qb_rows, hk = blockIdx.y, b = blockIdx.z / n_splits;
  const int n_rows = max(0, min(qb_rows, n_q - q0)) * g;   // rows in use; row r = (query q0 + r / g, head hk * g + r % g);
                                                           // none in the CTA that only completes a pair
  uint32_t crank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(crank));
  const bool leader = crank == 0;   // the CTA whose thread issues the MMAs and whose barriers collect the arrivals
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kPtMisc + 4);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kPtMisc);
  auto row_index = [&](int r) -> int64_t {               // offset of row r in q / out ([batch][n_q][n_q_heads][128])
    return (((int64_t)b * n_q + q0 + r / g) * a.n_q_heads + hk * g + r % g) * 128;
  };
  if (sb & 0xFFFFFFu) {   // the host asks for the place (window_as_mapped): never, and then NaN rather than anything (both CTAs leave alike)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int r = tid; r < n_rows; r += kPtThreads) a.part_lse[(int64_t)split * a.batch * a.n_q_heads + row_index(r) / 128] = CUDART_NAN_F;
    set_status(a.status, PQ_ERR_CUDA);
    return;
  }
  if (tid == 0) {
    for (int i = 0; i < kPtStages; ++i) {
      tc_mbar_init(sb + kPtBarKv + 8 * i, 2 * kPtGroups);    // one arrival per decoded piece (of both CTAs)
      tc_mbar_init(sb + kPtBarPv + 8 * i, 1);                // tcgen05.commit after the value MMA that read the stage
    }
    for (int i = 0; i < kPtRawBufs; ++i) {
      tc_mbar_init(sb + kPtBarRawFull + 8 * i, 1);           // the bytes of a bulk copy
      tc_mbar_init(sb + kPtBarRawEmpty + 8 * i, kPtGroups);  // one arrival per decoded piece
    }
    for (int i = 0; i < kPtScores; ++i) {
      tc_mbar_init(sb + kPtBarS + 8 * i, 1);   // tcgen05.commit
      tc_mbar_init(sb + kPtBarP + 8 * i, 8);   // one arrival per row-owner warp (of both CTAs)
    }
    tc_mbar_init(sb + kPtBarDrain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  build_fast_tables<kPtThreads>(smem + kPtTab, a.tables);   // from the caller's tables, which no kernel writes
  if (warp == 15) {   // the same warp of both CTAs, the same destination offset
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(sb + kPtMisc) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  // a programmatic dependent of the kernel before it: its results (lengths, cache, queries) are read only after this wait
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int len = a.lens[b];
  // ---- Q' (fp16 value | residual, rotate_rows_kernel) of this CTA's rows: staged in shared memory with coalesced copies, then
  // written to tensor memory by the row owners (lane = row, two k values per column).  Rows that do not exist repeat the
  // last one (they are not stored).
  for (int i = tid; i < kPtRows * 32; i += kPtThreads) {
    const int r = i >> 5, piece = i & 31;
    const uint32_t dst = sb + kPtKv + r * (2 * kPtQStride * 2) + (piece >> 4) * (kPtQStride * 2) + (piece & 15) * 16;
    if (n_rows > 0) pf_cp16(dst, a.qrot + row_index(min(r, n_rows - 1)) * 2 + 8 * piece);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();   // Q' is staged, tensor memory is allocated
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = *tmem_slot;
  if (warp < 4) {
    const uint32_t trow = tmem_base + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
    for (int c = 0; c < 4; ++c) {   // hi columns 0..31, 32..63, then lo
      const uint4* src = reinterpret_cast<const uint4*>(smem + kPtKv + tid * (2 * kPtQStride * 2) + (c >> 1) * (kPtQStride * 2) + (c & 1) * 128);
      uint32_t v[32];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const uint4 w = src[i];
        v[4 * i] = w.x; v[4 * i + 1] = w.y; v[4 * i + 2] = w.z; v[4 * i + 3] = w.w;
      }
      tc_st32u(trow + (c < 2 ? kPtTmQhi : kPtTmQlo) + 32 * (c & 1), v);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();   // Q' is in tensor memory; the staging is dead: the stages may be written
  pt_cluster_sync();   // both CTAs' barriers are initialised and both halves of Q' are in place
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  // the last query of the pair sees the most
  const int q_last = min(n_q, ((int)(blockIdx.x | 1u) + 1) * qb_rows) - 1;
  const int vis_cta = max(0, len - (n_q - 1 - q_last));
  const int all_blocks = (vis_cta + kTokenBlock - 1) / kTokenBlock;
  const int jb0 = (int)((int64_t)all_blocks * split / n_splits);                       // this pair's blocks are jb0 + jb,
  const int n_blocks = (int)((int64_t)all_blocks * (split + 1) / n_splits) - jb0;      // 0 <= jb < n_blocks
  // where this CTA's warps announce themselves: the barriers of the even CTA
  const uint32_t to_leader = pt_mapa(sb + kPtBase, 0u) - (sb + kPtBase);   // + a local shared address: that place in the even CTA (cluster window)
  const Layout L = make_layout(128, a.pg.page_tokens);

  float l_run = 0.f, m_run = -CUDART_INF_F;   // row owners: denominator and reference of this thread's row
  if (warp < 4) {
    // ================= row owners: softmax of row `tid` =================
    const int r = tid;
    const int vis = r < n_rows ? max(0, len - (n_q - 1 - (q0 + r / g))) : 0;
    const uint32_t trow = tmem_base + ((uint32_t)(warp * 32) << 16);
    const int vis_min = __reduce_min_sync(0xffffffffu, vis);
    for (int jb = 0; jb < n_blocks; ++jb) {
      const int t = jb % kPtScores;
      const uint32_t ph = (uint32_t)(jb / kPtScores) & 1u;
      bool ok = __all_sync(0xffffffffu, tc_mbar_wait(sb + kPtBarS + 8 * t, ph, abort_flag));
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      float s[64];
#pragma unroll
      for (int c = 0; c < 2; ++c) tc_ld32(trow + kPtTmS + 64 * t + 32 * c, s + 32 * c);
      // the causal mask touches only the last blocks of a row: one uniform test per warp skips it elsewhere
      if ((jb0 + jb + 1) * kTokenBlock > vis_min) {
#pragma unroll
        for (int i = 0; i < 64; ++i) s[i] = (jb0 + jb) * kTokenBlock + i < vis ? s[i] : -CUDART_INF_F;
      }
      float mx4[4] = {-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};   // four chains: no 64-long dependency
#pragma unroll
      for (int i = 0; i < 64; i += 8) {
#pragma unroll
        for (int c = 0; c < 4; ++c) mx4[c] = fmaxf(mx4[c], fmaxf(s[i + 2 * c], s[i + 2 * c + 1]));
      }
      const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
      // lazy reference: move it only when some score exceeds it by more than 8 (p <= 2^8 otherwise)
      const bool grow = mx > m_run + 8.f || (m_run == -CUDART_INF_F && mx > -CUDART_INF_F);
      if (__any_sync(0xffffffffu, grow)) {
        const float m_new = grow ? mx : m_run;
        const float corr = m_run == -CUDART_INF_F ? 1.f : fast_exp2(m_run - m_new);   // nothing accumulated yet: nothing to scale
        if (jb > 0) {
          // the value MMAs up to block jb - 1 must have completed before the accumulator is touched
          ok = __all_sync(0xffffffffu, tc_mbar_wait(sb + kPtBarPv + 8 * ((jb - 1) % kPtStages), (uint32_t)((jb - 1) / kPtStages) & 1u, abort_flag));
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
          for (int c = 0; c < 4; ++c) {
            float o[32];
            tc_ld32(trow + kPtTmO + 32 * c, o);
#pragma unroll
            for (int i = 0; i < 32; ++i) o[i] *= corr;
            tc_st32(trow + kPtTmO + 32 * c, o);
          }
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        }
        l_run *= corr;
        m_run = m_new;
      }
      const float m_use = m_run == -CUDART_INF_F ? 0.f : m_run;   // nothing visible yet: every p is 0
      // P_jb takes the first 32 columns of the accumulator it was computed from (all of it is in registers): the value
      // MMA of block jb - kPtScores, which read them last, was issued before the score MMAs that were waited for
      float sum4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {   // the store of the first half runs while the second half is computed
        uint32_t pw[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const int i = 32 * hf + 2 * e;
          float x0, x1;
          pt_add2(s[i], s[i + 1], -m_use, -m_use, x0, x1);
          const __half2 p2 = __floats2half2_rn(fast_exp2(x0), fast_exp2(x1));
          pw[e] = as_u32(p2);
          pt_add_halves(sum4[e & 3], pw[e]);   // the denominator of what the MMA will see
        }
        tc_st16u_nowait(trow + kPtTmS + 64 * t + 16 * hf, pw);
      }
      l_run += (sum4[0] + sum4[1]) + (sum4[2] + sum4[3]);
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) {
        pt_arrive_cluster(sb + kPtBarP + 8 * t + to_leader);
      }
    }
  } else if (warp < 15) {
    // ================= decoders: packed block -> K_hat hi / lo, V_hat^T =================
    // Pieces of 1 / kPtGroups of this CTA's half of a block, counted through all blocks, go to the decoder warps in turn (eleven
    // warps share sixteen pieces evenly only across blocks).  A piece is 16 coordinates of 32 lanes: 8 tokens x the 4
    // 16-blocks of one coordinate half (the code words of a warp then sit in few shared-memory rows, and the 8 lanes with one
    // 16-block store to 8 distinct swizzled positions).  Pieces 0-7: the keys of tokens 32 rank .. + 31; pieces 8-15: the
    // values of coordinates 64 rank .. + 63 of all 64 tokens.
    const int dw = warp - 4, bi = lane >> 3, t8 = lane & 7;
    const uint32_t rep = (uint32_t)(lane & 15) * 8u, t1 = (sb + kPtT1) | rep, ub = (sb + kPtU) | rep;
    const uint32_t swz = (uint32_t)(t8 * 128 + (((2 * bi) ^ t8) << 4));   // chunk 2 bi of a row's 64-coordinate half, swizzled by the row
    int fetched = 0, ready = -1;   // blocks requested (decoder warp 0, lane 0); the last block known to have landed and to have a stage
    for (int n = dw; n < kPtGroups * n_blocks; n += kPtDecoderWarps) {
      const int jb = n / kPtGroups, i = n % kPtGroups, st = jb % kPtStages, buf = jb % kPtRawBufs;
      bool ok = true;
      if (dw == 0) {   // keep up to kPtRawBufs packed blocks in flight; wait only for the one needed now
        if (lane == 0)
          while (ok && fetched < n_blocks && fetched < jb + kPtRawBufs) {
            const int f = fetched % kPtRawBufs;
            if (fetched >= kPtRawBufs) {
              const uint32_t ph = (uint32_t)(fetched / kPtRawBufs - 1) & 1u;
              if (fetched <= jb) ok = tc_mbar_wait(sb + kPtBarRawEmpty + 8 * f, ph, abort_flag);
              else if (!tc_mbar_test(sb + kPtBarRawEmpty + 8 * f, ph)) break;
            }
            if (ok) {
              tc_mbar_expect_tx(sb + kPtBarRawFull + 8 * f, kPtRawBytes);
              bulk_load(sb + kPtRaw + f * kPtRawBytes, a.cache + kv_block_pair_offset(L, a.pg, a.n_kv_heads, b, hk, jb0 + fetched, a.status),
                        kPtRawBytes, sb + kPtBarRawFull + 8 * f);
              ++fetched;
            }
          }
        ok = __all_sync(0xffffffffu, ok);
      }
      if (jb != ready) {
        // stage st is free once the value MMA of block jb - kPtStages has completed (it also covers that block's score MMAs)
        if (ok && jb >= kPtStages) ok = tc_mbar_wait(sb + kPtBarPv + 8 * st, (uint32_t)(jb / kPtStages - 1) & 1u, abort_flag);
        if (ok) ok = tc_mbar_wait(sb + kPtBarRawFull + 8 * buf, (uint32_t)(jb / kPtRawBufs) & 1u, abort_flag);
        ready = jb;
      }
      if (!__all_sync(0xffffffffu, ok)) break;
      const bool is_v = i >= 8;
      const int half = is_v ? (int)crank : (i >> 2) & 1, tok = 8 * (is_v ? i & 7 : (i & 3) + 4 * (int)crank) + t8, blk = 4 * half + bi;
      const bool live = (jb0 + jb) * kTokenBlock + tok < len;   // stale bytes past the sequence end must not reach the MMAs
      const uint32_t raw = sb + kPtRaw + buf * kPtRawBytes + (is_v ? kBlockBytes128 : 0);
      const uint32_t l1 = lds32(raw + tok * 32 + blk * 4);
      const uint32_t c2 = lds8(raw + kO2 + tok * 8 + blk);
      const uint32_t c3 = lds8(raw + kO3 + tok * 4 + (blk >> 1)) >> (4 * (blk & 1));
      const uint32_t c4 = (lds16(raw + kO4 + tok * 2) >> (2 * blk)) & 3u;
      const uint32_t rbits = lds16(raw + kORad + tok * 16 + blk * 2);
      const uint32_t rr = live ? rbits | (rbits << 16) : 0u;
      const BlockRef ref = make_block_ref(l1, c2, c3, c4, as_h2(rr), ub);
      if (!is_v) {
        // the key as an unevaluated sum hi + lo, coordinates in the order of the lookups: (4s, 4s+2), (4s+1, 4s+3)
        __half2 h[8], l[8];
        sub_block_hilo<0>(ref, t1, h[0], h[1], l[0], l[1]);
        sub_block_hilo<1>(ref, t1, h[2], h[3], l[2], l[3]);
        sub_block_hilo<2>(ref, t1, h[4], h[5], l[4], l[5]);
        sub_block_hilo<3>(ref, t1, h[6], h[7], l[6], l[7]);
        const uint32_t dst = sb + kPtKv + st * kPtStage + half * kPtKHalf + (i & 3) * 1024 + swz;
        pt_sts128(dst, as_u32(h[0]), as_u32(h[1]), as_u32(h[2]), as_u32(h[3]));
        pt_sts128(dst ^ 16u, as_u32(h[4]), as_u32(h[5]), as_u32(h[6]), as_u32(h[7]));
        pt_sts128(dst + kPtKLo, as_u32(l[0]), as_u32(l[1]), as_u32(l[2]), as_u32(l[3]));
        pt_sts128((dst + kPtKLo) ^ 16u, as_u32(l[4]), as_u32(l[5]), as_u32(l[6]), as_u32(l[7]));
      } else {
        __half2 x[4], y[4];
        sub_block_h2<0>(ref, t1, x[0], y[0]);
        sub_block_h2<1>(ref, t1, x[1], y[1]);
        sub_block_h2<2>(ref, t1, x[2], y[2]);
        sub_block_h2<3>(ref, t1, x[3], y[3]);
        // coordinates in natural order: (4s, 4s+1) = (x.lo, y.lo), (4s+2, 4s+3) = (x.hi, y.hi)
        uint32_t w[8];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          w[2 * s] = __byte_perm(as_u32(x[s]), as_u32(y[s]), 0x5410);
          w[2 * s + 1] = __byte_perm(as_u32(x[s]), as_u32(y[s]), 0x7632);
        }
        const uint32_t dst = sb + kPtKv + st * kPtStage + kPtKTile + (i & 7) * 1024 + swz;
        pt_sts128(dst, w[0], w[1], w[2], w[3]);
        pt_sts128(dst ^ 16u, w[4], w[5], w[6], w[7]);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) {
        pt_arrive_cluster(sb + kPtBarKv + 8 * st + to_leader);
        tc_mbar_arrive(sb + kPtBarRawEmpty + 8 * buf);
      }
    }
    if (dw == 0 && lane == 0)   // no copy may be in flight when the CTA ends (they are, where a wait gave up)
      for (int f = max(0, fetched - kPtRawBufs); f < fetched; ++f)
        for (int i = 0; i < (1 << 20) && !tc_mbar_try(sb + kPtBarRawFull + 8 * (f % kPtRawBufs), (uint32_t)(f / kPtRawBufs) & 1u); ++i)
          __nanosleep(32);
  } else if (leader) {
    // ================= MMA issuer =================
    // The whole warp goes through the loop and one elected lane issues: the operands of the MMAs are then warp-uniform values.
    // From a single thread's registers every MMA took 60 cycles to issue, more than it runs.
    // the value operand is MN-major: [token][coordinate] rows of 64 coordinates, one half per CTA
    constexpr uint32_t idesc_qk = tc_idesc(false, 256, 64);   // 64 tokens
    constexpr uint32_t idesc_pv = tc_idesc(false, 256, 128) | (1u << 16);
    uint64_t vdesc_hi = (uint64_t)(1024 >> 4) << 32;   // stride between groups of 8 tokens
    vdesc_hi |= (uint64_t)1 << 46;
    vdesc_hi |= (uint64_t)2 << 61;
    const uint32_t vdesc_lbo = (8192u >> 4) << 16;     // leading-dimension offset: the next 64 coordinates
    const uint64_t desc_hi = tc_smem_desc(0u) & 0xFFFFFFFF00000000ull;
    const int blocks = __shfl_sync(0xffffffffu, n_blocks, 0);
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem_base, 0);
    auto issue_pv = [&](int jb) {   // O (+)= P_jb V_hat_jb
      const int t = jb % kPtScores, st = jb % kPtStages;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t v_lo = ((kPtKv + st * kPtStage + kPtKTile) >> 4) | vdesc_lbo;
      if (tc_elect()) {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)   // 16 tokens = 8 columns of P = 16 rows of 128 bytes of V_hat per step
          tc_mma_ts_pair(tm + kPtTmO, tm + kPtTmS + 64 * t + 8 * kk, vdesc_hi | (v_lo + 128 * kk), idesc_pv, (jb > 0 || kk > 0) ? 1u : 0u);
        tc_commit_pair(sb + kPtBarPv + 8 * st);   // the stage is free, the output accumulator holds block jb
      }
    };
    auto issue_qk = [&](int jb) {   // S_jb = Q'lo K_hi^T + Q'hi K_lo^T + Q'hi K_hi^T, the small terms first
      const int t = jb % kPtScores, st = jb % kPtStages;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t kb = (uint32_t)tc_smem_desc(kPtKv + st * kPtStage);
      if (tc_elect()) {
#pragma unroll
        for (int term = 0; term < 3; ++term) {
          const uint32_t qa = tm + (term == 0 ? kPtTmQlo : kPtTmQhi);
#pragma unroll
          for (int ks = 0; ks < 8; ++ks) {   // 16 k values = 8 columns of Q' per step; step ks: half ks >> 2, 32 bytes per step
            const uint32_t koff = (uint32_t)((ks >> 2) * kPtKHalf + (ks & 3) * 32 + (term == 1 ? kPtKLo : 0)) >> 4;
            tc_mma_ts_pair(tm + kPtTmS + 64 * t, qa + 8 * ks, desc_hi | (kb + koff), idesc_qk, (term | ks) ? 1u : 0u);
          }
        }
        tc_commit_pair(sb + kPtBarS + 8 * t);
      }
    };
    // Value MMAs go first when their P is ready (they free a stage for the decoders); the score MMAs run up to kPtScores - 1
    // blocks ahead of them and keep the tensor core and the row owners busy.  Accumulator t is free for block jb once the
    // value MMA of block jb - kPtScores, which reads P from its columns, has been issued (MMAs of one thread execute in order).
    bool ok = true;
    int qk = 0, pv = 0, idle = 0;
    while (pv < blocks && ok) {
      if (pv < qk && __all_sync(0xffffffffu, tc_mbar_test(sb + kPtBarP + 8 * (pv % kPtScores), (uint32_t)(pv / kPtScores) & 1u))) {
        issue_pv(pv++);
        idle = 0;
      } else if (qk < blocks && qk < pv + kPtScores &&
                 __all_sync(0xffffffffu, tc_mbar_test(sb + kPtBarKv + 8 * (qk % kPtStages), (uint32_t)(qk / kPtStages) & 1u))) {
        if ((a.debug & 2u) && (blockIdx.x | blockIdx.y | blockIdx.z) == 0 && qk == min(2, blocks - 1)) {
          *abort_flag = 1;   // test hook: this wait counts as failed (what it waited for has arrived)
          ok = false;
        } else {
          issue_qk(qk++);
          idle = 0;
        }
      } else if (++idle > 32) {   // bounded like every wait
        __nanosleep(32);
        if (__any_sync(0xffffffffu, *abort_flag != 0) || idle > kTcSpin) {
          *abort_flag = 1;
          ok = false;
        }
      }
    }
    if (blocks > 0) {
      // every MMA issued above has completed when this commit arrives (nothing was issued without blocks: no commit)
      if (tc_elect()) tc_commit_pair(sb + kPtBarDrain);
      bool drained = false;
      for (int i = 0; i < (1 << 20) && !drained; ++i) {
        drained = tc_mbar_try(sb + kPtBarDrain, 0);
        if (!drained) __nanosleep(32);
      }
      if (!drained) *abort_flag = 1;
    }
    __syncwarp();
    if (lane == 0 && *abort_flag)   // tell the other CTA, whose warps wait for commits that will not come
      asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" ::"r"(kPtMisc + 4 - kPtBase + pt_mapa(sb + kPtBase, 1u)), "r"(1u) : "memory");
  } else if (lane == 0) {
    // the odd CTA of a pair: its operands are read until the even CTA's last commit arrives here too
    if (n_blocks > 0) {
      bool drained = false;
      for (int i = 0; i < kTcSpin && !drained && !*abort_flag; ++i) {
        drained = tc_mbar_try(sb + kPtBarDrain, 0);
        if (!drained) __nanosleep(64);
      }
      if (!drained) *abort_flag = 1;
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();   // all MMAs have completed (the issuer waited for its last commit), the stages are idle
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const bool aborted = *abort_flag != 0;
  // ---- normalise; merge_unrotate_kernel merges the ranges' parts and rotates back
  float* osm = reinterpret_cast<float*>(smem + kPtKv);
  if (warp < 4) {
    const int r = tid;
    const float inv = (!aborted && l_run > 0.f) ? 1.f / l_run : 0.f;
    const uint32_t trow = tmem_base + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
    for (int c = 0; c < 4; ++c) {
      float o[32];
      if (n_blocks > 0 && !aborted) {
        tc_ld32(trow + kPtTmO + 32 * c, o);
      } else {
#pragma unroll
        for (int i = 0; i < 32; ++i) o[i] = 0.f;
      }
#pragma unroll
      for (int i = 0; i < 32; i += 4)
        *reinterpret_cast<float4*>(osm + r * kPtOStride + 32 * c + i) = make_float4(o[i] * inv, o[i + 1] * inv, o[i + 2] * inv, o[i + 3] * inv);
    }
    if (r < n_rows)   // scores are in the log2 domain
      a.part_lse[(int64_t)split * a.batch * a.n_q_heads + row_index(r) / 128] =
          l_run > 0.f ? (m_run + log2f(l_run)) * 0.693147180559945309f : l_run == 0.f ? -CUDART_INF_F : l_run;   // NaN stays NaN
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  // Neither CTA may release tensor memory or leave while the other may still arrive on its barriers or
  // have its operands read: both have drained here.
  pt_cluster_sync();
  if (warp == 15) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
  }
  if (tid == 0 && aborted) set_status(a.status, PQ_ERR_TIMEOUT);
  for (int i = tid; i < n_rows * 32; i += kPtThreads)
    *reinterpret_cast<float4*>(a.part_out + (int64_t)split * a.batch * a.n_q_heads * 128 + row_index(i >> 5) + 4 * (i & 31)) =
        *reinterpret_cast<const float4*>(osm + (i >> 5) * kPtOStride + 4 * (i & 31));
}

}  // namespace pq
