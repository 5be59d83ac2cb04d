// Encoder of few rows (append: one per sequence; drafted tokens; short chunks), any head_dim of the packed cache (included by
// pq_encode.cu).  A call of this kind is all latency, so everything that does not depend on the rows is in registers
// before the kernel ahead in the stream has finished (S and the quantiser's constants; the kernel is its programmatic
// dependent), and where one block -- or a cluster of up to eight -- takes all the vectors of a sequence in a pass, it also
// advances the sequence's length: no second launch.
//
// A pass of a block is kVec vectors.  Rotation: thread = (column, slice of 16 rows of S) with its 16 entries of S in
// registers, all slices in flight at once; the slices' partial sums meet in shared memory.  So the error of a
// coordinate is at most (16 + D / 16) 2^-24 sum_k |x_k||S_kj| <= that factor times ||x||_2.  Then a thread per
// 16-coordinate block runs the certified quantiser; a block with an uncertified decision is rotated again in float64 by
// the whole thread block (two or fewer terms per thread) and decided by one warp.
// Measured (device time behind another kernel, 8 kv heads; a block per vector, float64 below head_dim 128, and a second launch for the
// lengths before): append of one token at head_dim 128 5.3 -> 4.9 us, of 16 10.9 -> 7.9 us; 31 tokens in one sequence 15.0 -> 7.9 us;
// at head_dim 64 one token 16.9 -> 7.5 us, 256 tokens 21.5 -> 15.3 us.  Rows that the tensor-core encoder does not take, at head_dim 128
// (tiles of 128 rows in encode_ffma_kernel before): 64 tokens 107 -> 13.9 us, 1024 114 -> 57; the neighbours among the radii fall from
// 0.009 to 0.003 %.
#pragma once

namespace pq {

static int32_t launch_advance_lens(const EncodeArgs& a, int32_t* lens, cudaStream_t stream);

constexpr int kRowsThreads = 1024;
template <int D, int kMin>
struct RowsShape {
  static constexpr int kBlocks = D / 16, kSlices = D / 16;          // 16-coordinate blocks; slices of 16 rows of S
  static constexpr int kGroups = kRowsThreads / (D * kSlices);      // vectors that are rotated side by side
  static constexpr int kVec = kGroups > kMin ? kGroups : kMin;      // vectors of a pass
  static constexpr int kPer = kVec / kGroups;                       // ... of a thread
  static constexpr int kQuant = kVec * kBlocks;                     // threads that quantise (a multiple of 32)
  static constexpr int kYFloats = kVec * kBlocks * 20;              // rotated blocks, 20 floats apart (conflict-free 16-byte reads)
  static constexpr int kSmem = 4 * (kVec * D + kSlices * kVec * D + kYFloats);
};

// One warp: codes and radius of a block from its 16 float64 coordinates (lane i holds coordinate i & 15), as
// polar_quant_block_exact; every lane returns them.
__device__ __forceinline__ double warp_quant_exact(double y, const Tables& tb, int lane, BlockCodes* c) {
  uint32_t code = 0;
  c->l1 = c->l2 = c->l3 = 0u;
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    const int n = 8 >> l;
    const double p = __shfl_sync(0xffffffffu, y, (2 * lane) & 31), q = __shfl_sync(0xffffffffu, y, (2 * lane + 1) & 31);
    code = l == 0 ? quant_level1_exact(p, q, tb) : quant_upper_exact(p, q, l + 1, tb);
    y = sqrt(p * p + q * q);
    uint32_t word = lane < n ? code << ((l == 0 ? 4 : 2) * lane) : 0u;
#pragma unroll
    for (int m = 1; m < 8; m <<= 1) word |= __shfl_xor_sync(0xffffffffu, word, m);
    word = __shfl_sync(0xffffffffu, word, 0);
    if (l == 0) c->l1 = word;
    else if (l == 1) c->l2 = word;
    else if (l == 2) c->l3 = word;
    else c->l4 = word;
  }
  return __shfl_sync(0xffffffffu, y, 0);
}

// kFlat: the blocks share all rows evenly, whatever sequences they belong to, and another launch advances the lengths.
template <int D, int kMin, bool kFlat>
__global__ void __launch_bounds__(kRowsThreads, 1) encode_rows_kernel(const __grid_constant__ EncodeArgs a, int32_t* lens) {
  using R = RowsShape<D, kMin>;
  static_assert(R::kQuant % 32 == 0, "whole warps quantise");
  extern __shared__ __align__(16) float rows_smem[];
  float* xs = rows_smem;                       // [kVec][D]
  float* part = xs + R::kVec * D;              // [kSlices][kVec][D]
  float* ys = part + R::kSlices * R::kVec * D; // [kVec * kBlocks][20]
  __shared__ FastQuant fq;
  __shared__ double exact_part[64][17];
  __shared__ BlockCodes exact_codes;
  __shared__ double exact_radius;
  __shared__ int n_list;
  __shared__ uint16_t list[R::kQuant];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int col = tid % D, slice = (tid / D) % R::kSlices, vgrp = tid / (D * R::kSlices);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  float s[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) s[i] = __ldg(a.S + (slice * 16 + i) * D + col);
  if (warp == 0) load_fast_quant(a.tables, &fq, lane, &a.tables->l1_cells[0][0]);
  if (tid == 0) n_list = 0;
  asm volatile("griddepcontrol.wait;" ::: "memory");

  const int b = blockIdx.y, rank = blockIdx.x, C = gridDim.x;   // the cluster spans x
  int first = 0, count = 0, rows = a.total_tokens, start = 0;
  bool fits = false;
  if (!kFlat) {
    first = b;
    count = 1;
    if (a.cu_seqlens != nullptr) {
      first = a.cu_seqlens[b];
      count = a.cu_seqlens[b + 1] - first;
    }
    rows = first < 0 ? 0 : min(count, a.total_tokens - first);   // no row outside the inputs, whatever cu_seqlens says
    start = a.cache_lens[b];
    fits = start >= 0 && start + count <= a.capacity;
    if (!fits && count > 0 && tid == 0) set_status(a.status, PQ_ERR_CAPACITY);
  }
  const int per_row = 2 * a.n_kv_heads, n_vec = rows > 0 ? rows * per_row : 0;
  const Layout L = make_layout(D, a.pg.page_tokens);
  int bad_page = 0;
  for (int v0 = rank * R::kVec; v0 < n_vec; v0 += C * R::kVec) {
    int bad = 0;
    for (int i = tid; i < R::kVec * D; i += kRowsThreads) {
      const int v = v0 + i / D, k = i % D;
      float x = 0.f;
      if (v < n_vec) {
        const int r = v / per_row, w = v - r * per_row, kv = w / a.n_kv_heads, head = w - kv * a.n_kv_heads;
        x = load_elem(kv ? a.V : a.K, a.in_dtype, (int64_t)(first + r) * a.token_stride + (int64_t)head * a.head_stride + k);
      }
      bad += !(fabsf(x) < CUDART_INF_F);
      xs[i] = x;
    }
    if (bad) {
      atomicAdd(a.status + 1, bad);
      set_status(a.status, PQ_ERR_NONFINITE);
    }
    // a thread per (vector, block) quantises; the blocks of a vector are neighbouring lanes
    const int v = v0 + tid / R::kBlocks, blk = tid % R::kBlocks;
    int seq = b, pos = start + v / per_row;
    bool goes = fits;
    if (kFlat && tid < R::kQuant && v < n_vec) {
      row_destination(a, v / per_row, &seq, &pos);
      goes = pos >= 0;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < R::kPer; ++j) {
      const int w = vgrp + j * R::kGroups;
      const float4* xv = reinterpret_cast<const float4*>(xs + w * D + slice * 16);
      float acc = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 x4 = xv[i];
        acc = fmaf(x4.x, s[4 * i], acc);
        acc = fmaf(x4.y, s[4 * i + 1], acc);
        acc = fmaf(x4.z, s[4 * i + 2], acc);
        acc = fmaf(x4.w, s[4 * i + 3], acc);
      }
      part[(slice * R::kVec + w) * D + col] = acc;
    }
    __syncthreads();
    for (int i = tid; i < R::kVec * D; i += kRowsThreads) {
      float y = part[i];
#pragma unroll
      for (int q = 1; q < R::kSlices; ++q) y += part[q * R::kVec * D + i];
      ys[(i >> 4) * 20 + (i & 15)] = y;
    }
    __syncthreads();
    FastBlock fb = {0u, 0u, 0u, 0u, 0u, 0.f};
    bool mine = false, unsure = false;
    uint8_t* tb = nullptr;
    int tok = 0;
    if (tid < R::kQuant) {
      float yb[16];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 w = *reinterpret_cast<const float4*>(ys + tid * 20 + 4 * i);
        yb[4 * i] = w.x; yb[4 * i + 1] = w.y; yb[4 * i + 2] = w.z; yb[4 * i + 3] = w.w;
      }
      float sq[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int i = 0; i < 16; ++i) sq[i & 3] = fmaf(yb[i], yb[i], sq[i & 3]);
      float n2 = (sq[0] + sq[1]) + (sq[2] + sq[3]);
#pragma unroll
      for (int m = 1; m < R::kBlocks; m <<= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, m);
      const float norm = 1.0001f * sqrtf(n2);
      const RowMargins rm = make_row_margins(norm, 1.1f * (16 + R::kSlices) * 5.9604644775390625e-08f, fq);
      if (fq.analytic) polar_quant_block_fast<true>(yb, rm, fq, &fb);
      else polar_quant_block_fast<false>(yb, rm, fq, &fb);
      const float block_err = rotation_block_error(16, R::kSlices) * norm;
      bool zero = false;   // EncodeArgs::zero_bad_rows; the eight lanes of a vector look at its inputs together
      if (D == 128 && a.zero_bad_rows && !(n2 < CUDART_INF_F)) {
        const unsigned of_vector = 0xFFu << (lane & 24);
        for (int i = 0; i < 16; ++i) zero = zero || !(fabsf(xs[16 * tid + i]) < CUDART_INF_F);
        zero = __any_sync(of_vector, zero);
        if (zero) fb = {0u, 0u, 0u, 0u, 0u, 0.f};
      }
      if (v < n_vec) {
        const int w = v % per_row, kv = w / a.n_kv_heads, head = w - kv * a.n_kv_heads;
        if (goes) {
          const int64_t off = block_offset(L, a.pg, a.n_kv_heads, seq, head, kv, pos);
          if (off < 0) bad_page = 1;   // a page outside the pool: nothing of the row is written
          else {
            tb = a.cache + off;
            tok = pos % kTokenBlock;
            mine = true;
          }
        }
        // head dims below 128: radii as rounded once from float64; at 128 as the tensor-core encoder forms them
        unsure = fb.amb != 0u || (D < 128 && radius_unsure(fb.radius, block_err));
        if (mine && unsure && !zero) list[atomicAdd(&n_list, 1)] = (uint16_t)tid;
      }
    }
    __syncthreads();
    const int n_exact = n_list;
    for (int e = 0; e < n_exact; ++e) {
      const int item = list[e], ev = v0 + item / R::kBlocks, eb = item % R::kBlocks;
      {   // thread = (coordinate, one of 64 slices of the sum)
        const int c16 = tid & 15, sl = tid >> 4;
        double p = 0.0;
        for (int k = sl; k < D; k += 64) p = fma((double)xs[(ev - v0) * D + k], (double)__ldg(a.S + k * D + 16 * eb + c16), p);
        exact_part[sl][c16] = p;
      }
      __syncthreads();
      if (warp < 16) {   // warp = coordinate
        double p = exact_part[lane][warp] + exact_part[lane + 32][warp];
#pragma unroll
        for (int m = 16; m > 0; m >>= 1) p += __shfl_xor_sync(0xffffffffu, p, m);
        __syncwarp();
        if (lane == 0) exact_part[0][warp] = p;   // column `warp` belongs to this warp alone
      }
      __syncthreads();
      if (warp == 0) {
        BlockCodes c;
        const double r = warp_quant_exact(exact_part[0][lane & 15], *a.tables, lane, &c);
        if (lane == 0) {
          exact_codes = c;
          exact_radius = r;
        }
      }
      __syncthreads();
      if (tid == item) {
        if (fb.amb) atomicAdd(a.status + 3, __popc(fb.amb));
        fb.l1 = exact_codes.l1; fb.l2 = exact_codes.l2; fb.l3 = exact_codes.l3; fb.l4 = exact_codes.l4;
        if (exact_radius > 65504.0) fb.radius = CUDART_INF_F;
        else fb.radius = __half2float(__double2half(exact_radius));   // the one rounding of the radius
      }
    }
    if (tid < R::kQuant) {
      float rv = fb.radius;
      if (mine && rv > 65504.f) {
        rv = 65504.f;
        atomicAdd(a.status + 2, 1);
      }
      const BlockCodes c = {fb.l1, fb.l2, fb.l3, fb.l4};
      store_block(tb, L, tok, blk, c, __float2half_rn(rv), mine);
    }
    __syncthreads();
    if (tid == 0) n_list = 0;
  }
  if (kFlat) return;   // row_destination has looked at the pages
  // ---- the sequence's length (every block of the cluster has read it and written its vectors)
  bad_page = __syncthreads_or(bad_page);
  if (bad_page && tid == 0) set_status(a.status, PQ_ERR_INVALID_ARG);
  if (C > 1) {
    cluster_arrive();
    cluster_wait();
  }
  if (rank == 0 && tid == 0 && fits && count > 0) {
    bool ok = true;
    if (a.pg.table != nullptr)
      for (int p = start / a.pg.page_tokens; p <= (start + count - 1) / a.pg.page_tokens; ++p)
        ok = ok && (unsigned)a.pg.table[(int64_t)b * a.pg.pages_per_seq + p] < (unsigned)a.pg.n_pages;
    if (ok) lens[b] = start + count;
  }
}

template <int D, int kMin, bool kFlat>
static int32_t launch_encode_rows_as(const EncodeArgs& a, int32_t* lens, dim3 grid, cudaStream_t stream) {
  using R = RowsShape<D, kMin>;
  static DeviceMemo configured;
  if (configure_for_device(encode_rows_kernel<D, kMin, kFlat>, R::kSmem, configured) == 0) return PQ_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kRowsThreads);
  cfg.dynamicSmemBytes = R::kSmem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // set up while the kernel before it finishes (it waits inside)
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = grid.x;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = !kFlat && grid.x > 1 ? 2 : 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, encode_rows_kernel<D, kMin, kFlat>, a, lens);
  if (e != cudaSuccess) {
    note_cuda_error(e);
    cudaGetLastError();
    return PQ_ERR_CUDA;
  }
  return kFlat ? launch_advance_lens(a, lens, stream) : PQ_OK;
}

// A block or cluster per sequence where that is a single pass whatever the rows are: an append, or all rows in one sequence,
// of at most eight blocks' vectors (the portable cluster size).  Otherwise -- the host does not know how the rows of an encode
// are spread over its sequences -- the rows evenly over all blocks, and a second launch for the lengths.
template <int D, int kMin>
static int32_t launch_encode_rows_of(const EncodeArgs& a, int32_t* lens, cudaStream_t stream) {
  constexpr int kVec = RowsShape<D, kMin>::kVec;
  const int64_t all = (int64_t)a.total_tokens * 2 * a.n_kv_heads, per_seq = a.cu_seqlens == nullptr ? 2 * (int64_t)a.n_kv_heads : all;
  if ((a.cu_seqlens == nullptr || a.batch == 1) && per_seq <= 8 * kVec && (a.cu_seqlens != nullptr || a.batch <= 65535)) {
    int C = 1;
    while (C * kVec < per_seq) C *= 2;
    return launch_encode_rows_as<D, kMin, false>(a, lens, dim3(C, a.batch), stream);
  }
  return launch_encode_rows_as<D, kMin, true>(a, lens, dim3((unsigned)((all + kVec - 1) / kVec)), stream);
}

// A pass takes as long as its vectors: fewer of them where the blocks still have an SM each (one sequence, 8 kv heads, head_dim 128:
// 7.1 us with 16 vectors in one block, 4.9 with a cluster of four).
template <int D, int kFew>
static int32_t launch_encode_rows_by_size(const EncodeArgs& a, int32_t* lens, int n_sm, cudaStream_t stream) {
  const int64_t all = (int64_t)a.total_tokens * 2 * a.n_kv_heads;
  return all <= (int64_t)kFew * n_sm ? launch_encode_rows_of<D, kFew>(a, lens, stream) : launch_encode_rows_of<D, 16>(a, lens, stream);
}

static bool encode_rows_in_passes(const EncodeArgs& a, int n_sm, int passes) {   // of 16 vectors (RowsShape's kVec at head_dim 16) per SM
  const int per_pass = a.head_dim == 16 ? RowsShape<16, 16>::kVec : 16;
  return (int64_t)a.total_tokens * 2 * a.n_kv_heads <= passes * (int64_t)n_sm * per_pass;
}
// Calls that this kernel takes before any other: fewer than 32 tokens; below head_dim 128 as long as two passes of every SM hold them,
// at head_dim 128 as long as four vectors per SM do.  There the tensor-core encoder takes 16.4 us for its first tile (bf16, 2 kv heads,
// 128 tokens: 8.8 us here); with sixteen per SM it would be 17.2 -> 13.9, but 18.6 -> 24.8 without a preconditioner, when one pair in a
// thousand lies on a boundary.
static bool encode_rows_takes(const EncodeArgs& a, int n_sm) {
  return a.total_tokens < 32 || (a.head_dim == 128 ? (int64_t)a.total_tokens * 2 * a.n_kv_heads <= 4 * (int64_t)n_sm
                                                   : encode_rows_in_passes(a, n_sm, 2));
}
static int32_t launch_encode_rows(const EncodeArgs& a, int32_t* lens, int n_sm, cudaStream_t stream) {
  switch (a.head_dim) {
    case 16: return launch_encode_rows_of<16, 16>(a, lens, stream);
    case 32: return launch_encode_rows_of<32, 16>(a, lens, stream);
    case 64: return launch_encode_rows_by_size<64, 8>(a, lens, n_sm, stream);
    default: return launch_encode_rows_by_size<128, 4>(a, lens, n_sm, stream);
  }
}

}  // namespace pq
