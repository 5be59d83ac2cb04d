// Attention of one query per sequence over the uncompressed window, bf16 rows of head_dim 128, up to four query heads per kv head
// (included by pq_decode.cu after tail_attention, which takes everything else).
//
// Every warp of a block is a stream of its own over tiles of 16 tokens: it copies its tiles (16-byte cp.async, K and V pieces of 4 KB through
// a ring of three), multiplies on tensor cores and keeps its own maximum, denominator and output; the four warps meet once, at the
// end.  The operands are exact: keys and values are bf16 as they are, a float32 query coordinate and a float32 probability are
// three bf16 terms each (24 bits), products of bf16 are exact in float32 and summed there.
//   scores (tokens x columns) = K (16 x 128) times the query terms: column 2h = first, 2h + 1 = second term of head h, and in a second
//     MMA column 2h = third term, so all terms of a (token, head) land in one thread;
//   output (rows x coordinates) = P (16 x 16 tokens) times V: row 4 t + h = term t of head h's probabilities.
// A 0 of a term times an infinite key or value is a NaN that the product itself would not be, so a block whose result holds a NaN is
// computed again by tail_attention.
// Bound by the memory latency of a window's few steps.  As float32 multiply-adds over rows in shared memory, the query and the
// probabilities read as broadcasts, the kernel took 15.3 us (batch 8, 1024 tokens, 32/8 heads, 8 splits, 33 MB), now about 10.5: with the
// attention over up to 16384 compressed tokens and the merge 91.9 -> 87.2 us.
#pragma once

namespace pq {

constexpr int kTmTile = 16, kTmPiece = kTmTile * 256, kTmRing = 3, kTmWarps = kTailThreads / 32;
constexpr int kTmSmQ = 0;                                     // query fragments [k-step][lane], 16 bytes
constexpr int kTmSmMl = kTmSmQ + 8 * 32 * 16;                 // (m, l) [warp][head]
constexpr int kTmSmRing = kTmSmMl + kTmWarps * 4 * 8;         // the pieces; the warps' outputs at the end
constexpr int kTmSmTotal = kTmSmRing + kTmWarps * kTmRing * kTmPiece;
static_assert(kTmSmRing % 128 == 0 && kTmWarps * 4 * 128 * 4 <= kTmWarps * kTmRing * kTmPiece, "map");

// Term t of the pair (a, b) as bf16, a in the low half.
__device__ __forceinline__ uint32_t tm_term(float a, float b, int t) {
  uint32_t w[3];
  bf16_terms(a, b, w);
  return t == 0 ? w[0] : t == 1 ? w[1] : w[2];
}

__device__ __noinline__ void tail_attention_again(const TailArgs& a, float* sm) { tail_attention<1>(a, sm); }

__global__ void __launch_bounds__(kTailThreads, 4) tail_mma_kernel(const __grid_constant__ TailArgs a) {
  extern __shared__ __align__(128) uint8_t tm_smem[];
  const int g_heads = a.n_q_heads / a.n_kv_heads, hk = blockIdx.x, b = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, c = lane & 3;
  const uint32_t sm = (uint32_t)__cvta_generic_to_shared(tm_smem);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  int len_all = a.lens[b];
  len_all = len_all < 0 ? 0 : (len_all > a.capacity ? a.capacity : len_all);
  const int per = (len_all + (int)gridDim.z - 1) / (int)gridDim.z;
  const int t_begin = min(len_all, (int)blockIdx.z * per), len = min(len_all, t_begin + per) - t_begin;
  const int64_t row_stride = (int64_t)a.n_kv_heads * 256, base = (((int64_t)b * a.capacity + t_begin) * a.n_kv_heads + hk) * 256;
  const int n_tiles = (len + kTmTile - 1) / kTmTile, mine = n_tiles > warp ? (n_tiles - warp + kTmWarps - 1) / kTmWarps : 0;
  const uint32_t ring = sm + kTmSmRing + warp * (kTmRing * kTmPiece);
  // Piece 2k is the keys of the warp's tile k, 2k + 1 its values: 16 rows of 256 bytes, 16-byte chunk x of a row at x ^ (row & 7);
  // rows past the end are zeros.
  auto request = [&](int piece) {
    if (piece < 2 * mine) {
      const int t0 = (warp + (piece >> 1) * kTmWarps) * kTmTile;
      const uint8_t* src = reinterpret_cast<const uint8_t*>(piece & 1 ? a.v : a.k) + base;
      const uint32_t dst = ring + (piece % kTmRing) * kTmPiece;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int row = 2 * i + (lane >> 4), chunk = lane & 15, t = t0 + row;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + row * 256 + ((chunk ^ (row & 7)) << 4)),
                     "l"(src + min(t, len - 1) * row_stride + 16 * chunk), "r"(t < len ? 16 : 0)
                     : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int i = 0; i < kTmRing; ++i) request(i);
  // the queries' terms in fragment order: lane (n, c) of a k-step holds rows 2c, 2c + 1 and 2c + 8, 2c + 9 of column n of both MMAs
  for (int i = tid; i < 8 * 32; i += kTailThreads) {
    const int ks = i >> 5, n = (i >> 2) & 7, h = n >> 1, k = 16 * ks + 2 * (i & 3);
    float f[4] = {0.f, 0.f, 0.f, 0.f};
    if (h < g_heads) {
      const int64_t q0 = ((int64_t)b * a.n_q_heads + hk * g_heads + h) * 128 + k;
#pragma unroll
      for (int e = 0; e < 4; ++e) f[e] = tail_elem(a.q, a.io_dtype, q0 + (e & 1) + 8 * (e >> 1)) * a.scale * 1.4426950408889634f;
    }
    const int part = n & 1;
    *reinterpret_cast<uint4*>(tm_smem + kTmSmQ + i * 16) =
        make_uint4(tm_term(f[0], f[1], part), tm_term(f[2], f[3], part), part ? 0u : tm_term(f[0], f[1], 2), part ? 0u : tm_term(f[2], f[3], 2));
  }
  __syncthreads();

  float o[16][4], m_run = -CUDART_INF_F, l_run = 0.f;   // o: rows g and g + 8; m, l: of head c, l this thread's share
#pragma unroll
  for (int j = 0; j < 16; ++j) o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.f;
  const int frag_row = (lane & 7) + (lane & 8);
  const uint32_t frag = ring + frag_row * 256;
#pragma unroll 1
  for (int i = 0; i < mine; ++i) {
    const int t0 = (warp + i * kTmWarps) * kTmTile;
    asm volatile("cp.async.wait_group %0;" ::"n"(kTmRing - 1) : "memory");
    __syncwarp();
    float s0[4] = {0.f, 0.f, 0.f, 0.f}, s1[4] = {0.f, 0.f, 0.f, 0.f};
    {
      const uint32_t at = frag + (2 * i % kTmRing) * kTmPiece;
#pragma unroll
      for (int ks = 0; ks < 8; ++ks) {
        uint32_t k4[4];
        ldmatrix_x4<false>(at + (((2 * ks + (lane >> 4)) ^ (frag_row & 7)) << 4), k4);
        const uint4 q = *reinterpret_cast<const uint4*>(tm_smem + kTmSmQ + (ks * 32 + lane) * 16);
        mma_bf16_16816(s1, k4, q.z, q.w);
        mma_bf16_16816(s0, k4, q.x, q.y);
      }
    }
    __syncwarp();
    request(2 * i + kTmRing);   // takes the keys' place
    float p0 = (s1[0] + s0[1]) + s0[0], p1 = (s1[2] + s0[3]) + s0[2];   // head c of tokens g and g + 8, small terms first
    if (t0 + g >= len) p0 = -CUDART_INF_F;
    if (t0 + g + 8 >= len) p1 = -CUDART_INF_F;
    if (__any_sync(0xffffffffu, fmaxf(p0, p1) > m_run + kLazyMax)) {   // the reference moves only when a score is well above it
      float mx = fmaxf(p0, p1);
#pragma unroll
      for (int w = 4; w < 32; w <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, w));
      const float m_new = fmaxf(m_run, mx), corr = exp2f(m_run - m_new);   // 0 on the first tile; m_new is finite
      m_run = m_new;
      l_run *= corr;
      const float k = __shfl_sync(0xffffffffu, corr, g & 3);   // of the head of rows g and g + 8
#pragma unroll
      for (int j = 0; j < 16; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[j][e] *= k;
    }
    p0 = exp2f(p0 - m_run);
    p1 = exp2f(p1 - m_run);
    l_run += p0 + p1;
    // A operand: rows g (term g / 4 of head g & 3) and g + 8 (third term; rows 12 .. 15 are zeros), tokens 2c, 2c + 1 and 2c + 8, 2c + 9
    const int from = 8 * c + (g & 3);
    const float x0 = __shfl_sync(0xffffffffu, p0, from), x1 = __shfl_sync(0xffffffffu, p0, from + 4);
    const float x2 = __shfl_sync(0xffffffffu, p1, from), x3 = __shfl_sync(0xffffffffu, p1, from + 4);
    const uint32_t pa[4] = {tm_term(x0, x1, g >> 2), g < 4 ? tm_term(x0, x1, 2) : 0u, tm_term(x2, x3, g >> 2), g < 4 ? tm_term(x2, x3, 2) : 0u};
    asm volatile("cp.async.wait_group %0;" ::"n"(kTmRing - 1) : "memory");
    __syncwarp();
    {
      const uint32_t at = frag + ((2 * i + 1) % kTmRing) * kTmPiece;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        uint32_t v4[4];
        ldmatrix_x4<true>(at + (((2 * j + (lane >> 4)) ^ (frag_row & 7)) << 4), v4);
        mma_bf16_16816(o[2 * j], pa, v4[0], v4[1]);
        mma_bf16_16816(o[2 * j + 1], pa, v4[2], v4[3]);
      }
    }
    __syncwarp();
    request(2 * i + 1 + kTmRing);   // takes the values' place
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
  for (int w = 4; w < 32; w <<= 1) l_run += __shfl_xor_sync(0xffffffffu, l_run, w);
  __syncthreads();   // the ring is free
  float* out_w = reinterpret_cast<float*>(tm_smem + kTmSmRing) + warp * 4 * 128;   // [head][128]
  float2* ml = reinterpret_cast<float2*>(tm_smem + kTmSmMl);                       // [warp][head]
  if (lane < 4) ml[warp * 4 + lane] = make_float2(m_run, l_run);
#pragma unroll
  for (int j = 0; j < 16; ++j)
#pragma unroll
    for (int e = 0; e < 2; ++e) {   // the three terms: rows g, g + 4 and g + 8
      const float v = (o[j][2 + e] + __shfl_xor_sync(0xffffffffu, o[j][e], 16)) + o[j][e];
      if (g < 4) out_w[g * 128 + 8 * j + 2 * c + e] = v;
    }
  __syncthreads();
  float res[4];
  bool nan = false;
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    float M = -CUDART_INF_F, L = 0.f, acc = 0.f;
#pragma unroll
    for (int w = 0; w < kTmWarps; ++w) M = fmaxf(M, ml[w * 4 + h].x);
#pragma unroll
    for (int w = 0; w < kTmWarps; ++w) {
      const float2 v = ml[w * 4 + h];
      const float k = v.x == -CUDART_INF_F ? 0.f : exp2f(v.x - M);
      L = fmaf(v.y, k, L);
      acc = fmaf(reinterpret_cast<const float*>(tm_smem + kTmSmRing)[(w * 4 + h) * 128 + tid], k, acc);
    }
    res[h] = len > 0 ? acc / L : 0.f;
    nan = nan || (h < g_heads && res[h] != res[h]);
    if (tid == h) {   // log-sum-exp of the part
      const int64_t li = ((int64_t)blockIdx.z * a.batch + b) * a.n_q_heads + hk * g_heads + h;
      if (h < g_heads && a.lse != nullptr) a.lse[li] = len > 0 ? (M + log2f(L)) * 0.693147180559945309f : -CUDART_INF_F;
      else if (h < g_heads && len <= 0) set_status(a.status, PQ_ERR_EMPTY);
    }
  }
  if (__syncthreads_or(nan)) {
    tail_attention_again(a, reinterpret_cast<float*>(tm_smem));
    return;
  }
#pragma unroll
  for (int h = 0; h < 4; ++h)
    if (h < g_heads) {
      const int64_t oi = (((int64_t)blockIdx.z * a.batch + b) * a.n_q_heads + hk * g_heads + h) * 128 + tid;
      if (a.io_dtype == PQ_DTYPE_BF16) reinterpret_cast<__nv_bfloat16*>(a.out)[oi] = __float2bfloat16(res[h]);
      else reinterpret_cast<float*>(a.out)[oi] = res[h];
    }
}

}  // namespace pq
