// Decode attention in float32 over any packed layout (included by pq_decode.cu and pq_general.cu): one cluster of
// thread blocks per (kv head, sequence), the tokens cut into one contiguous range per block of the cluster.
//
// A block keeps a chunk of packed keys and values in shared memory (16-byte cp.async, the next chunk's copies in flight
// while the current one is used) and works on "groups" of 16 coordinates:
//   * scores: thread = (token, group or several groups); the 16 coordinates are decoded into registers and multiplied
//     into the group's query heads there (packed float32 multiply-adds), partial scores meet in shuffles;
//   * softmax: a warp per head, once per chunk (log2 domain);
//   * values: warp = group, lane = token; every thread accumulates heads x 16 coordinates of its own tokens in registers,
//     and the 32 lanes are summed once per chunk by halving exchanges.
// No decoded coordinate is ever stored: per token and kv head the work is the angle lookups (one 8-byte (cos, sin) entry
// each), two multiplications per angle and 2 x heads x d multiply-adds.
// The blocks of a cluster share the rotation of the query (each forms d / C coordinates of q' = q S and sends them to
// the others), merge their partial softmaxes through distributed shared memory, and each un-rotates d / C coordinates
// of the output.  So a call is one launch and needs no scratch in global memory.
// Bound by instruction issue (angle decode); the figures are beside the launch code of the two layouts.
#pragma once

namespace pq {

constexpr int kSplitThreads = 256;
constexpr int kSplitWarps = kSplitThreads / 32;
constexpr int kGroupStride = 20;  // floats between the 16-coordinate groups of q': eight groups start in eight bank quads

// What the kernel needs beside the layout.
struct SplitCommon {
  int d, n_q_heads, n_kv_heads, io_dtype;
  int chunk;   // tokens staged at a time (a multiple of 64)
  float scale;
  const float* S;
  const void* q;
  void* out;
  float* lse;  // may be null; with it an empty sequence is not an error
  int32_t* status;
};

constexpr int kSplitSmemMax = 200 * 1024;

__host__ __device__ inline int split_groups(int d) { return d < 16 ? 1 : d / 16; }
// Shared memory of a block in bytes: tables, q', scores, partial sums, three [heads][d] vectors, running (m, l, corr),
// the two staging buffers.
__host__ __device__ inline int split_smem_bytes(int d, int kh, int n_tab, int chunk, int stage_bytes) {
  const int ng = split_groups(d);
  const int floats = 2 * n_tab + kh * ng * kGroupStride + chunk * kh + kSplitThreads * kh + 3 * kh * 16 * ng + 4 * kh;
  return ((floats * 4 + 15) & ~15) + 2 * stage_bytes;
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
__device__ __forceinline__ void cluster_st(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void split_cp16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void split_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void split_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(kPending) : "memory");
}
__device__ __forceinline__ uint32_t split_lds32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ float2 split_lds_f2(uint32_t addr) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr));
  return v;
}
__device__ __forceinline__ uint32_t split_lds16(uint32_t addr) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ uint32_t split_lds8(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}

// Sum of v[0 .. kN) over the 32 lanes by halving exchanges: lane L ends with the kN / 32 sums from L * kN / 32 on in
// v[0 ..] (kN = 16: lanes 2 i and 2 i + 1 both with sum i).  The order of the additions is fixed.
template <int kN>
__device__ __forceinline__ void lane_sums(float* v, int lane) {
  int half = kN / 2;
#pragma unroll
  for (int mask = 16; mask >= 1; mask >>= 1) {
    if (half >= 1) {
      const bool up = lane & mask;
#pragma unroll
      for (int i = 0; i < kN / 2; ++i)
        if (i < half) v[i] = (up ? v[i + half] : v[i]) + __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + half], mask);
      half >>= 1;
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], mask);
    }
  }
}

// Layout policies (template parameter P, passed by value) provide
//   SplitCommon c;
//   int stage_bytes                   size of a staging buffer (keys or values of a chunk)
//   int len(pair)                     tokens the pair's query sees
//   int n_tab                         entries of the (cos, sin) table (even)
//   void fill_tables(tab, tid)        kEarlyTables: before the kernel ahead in the stream has finished (it may not write them)
//   void stage(buf, pair, hk, kv, t0, n, tid)   issue the copies of the keys (kv = 0) or values (1) of tokens t0 .. t0 + n - 1
//   int shift(pair, hk, kv, t0)       where in the buffer the chunk that starts at token t0 begins
//   int lanes_per_token(ng)           least number of lanes that should share a token in the score phase
//   void decode(buf, t, g, tab, y)    16 rotated coordinates of group g of the chunk's token t
template <class P, int kH>
__global__ void __launch_bounds__(kSplitThreads, kH == 8 ? 1 : 2) split_attention_kernel(const __grid_constant__ P p) {
  extern __shared__ __align__(16) uint8_t split_smem[];
  const SplitCommon& c = p.c;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int C = gridDim.x, rank = blockIdx.x, hk = blockIdx.y, pair = blockIdx.z;   // the cluster spans the x dimension
  const int d = c.d, ng = split_groups(d), dp = 16 * ng, grp = c.n_q_heads / c.n_kv_heads;
  float2* tab = reinterpret_cast<float2*>(split_smem);
  float* qg = reinterpret_cast<float*>(tab + p.n_tab);   // [kH][ng * kGroupStride]
  float* sc = qg + kH * ng * kGroupStride;                 // [chunk][kH]
  float* part = sc + c.chunk * kH;                         // [kSplitThreads * kH]
  float* o_sm = part + kSplitThreads * kH;                 // [kH][dp]
  float* y_sm = o_sm + kH * dp;                            // [kH][dp]
  float* q_in = y_sm + kH * dp;                            // [kH][dp]
  float* m_sm = q_in + kH * dp;                            // [kH] running maximum, [kH] denominator, [kH] rescale
  float* l_sm = m_sm + kH;
  float* corr_sm = l_sm + kH;
  const uint32_t tab_s = (uint32_t)__cvta_generic_to_shared(split_smem);
  const int head_floats = (int)(corr_sm + 2 * kH - reinterpret_cast<float*>(split_smem));
  const uint32_t kbuf = tab_s + ((head_floats * 4 + 15) & ~15), vbuf = kbuf + p.stage_bytes;

  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (P::kEarlyTables) p.fill_tables(tab, tid);
  asm volatile("griddepcontrol.wait;" ::: "memory");   // lengths, cache and queries may come from the kernel before this one
  const int len = p.len(pair);
  const int per = ((len + C - 1) / C + 63) & ~63;
  const int t_first = min(len, rank * per), n_mine = min(len, t_first + per) - t_first;
  if (n_mine > 0) p.stage(kbuf, pair, hk, 0, t_first, min(n_mine, c.chunk), tid);
  split_commit();
  if (n_mine > 0) p.stage(vbuf, pair, hk, 1, t_first, min(n_mine, c.chunk), tid);
  split_commit();
  if (!P::kEarlyTables) p.fill_tables(tab, tid);

  // ---- q' = q S * scale * log2(e): this block's d / C columns, sent to every block of the cluster
  const int64_t q0 = ((int64_t)pair * c.n_q_heads + hk * grp) * d;
  for (int i = tid; i < kH * dp; i += kSplitThreads) {
    const int h = i / dp, k = i - h * dp;
    float v = 0.f;
    if (h < grp && k < d)
      v = c.io_dtype == PQ_DTYPE_BF16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(c.q)[q0 + h * d + k])
                                      : reinterpret_cast<const float*>(c.q)[q0 + h * d + k];
    q_in[i] = v;
    o_sm[i] = 0.f;
  }
  for (int i = tid; i < kH * ng * kGroupStride; i += kSplitThreads)   // coordinates past d (head dims below 16) stay zero
    if (d < 16) qg[i] = 0.f;
  if (tid < kH) {
    m_sm[tid] = -CUDART_INF_F;
    l_sm[tid] = 0.f;
  }
  cluster_arrive();   // (A) every block of the cluster runs and has cleared its q'; waited for before the first remote store
  __syncthreads();
  const int nc = d / C, j0 = rank * nc, kparts = kSplitThreads / nc;   // C divides d
  {
    const int cc = tid % nc, kp = tid / nc;
    float acc[kH];
#pragma unroll
    for (int h = 0; h < kH; ++h) acc[h] = 0.f;
    for (int k = kp; k < d; k += kparts) {
      const float s = __ldg(c.S + (int64_t)k * d + j0 + cc);
#pragma unroll
      for (int h = 0; h < kH; ++h) acc[h] = fmaf(q_in[h * dp + k], s, acc[h]);
    }
#pragma unroll
    for (int h = 0; h < kH; ++h) part[(kp * nc + cc) * kH + h] = acc[h];
  }
  cluster_wait();   // (A)
  __syncthreads();
  for (int i = tid; i < nc * kH; i += kSplitThreads) {
    const int cc = i / kH, h = i - cc * kH, j = j0 + cc;
    float v = 0.f;
    const int n_kp = min(kparts, d);
    for (int kp = 0; kp < n_kp; ++kp) v += part[(kp * nc + cc) * kH + h];
    v *= c.scale * 1.4426950408889634f;
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(qg + h * ng * kGroupStride + (j >> 4) * kGroupStride + (j & 15));
    for (int r = 0; r < C; ++r) cluster_st(cluster_map(dst, r), v);
  }
  cluster_arrive();   // (B) q' is complete everywhere
  cluster_wait();

  // ---- chunks of this block's tokens
  const int n_slice = ng < kSplitWarps ? kSplitWarps / ng : 1;
  const uint32_t qg_s = (uint32_t)__cvta_generic_to_shared(qg);
  for (int c0 = 0; c0 < n_mine; c0 += c.chunk) {
    const int n = min(c.chunk, n_mine - c0), t0 = t_first + c0, n_next = min(c.chunk, n_mine - c0 - c.chunk);
    split_wait<1>();   // the keys have landed (the values are the younger group)
    __syncthreads();
    {
      // scores: gs consecutive lanes share a token; more of them when there are few tokens
      const uint32_t kb = kbuf + p.shift(pair, hk, 0, t0);
      int gs = p.lanes_per_token(ng);
      while (gs < ng && n * gs < 2 * kSplitThreads) gs <<= 1;
      const int gs_log = 31 - __clz(gs);
      for (int i0 = 0; i0 < (n << gs_log); i0 += kSplitThreads) {
        const int t = (i0 + tid) >> gs_log, g0 = (i0 + tid) & (gs - 1);
        uint64_t s2[kH];
#pragma unroll
        for (int h = 0; h < kH; ++h) s2[h] = 0ull;
        if (t < n)
          for (int g = g0; g < ng; g += gs) {
            float y[16];
            p.decode(kb, t, g, tab_s, y);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const uint64_t ya = f2_pack(y[4 * i], y[4 * i + 1]), yb = f2_pack(y[4 * i + 2], y[4 * i + 3]);
#pragma unroll
              for (int h = 0; h < kH; ++h) {
                uint64_t qa, qb;
                asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];"
                             : "=l"(qa), "=l"(qb)
                             : "r"(qg_s + ((h * ng + g) * kGroupStride + 4 * i) * 4));
                s2[h] = f2_fma(ya, qa, s2[h]);
                s2[h] = f2_fma(yb, qb, s2[h]);
              }
            }
          }
#pragma unroll
        for (int h = 0; h < kH; ++h) {
          float a, b;
          f2_unpack(s2[h], a, b);
          float s = a + b;
          for (int m = 1; m < gs; m <<= 1) s += __shfl_xor_sync(0xffffffffu, s, m);
          if (t < n && g0 == 0) sc[t * kH + h] = s;
        }
      }
    }
    __syncthreads();
    // the keys have been used: the next chunk's keys may arrive
    if (n_next > 0) p.stage(kbuf, pair, hk, 0, t0 + c.chunk, n_next, tid);
    split_commit();
    if (warp < kH) {
      const int h = warp;
      float mx = -CUDART_INF_F;
      for (int t = lane; t < n; t += 32) mx = fmaxf(mx, sc[t * kH + h]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      const float m_old = m_sm[h], m_new = fmaxf(m_old, mx);
      float sum = 0.f;
      for (int t = lane; t < n; t += 32) {
        const float e = exp2f(sc[t * kH + h] - m_new);
        sc[t * kH + h] = e;
        sum += e;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      __syncwarp();
      if (lane == 0) {
        const float corr = exp2f(m_old - m_new);   // 0 on the first chunk
        corr_sm[h] = corr;
        l_sm[h] = l_sm[h] * corr + sum;
        m_sm[h] = m_new;
      }
    }
    split_wait<1>();   // the values have landed
    __syncthreads();
    const uint32_t vb = vbuf + p.shift(pair, hk, 1, t0);
    for (int g = ng < kSplitWarps ? warp % ng : warp; g < ng; g += kSplitWarps) {
      const int slice = ng < kSplitWarps ? warp / ng : 0;
      uint64_t acc[kH][8];
#pragma unroll
      for (int h = 0; h < kH; ++h)
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[h][i] = 0ull;
      for (int t = lane + 32 * slice; t < n; t += 32 * n_slice) {
        float y[16];
        p.decode(vb, t, g, tab_s, y);
        float pr[kH];
        if (kH >= 4) {
#pragma unroll
          for (int h = 0; h < kH / 4; ++h) {
            const float4 p4 = *reinterpret_cast<const float4*>(sc + t * kH + 4 * h);
            pr[4 * h] = p4.x; pr[(4 * h + 1) % kH] = p4.y; pr[(4 * h + 2) % kH] = p4.z; pr[(4 * h + 3) % kH] = p4.w;
          }
        } else {
#pragma unroll
          for (int h = 0; h < kH; ++h) pr[h] = sc[t * kH + h];
        }
#pragma unroll
        for (int h = 0; h < kH; ++h) {
          const uint64_t pp = f2_pack(pr[h], pr[h]);
#pragma unroll
          for (int i = 0; i < 8; ++i) acc[h][i] = f2_fma(pp, f2_pack(y[2 * i], y[2 * i + 1]), acc[h][i]);
        }
      }
      float v[16 * kH];
#pragma unroll
      for (int h = 0; h < kH; ++h)
#pragma unroll
        for (int i = 0; i < 8; ++i) f2_unpack(acc[h][i], v[16 * h + 2 * i], v[16 * h + 2 * i + 1]);
      lane_sums<16 * kH>(v, lane);
      float* dst = part + (g * n_slice + slice) * 16 * kH;
      if (kH == 1) {
        if ((lane & 1) == 0) dst[lane >> 1] = v[0];
      } else {
#pragma unroll
        for (int i = 0; i < kH / 2; ++i) dst[lane * (kH / 2) + i] = v[i];
      }
    }
    __syncthreads();
    if (n_next > 0) p.stage(vbuf, pair, hk, 1, t0 + c.chunk, n_next, tid);
    split_commit();
    for (int i = tid; i < kH * dp; i += kSplitThreads) {
      const int h = i / dp, j = i - h * dp;
      float v = 0.f;
      for (int s = 0; s < n_slice; ++s) v += part[((j >> 4) * n_slice + s) * 16 * kH + h * 16 + (j & 15)];
      o_sm[i] = fmaf(o_sm[i], corr_sm[h], v);
    }
  }
  // ---- merge over the cluster: this block's d / C coordinates of every head, in rank order
  __syncthreads();
  cluster_arrive();   // (C) partial results are complete everywhere
  cluster_wait();
  for (int i = tid; i < nc * kH; i += kSplitThreads) {
    const int h = i / nc, j = j0 + (i - h * nc);
    const uint32_t m_a = (uint32_t)__cvta_generic_to_shared(m_sm + h), l_a = (uint32_t)__cvta_generic_to_shared(l_sm + h);
    const uint32_t o_a = (uint32_t)__cvta_generic_to_shared(o_sm + h * dp + j);
    float M = -CUDART_INF_F;
#pragma unroll 4
    for (int r = 0; r < C; ++r) M = fmaxf(M, cluster_ld(cluster_map(m_a, r)));
    float L = 0.f, y = 0.f;
#pragma unroll 4
    for (int r = 0; r < C; ++r) {
      const float m = cluster_ld(cluster_map(m_a, r));
      const float w = m == -CUDART_INF_F ? 0.f : exp2f(m - M);
      L = fmaf(cluster_ld(cluster_map(l_a, r)), w, L);
      y = fmaf(cluster_ld(cluster_map(o_a, r)), w, y);
    }
    y = len > 0 ? y / L : 0.f;
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(y_sm + h * dp + j);
    for (int r = 0; r < C; ++r) cluster_st(cluster_map(dst, r), y);
    if (c.lse != nullptr && j == 0 && h < grp)   // scores are in the log2 domain
      c.lse[(int64_t)pair * c.n_q_heads + hk * grp + h] = len > 0 ? (M + log2f(L)) * 0.693147180559945309f : -CUDART_INF_F;
  }
  if (rank == 0 && tid == 0 && len <= 0 && c.lse == nullptr) set_status(c.status, PQ_ERR_EMPTY);
  cluster_arrive();   // (D) the merged output is complete everywhere; no block reads another's shared memory after this
  cluster_wait();
  // ---- x_hat_j = sum_k y_k S[j][k] for this block's coordinates: a warp per row of S
  for (int jj = warp; jj < nc; jj += kSplitWarps) {
    const int j = j0 + jj;
    float acc[kH];
#pragma unroll
    for (int h = 0; h < kH; ++h) acc[h] = 0.f;
    for (int k = lane; k < d; k += 32) {
      const float s = __ldg(c.S + (int64_t)j * d + k);
#pragma unroll
      for (int h = 0; h < kH; ++h) acc[h] = fmaf(y_sm[h * dp + k], s, acc[h]);
    }
#pragma unroll
    for (int h = 0; h < kH; ++h) {
      float v = acc[h];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0 && h < grp) {
        const int64_t idx = q0 + h * d + j;
        if (c.io_dtype == PQ_DTYPE_BF16) reinterpret_cast<__nv_bfloat16*>(c.out)[idx] = __float2bfloat16(v);
        else reinterpret_cast<float*>(c.out)[idx] = v;
      }
    }
  }
}

// Blocks per cluster: enough to give every SM two blocks, a power of two that divides d, at least 64 tokens per block,
// at most 8 (the portable limit) or 16 where the call has so few (kv head, sequence) pairs that 8 leave SMs idle.
inline int split_cluster_size(int d, int64_t units, int max_len, int n_sm, int smem_bytes) {
  int C = 1;
  while (C < 8 && C * 2 <= d && C * 64 < max_len && C * units < 2 * n_sm) C *= 2;
  if (C == 8 && d >= 16 && C * 64 < max_len && C * units < n_sm && smem_bytes <= 100 * 1024) C = 16;
  return C;
}

// `configured`: one DeviceMemo per instantiation.
template <class P, int kH>
int32_t launch_split_attention(const P& p, int64_t pairs, int max_len, int smem, cudaStream_t stream) {
  static DeviceMemo configured;
  auto kernel = split_attention_kernel<P, kH>;
  const int n_sm = configure_for_device(kernel, kSplitSmemMax, configured, true);
  if (n_sm == 0) return PQ_ERR_CUDA;
  const int C = split_cluster_size(p.c.d, pairs * p.c.n_kv_heads, max_len, n_sm, smem);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(C, p.c.n_kv_heads, (unsigned)pairs);
  cfg.blockDim = dim3(kSplitThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // set up while the kernel before it finishes (it waits inside)
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, p);
  if (e != cudaSuccess) {
    note_cuda_error(e);
    cudaGetLastError();
    return PQ_ERR_CUDA;
  }
  return launch_status();
}

}  // namespace pq
