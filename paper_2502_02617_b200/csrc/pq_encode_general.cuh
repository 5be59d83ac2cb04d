// Encoder for any head_dim <= 256, recursion depth and bits per level, and for the packed cache at head dims below 128
// (included by pq_general.cu): float32 rotation and float32 decisions with certified margins, float64
// for what a margin does not cover, so the codes are those of a float64 evaluation of Algorithm 1.
//
// A thread block takes a tile of vectors (consecutive rows of one head, K or V):
//   * y = x S.  bf16 rows, where there are enough for four vectors a thread: on tensor cores (mma.sync), S split into three bf16 terms
//     as its slices of 32 rows arrive in shared memory (ge_product_mma; its error bound there).  Otherwise on the FMA pipe: thread =
//     kVT vectors x 8 columns, the sum over k formed per slice and the slices added, so |y - y_exact| <= (32 + d / 32) 2^-24
//     sum_k |x_k||S_kj|, which is at most that factor times ||x||_2 (Cauchy-Schwarz; the columns of an orthogonal S have unit norm).
//   * quantise: thread = (vector, group of 16 coordinates), the four lowest levels in registers.  A code is found by
//     binary search over the level's boundary lines: psi > beta iff r_b cos(beta) - r_a sin(beta) > 0 (with the
//     half-plane bookkeeping of level 1), which needs no arc tangent.  The search tests both neighbours of the cell it
//     ends in, so the smallest |r_b cos - r_a sin| it met bounds the distance to the next boundary.
//   * levels 5 and up: a thread per vector on the groups' norms.
//   * a (vector, group) with any decision inside its margin, or a block radius that close to a rounding boundary of
//     fp16, is taken again by a warp in float64 from the inputs; the same for the upper levels of a (vector, block).
// Margins: moving every coordinate by at most dy moves the norm of n of them by at most sqrt(n) dy, so a test on the
// radii of n-coordinate halves moves by at most sqrt(2 n) dy; 1.1 x that, plus 1e-6 (r_a + r_b) for the float32
// roundings of radii (squares, sums, square root: below 6e-7), table entries and the test itself.
// A radius is certified by radius_unsure, with the bound of rotation_block_error: 1.4 to 5 % of them are not, according to the slices
// of S and the blocks of a vector.
// Bound by the latency of its phases and of the float64 re-decisions, the barriers around them and the fetch of code that a block walks
// through once.  Measured (8 heads; a block per vector in float64 before): 512 tokens, seven levels of three bits 89.7 -> 43.4 us;
// packed cache, 2048 tokens at head_dim 64 67 -> 40 us.  Product on tensor cores instead of the FMA pipe: 8 x 512 tokens, seven levels
// of three bits 206.9 -> 158.9 us.
#pragma once
#include <math_constants.h>

#include "pq_general_common.cuh"

namespace pq {

constexpr int kGeThreads = 256;
constexpr int kGeSlice = 32;              // rows of S per slice

// A slice in shared memory: float32, or its three bf16 terms with rows of dc + 8.
__host__ __device__ constexpr int ge_slice_floats(int dc) { return 3 * kGeSlice * (dc + 8) / 2; }

struct GeShape {
  int dc, ng, vecs, x_stride, row_words, floats_xy;
};
// dc: columns of the tile (head dims below 16 are padded); x rows are dc + 4 floats apart, the 16-coordinate groups of
// a y row 20 floats (conflict-free 16-byte reads in both cases).
__host__ __device__ inline GeShape ge_shape(int d, int row_bytes, int vt) {
  GeShape s;
  s.dc = d < 16 ? 16 : d;
  s.ng = s.dc / 16;
  s.vecs = kGeThreads / (s.dc / 8) * vt;
  s.x_stride = s.dc + 4;
  s.row_words = ((row_bytes + 3) / 4) | 1;
  const int fx = s.vecs * s.x_stride, fy = s.vecs * s.ng * 20;
  s.floats_xy = fx > fy ? fx : fy;
  return s;
}
__host__ inline int ge_smem_bytes(const GeShape& s, int n_bnd) {
  return 4 * (s.floats_xy + ge_slice_floats(s.dc) + s.vecs * s.row_words + s.vecs * s.ng + 2 * s.vecs + 2 * ((n_bnd + 1) & ~1)) +
         8 * s.vecs + 8 * s.vecs * s.ng + 6 * s.vecs * s.ng + 64;
}

__device__ __forceinline__ float ge_load(const void* base, int dtype, int64_t i) {
  return dtype == PQ_DTYPE_BF16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(base)[i])
                                : reinterpret_cast<const float*>(base)[i];
}
// OR `value` (at most 32 bits) into a row at bit `bit`.
__device__ __forceinline__ void ge_put(uint32_t* row, int bit, uint32_t value) {
  const int sh = bit & 31;
  atomicOr(row + (bit >> 5), value << sh);
  const uint32_t hi = sh ? value >> (32 - sh) : 0u;
  if (hi) atomicOr(row + (bit >> 5) + 1, hi);
}
// Put `value` in the place of the `width` (at most 16) bits from bit `bit` on.
__device__ __forceinline__ void ge_replace(uint32_t* row, int bit, int width, uint32_t value) {
  const int sh = bit & 31;
  const uint32_t mask = (1u << width) - 1u;
  atomicAnd(row + (bit >> 5), ~(mask << sh));
  if (sh + width > 32) atomicAnd(row + (bit >> 5) + 1, ~(mask >> (32 - sh)));
  ge_put(row, bit, value);
}
__device__ __forceinline__ float ge_sqrt(float x) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Code of (a, b) at one level: `tab` = (cos, sin) of the level's boundaries, 2^bits - 1 of them; level 1 (kFirst): the first
// n_upper lie in [0, pi].  `near` becomes the smallest distance met.
template <bool kFirst>
__device__ __forceinline__ uint32_t ge_search(float a, float b, const float2* tab, int bits, int n_upper, float& near) {
  uint32_t pos = 0;
  const bool neg = kFirst && b < 0.f;
  near = kFirst ? fabsf(b) : CUDART_INF_F;
  for (int s = bits - 1; s >= 0; --s) {
    const int k = (int)pos + (1 << s) - 1;
    const float2 cs = tab[k];
    const float cross = fmaf(b, cs.x, -a * cs.y);
    near = fminf(near, fabsf(cross));
    bool above = cross > 0.f;
    if (kFirst) above = k < n_upper ? (neg || above) : (neg && above);
    pos += above ? 1u << s : 0u;
  }
  return pos;
}

// The exact code of the pair (a, b) at level l (0-based); kShared: the boundaries lie in shared memory.
template <bool kShared = false>
__device__ __forceinline__ uint32_t ge_exact_code(double a, double b, const GenConfig& g, int l, const double* boundaries) {
  double psi = atan2(b, a);
  if (l == 0 && psi < 0.0) psi += 6.283185307179586476925286766559;
  const double* bnd = boundaries + g.bnd_off[l];
  uint32_t code = 0;
  for (int k = 0; k < (1 << g.bits[l]) - 1; ++k) code += psi > (kShared ? bnd[k] : __ldg(bnd + k));
  return code;
}

// One warp: coordinate 16 grp + (lane & 15) of x S in float64 (each half-warp sums half of the terms, in four chains: a
// float64 multiply-add has several times the latency of a float32 one).
__device__ __forceinline__ double ge_exact_coord(const GenEncodeArgs& a, const void* xbase, int64_t xoff, int grp, int lane) {
  const int d = a.g.d, col = 16 * grp + (lane & 15), half = d >> 1, k0 = (lane >> 4) * half;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  if (col < d) {
    const float* s = a.S + (int64_t)k0 * d + col;
    const int n4 = half & ~3;
#pragma unroll 8   // the loads of 32 terms in flight together: an item is a chain of round trips to L2
    for (int k = 0; k < n4; k += 4)
#pragma unroll
      for (int i = 0; i < 4; ++i)
        acc[i] = fma((double)ge_load(xbase, a.in_dtype, xoff + k0 + k + i), (double)__ldg(s + (int64_t)(k + i) * d), acc[i]);
    for (int k = n4; k < half; ++k) acc[0] = fma((double)ge_load(xbase, a.in_dtype, xoff + k0 + k), (double)__ldg(s + (int64_t)k * d), acc[0]);
  }
  const double sum = (acc[0] + acc[1]) + (acc[2] + acc[3]);
  return sum + __shfl_xor_sync(0xffffffffu, sum, 16);
}

// Where packed row `row` goes, head `head`, K (kv = 0) or V: the byte offset of its general row in the cache; in the packed cache
// token-block and token in one number; -1 if it is not written.
__device__ __forceinline__ int64_t ge_destination(const GenEncodeArgs& a, int row, int head, int kv) {
  int b = row, first = row, count = 1;
  if (a.cu_seqlens != nullptr) {   // the sequence that owns the row: largest b with cu[b] <= row
    int lo = 0, hi = a.batch - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (a.cu_seqlens[mid] <= row) lo = mid; else hi = mid - 1;
    }
    b = lo; first = a.cu_seqlens[lo]; count = a.cu_seqlens[lo + 1] - first;
  }
  const int start = a.lens[b];
  if (start < 0 || start + count > a.capacity) {
    set_status(a.status, PQ_ERR_CAPACITY);
    return -1;
  }
  const int pos = start + (row - first);
  if (!a.packed) return ((((int64_t)b * a.n_kv_heads + head) * 2 + kv) * a.capacity + pos) * a.g.row_bytes;
  const Layout P = make_layout(a.g.d, a.pg.page_tokens);
  const int64_t off = block_offset(P, a.pg, a.n_kv_heads, b, head, kv, pos);
  if (off < 0) {
    set_status(a.status, PQ_ERR_INVALID_ARG);   // a page outside the pool
    return -1;
  }
  return off * kTokenBlock + pos % kTokenBlock;
}

// Bounds on the error of the product on tensor cores relative to ||x||_2 (rot_err in the kernel, and as rotation_block_error).  The
// hardware's sum is not IEEE's: mma.sync m16n8k16 of bf16 truncates its sixteen products, which are exact, and C to multiples of 2^(e - 25),
// e the largest exponent among them (of a product: the sum of its factors' exponents), adds them exactly and truncates the sum to
// float32.  An emulation of that agrees with the device on three million sums (normal, wide ranges of exponents, cancelling pairs beside terms
// at the cut, positive, geometric), bit for bit.  So with M the largest of the terms in magnitude and R the result an MMA is off
// by at most 16 * 2^-25 M + 2^-23 |R| = 2^-24 (8 M + 2 |R|).
// Three bf16 terms hold a float32 S exactly (24 bits), the second at most 2^-9 and the third 2^-18 of the first.  A k-step of 16 rows
// starts from 0 and takes the smallest term first, so M and R are those of the k-step, not of the whole sum:
//   * a coordinate: M and |R| are at most ||x_k|| ||S_kj|| of the k-step (Cauchy-Schwarz), and these add up to ||x|| ||S_j|| = ||x||: 10.1
//     with the smaller terms; then a rounding of 2^-24 for each addition of a k-step but the first;
//   * the coordinates of a block in the 2-norm: the squares of M add up to at most sum_k x_k^2 sum_j S_kj^2 <= ||x_k||^2, those of R too
//     (spectral norm), and the k-steps' norms to sqrt(k-steps) ||x|| at most.
// 10 % and 2 % for the rounding of S (its columns are unit vectors to float32) and second order.
__host__ __device__ constexpr int ge_mma_steps(int dc) { return dc / 16; }
__host__ __device__ constexpr float ge_mma_error(int dc) { return 1.1f * (10.1f + ge_mma_steps(dc)) * 5.9604644775390625e-08f; }
__host__ __device__ constexpr float ge_mma_block_error(int dc) {
  return 1.02f * (10.1f * const_sqrt(ge_mma_steps(dc)) + ge_mma_steps(dc)) * 5.9604644775390625e-08f;
}

// y = x S of a tile of V bf16 vectors (xh [V][dc + 8]) on tensor cores, into y [V][dc / 16][20] over the same memory.  S goes through
// shared memory in slices of 32 rows, split into three bf16 terms as it arrives; a warp owns eight 16 x 8 tiles of y, smallest terms
// first, a fresh accumulator per k-step (see the bounds).
__device__ __forceinline__ void ge_product_mma(const GenEncodeArgs& a, int V, int dc, float* xy, float* Ss, int tid) {
  const int lane = tid & 31, warp = tid >> 5, stride = dc + 8;
  const __nv_bfloat16* xh = reinterpret_cast<const __nv_bfloat16*>(xy);
  uint32_t* Sw = reinterpret_cast<uint32_t*>(Ss);   // [term][32][stride / 2] pairs
  const int m_tiles = V >> 4, per_m = m_tiles >= 8 ? 1 : 8 / m_tiles;      // warps that share 16 vectors
  const int pairs = m_tiles >= 8 ? 32 / m_tiles : 4;                       // pairs of 8-column tiles per 16 vectors of a warp
  const int m0 = m_tiles >= 8 ? warp * (m_tiles >> 3) : warp / per_m, n0 = m_tiles >= 8 ? 0 : (warp % per_m) * 64;
  const int lr = (lane & 7) + (lane & 8), lc = (lane >> 4) * 8;            // this lane's row and column of a 16 x 16 ldmatrix
  const bool aligned = ((uintptr_t)a.S & 15) == 0;
  float tot[8][4];
#pragma unroll
  for (int t = 0; t < 8; ++t)
#pragma unroll
    for (int e = 0; e < 4; ++e) tot[t][e] = 0.f;
#pragma unroll 1
  for (int k0 = 0; k0 < dc; k0 += kGeSlice) {
    const int nk = min(kGeSlice, dc - k0);
    __syncthreads();   // x is complete; the slice before has been used
#pragma unroll 4
    for (int i = 4 * tid; i < nk * dc; i += 4 * kGeThreads) {
      const int k = i / dc, n = i - k * dc;   // four columns of a row
      const float* src = a.S + (int64_t)k0 * dc + i;
      float4 v;
      if (aligned) v = __ldg(reinterpret_cast<const float4*>(src));
      else v = make_float4(__ldg(src), __ldg(src + 1), __ldg(src + 2), __ldg(src + 3));
      uint32_t lo[3], hi[3];
      bf16_terms(v.x, v.y, lo);
      bf16_terms(v.z, v.w, hi);
#pragma unroll
      for (int t = 0; t < 3; ++t)
        *reinterpret_cast<uint2*>(Sw + ((t * kGeSlice + k) * stride + n) / 2) = make_uint2(lo[t], hi[t]);
    }
    __syncthreads();
#pragma unroll 1
    for (int ks = 0; ks < nk; ks += 16) {
      uint32_t A[4];
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const int m = m0 + p / pairs, n = n0 + (p % pairs) * 16;
        if (p % pairs == 0) ldmatrix_x4<false>((uint32_t)__cvta_generic_to_shared(xh + (m * 16 + lr) * stride + k0 + ks + lc), A);
        float acc[2][4] = {};
#pragma unroll
        for (int t = 2; t >= 0; --t) {
          uint32_t B[4];
          ldmatrix_x4<true>((uint32_t)__cvta_generic_to_shared(reinterpret_cast<const __nv_bfloat16*>(Sw) + (t * kGeSlice + ks + lr) * stride + n + lc), B);
          mma_bf16_16816(acc[0], A, B[0], B[1]);
          mma_bf16_16816(acc[1], A, B[2], B[3]);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          tot[2 * p][e] += acc[0][e];
          tot[2 * p + 1][e] += acc[1][e];
        }
      }
    }
  }
  __syncthreads();   // x has been used: y takes its place
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    const int p = t >> 1, row = (m0 + p / pairs) * 16 + (lane >> 2), col = n0 + (p % pairs) * 16 + 8 * (t & 1) + 2 * (lane & 3);
    float* y = xy + (row * (dc >> 4) + (col >> 4)) * 20 + (col & 15);
    *reinterpret_cast<float2*>(y) = make_float2(tot[t][0], tot[t][1]);
    *reinterpret_cast<float2*>(y + 8 * (dc >> 4) * 20) = make_float2(tot[t][2], tot[t][3]);
  }
}

// kVT: vectors per thread in the product (4; 1 for few rows).  kSub: levels inside a group, min(L, 4).
template <int kVT, int kSub>
__global__ void __launch_bounds__(kGeThreads, 2) gen_encode_kernel(const __grid_constant__ GenEncodeArgs a) {
  extern __shared__ __align__(16) uint8_t ge_smem[];
  const GenConfig& g = a.g;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, d = g.d, L = g.L;
  const GeShape s = ge_shape(d, g.row_bytes, kVT);
  const int V = s.vecs, ng = s.ng, dc = s.dc;
  float* xy = reinterpret_cast<float*>(ge_smem);                        // x [V][x_stride], then y [V][ng * 20]
  float* Ss = xy + s.floats_xy;                                         // a slice of S
  uint32_t* rows = reinterpret_cast<uint32_t*>(Ss + ge_slice_floats(dc)); // [V][row_words]
  float* gsum = reinterpret_cast<float*>(rows + V * s.row_words);       // [V][ng] squared norms of the groups
  float* dy_sm = gsum + V * ng;                                         // [V] bound on the error of a coordinate, [V] on that of a block
  float2* tab = reinterpret_cast<float2*>(dy_sm + 2 * V);               // boundaries
  const int n_bnd = g.n_cen - L;
  int64_t* dest = reinterpret_cast<int64_t*>(tab + ((n_bnd + 1) & ~1)); // [V] where the row goes (-1: nowhere)
  double* norm_up = reinterpret_cast<double*>(dest + V);                // [V * ng] exact norms of groups, where needed
  uint16_t* list = reinterpret_cast<uint16_t*>(norm_up + V * ng);       // [V * ng] (vector, group) pairs to take again
  uint16_t* norms = list + V * ng;                                      // [V * ng] (vector, group) pairs of which the norm is needed
  uint16_t* list_up = norms + V * ng;                                   // [V * ng] (vector, block) pairs whose upper levels are taken again
  __shared__ int n_list, n_norms, n_list_up, n_upper;
  const int head = blockIdx.y, kv = blockIdx.z, row0 = blockIdx.x * V;
  const void* xbase = kv ? a.V : a.K;

  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (tid == 0) n_list = n_norms = n_list_up = n_upper = 0;
  for (int i = tid; i < V * s.row_words; i += kGeThreads) rows[i] = 0u;
  __syncthreads();
  asm volatile("griddepcontrol.wait;" ::: "memory");   // the inputs may come from the kernel before this one
  for (int i = tid; i < n_bnd; i += kGeThreads) {
    const double beta = a.boundaries[i];
    tab[i] = cos_sin_table(beta);
    if (i < (1 << g.bits[0]) - 1 && beta <= 3.14159265358979323846) atomicAdd(&n_upper, 1);
  }

  // ---- destinations and inputs
  for (int v = tid; v < V; v += kGeThreads) {
    const int row = row0 + v;
    dest[v] = row < a.total_tokens ? ge_destination(a, row, head, kv) : -1;
  }
  const bool vec8 = a.in_dtype == PQ_DTYPE_BF16 && d >= 16 && ((a.token_stride | a.head_stride) & 7) == 0 &&
                    ((uintptr_t)xbase & 15) == 0;
  const bool tc = kVT == 4 && a.in_dtype == PQ_DTYPE_BF16 && d >= 16;   // the product on tensor cores: x stays bf16
  __nv_bfloat16* xh = reinterpret_cast<__nv_bfloat16*>(xy);
  int bad = 0;
  if (vec8) {
    const int per_row = d / 8;
    for (int i = tid; i < V * per_row; i += kGeThreads) {
      const int v = i / per_row, p = i - v * per_row, row = row0 + v;
      uint4 w = make_uint4(0u, 0u, 0u, 0u);
      if (row < a.total_tokens)
        w = __ldg(reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(xbase) + (int64_t)row * a.token_stride +
                                                 (int64_t)head * a.head_stride + 8 * p));
      const uint32_t u[4] = {w.x, w.y, w.z, w.w};
      float f[8];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        f[2 * e] = __uint_as_float(u[e] << 16);
        f[2 * e + 1] = __uint_as_float(u[e] & 0xFFFF0000u);
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) bad += !(fabsf(f[e]) < CUDART_INF_F);
      if (tc) {
        *reinterpret_cast<uint4*>(xh + v * (dc + 8) + 8 * p) = w;
        continue;
      }
      float4* dst = reinterpret_cast<float4*>(xy + v * s.x_stride + 8 * p);
      dst[0] = make_float4(f[0], f[1], f[2], f[3]);
      dst[1] = make_float4(f[4], f[5], f[6], f[7]);
    }
  } else {
    for (int i = tid; i < V * dc; i += kGeThreads) {
      const int v = i / dc, k = i - v * dc, row = row0 + v;
      float f = 0.f;
      if (row < a.total_tokens && k < d)
        f = ge_load(xbase, a.in_dtype, (int64_t)row * a.token_stride + (int64_t)head * a.head_stride + k);
      bad += !(fabsf(f) < CUDART_INF_F);
      if (tc) xh[v * (dc + 8) + k] = __float2bfloat16(f);
      else xy[v * s.x_stride + k] = f;
    }
  }
  if (bad) {
    atomicAdd(a.status + 1, bad);
    set_status(a.status, PQ_ERR_NONFINITE);
  }

  if (tc) {
    ge_product_mma(a, V, dc, xy, Ss, tid);
  } else {
    // ---- y = x S: thread = kVT vectors x 8 columns (four packed pairs)
    const int tx = tid % (dc / 8), ty = tid / (dc / 8);
    float tot[kVT][8];
#pragma unroll
    for (int v = 0; v < kVT; ++v)
#pragma unroll
      for (int j = 0; j < 8; ++j) tot[v][j] = 0.f;
    for (int k0 = 0; k0 < dc; k0 += kGeSlice) {
      const int nk = min(kGeSlice, dc - k0);
      __syncthreads();
      if (d >= 16) {
        const float4* src = reinterpret_cast<const float4*>(a.S + (int64_t)k0 * d);
        float4* dst = reinterpret_cast<float4*>(Ss);
        if (((uintptr_t)a.S & 15) == 0) {
          for (int i = tid; i < nk * dc / 4; i += kGeThreads) dst[i] = __ldg(src + i);
        } else {
          for (int i = tid; i < nk * dc; i += kGeThreads) Ss[i] = __ldg(a.S + (int64_t)k0 * d + i);
        }
      } else {
        for (int i = tid; i < nk * dc; i += kGeThreads) {
          const int k = k0 + i / dc, j = i % dc;
          Ss[i] = k < d && j < d ? __ldg(a.S + k * d + j) : 0.f;
        }
      }
      __syncthreads();
      uint64_t acc[kVT][4];
#pragma unroll
      for (int v = 0; v < kVT; ++v)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[v][j] = 0ull;
#pragma unroll 2
      for (int k = 0; k < nk; k += 4) {
        float4 xv[kVT];
#pragma unroll
        for (int v = 0; v < kVT; ++v) xv[v] = *reinterpret_cast<const float4*>(xy + (ty * kVT + v) * s.x_stride + k0 + k);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const ulonglong2 sa = *reinterpret_cast<const ulonglong2*>(Ss + (k + kk) * dc + 8 * tx);
          const ulonglong2 sb = *reinterpret_cast<const ulonglong2*>(Ss + (k + kk) * dc + 8 * tx + 4);
#pragma unroll
          for (int v = 0; v < kVT; ++v) {
            const float xk = kk == 0 ? xv[v].x : kk == 1 ? xv[v].y : kk == 2 ? xv[v].z : xv[v].w;
            const uint64_t xx = f2_pack(xk, xk);
            acc[v][0] = f2_fma(xx, sa.x, acc[v][0]);
            acc[v][1] = f2_fma(xx, sa.y, acc[v][1]);
            acc[v][2] = f2_fma(xx, sb.x, acc[v][2]);
            acc[v][3] = f2_fma(xx, sb.y, acc[v][3]);
          }
        }
      }
#pragma unroll
      for (int v = 0; v < kVT; ++v)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float lo, hi;
          f2_unpack(acc[v][j], lo, hi);
          tot[v][2 * j] += lo;
          tot[v][2 * j + 1] += hi;
        }
    }
    __syncthreads();   // x has been used: y takes its place
#pragma unroll
    for (int v = 0; v < kVT; ++v) {
      float* dst = xy + ((ty * kVT + v) * ng + (tx >> 1)) * 20 + 8 * (tx & 1);
      *reinterpret_cast<float4*>(dst) = make_float4(tot[v][0], tot[v][1], tot[v][2], tot[v][3]);
      *reinterpret_cast<float4*>(dst + 4) = make_float4(tot[v][4], tot[v][5], tot[v][6], tot[v][7]);
    }
  }
  __syncthreads();
  for (int i = tid; i < V * ng; i += kGeThreads) {   // squared norms of the groups
    const float4* src = reinterpret_cast<const float4*>(xy + i * 20);
    float q[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float4 w = src[j];
      q[j] = fmaf(w.x, w.x, w.y * w.y) + fmaf(w.z, w.z, w.w * w.w);
    }
    gsum[i] = (q[0] + q[1]) + (q[2] + q[3]);
  }
  __syncthreads();
  const float rot_err = tc ? ge_mma_error(dc) : 1.1f * (float)(kGeSlice + dc / kGeSlice) * 5.9604644775390625e-08f;
  const float blk_err = tc ? ge_mma_block_error(dc) : rotation_block_error(kGeSlice, (dc + kGeSlice - 1) / kGeSlice);
  for (int v = tid; v < V; v += kGeThreads) {
    float t = 0.f;
    for (int i = 0; i < ng; ++i) t += gsum[v * ng + i];
    // the floor: where squares leave the float32 range (below 4e-20), nothing is certified
    dy_sm[v] = fmaf(rot_err * 1.0001f, sqrtf(t), 1e-19f);
    dy_sm[V + v] = blk_err * 1.0001f * sqrtf(t);
  }
  __syncthreads();

  // ---- the levels inside a group of 16 coordinates
  for (int i = tid; i < V * ng; i += kGeThreads) {
    const int v = i / ng, grp = i - v * ng;
    if (dest[v] < 0) continue;
    const float dy = dy_sm[v];
    float r[16];
    const float4* src = reinterpret_cast<const float4*>(xy + i * 20);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float4 w = src[j];
      r[4 * j] = w.x; r[4 * j + 1] = w.y; r[4 * j + 2] = w.z; r[4 * j + 3] = w.w;
    }
    bool sure = true;
    uint32_t lo[kSub], hi[kSub];   // the level's codes in the group: the first half of them in lo, the second in hi
    float s2[8];                   // squared radii of the level
#pragma unroll
    for (int l = 0; l < kSub; ++l) {
      const int n = 8 >> l, b = g.bits[l];
      const float m_dy = 1.1f * (l == 0 ? 1.41421356f : l == 1 ? 2.f : l == 2 ? 2.82842712f : 4.f) * dy;
      lo[l] = hi[l] = 0u;
#pragma unroll
      for (int j = 0; j < n; ++j) {
        const float p = r[2 * j], q = r[2 * j + 1];
        float near;
        const uint32_t code = l == 0 ? ge_search<true>(p, q, tab, b, n_upper, near) : ge_search<false>(p, q, tab + g.bnd_off[l], b, 0, near);
        if (l == 0 && 16 * grp + 2 * j >= d) near = CUDART_INF_F;   // padding of a head_dim below 16
        if (l > 0 && 16 * grp + (j << (l + 1)) >= d) near = CUDART_INF_F;
        sure = sure && near > fmaf(1e-6f, fabsf(p) + fabsf(q), m_dy);
        if (n == 1 || j < n / 2) lo[l] |= code << (j * b);
        else hi[l] |= code << ((j - n / 2) * b);
        s2[j] = l == 0 ? fmaf(p, p, q * q) : s2[2 * j] + s2[2 * j + 1];
      }
      // radii of the next level (in place: r[j] is read before r[j] of the next level is needed)
#pragma unroll
      for (int j = 0; j < n; ++j) r[j] = ge_sqrt(s2[j]);
    }
    const int n_blk = 16 >> kSub;
    uint32_t rad[n_blk];
    if (L == kSub) {
#pragma unroll
      for (int j = 0; j < n_blk; ++j) {
        if (grp * n_blk + j < g.nb) sure = sure && !radius_unsure(r[j], dy_sm[V + v]);
        rad[j] = __half_as_ushort(__float2half_rn(r[j]));
      }
    }
    if (!sure) {
      list[atomicAdd(&n_list, 1)] = (uint16_t)i;
      continue;
    }
    uint32_t* row = rows + v * s.row_words;
#pragma unroll
    for (int l = 0; l < kSub; ++l) {
      const int n = 8 >> l, b = g.bits[l], bit = g.byte_off[l] * 8 + grp * n * b;
      if (16 * grp >= d) continue;
      ge_put(row, bit, lo[l]);
      if (n > 1) ge_put(row, bit + (n / 2) * b, hi[l]);
    }
    if (L == kSub) {
#pragma unroll
      for (int j = 0; j < n_blk; ++j)
        if (grp * n_blk + j < g.nb) ge_put(row, g.rad_off * 8 + 16 * (grp * n_blk + j), rad[j]);
    }
  }
  // ---- levels above the groups: a thread per vector, the squared norms halved in place
  const int gpb = L > 4 ? 1 << (L - 4) : 1;   // groups of a block
  if (L > 4) {
    __syncthreads();
    for (int v = tid; v < V; v += kGeThreads) {
      if (dest[v] < 0) continue;
      float* q2 = gsum + v * ng;
      uint32_t* row = rows + v * s.row_words;
      uint32_t unsure = 0u;   // blocks with a decision or a radius that is not certified
      const float dy = dy_sm[v];
      for (int l = 4; l < L; ++l) {
        const int n = d >> (l + 1), b = g.bits[l];
        const float m_dy = 1.1f * ge_sqrt((float)(2 << l)) * dy;
        uint32_t word = 0u;
        int fill = 0, bit = g.byte_off[l] * 8;
        for (int j = 0; j < n; ++j) {
          const float sa = q2[2 * j], sb = q2[2 * j + 1], p = ge_sqrt(sa), q = ge_sqrt(sb);
          float near;
          const uint32_t code = ge_search<false>(p, q, tab + g.bnd_off[l], b, 0, near);
          if (!(near > fmaf(1e-6f, p + q, m_dy))) unsure |= 1u << (j >> (L - 1 - l));
          word |= code << fill;
          fill += b;
          if (fill > 24 || j + 1 == n) {
            ge_put(row, bit, word);
            bit += fill;
            word = 0u;
            fill = 0;
          }
          q2[j] = sa + sb;
        }
      }
      for (int j = 0; j < g.nb; ++j) {
        const float r = ge_sqrt(q2[j]);
        if (radius_unsure(r, dy_sm[V + v])) unsure |= 1u << j;
        ge_put(row, g.rad_off * 8 + 16 * j, __half_as_ushort(__float2half_rn(r)));
      }
      for (; unsure; unsure &= unsure - 1) {
        const int j = __ffs(unsure) - 1;
        list_up[atomicAdd(&n_list_up, 1)] = (uint16_t)(v * g.nb + j);
        const int at = atomicAdd(&n_norms, gpb);
        for (int i = 0; i < gpb; ++i) norms[at + i] = (uint16_t)(v * ng + j * gpb + i);
      }
    }
  }
  __syncthreads();

  // ---- float64 for what the margins do not cover: a warp per (vector, group)
  for (int e = warp; e < n_list; e += kGeThreads / 32) {
    const int i = list[e], v = i / ng, grp = i - v * ng;
    const int64_t xoff = (int64_t)(row0 + v) * a.token_stride + (int64_t)head * a.head_stride;
    double y = ge_exact_coord(a, xbase, xoff, grp, lane);   // of coordinate 16 grp + (lane & 15)
    uint32_t* row = rows + v * s.row_words;
#pragma unroll
    for (int l = 0; l < kSub; ++l) {
      const int n = 8 >> l;
      const double p = __shfl_sync(0xffffffffu, y, (2 * lane) & 31), q = __shfl_sync(0xffffffffu, y, (2 * lane + 1) & 31);
      if (lane < n && 16 * grp + (lane << (l + 1)) < d)
        ge_put(row, g.byte_off[l] * 8 + (grp * n + lane) * g.bits[l], ge_exact_code(p, q, g, l, a.boundaries));
      y = sqrt(p * p + q * q);
    }
    const int n_blk = 16 >> kSub;
    if (L == kSub && lane < n_blk && grp * n_blk + lane < g.nb) {
      double r = y;
      if (r > 65504.0) {
        r = 65504.0;
        atomicAdd(a.status + 2, 1);
      }
      ge_put(row, g.rad_off * 8 + 16 * (grp * n_blk + lane), __half_as_ushort(__double2half(r)));
    }
    if (lane == 0) atomicAdd(a.status + 3, 1);
  }
  if (L > 4) {
    // the norms of all groups of the vectors whose upper levels are taken again, then those levels, a warp per vector
    for (int e = warp; e < n_norms; e += kGeThreads / 32) {
      const int i = norms[e], v = i / ng;
      double y = ge_exact_coord(a, xbase, (int64_t)(row0 + v) * a.token_stride + (int64_t)head * a.head_stride, i - v * ng, lane);
#pragma unroll
      for (int l = 0; l < 4; ++l) {   // radius of a pair, of four coordinates, ... as the recursion forms them
        const double p = __shfl_sync(0xffffffffu, y, (2 * lane) & 31), q = __shfl_sync(0xffffffffu, y, (2 * lane + 1) & 31);
        y = sqrt(p * p + q * q);
      }
      if (lane == 0) norm_up[i] = y;
    }
    __syncthreads();
    for (int e = warp; e < n_list_up; e += kGeThreads / 32) {
      const int v = list_up[e] / g.nb, blk = list_up[e] - v * g.nb;
      uint32_t* row = rows + v * s.row_words;
      double mine = lane < gpb ? norm_up[v * ng + blk * gpb + lane] : 0.0;
      for (int l = 4; l < L; ++l) {
        const int n = gpb >> (l - 3);   // the block's angles at this level
        const double p = __shfl_sync(0xffffffffu, mine, (2 * lane) & 31), q = __shfl_sync(0xffffffffu, mine, (2 * lane + 1) & 31);
        if (lane < n) ge_replace(row, g.byte_off[l] * 8 + (blk * n + lane) * g.bits[l], g.bits[l], ge_exact_code(p, q, g, l, a.boundaries));
        mine = sqrt(p * p + q * q);
      }
      if (lane == 0) {
        double r = mine;
        if (r > 65504.0) {
          r = 65504.0;
          atomicAdd(a.status + 2, 1);
        }
        ge_replace(row, g.rad_off * 8 + 16 * blk, 16, __half_as_ushort(__double2half(r)));
        atomicAdd(a.status + 3, 1);
      }
    }
  }
  __syncthreads();

  // ---- rows out
  if (a.packed) {
    const Layout P = make_layout(d, a.pg.page_tokens);
    for (int i = tid; i < V * g.row_bytes; i += kGeThreads) {
      const int v = i / g.row_bytes, t = i - v * g.row_bytes;
      const int64_t at = dest[v];
      if (at < 0) continue;
      uint8_t* tb = a.cache + at / kTokenBlock;
      const int tok = (int)(at % kTokenBlock);
      const uint8_t byte = reinterpret_cast<const uint8_t*>(rows + v * s.row_words)[t];
      if (t < P.b1) tb[tok * P.b1 + t] = byte;
      else if (t < P.b1 + P.b2) tb[P.o2 + tok * P.b2 + t - P.b1] = byte;
      else if (t < P.b1 + P.b2 + P.b3) tb[P.o3 + tok * P.b3 + t - P.b1 - P.b2] = byte;
      else if (t < P.b1 + P.b2 + P.b3 + P.b4) tb[P.o4 + tok * P.b4 + t - P.b1 - P.b2 - P.b3] = byte;
      else if (t >= g.rad_off) tb[P.orad + tok * P.br + t - g.rad_off] = byte;
    }
  } else if ((g.row_bytes & 3) == 0 && ((uintptr_t)a.cache & 3) == 0) {
    const int per = g.row_bytes >> 2;
    for (int i = tid; i < V * per; i += kGeThreads) {
      const int v = i / per, t = i - v * per;
      if (dest[v] >= 0) reinterpret_cast<uint32_t*>(a.cache + dest[v])[t] = rows[v * s.row_words + t];
    }
  } else {
    const int per = g.row_bytes >> 1;
    for (int i = tid; i < V * per; i += kGeThreads) {
      const int v = i / per, t = i - v * per;
      if (dest[v] >= 0)
        reinterpret_cast<uint16_t*>(a.cache + dest[v])[t] = reinterpret_cast<const uint16_t*>(rows + v * s.row_words)[t];
    }
  }
}

// Few vectors, general rows: one thread block of max(d, 32) threads per vector (row, K | V, head), float64 throughout: y = x S, then
// the polar tree level by level (thread j forms angle j of the level, code = number of boundaries below it), then the bit streams.
// A chain of d float64 multiply-adds and log2 d levels, hardly longer for a thousand vectors than for one: see launch_gen_encode.
__global__ void gen_encode_vector_kernel(const __grid_constant__ GenEncodeArgs a) {
  __shared__ double ra[kGenMaxDim], rb[kGenMaxDim], bnd[kGenMaxCentroids];
  __shared__ uint8_t codes[kGenMaxDim];
  __shared__ int64_t dest;
  const GenConfig& g = a.g;
  const int j = threadIdx.x, d = g.d;
  const int64_t v = blockIdx.x;
  const int head = (int)(v % a.n_kv_heads), kv = (int)((v / a.n_kv_heads) & 1);
  const int row = (int)(v / (2 * a.n_kv_heads));
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");   // the inputs may come from the kernel before this one
  if (j == 0) dest = ge_destination(a, row, head, kv);
  for (int i = j; i < g.n_cen - g.L; i += blockDim.x) bnd[i] = a.boundaries[i];
  if (j < d) {
    const float x = ge_load(kv ? a.V : a.K, a.in_dtype, (int64_t)row * a.token_stride + (int64_t)head * a.head_stride + j);
    if (!(fabsf(x) < CUDART_INF_F)) {
      atomicAdd(a.status + 1, 1);
      set_status(a.status, PQ_ERR_NONFINITE);
    }
    ra[j] = (double)x;
  }
  __syncthreads();
  if (j < d) {
    double acc = 0.0;
    for (int k = 0; k < d; ++k) acc = fma(ra[k], (double)__ldg(a.S + (int64_t)k * d + j), acc);
    rb[j] = acc;
  }
  __syncthreads();
  double* src = rb;
  double* dst = ra;
  for (int l = 0; l < g.L; ++l) {
    if (j < (d >> (l + 1))) {
      const double p = src[2 * j], q = src[2 * j + 1];
      codes[g.code_off[l] + j] = (uint8_t)ge_exact_code<true>(p, q, g, l, bnd);
      dst[j] = sqrt(p * p + q * q);
    }
    __syncthreads();
    double* t = src; src = dst; dst = t;
  }
  if (dest < 0) return;
  uint8_t* out = a.cache + dest;
  for (int t = j; t < g.rad_off; t += blockDim.x) {   // byte t of the row: gather its bits
    int l = g.L - 1;
    while (l > 0 && t < g.byte_off[l]) --l;
    uint32_t byte = 0;
    if (t < g.byte_off[l] + g.level_bytes[l]) {
      const int b = g.bits[l], n = d >> (l + 1);
      for (int bit = 0; bit < 8; ++bit) {
        const int at = (t - g.byte_off[l]) * 8 + bit, idx = at / b;
        if (idx < n) byte |= (((uint32_t)codes[g.code_off[l] + idx] >> (at % b)) & 1u) << bit;
      }
    }
    out[t] = (uint8_t)byte;
  }
  if (j < g.nb) {
    double r = src[j];
    if (r > 65504.0) {
      r = 65504.0;
      atomicAdd(a.status + 2, 1);
    }
    reinterpret_cast<__half*>(out + g.rad_off)[j] = __double2half(r);
  }
}

// A kernel as a programmatic dependent launch: set up while the kernel before it in the stream finishes (it waits inside).
static int32_t launch_gen_kernel(void (*kernel)(GenEncodeArgs), dim3 grid, int threads, int smem, const GenEncodeArgs& a, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
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
  return PQ_OK;
}

template <int kVT, int kSub>
static int32_t launch_gen_encode_as(const GenEncodeArgs& a, cudaStream_t stream) {
  const GeShape s = ge_shape(a.g.d, a.g.row_bytes, kVT);
  static DeviceMemo configured;
  if (configure_for_device(gen_encode_kernel<kVT, kSub>, 113 * 1024, configured) == 0) return PQ_ERR_CUDA;
  return launch_gen_kernel(gen_encode_kernel<kVT, kSub>, dim3((a.total_tokens + s.vecs - 1) / s.vecs, a.n_kv_heads, 2), kGeThreads,
                           ge_smem_bytes(s, a.g.n_cen - a.g.L), a, stream);
}

// A block per vector until the tiled kernel, which starts at 14 to 60 us, is faster.  Measured (vector against tiled kernel): head_dim
// 256, bits 4,2,2,2,2 128 vectors 18.6 / 53 us, 2048 72 / 78, 4096 135 / 88; 128, seven levels of three bits 128 vectors 16.2 / 35 us,
// 2048 30 / 40, 4096 50 / 46; 64, bits 4,3,2 4096 vectors 23 / 25 us, 8192 41 / 29; 16 4096 10 / 14 us, 8192 16 / 14.
// In the tiled kernel one vector per thread in the product instead of four as long as that many blocks fit on the device at
// once: a short chunk then spreads over four times as many SMs.
static int32_t launch_gen_encode(const GenEncodeArgs& a, cudaStream_t stream) {
  const int64_t n_vec = (int64_t)a.total_tokens * 2 * a.n_kv_heads;
  if (!a.packed && n_vec <= (a.g.d > 128 ? 2048 : a.g.d > 64 ? 3072 : 4096))
    return launch_gen_kernel(gen_encode_vector_kernel, dim3((unsigned)n_vec), a.g.d < 32 ? 32 : a.g.d, 0, a, stream);
  static DeviceMemo sm_count;
  const int n_sm = sm_count_of_device(sm_count);
  if (n_sm == 0) return PQ_ERR_CUDA;
  const GeShape s1 = ge_shape(a.g.d, a.g.row_bytes, 1);
  const bool few = (int64_t)((a.total_tokens + s1.vecs - 1) / s1.vecs) * 2 * a.n_kv_heads <= 2 * n_sm;
  switch (a.g.L < 4 ? a.g.L : 4) {
    case 1: return few ? launch_gen_encode_as<1, 1>(a, stream) : launch_gen_encode_as<4, 1>(a, stream);
    case 2: return few ? launch_gen_encode_as<1, 2>(a, stream) : launch_gen_encode_as<4, 2>(a, stream);
    case 3: return few ? launch_gen_encode_as<1, 3>(a, stream) : launch_gen_encode_as<4, 3>(a, stream);
    default: return few ? launch_gen_encode_as<1, 4>(a, stream) : launch_gen_encode_as<4, 4>(a, stream);
  }
}

}  // namespace pq
