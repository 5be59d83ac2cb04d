// The query rotation before, and the merge and un-rotation after, the tcgen05 multi-query kernel, for all (query, head) rows of
// a call (included by pq_decode.cu): plain float32 products of [rows][128] with S or S^T, spread over all SMs.  Inside the
// attention kernel, where a CTA needs them for its own 128 rows and repeats them for every range of the blocks, they took 90 us
// of every CTA's time.
// A block of 256 threads takes kTile rows.  64 rows: thread = 4 columns x 8 rows (a warp shares its rows, so its reads of them
// are broadcasts, and reads 512 consecutive bytes of S), bound by the multiply-adds.  8, 16 or 32 rows, while that many blocks do not fill
// the device: thread = one column x half of the rows; every warp reading all of S takes twice as many shared-memory wavefronts,
// which bound such a block.  As long as every block can have an SM to itself it asks for more than half of the shared memory: two or
// three on the SMs that the attention kernel left first took 7 us each for a product of 2.
// Attention of 32 queries in four sequences of 150 tokens, 32/8 heads, 4096 rows: 34 us with tiles of 32, 39 with 16 or 64 (tcgen05 kernel).
#pragma once

namespace pq {

constexpr int kRotThreads = 256, kRotSStride = 132;
constexpr int kRotAlone = 116 * 1024;
template <int kTile>
inline int rot_smem_bytes(int64_t n_rows, int n_sm) {
  constexpr int need = (128 * kRotSStride + kTile * 128) * 4;
  static_assert(need <= kRotAlone, "the limit that the kernels are configured for");
  return n_rows <= (int64_t)n_sm * kTile ? kRotAlone : need;
}

// What a thread computes of the tile's product: kRows rows from r0 on, kCols columns from c0 on.
template <int kTile>
struct RotShare {
  static constexpr int kCols = kTile == 64 ? 4 : 1, kRows = kTile == 64 ? 8 : kTile / 2;
  int r0, c0;
  __device__ __forceinline__ RotShare(int lane, int warp) {
    r0 = kTile == 64 ? warp * 8 : (warp >> 2) * kRows;
    c0 = kTile == 64 ? 4 * lane : 32 * (warp & 3) + lane;
  }
};
// out[r][e] = sum_k x[r0 + r][k] s[k][c0 + e]
template <int kTile>
__device__ __forceinline__ void rot_product(const float* x, const float* s, const RotShare<kTile>& t,
                                            float (&out)[RotShare<kTile>::kRows][RotShare<kTile>::kCols]) {
  constexpr int kRows = RotShare<kTile>::kRows;
  if constexpr (kTile == 64) {
    uint64_t acc[kRows][2];
#pragma unroll
    for (int r = 0; r < kRows; ++r) acc[r][0] = acc[r][1] = 0ull;
#pragma unroll 2
    for (int k = 0; k < 128; k += 4) {
      ulonglong2 b[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) b[e] = *reinterpret_cast<const ulonglong2*>(s + (k + e) * kRotSStride + t.c0);
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        const float4 v = *reinterpret_cast<const float4*>(x + (t.r0 + r) * 128 + k);
        const uint64_t v0 = f2_pack(v.x, v.x), v1 = f2_pack(v.y, v.y), v2 = f2_pack(v.z, v.z), v3 = f2_pack(v.w, v.w);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          acc[r][h] = f2_fma(v0, h ? b[0].y : b[0].x, acc[r][h]);
          acc[r][h] = f2_fma(v1, h ? b[1].y : b[1].x, acc[r][h]);
          acc[r][h] = f2_fma(v2, h ? b[2].y : b[2].x, acc[r][h]);
          acc[r][h] = f2_fma(v3, h ? b[3].y : b[3].x, acc[r][h]);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      f2_unpack(acc[r][0], out[r][0], out[r][1 % RotShare<kTile>::kCols]);
      f2_unpack(acc[r][1], out[r][2 % RotShare<kTile>::kCols], out[r][3 % RotShare<kTile>::kCols]);
    }
  } else {
#pragma unroll
    for (int r = 0; r < kRows; ++r) out[r][0] = 0.f;
#pragma unroll 4
    for (int k = 0; k < 128; k += 4) {
      float b[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) b[e] = s[(k + e) * kRotSStride + t.c0];
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        const float4 v = *reinterpret_cast<const float4*>(x + (t.r0 + r) * 128 + k);
        out[r][0] = fmaf(v.w, b[3], fmaf(v.z, b[2], fmaf(v.y, b[1], fmaf(v.x, b[0], out[r][0]))));
      }
    }
  }
}

// q' = (q S) * factor of every row as fp16 value and residual: qrot [row][value | residual][128], coordinate j at position
// (j & ~3) | (0, 2, 1, 3)[j & 3] -- the order in which the decoders deliver the keys.
template <int kTile>
__global__ void __launch_bounds__(kRotThreads) rotate_rows_kernel(const float* S, const void* q, int io_dtype, int64_t n_rows, float factor,
                                                                  __half* qrot) {
  extern __shared__ __align__(16) float rot_smem[];
  float* s = rot_smem;
  float* x = rot_smem + 128 * kRotSStride;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t row0 = (int64_t)blockIdx.x * kTile;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
#pragma unroll 4
  for (int i = tid; i < 128 * 32; i += kRotThreads) {   // S is a constant of the caller: read before the wait
    const int k = i >> 5, c = 4 * (i & 31);
    *reinterpret_cast<float4*>(s + k * kRotSStride + c) = __ldg(reinterpret_cast<const float4*>(S + k * 128 + c));
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  for (int i = tid; i < kTile * 32; i += kRotThreads) {
    const int64_t row = row0 + (i >> 5);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row < n_rows) {
      const int64_t at = row * 128 + 4 * (i & 31);
      if (io_dtype == PQ_DTYPE_BF16) {
        const uint2 w = *reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(q) + at);
        v = make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xFFFF0000u), __uint_as_float(w.y << 16),
                        __uint_as_float(w.y & 0xFFFF0000u));
      } else {
        v = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(q) + at);
      }
    }
    *reinterpret_cast<float4*>(x + 4 * i) = v;
  }
  __syncthreads();
  const RotShare<kTile> t(lane, warp);
  float out[RotShare<kTile>::kRows][RotShare<kTile>::kCols];
  rot_product<kTile>(x, s, t, out);
#pragma unroll
  for (int r = 0; r < RotShare<kTile>::kRows; ++r) {
    const int64_t row = row0 + t.r0 + r;
    if (row >= n_rows) break;
    if constexpr (kTile == 64) {
      __half hi[4], lo[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int at = ((e & 1) << 1) | (e >> 1);
        const float v = out[r][e] * factor;
        hi[at] = __float2half_rn(v);
        lo[at] = __float2half_rn(v - __half2float(hi[at]));
      }
      *reinterpret_cast<uint2*>(qrot + row * 256 + t.c0) = *reinterpret_cast<const uint2*>(hi);
      *reinterpret_cast<uint2*>(qrot + row * 256 + 128 + t.c0) = *reinterpret_cast<const uint2*>(lo);
    } else {
      const int at = (t.c0 & ~3) | (t.c0 & 1) << 1 | (t.c0 >> 1 & 1);
      const float v = out[r][0] * factor;
      const __half hi = __float2half_rn(v);
      qrot[row * 256 + at] = hi;
      qrot[row * 256 + 128 + at] = __float2half_rn(v - __half2float(hi));
    }
  }
}

// S^T in shared memory.
__device__ __forceinline__ void load_transposed(const float* S, float* s, int tid) {
#pragma unroll 4
  for (int i = tid; i < 128 * 32; i += kRotThreads) {
    const int n = i & 127, k = 4 * (i >> 7);   // neighbouring threads write neighbouring columns
    const float4 v = __ldg(reinterpret_cast<const float4*>(S + n * 128 + k));
    s[k * kRotSStride + n] = v.x;
    s[(k + 1) * kRotSStride + n] = v.y;
    s[(k + 2) * kRotSStride + n] = v.z;
    s[(k + 3) * kRotSStride + n] = v.w;
  }
}

// The tile (x) times S^T (s), to the rows from row0 on of out.
template <int kTile>
__device__ __forceinline__ void store_unrotated(const float* x, const float* s, int64_t row0, int64_t n_rows, int lane, int warp, void* out,
                                                int out_dtype) {
  const RotShare<kTile> t(lane, warp);
  float y[RotShare<kTile>::kRows][RotShare<kTile>::kCols];
  rot_product<kTile>(x, s, t, y);
#pragma unroll
  for (int r = 0; r < RotShare<kTile>::kRows; ++r) {
    const int64_t row = row0 + t.r0 + r;
    if (row >= n_rows) break;
    const int64_t at = row * 128 + t.c0;
    if constexpr (kTile == 64) {
      if (out_dtype == PQ_DTYPE_BF16) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(y[r][0], y[r][1]), b = __floats2bfloat162_rn(y[r][2], y[r][3]);
        *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(out) + at) =
            make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
      } else {
        *reinterpret_cast<float4*>(reinterpret_cast<float*>(out) + at) = make_float4(y[r][0], y[r][1], y[r][2], y[r][3]);
      }
    } else if (out_dtype == PQ_DTYPE_BF16) {
      reinterpret_cast<__nv_bfloat16*>(out)[at] = __float2bfloat16(y[r][0]);
    } else {
      reinterpret_cast<float*>(out)[at] = y[r][0];
    }
  }
}

// out = (sum_p exp(lse_p - lse) part_p) S^T of every row; parts [part][row][128], lse [part][row] (natural log, -inf: nothing seen).
template <int kTile>
__global__ void __launch_bounds__(kRotThreads) merge_unrotate_kernel(const float* S, const float* parts, const float* lse, int n_parts,
                                                                     int64_t n_rows, void* out, int out_dtype, int32_t* status) {
  extern __shared__ __align__(16) float rot_smem[];
  float* s = rot_smem;   // S^T
  float* x = rot_smem + 128 * kRotSStride;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t row0 = (int64_t)blockIdx.x * kTile;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  load_transposed(S, s, tid);
  asm volatile("griddepcontrol.wait;" ::: "memory");   // the parts come from the kernel before this one
#pragma unroll 2
  for (int i = tid; i < kTile * 32; i += kRotThreads) {   // a warp per row
    const int64_t row = row0 + (i >> 5);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row < n_rows) {
      const float mine = lane < n_parts ? lse[(int64_t)lane * n_rows + row] : -CUDART_INF_F;   // at most 32 parts
      float mx = mine;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      if (mx > -CUDART_INF_F || __any_sync(0xffffffffu, mine != mine)) {   // a NaN part makes the row NaN
        const float w_mine = __expf(mine - mx);
        float wsum = w_mine;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) wsum += __shfl_xor_sync(0xffffffffu, wsum, o);
#pragma unroll 4
        for (int p = 0; p < n_parts; ++p) {
          const float4 v = *reinterpret_cast<const float4*>(parts + ((int64_t)p * n_rows + row) * 128 + 4 * lane);
          const float w = __shfl_sync(0xffffffffu, w_mine, p);
          acc.x = fmaf(w, v.x, acc.x);
          acc.y = fmaf(w, v.y, acc.y);
          acc.z = fmaf(w, v.z, acc.z);
          acc.w = fmaf(w, v.w, acc.w);
        }
        const float k = 1.f / wsum;
        acc = make_float4(acc.x * k, acc.y * k, acc.z * k, acc.w * k);
      } else if (lane == 0) {
        set_status(status, PQ_ERR_EMPTY);   // a query that sees no token: zeros
      }
    }
    *reinterpret_cast<float4*>(x + 4 * i) = acc;
  }
  __syncthreads();
  store_unrotated<kTile>(x, s, row0, n_rows, lane, warp, out, out_dtype);
}

// The same for the parts that rows_attention_kernel leaves: row i (pair i / n_q_heads) belongs to a unit whose parts are the slots
// unit_parts[unit].x .. + unit_parts[unit].y - 1, each with (reference, denominator) in the log2 domain and an output relative to it.
template <int kTile>
__global__ void __launch_bounds__(kRotThreads) merge_rows_kernel(const float* S, DecodeArgs a) {
  extern __shared__ __align__(16) float rot_smem[];
  float* s = rot_smem;   // S^T
  float* x = rot_smem + 128 * kRotSStride;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int row0 = blockIdx.x * kTile, n_rows = a.batch * a.n_q_heads, g = a.n_q_heads / a.n_kv_heads, R = a.rows_per_block;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  load_transposed(S, s, tid);
  asm volatile("griddepcontrol.wait;" ::: "memory");   // the parts come from the kernel before this one
#pragma unroll 2
  for (int i = tid; i < kTile * 32; i += kRotThreads) {   // a warp per row
    const int row = row0 + (i >> 5);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row < n_rows) {
      const int pair = row / a.n_q_heads, head = row - pair * a.n_q_heads, hk = head / g, seq = pair / a.n_q, j = pair - seq * a.n_q;
      const int r_all = j * g + head - hk * g, rb = r_all / R, r = r_all - rb * R;
      const int2 unit = a.unit_parts[(seq * a.n_kv_heads + hk) * a.n_row_blocks + rb];
      const float2* ml = reinterpret_cast<const float2*>(a.ws.ml) + (int64_t)unit.x * R + r;
      const float4* o = reinterpret_cast<const float4*>(a.ws.o + ((int64_t)unit.x * R + r) * 128) + lane;
      float M = -CUDART_INF_F, L = 0.f;
      for (int p0 = 0; p0 < unit.y; p0 += 32) {   // 32 parts at a time, in slot order
        const float2 mine = p0 + lane < unit.y ? ml[(int64_t)(p0 + lane) * R] : make_float2(-CUDART_INF_F, 0.f);
        float m_new = mine.x;   // a NaN is passed over here and makes the row NaN by its weight
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) m_new = fmaxf(m_new, __shfl_xor_sync(0xffffffffu, m_new, off));
        m_new = fmaxf(M, m_new);
        const float k = M == -CUDART_INF_F ? 0.f : fast_exp2(M - m_new);
        const float w_mine = mine.x == -CUDART_INF_F ? 0.f : fast_exp2(mine.x - m_new);
        float l = mine.y * w_mine;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
        L = L * k + l;
        M = m_new;
        acc = make_float4(acc.x * k, acc.y * k, acc.z * k, acc.w * k);
        const int n = min(32, unit.y - p0);
#pragma unroll 4
        for (int p = 0; p < n; ++p) {
          const float4 v = o[(int64_t)(p0 + p) * R * 32];
          const float w = __shfl_sync(0xffffffffu, w_mine, p);
          acc.x = fmaf(w, v.x, acc.x);
          acc.y = fmaf(w, v.y, acc.y);
          acc.z = fmaf(w, v.z, acc.z);
          acc.w = fmaf(w, v.w, acc.w);
        }
      }
      const float inv = L > 0.f ? 1.f / L : 0.f;   // 0 times a NaN output stays NaN
      acc = make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
      if (lane == 0 && a.lens[seq] - (a.n_q - 1 - j) <= 0) set_status(a.status, PQ_ERR_EMPTY);   // a query that sees no token: zeros
    }
    *reinterpret_cast<float4*>(x + 4 * i) = acc;
  }
  __syncthreads();
  store_unrotated<kTile>(x, s, row0, n_rows, lane, warp, a.out, a.io_dtype);
}

// Launches `kernel` as a programmatic dependent (it waits inside for the kernel before it in the stream).
template <class... Params, class... Args>
static int32_t launch_dependent(void (*kernel)(Params...), dim3 grid, int threads, int smem, cudaStream_t stream, Args... args) {
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
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
  if (e != cudaSuccess) {
    note_cuda_error(e);
    cudaGetLastError();
    return PQ_ERR_CUDA;
  }
  return launch_status();
}

// `launch` with the tile for the number of rows as a constant, and the device's SMs.
template <class Launch>
static int32_t with_rot_tile(int64_t n_rows, Launch launch) {
  static DeviceMemo sm_count;
  const int n_sm = sm_count_of_device(sm_count);
  if (n_sm == 0) return PQ_ERR_CUDA;
  if (n_rows <= 8 * (int64_t)n_sm) return launch(std::integral_constant<int, 8>{}, n_sm);
  if (n_rows <= 16 * (int64_t)n_sm) return launch(std::integral_constant<int, 16>{}, n_sm);
  if (n_rows <= 32 * (int64_t)n_sm) return launch(std::integral_constant<int, 32>{}, n_sm);
  return launch(std::integral_constant<int, 64>{}, n_sm);
}
template <int kTile, typename... Params, typename... Args>
static int32_t launch_rot_kernel(void (*kernel)(Params...), DeviceMemo& configured, int64_t n_rows, int n_sm, cudaStream_t stream, Args... args) {
  if (configure_for_device(kernel, kRotAlone, configured) == 0) return PQ_ERR_CUDA;
  return launch_dependent(kernel, dim3((unsigned)((n_rows + kTile - 1) / kTile)), kRotThreads, rot_smem_bytes<kTile>(n_rows, n_sm), stream, args...);
}
static int32_t launch_rotate(const float* S, const void* q, int io_dtype, int64_t n_rows, float factor, __half* qrot, cudaStream_t stream) {
  return with_rot_tile(n_rows, [&](auto tile, int n_sm) {
    static DeviceMemo configured;
    return launch_rot_kernel<tile>(rotate_rows_kernel<tile>, configured, n_rows, n_sm, stream, S, q, io_dtype, n_rows, factor, qrot);
  });
}
static int32_t launch_unrotate(const float* S, const float* parts, const float* lse, int n_parts, int64_t n_rows, void* out, int out_dtype,
                               int32_t* status, cudaStream_t stream) {
  return with_rot_tile(n_rows, [&](auto tile, int n_sm) {
    static DeviceMemo configured;
    return launch_rot_kernel<tile>(merge_unrotate_kernel<tile>, configured, n_rows, n_sm, stream, S, parts, lse, n_parts, n_rows, out, out_dtype,
                                   status);
  });
}
static int32_t launch_merge_rows(const DecodeArgs& a, cudaStream_t stream) {
  const int64_t n_rows = (int64_t)a.batch * a.n_q_heads;
  return with_rot_tile(n_rows, [&](auto tile, int n_sm) {
    static DeviceMemo configured;
    return launch_rot_kernel<tile>(merge_rows_kernel<tile>, configured, n_rows, n_sm, stream, a.S, a);
  });
}

}  // namespace pq
