// The query rotation before, and the merge and un-rotation after, the tcgen05 multi-query kernel, for all (query, head) rows of
// a call (included by pq_decode.cu): plain float32 products of [rows][128] with S or S^T, spread over all SMs.  Inside the
// attention kernel, where a CTA needs them for its own 128 rows and repeats them for every range of the blocks, they took 90 us
// of every CTA's time.
// A block of 256 threads takes kTile rows; thread = 4 columns x kTile / 8 rows (a warp shares its rows, so its reads of them
// are broadcasts, and reads 512 consecutive bytes of S).  kTile = 16 while that many blocks do not fill the device, else
// 64: bound by the shared-memory reads of S at 16 rows, by the multiply-adds at 64.
#pragma once

namespace pq {

constexpr int kRotThreads = 256, kRotSStride = 132;
template <int kTile>
constexpr int rot_smem_bytes() {
  return (128 * kRotSStride + kTile * 128) * 4;
}

// acc[r][0 .. 3] = sum_k x[r0 + r][k] s[k][4 lane .. 4 lane + 3] for the warp's kTile / 8 rows
template <int kTile>
__device__ __forceinline__ void rot_product(const float* x, const float* s, int r0, int lane, float (&out)[kTile / 8][4]) {
  uint64_t acc[kTile / 8][2];
#pragma unroll
  for (int r = 0; r < kTile / 8; ++r) acc[r][0] = acc[r][1] = 0ull;
#pragma unroll 2
  for (int k = 0; k < 128; k += 4) {
    ulonglong2 b[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) b[e] = *reinterpret_cast<const ulonglong2*>(s + (k + e) * kRotSStride + 4 * lane);
#pragma unroll
    for (int r = 0; r < kTile / 8; ++r) {
      const float4 v = *reinterpret_cast<const float4*>(x + (r0 + r) * 128 + k);
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
  for (int r = 0; r < kTile / 8; ++r) {
    f2_unpack(acc[r][0], out[r][0], out[r][1]);
    f2_unpack(acc[r][1], out[r][2], out[r][3]);
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
  float out[kTile / 8][4];
  const int r0 = warp * (kTile / 8);
  rot_product<kTile>(x, s, r0, lane, out);
#pragma unroll
  for (int r = 0; r < kTile / 8; ++r) {
    const int64_t row = row0 + r0 + r;
    if (row >= n_rows) break;
    __half hi[4], lo[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int at = ((e & 1) << 1) | (e >> 1);
      const float v = out[r][e] * factor;
      hi[at] = __float2half_rn(v);
      lo[at] = __float2half_rn(v - __half2float(hi[at]));
    }
    *reinterpret_cast<uint2*>(qrot + row * 256 + 4 * lane) = *reinterpret_cast<const uint2*>(hi);
    *reinterpret_cast<uint2*>(qrot + row * 256 + 128 + 4 * lane) = *reinterpret_cast<const uint2*>(lo);
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
  for (int i = tid; i < 128 * 32; i += kRotThreads) {
    const int n = i & 127, k = 4 * (i >> 7);   // neighbouring threads write neighbouring columns
    const float4 v = __ldg(reinterpret_cast<const float4*>(S + n * 128 + k));
    s[k * kRotSStride + n] = v.x;
    s[(k + 1) * kRotSStride + n] = v.y;
    s[(k + 2) * kRotSStride + n] = v.z;
    s[(k + 3) * kRotSStride + n] = v.w;
  }
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
  float y[kTile / 8][4];
  const int r0 = warp * (kTile / 8);
  rot_product<kTile>(x, s, r0, lane, y);
#pragma unroll
  for (int r = 0; r < kTile / 8; ++r) {
    const int64_t row = row0 + r0 + r;
    if (row >= n_rows) break;
    const int64_t at = row * 128 + 4 * lane;
    if (out_dtype == PQ_DTYPE_BF16) {
      const __nv_bfloat162 a = __floats2bfloat162_rn(y[r][0], y[r][1]), b = __floats2bfloat162_rn(y[r][2], y[r][3]);
      *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(out) + at) =
          make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
    } else {
      *reinterpret_cast<float4*>(reinterpret_cast<float*>(out) + at) = make_float4(y[r][0], y[r][1], y[r][2], y[r][3]);
    }
  }
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

template <int kTile>
static int32_t launch_rotate_as(const float* S, const void* q, int io_dtype, int64_t n_rows, float factor, __half* qrot, cudaStream_t stream) {
  static DeviceMemo configured;
  if (configure_for_device(rotate_rows_kernel<kTile>, rot_smem_bytes<kTile>(), configured) == 0) return PQ_ERR_CUDA;
  return launch_dependent(rotate_rows_kernel<kTile>, dim3((unsigned)((n_rows + kTile - 1) / kTile)), kRotThreads, rot_smem_bytes<kTile>(),
                          stream, S, q, io_dtype, n_rows, factor, qrot);
}
static int32_t launch_rotate(const float* S, const void* q, int io_dtype, int64_t n_rows, float factor, __half* qrot, cudaStream_t stream) {
  return n_rows <= 16 * 2 * 148 ? launch_rotate_as<16>(S, q, io_dtype, n_rows, factor, qrot, stream)
                                : launch_rotate_as<64>(S, q, io_dtype, n_rows, factor, qrot, stream);
}
template <int kTile>
static int32_t launch_unrotate_as(const float* S, const float* parts, const float* lse, int n_parts, int64_t n_rows, void* out, int out_dtype,
                                  int32_t* status, cudaStream_t stream) {
  static DeviceMemo configured;
  if (configure_for_device(merge_unrotate_kernel<kTile>, rot_smem_bytes<kTile>(), configured) == 0) return PQ_ERR_CUDA;
  return launch_dependent(merge_unrotate_kernel<kTile>, dim3((unsigned)((n_rows + kTile - 1) / kTile)), kRotThreads, rot_smem_bytes<kTile>(),
                          stream, S, parts, lse, n_parts, n_rows, out, out_dtype, status);
}
static int32_t launch_unrotate(const float* S, const float* parts, const float* lse, int n_parts, int64_t n_rows, void* out, int out_dtype,
                               int32_t* status, cudaStream_t stream) {
  return n_rows <= 16 * 2 * 148 ? launch_unrotate_as<16>(S, parts, lse, n_parts, n_rows, out, out_dtype, status, stream)
                                : launch_unrotate_as<64>(S, parts, lse, n_parts, n_rows, out, out_dtype, status, stream);
}

}  // namespace pq
