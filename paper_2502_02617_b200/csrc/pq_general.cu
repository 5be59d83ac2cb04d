// General recursion depth and bit tables (Definition 1 and Algorithm 1 with any L <= log2 d levels and any bits per
// level; Section 4 counts b_FPN + (d - 1) b bits per vector for L = log2 d and b bits everywhere).  The encoder decides
// in float32 with certified margins and takes the rest in float64 (pq_encode_general.cuh), attention is float32
// throughout (pq_split_attention.cuh).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <math_constants.h>
#include <vector>

#include "pq_encode_general.cuh"
#include "pq_split_attention.cuh"

namespace pq {

static int32_t make_gen_config(const pq_general_config* c, GenConfig* g) {
  if (c == nullptr) return PQ_ERR_INVALID_ARG;
  const int d = c->head_dim, L = c->n_levels;
  if (d < 2 || d > kGenMaxDim || (d & (d - 1)) || L < 1 || L > kGenMaxLevels || (1 << L) > d) return PQ_ERR_UNSUPPORTED;
  std::memset(g, 0, sizeof(*g));
  g->d = d; g->L = L; g->nb = d >> L; g->n_codes = d - g->nb;
  int cen = 0, bnd = 0, code = 0, byte = 0;
  for (int l = 0; l < L; ++l) {
    const int b = c->bits[l];
    if (b < 1 || b > kGenMaxBits) return PQ_ERR_UNSUPPORTED;
    g->bits[l] = b;
    g->cen_off[l] = cen; g->bnd_off[l] = bnd; g->code_off[l] = code; g->byte_off[l] = byte;
    g->level_bytes[l] = ((d >> (l + 1)) * b + 7) / 8;
    cen += 1 << b; bnd += (1 << b) - 1; code += d >> (l + 1); byte += g->level_bytes[l];
  }
  g->n_cen = cen;
  g->rad_off = (byte + 1) & ~1;
  g->row_bytes = g->rad_off + 2 * g->nb;
  return PQ_OK;
}

__host__ __device__ inline int64_t gen_row_offset(const GenConfig& g, int n_kv_heads, int capacity, int b, int h, int kv, int tok) {
  return ((((int64_t)b * n_kv_heads + h) * 2 + kv) * capacity + tok) * g.row_bytes;
}

// Code `idx` of level l (0-based) of a row.
__device__ __forceinline__ uint32_t gen_get_code(const uint8_t* row, const GenConfig& g, int l, int idx) {
  const int bit = idx * g.bits[l];
  const uint8_t* p = row + g.byte_off[l] + (bit >> 3);
  const uint32_t two = (uint32_t)p[0] | ((bit & 7) + g.bits[l] > 8 ? (uint32_t)p[1] << 8 : 0u);
  return (two >> (bit & 7)) & ((1u << g.bits[l]) - 1u);
}

// Rotated coordinate i of a row: the block radius times, level by level from the top, cos or sin of the centroid of
// the angle above coordinate i (Algorithm 1, DeQuant).
__device__ __forceinline__ float gen_decode_coord(const uint8_t* row, const GenConfig& g, int i, const float* cen_cos,
                                                  const float* cen_sin) {
  float v = __half2float(reinterpret_cast<const __half*>(row + g.rad_off)[i >> g.L]);
  for (int l = g.L - 1; l >= 0; --l) {
    const uint32_t code = gen_get_code(row, g, l, i >> (l + 1));
    v *= ((i >> l) & 1) ? cen_sin[g.cen_off[l] + code] : cen_cos[g.cen_off[l] + code];
  }
  return v;
}

__global__ void gen_advance_lens_kernel(const int32_t* cu_seqlens, int batch, int capacity, int32_t* lens) {
  asm volatile("griddepcontrol.wait;" ::: "memory");   // launched ahead of time: the encoder reads the lengths
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= batch) return;
  const int count = cu_seqlens[b + 1] - cu_seqlens[b], start = lens[b];
  if (start >= 0 && start + count <= capacity) lens[b] = start + count;
}

__global__ void gen_unpack_kernel(GenConfig g, int n_kv_heads, const uint8_t* cache, int batch, int capacity, int n_tokens,
                                  uint8_t* codes, __half* radii) {
  const int64_t n = (int64_t)batch * n_kv_heads * 2 * n_tokens;
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  const int tok = (int)(v % n_tokens), kv = (int)((v / n_tokens) & 1);
  const int h = (int)((v / (2 * (int64_t)n_tokens)) % n_kv_heads), b = (int)(v / (2 * (int64_t)n_tokens * n_kv_heads));
  const uint8_t* row = cache + gen_row_offset(g, n_kv_heads, capacity, b, h, kv, tok);
  for (int l = 0; l < g.L; ++l)
    for (int i = 0; i < (g.d >> (l + 1)); ++i) codes[v * g.n_codes + g.code_off[l] + i] = (uint8_t)gen_get_code(row, g, l, i);
  for (int i = 0; i < g.nb; ++i) radii[v * g.nb + i] = reinterpret_cast<const __half*>(row + g.rad_off)[i];
}

// DeQuant of one vector per thread block, including the final S^T.
__global__ void gen_dequant_kernel(GenConfig g, int n_kv_heads, const float* S, const double* centroids, const uint8_t* cache,
                                   int capacity, int n_tokens, float* x_hat) {
  __shared__ float cc[kGenMaxCentroids], cs[kGenMaxCentroids], ys[kGenMaxDim];
  const int j = threadIdx.x, d = g.d;
  for (int i = j; i < g.n_cen; i += blockDim.x) {
    const float2 e = cos_sin_table(centroids[i]);
    cc[i] = e.x;
    cs[i] = e.y;
  }
  __syncthreads();
  const int64_t v = blockIdx.x;
  const int tok = (int)(v % n_tokens), kv = (int)((v / n_tokens) & 1);
  const int h = (int)((v / (2 * (int64_t)n_tokens)) % n_kv_heads), b = (int)(v / (2 * (int64_t)n_tokens * n_kv_heads));
  const uint8_t* row = cache + gen_row_offset(g, n_kv_heads, capacity, b, h, kv, tok);
  if (j < d) ys[j] = gen_decode_coord(row, g, j, cc, cs);
  __syncthreads();
  if (j < d) {
    float acc = 0.f;
    for (int k = 0; k < d; ++k) acc = fmaf(ys[k], __ldg(S + (int64_t)j * d + k), acc);
    x_hat[v * d + j] = acc;
  }
}

// General rows for split_attention_kernel.  Rows are only 2-byte aligned: a tile is copied as the aligned 16-byte pieces that
// hold a byte of it, to the same position modulo 16 in the buffer.  (An aligned 16-byte piece never crosses the end of an
// allocation, so the few bytes beside the tile are readable; they are not used.)
// kSub = min(L, 4): the levels inside a group of 16 coordinates (the angles above it are walked one by one).  kB: bits per
// angle where every level has the same number (2, 3 or 4: shifts and masks become constants; eight sequences of 4096 tokens, 32/8 heads of
// 128: 102.6 -> 92.5, 102.6 -> 93.6 and 103.5 -> 92.4 us), 0 for any table.
template <int kSub, int kB>
struct GenSplit {
  static constexpr bool kEarlyTables = false, kPairs = false;
  static constexpr int kTabMax = kB ? kGenMaxLevels << kB : kGenMaxCentroids, kDim = 0;
  SplitCommon c;
  GenConfig g;
  int capacity;
  const double* centroids;
  const uint8_t* cache;
  const int32_t* lens;

  int tile_bytes(int n) const { return (n * g.row_bytes + 15 + 8 + 15) & ~15; }   // + the shift, + what a window reads past a row
  __device__ __forceinline__ int len(int pair) const { return max(0, min(lens[pair], capacity)); }
  __device__ __forceinline__ void fill_tables(float2* tab, int tid) const {
    for (int i = tid; i < g.n_cen; i += blockDim.x) tab[i] = cos_sin_table(centroids[i]);
  }
  __device__ __forceinline__ int64_t row_offset(int pair, int hk, int kv, int t) const {
    return gen_row_offset(g, c.n_kv_heads, capacity, pair, hk, kv, t);
  }
  __device__ __forceinline__ int shift(int pair, int hk, int kv, int t0) const {
    return (int)((reinterpret_cast<uintptr_t>(cache) + row_offset(pair, hk, kv, t0)) & 15);
  }
  __device__ __forceinline__ void stage(uint8_t* buf, int pair, int hk, int kv, int t0, int n, int lane) const {
    const uint8_t* src = cache + row_offset(pair, hk, kv, t0);
    const int sh = (int)(reinterpret_cast<uintptr_t>(src) & 15);
    src -= sh;
#pragma unroll 1
    for (int i = 16 * lane; i < sh + n * g.row_bytes; i += 512) split_cp16(buf + i, src + i);
  }
  __device__ __forceinline__ int bits(int l) const { return kB ? kB : g.bits[l]; }
  __device__ __forceinline__ const float2* level(const float2* tab, int l) const { return tab + (kB ? l << kB : g.cen_off[l]); }
  // 32 bits from bit `bit` of the row at buf + row on
  __device__ __forceinline__ static uint32_t window(const uint8_t* buf, int row, int bit) {
    const int at = row + (bit >> 3);
    const uint32_t* w = reinterpret_cast<const uint32_t*>(buf + (at & ~3));
    return __funnelshift_r(w[0], w[1], ((at & 3) << 3) + (bit & 7));
  }
  template <int kU>
  __device__ __forceinline__ void decode(const uint8_t* buf, int at, int t, int unit, const float2* tab, const float4*, float* y) const {
    constexpr int kTop = kU == 16 ? 4 : 3;                 // levels a unit of kU coordinates spans
    constexpr int kIn = kSub < kTop ? kSub : kTop;         // ... and those of them that exist
    constexpr int kBlk = kU >> kIn;                        // subtrees whose root starts inside the unit
    const int row = at + t * g.row_bytes;
    const __half* radii = reinterpret_cast<const __half*>(buf + row + g.rad_off);
    float v[kU];
    if (kIn == kTop) {
      float r = __half2float(radii[unit >> (g.L - kTop)]);
      for (int l = g.L - 1; l >= kTop; --l) {   // the angles above the unit
        const int b = bits(l);
        const uint32_t code = window(buf, row, g.byte_off[l] * 8 + (unit >> (l + 1 - kTop)) * b) & ((1u << b) - 1u);
        const float2 cs = level(tab, l)[code];
        r *= (unit >> (l - kTop)) & 1 ? cs.y : cs.x;
      }
      v[0] = r;
    } else {
#pragma unroll
      for (int j = 0; j < kBlk; ++j) {
        const int blk = unit * kBlk + j;
        v[j] = blk < g.nb ? __half2float(radii[blk]) : 0.f;
      }
    }
#pragma unroll
    for (int l = kIn - 1; l >= 0; --l) {
      constexpr int kAngles = kU / 2;
      const int n = kAngles >> l, b = bits(l), bit = g.byte_off[l] * 8 + unit * n * b;   // n angles of the level in the unit
      const uint32_t mask = (1u << b) - 1u;
      const float2* entry = level(tab, l);
      const uint32_t w = window(buf, row, bit);
      uint32_t w2 = 0u;
      if (n == 8) w2 = b <= 4 ? w >> (4 * b) : window(buf, row, bit + 4 * b);   // 8 codes of up to 6 bits
#pragma unroll
      for (int j = n - 1; j >= 0; --j) {
        const float2 cs = entry[((j < 4 ? w : w2) >> ((j & 3) * b)) & mask];
        const float r = v[j];
        v[2 * j] = r * cs.x;
        v[2 * j + 1] = r * cs.y;
      }
    }
#pragma unroll
    for (int i = 0; i < kU; ++i) y[i] = v[i];
  }
};

template <int kSub, int kB>
static int32_t launch_gen_attention_as(const GenConfig& g, const SplitCommon& c, int batch, int capacity, const double* centroids,
                                       const void* cache, const int32_t* lens, cudaStream_t stream) {
  GenSplit<kSub, kB> p;
  p.c = c; p.g = g; p.capacity = capacity; p.centroids = centroids; p.cache = reinterpret_cast<const uint8_t*>(cache); p.lens = lens;
  return dispatch_split_attention(p, batch, capacity, stream);
}
static int32_t launch_gen_attention(const GenConfig& g, const SplitCommon& c, int batch, int capacity, const double* centroids,
                                    const void* cache, const int32_t* lens, cudaStream_t s) {
  bool same = true;
  for (int l = 1; l < g.L; ++l) same = same && g.bits[l] == g.bits[0];
  if (g.L >= 4 && same && g.bits[0] == 2) return launch_gen_attention_as<4, 2>(g, c, batch, capacity, centroids, cache, lens, s);
  if (g.L >= 4 && same && g.bits[0] == 3) return launch_gen_attention_as<4, 3>(g, c, batch, capacity, centroids, cache, lens, s);
  if (g.L >= 4 && same && g.bits[0] == 4) return launch_gen_attention_as<4, 4>(g, c, batch, capacity, centroids, cache, lens, s);
  switch (g.L < 4 ? g.L : 4) {
    case 1: return launch_gen_attention_as<1, 0>(g, c, batch, capacity, centroids, cache, lens, s);
    case 2: return launch_gen_attention_as<2, 0>(g, c, batch, capacity, centroids, cache, lens, s);
    case 3: return launch_gen_attention_as<3, 0>(g, c, batch, capacity, centroids, cache, lens, s);
    default: return launch_gen_attention_as<4, 0>(g, c, batch, capacity, centroids, cache, lens, s);
  }
}

int32_t launch_packed_encode(GenEncodeArgs a, int head_dim, cudaStream_t stream) {
  pq_general_config cfg = {head_dim, 4, {4, 2, 2, 2}};
  const int32_t st = make_gen_config(&cfg, &a.g);
  if (st != PQ_OK) return st;
  a.packed = 1;
  return launch_gen_encode(a, stream);
}

}  // namespace pq

namespace {
const double kPiG = 3.14159265358979323846264338327950288;
// Lloyd-Max centroids of the level's analytic density (Lemma 2) by Simpson quadrature; level is 1-based.
void gen_fit_level(int level, int n, double* theta, double* beta) {
  const double lo = 0.0, hi = level == 1 ? 2.0 * kPiG : 0.5 * kPiG;
  const int expo = (1 << (level - 1)) - 1;
  auto moments = [&](double a, double b, double* m0, double* m1) {
    const int panels = 2048;
    const double h = (b - a) / panels;
    double s0 = 0.0, s1 = 0.0;
    for (int i = 0; i <= panels; ++i) {
      const double p = a + h * i, w = (i == 0 || i == panels) ? 1.0 : ((i & 1) ? 4.0 : 2.0);
      const double f = level == 1 ? 1.0 : std::pow(std::sin(2.0 * p), expo);
      s0 += w * f;
      s1 += w * f * p;
    }
    *m0 = s0 * h / 3.0;
    *m1 = s1 * h / 3.0;
  };
  for (int k = 0; k < n; ++k) theta[k] = lo + (k + 0.5) * (hi - lo) / n;
  if (level > 1) {  // start inside the bulk of the density (it concentrates around pi/4 as the level grows)
    const double width = 4.0 / std::sqrt((double)(expo + 1));
    for (int k = 0; k < n; ++k) theta[k] = 0.25 * kPiG + (k + 0.5 - 0.5 * n) * std::fmin(hi / n, width / n);
  }
  for (int it = 0; it < 100000; ++it) {
    double delta = 0.0;
    for (int k = 0; k + 1 < n; ++k) beta[k] = 0.5 * (theta[k] + theta[k + 1]);
    for (int k = 0; k < n; ++k) {
      const double a = k == 0 ? lo : beta[k - 1], b = k == n - 1 ? hi : beta[k];
      double m0, m1;
      moments(a, b, &m0, &m1);
      const double t = m0 > 0.0 ? m1 / m0 : 0.5 * (a + b);
      delta = std::fmax(delta, std::fabs(t - theta[k]));
      theta[k] = t;
    }
    if (delta < 1e-14) break;
  }
  for (int k = 0; k + 1 < n; ++k) beta[k] = 0.5 * (theta[k] + theta[k + 1]);
}
}  // namespace

extern "C" {

int32_t pq_general_sizes(const pq_general_config* cfg, int32_t* n_centroids, int32_t* n_boundaries, int32_t* n_codes,
                         int32_t* n_radii, int32_t* row_bytes) {
  pq::GenConfig g;
  const int32_t st = pq::make_gen_config(cfg, &g);
  if (st != PQ_OK) return st;
  if (n_centroids) *n_centroids = g.n_cen;
  if (n_boundaries) *n_boundaries = g.n_cen - g.L;
  if (n_codes) *n_codes = g.n_codes;
  if (n_radii) *n_radii = g.nb;
  if (row_bytes) *row_bytes = g.row_bytes;
  return PQ_OK;
}

int32_t pq_general_fit_codebooks(const pq_general_config* cfg, double* centroids_host, double* boundaries_host) {
  pq::GenConfig g;
  const int32_t st = pq::make_gen_config(cfg, &g);
  if (st != PQ_OK) return st;
  if (centroids_host == nullptr || boundaries_host == nullptr) return PQ_ERR_INVALID_ARG;
  for (int l = 0; l < g.L; ++l) gen_fit_level(l + 1, 1 << g.bits[l], centroids_host + g.cen_off[l], boundaries_host + g.bnd_off[l]);
  return PQ_OK;
}

int64_t pq_general_cache_bytes(const pq_general_config* cfg, int32_t batch, int32_t n_kv_heads, int32_t capacity) {
  pq::GenConfig g;
  const int32_t st = pq::make_gen_config(cfg, &g);
  if (st != PQ_OK) return st;
  if (batch <= 0 || n_kv_heads <= 0 || capacity <= 0) return PQ_ERR_INVALID_ARG;
  return (int64_t)batch * n_kv_heads * 2 * capacity * g.row_bytes;
}

int32_t pq_general_encode_kv(const pq_general_config* cfg, int32_t n_kv_heads, const float* S_dev,
                             const double* boundaries_dev, const void* K_dev, const void* V_dev, int32_t in_dtype,
                             int64_t token_stride, int64_t head_stride, const int32_t* cu_seqlens_dev, int32_t batch,
                             int32_t total_tokens, void* cache_dev, int32_t* cache_lens_dev, int32_t capacity,
                             int32_t* status_dev, void* stream) {
  pq::GenEncodeArgs a;
  const int32_t st = pq::make_gen_config(cfg, &a.g);
  if (st != PQ_OK) return st;
  if (!S_dev || !boundaries_dev || !K_dev || !V_dev || !cu_seqlens_dev || !cache_dev || !cache_lens_dev || !status_dev)
    return PQ_ERR_INVALID_ARG;
  if (n_kv_heads <= 0 || batch <= 0 || total_tokens < 0 || capacity <= 0 || token_stride < 0 || head_stride < 0) return PQ_ERR_INVALID_ARG;
  if (in_dtype != PQ_DTYPE_F32 && in_dtype != PQ_DTYPE_BF16) return PQ_ERR_UNSUPPORTED;
  if ((int64_t)total_tokens * 2 * n_kv_heads >= (1ll << 31)) return PQ_ERR_UNSUPPORTED;
  if (((uintptr_t)boundaries_dev & 7) || ((uintptr_t)cache_dev & 1)) return PQ_ERR_ALIGNMENT;
  if (total_tokens == 0) return PQ_OK;
  a.K = K_dev; a.V = V_dev; a.in_dtype = in_dtype; a.token_stride = token_stride; a.head_stride = head_stride;
  a.cu_seqlens = cu_seqlens_dev; a.batch = batch; a.total_tokens = total_tokens; a.n_kv_heads = n_kv_heads; a.capacity = capacity;
  a.S = S_dev; a.boundaries = boundaries_dev; a.cache = reinterpret_cast<uint8_t*>(cache_dev); a.lens = cache_lens_dev;
  a.status = status_dev;
  a.packed = 0;
  a.pg = pq::contiguous_paging(capacity, batch);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int32_t launched = pq::launch_gen_encode(a, s);
  if (launched != PQ_OK) return launched;
  // the length update as a programmatic dependent launch of the encode kernel (its launch latency is hidden)
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3((batch + 127) / 128);
  lc.blockDim = dim3(128);
  lc.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = attr;
  lc.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&lc, pq::gen_advance_lens_kernel, cu_seqlens_dev, (int)batch, (int)capacity, cache_lens_dev);
  if (e != cudaSuccess) {
    pq::note_cuda_error(e);
    cudaGetLastError();
    return PQ_ERR_CUDA;
  }
  return pq::launch_status();
}

int32_t pq_general_decode_attention(const pq_general_config* cfg, int32_t n_q_heads, int32_t n_kv_heads, const float* S_dev,
                                    const double* centroids_dev, const void* q_dev, int32_t io_dtype, const void* cache_dev,
                                    const int32_t* cache_lens_dev, int32_t batch, int32_t capacity, float scale,
                                    void* out_dev, int32_t* status_dev, void* stream) {
  pq::GenConfig g;
  const int32_t st = pq::make_gen_config(cfg, &g);
  if (st != PQ_OK) return st;
  if (!S_dev || !centroids_dev || !q_dev || !cache_dev || !cache_lens_dev || !out_dev || !status_dev) return PQ_ERR_INVALID_ARG;
  if (batch <= 0 || batch > 65535 || n_q_heads <= 0 || n_kv_heads <= 0 || capacity <= 0 || n_q_heads % n_kv_heads) return PQ_ERR_INVALID_ARG;
  if (n_q_heads / n_kv_heads > pq::kMaxGroup) return PQ_ERR_UNSUPPORTED;
  if (io_dtype != PQ_DTYPE_F32 && io_dtype != PQ_DTYPE_BF16) return PQ_ERR_UNSUPPORTED;
  if (((uintptr_t)centroids_dev & 7) || ((uintptr_t)cache_dev & 1)) return PQ_ERR_ALIGNMENT;
  pq::SplitCommon c;
  c.d = g.d; c.n_q_heads = n_q_heads; c.n_kv_heads = n_kv_heads; c.io_dtype = io_dtype; c.scale = scale;
  c.S = S_dev; c.q = q_dev; c.out = out_dev; c.lse = nullptr; c.status = status_dev;
  return pq::launch_gen_attention(g, c, batch, capacity, centroids_dev, cache_dev, cache_lens_dev,
                                  reinterpret_cast<cudaStream_t>(stream));
}

int32_t pq_general_unpack_codes(const pq_general_config* cfg, int32_t n_kv_heads, const void* cache_dev, int32_t batch,
                                int32_t capacity, int32_t n_tokens, uint8_t* codes_dev, void* radii_dev, void* stream) {
  pq::GenConfig g;
  const int32_t st = pq::make_gen_config(cfg, &g);
  if (st != PQ_OK) return st;
  if (!cache_dev || !codes_dev || !radii_dev || batch <= 0 || n_kv_heads <= 0 || n_tokens <= 0 || n_tokens > capacity)
    return PQ_ERR_INVALID_ARG;
  const int64_t n = (int64_t)batch * n_kv_heads * 2 * n_tokens;
  pq::gen_unpack_kernel<<<(unsigned)((n + 127) / 128), 128, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      g, n_kv_heads, reinterpret_cast<const uint8_t*>(cache_dev), batch, capacity, n_tokens, codes_dev,
      reinterpret_cast<__half*>(radii_dev));
  return pq::launch_status();
}

int32_t pq_general_dequant_kv(const pq_general_config* cfg, int32_t n_kv_heads, const float* S_dev, const double* centroids_dev,
                              const void* cache_dev, int32_t batch, int32_t capacity, int32_t n_tokens, float* x_hat_dev,
                              void* stream) {
  pq::GenConfig g;
  const int32_t st = pq::make_gen_config(cfg, &g);
  if (st != PQ_OK) return st;
  if (!S_dev || !centroids_dev || !cache_dev || !x_hat_dev || batch <= 0 || n_kv_heads <= 0 || n_tokens <= 0 || n_tokens > capacity)
    return PQ_ERR_INVALID_ARG;
  const int64_t n = (int64_t)batch * n_kv_heads * 2 * n_tokens;
  if (n >= (1ll << 31)) return PQ_ERR_UNSUPPORTED;
  pq::gen_dequant_kernel<<<(unsigned)n, g.d < 32 ? 32 : g.d, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      g, n_kv_heads, S_dev, centroids_dev, reinterpret_cast<const uint8_t*>(cache_dev), capacity, n_tokens, x_hat_dev);
  return pq::launch_status();
}

}  // extern "C"
