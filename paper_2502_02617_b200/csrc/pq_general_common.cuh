// The general row layout (any recursion depth and bits per level) and what its encoder and its readers share.
#pragma once
#include <math_constants.h>

#include "pq_common.cuh"

namespace pq {

constexpr int kGenMaxLevels = PQ_GENERAL_MAX_LEVELS;
constexpr int kGenMaxBits = 6;
constexpr int kGenMaxDim = 256;
constexpr int kGenMaxCentroids = kGenMaxLevels << kGenMaxBits;

// A validated configuration with the derived sizes.  A row (one token of one head, K or V) holds, per level, the
// level's d / 2^l codes as one bit stream (code i at bits [i b, (i + 1) b), least significant first, padded to a
// byte), then padding to an even offset, then the d / 2^L block radii in fp16.  The cache is
// [sequence][kv head][K | V][token][row_bytes].
struct GenConfig {
  int d, L, nb, n_codes, n_cen, row_bytes, rad_off;
  int bits[kGenMaxLevels], cen_off[kGenMaxLevels], bnd_off[kGenMaxLevels], code_off[kGenMaxLevels], byte_off[kGenMaxLevels],
      level_bytes[kGenMaxLevels];
};

struct GenEncodeArgs {
  GenConfig g;
  const void* K;
  const void* V;
  int in_dtype;
  int64_t token_stride, head_stride;
  const int32_t* cu_seqlens;   // nullptr: one row per sequence
  int batch, total_tokens, n_kv_heads, capacity;
  const float* S;
  const double* boundaries;    // of all levels, concatenated
  uint8_t* cache;
  const int32_t* lens;
  int32_t* status;
  int packed;                  // 1: the planes of the packed cache (pg, head_dim < 128), 0: general rows
  Paging pg;
};

// Encode into the packed cache at head dims below 128 (levels and bits of Section 4.1); a.g and a.packed are filled in.
int32_t launch_packed_encode(GenEncodeArgs a, int head_dim, cudaStream_t stream);

// Would the block radius r round to another fp16 value if it moved by its error?  (NaN and infinite r: yes; near saturation: yes, it
// is counted from the exact value.)  `err` bounds the 2-norm of the error of the block's rotated coordinates, and so the error that
// their rotation brings into r; the sums of squares and the square root add less than 8 roundings of 2^-24, below 5e-7 r.
__device__ __forceinline__ bool radius_unsure(float r, float err) {
  const float slack = fmaf(5e-7f, r, err), lo = fminf(r - slack, 65504.f), hi = fminf(r + slack, 65504.f);
  return !(r < CUDART_INF_F) || __half_as_ushort(__float2half_rn(fmaxf(lo, 0.f))) != __half_as_ushort(__float2half_rn(hi)) || !(r <= 65000.f);
}
// That bound for y = x S summed in `slices` chains of `chain` fused multiply-adds whose results are added one by one, relative to
// ||x||_2: the rounding of step m of a chain moves the coordinates of any block by at most 2^-24 times the norm of the partial sums,
// which is at most that of the slice of x (the rows and columns of an orthogonal S that meet there have spectral norm 1 or less);
// the slices' norms add up to sqrt(slices) ||x|| at most, and each of the additions moves the block by 2^-24 ||x||.  2 % for the
// rounding of S and second order.
__host__ __device__ constexpr float const_sqrt(int n) {   // of 1, 2, 4, 8, 16 exactly enough, rounded up
  return n <= 1 ? 1.f : n <= 2 ? 1.4143f : n <= 4 ? 2.f : n <= 8 ? 2.8285f : 4.f;
}
__host__ __device__ constexpr float rotation_block_error(int chain, int slices) {
  return 1.02f * (chain * const_sqrt(slices) + slices) * 5.9604644775390625e-08f;
}

// (cos x, sin x) for 0 <= x <= 2 pi, rounded once to float32 from a float64 evaluation: x is reduced by a multiple of
// pi/2 and both functions of the remainder r (|r| <= pi/4) are summed from their Taylor series; the first terms left
// out are r^14 / 14! and r^13 / 13!, below 7e-12.  The float64 pipe is slow here: 16 operations against several times
// that in the library's full-precision functions, for tables that every thread block fills.
__device__ __forceinline__ float2 cos_sin_table(double x) {
  const double k = rint(x * 0.63661977236758134308);   // 2 / pi
  const double r = fma(-k, 1.57079632679489661923, x), z = r * r;
  double c = fma(z, 1.0 / 479001600.0, -1.0 / 3628800.0);
  c = fma(c, z, 1.0 / 40320.0);
  c = fma(c, z, -1.0 / 720.0);
  c = fma(c, z, 1.0 / 24.0);
  c = fma(c, z, -0.5);
  c = fma(c, z, 1.0);
  double s = fma(z, -1.0 / 39916800.0, 1.0 / 362880.0);
  s = fma(s, z, -1.0 / 5040.0);
  s = fma(s, z, 1.0 / 120.0);
  s = fma(s, z, -1.0 / 6.0);
  s = fma(s * z, r, r);
  const int q = (int)k & 3;
  const float cf = (float)c, sf = (float)s;
  const float a = (q & 1) ? sf : cf, b = (q & 1) ? cf : sf;
  return make_float2((q == 1 || q == 2) ? -a : a, (q & 2) ? -b : b);
}

}  // namespace pq
