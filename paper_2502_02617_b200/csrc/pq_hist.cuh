// Histograms of the observed angles (the sample the "online" codebook of Section 4.1 is clustered on); included by
// pq_encode.cu.  The angles of Algorithm 1's Polar are formed in float32 from the rotated coordinates and counted per
// level in n_bins bins of equal width over the level's range ([0, 2 pi) at level 1, [0, pi/2] above).  Against a
// float64 evaluation an angle within the float32 error of a bin edge (about 1e-5 rad) may fall in the neighbouring
// bin; the clustering sees a sample moved by less than a bin.
#pragma once

namespace pq {

constexpr int kHistMaxBins = PQ_HIST_MAX_BINS;

// Two of them at a time: the packed float32 instructions halve the polynomial's issue slots, and the chains of a block overlap.
// atan(t) for t in [0, 1]: t * P(t^2), P of degree 5 fitted by least squares at Chebyshev nodes; the absolute error is
// below 2e-6 rad, a few thousandths of the narrowest bin.
__device__ __forceinline__ void hist_atan01(float& t0, float& t1) {
  const uint64_t t = f2_pack(t0, t1), z = f2_mul(t, t);
  auto both = [](float c) { return f2_pack(c, c); };
  uint64_t p = both(-0.011465809307992458f);
  p = f2_fma(p, z, both(0.05195053294301033f));
  p = f2_fma(p, z, both(-0.1157294437289238f));
  p = f2_fma(p, z, both(0.19323529303073883f));
  p = f2_fma(p, z, both(-0.33256831765174866f));
  p = f2_fma(p, z, both(0.9999744892120361f));
  f2_unpack(f2_mul(p, t), t0, t1);
}

__device__ __forceinline__ float hist_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// The tangent of the angle of (b, a) folded into [0, pi/4] (0 for a = b = 0), and the bin of the angle from the folded one:
// of atan2(b, a) in [0, 2 pi), `scale` = n_bins / (2 pi), and of atan2(sqrt(sb), sqrt(sa)) in [0, pi/2] from the squared
// radii, `scale` = n_bins / (pi/2).
__device__ __forceinline__ float hist_fold_level1(float a, float b) {
  const float ax = fabsf(a), ay = fabsf(b), u = fmaxf(ax, ay);
  return u > 0.f ? fminf(fminf(ax, ay) * hist_rcp(u), 1.f) : 0.f;
}
__device__ __forceinline__ int hist_bin_level1(float phi, float a, float b, float scale, int n_bins) {
  if (fabsf(b) > fabsf(a)) phi = 1.57079632679489662f - phi;
  if (a < 0.f) phi = 3.14159265358979324f - phi;
  if (b < 0.f) phi = 6.28318530717958648f - phi;
  return min((int)(phi * scale), n_bins - 1);
}
__device__ __forceinline__ float hist_fold_upper(float sa, float sb) {
  const float M = fmaxf(sa, sb);
  // the approximate root's errors of 1e-7 stand beside the polynomial's 2e-6: centroids of 1024 to 16384 tokens differ from those of
  // float64 angles by 4.51e-6 at most (0.0394 % of the counts in another bin), with IEEE roots by 4.54e-6 (0.0395 %)
  return M > 0.f ? fminf(fast_sqrt(fminf(sa, sb) * hist_rcp(M)), 1.f) : 0.f;
}
__device__ __forceinline__ int hist_bin_upper(float phi, float sa, float sb, float scale, int n_bins) {
  if (sb > sa) phi = 1.57079632679489662f - phi;
  return min((int)(phi * scale), n_bins - 1);
}

// Count the 15 angles of one 16-coordinate block into h[level - 1][bin] (shared or global 32-bit counters).
// A block with a non-finite coordinate (or an overflowing norm) is skipped and reported by the return value.
__device__ __forceinline__ bool hist_block(const float* y, uint32_t* h, int n_bins, float scale1, float scale_up) {
  float s1[8], s2[4], s3[2];
#pragma unroll
  for (int j = 0; j < 8; ++j) s1[j] = fmaf(y[2 * j], y[2 * j], y[2 * j + 1] * y[2 * j + 1]);
#pragma unroll
  for (int j = 0; j < 4; ++j) s2[j] = s1[2 * j] + s1[2 * j + 1];
  s3[0] = s2[0] + s2[1];
  s3[1] = s2[2] + s2[3];
  if (!(s3[0] + s3[1] < CUDART_INF_F)) return false;
  // all fifteen bins first (independent dependency chains that overlap), then the fifteen counts
  int bin[16];
  auto upper = [&](int j, float* sa, float* sb) {   // the radii of angle j = 0 .. 6 above level 1
    *sa = j < 4 ? s1[(2 * j) & 7] : j < 6 ? s2[(2 * j) & 3] : s3[0];
    *sb = j < 4 ? s1[(2 * j + 1) & 7] : j < 6 ? s2[(2 * j + 1) & 3] : s3[1];
  };
#pragma unroll
  for (int j = 0; j < 8; j += 2) {
    float t0 = hist_fold_level1(y[2 * j], y[2 * j + 1]), t1 = hist_fold_level1(y[2 * j + 2], y[2 * j + 3]);
    hist_atan01(t0, t1);
    bin[j] = hist_bin_level1(t0, y[2 * j], y[2 * j + 1], scale1, n_bins);
    bin[j + 1] = hist_bin_level1(t1, y[2 * j + 2], y[2 * j + 3], scale1, n_bins);
  }
#pragma unroll
  for (int j = 0; j < 8; j += 2) {
    float a0, b0, a1, b1;
    upper(j, &a0, &b0);
    upper(j < 6 ? j + 1 : j, &a1, &b1);
    float t0 = hist_fold_upper(a0, b0), t1 = j < 6 ? hist_fold_upper(a1, b1) : 0.f;
    hist_atan01(t0, t1);
    bin[8 + j] = (j < 4 ? 1 : j < 6 ? 2 : 3) * n_bins + hist_bin_upper(t0, a0, b0, scale_up, n_bins);
    bin[9 + j] = (j < 4 ? 1 : 2) * n_bins + hist_bin_upper(t1, a1, b1, scale_up, n_bins);   // the last one is not counted
  }
#pragma unroll
  for (int j = 0; j < 15; ++j) atomicAdd(h + bin[j], 1u);
  return true;
}

// Add a CTA's 32-bit counters to the 64-bit histogram in global memory.
__device__ inline void hist_flush(const uint32_t* h, int n, unsigned long long* out, int tid, int n_threads) {
  for (int i = tid; i < n; i += n_threads)
    if (h[i]) atomicAdd(out + i, (unsigned long long)h[i]);
}

}  // namespace pq
