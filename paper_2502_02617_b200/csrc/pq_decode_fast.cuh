// Fast decode-attention kernel for head_dim 128 (included by pq_decode.cu).
//
// Persistent CTAs of 16 warps, each with a contiguous share of the (sequence, kv head) token streams.
// 128-token stages of the packed cache (K block, V block, K block, V block: one contiguous 15872-byte
// bulk copy) stream through a shared-memory ring.  The warps form two groups of 8 that take alternate
// stages; each group has two ring slots and one thread that issues its copies a stage ahead; each warp
// takes one 16-token tile of its group's stage.  (16 warps, not 17: the register file is split over
// four schedulers, and a fifth warp on one of them would cap every thread at 96 registers.)
//
// Per tile a warp
//   * decodes the keys of 16 tokens straight into mma.sync A fragments (fp16, rotated basis) with
//     shared-memory table lookups, and forms S = K_hat q'^T (tokens x heads) on tensor cores,
//   * runs the online softmax on the S fragment (log2 domain, fp32, lazily updated reference),
//   * decodes the values into A fragments (coordinates x (token, element of a decoded pair)) and
//     accumulates O^T += V_hat^T P on tensor cores (fp32 accumulators in registers).
// DeQuant (Algorithm 1) of one 16-coordinate block is a product tree r * t4 * t3 * t2 * t1.
// Levels 4..2 are folded into one lookup per half block (8 coordinates), level 1 is one lookup per byte of codes and a half2
// multiply by it:
//   U  index = the half's level-2 codes (4 bits) | level-3 code << 4 | level-4 code << 6 -> the multipliers of its four level-1
//      pairs as (half2 values, half2 rounding residuals)
//   T  index = one byte of level-1 codes (pair a = 2s | pair b = 2s+1 << 4) -> (cos a, cos b), (sin a, sin b) in fp16: a half2
//      (u_a, u_b) of the table above multiplies them element-wise; for the keys the fp16 rounding residuals of the same stand beside them
// replicated so that the lanes that read together read their own banks (16 copies of 8-byte entries, 8 of 16-byte ones).  Bound by
// the shared-memory pipe and by instruction issue together, so a lookup's work is what counts: index bytes are put together four
// at a time, and a row of both tables is 256 bytes, so that one byte permute makes an address.  One lookup per 4-coordinate sub-block at level 2..4, values and residuals of level
// 1 in tables of their own and shift-and-mask addresses took 770 instructions and 210 shared-memory wavefronts per tile (8 x 32768
// tokens, 32/8 heads: 141.4 us; now 129.4).  Without the residuals of level 1 it is 119.5 us, but the scores are then off by 1e-5 of
// their terms: the log-sum-exp by 4e-5 where it is off by 2e-6 now (2 x 4096 tokens, scores up to 16), and outputs of scores in the
// thousands by 4.5e-4 instead of 3.8e-4.  The rows and tcgen05 kernels keep a table
// per sub-block (u [4][64][16], t1hi and t1lo [256][16]): the first is bound by its start and end and the MMAs of its rows, the second
// has no room for rows of 256 bytes.
// Values use the fp16 parts only.  Keys feed the softmax exponent, where an fp16-rounded operand
// costs ~3x its relative error in the output, so they are decoded as an unevaluated sum hi + lo
// (error-free fp16 transformations with fused multiply-adds) and contracted with two MMAs.
#pragma once

namespace pq {

constexpr int kFastConsumerWarps = 16;
constexpr int kFastThreads = kFastConsumerWarps * 32;
constexpr int kStageTokens = 2 * kTokenBlock;       // 128
constexpr int kBlockBytes128 = 62 * kTokenBlock;    // 3968: one K or V token-block at d = 128
constexpr int kStageBytes = 4 * kBlockBytes128;     // 15872
constexpr int kStages = 4;                          // two per group of 8 warps
constexpr int kSpinLimit = 1 << 22;

// Tables per sub-block, of the rows and the tcgen05 kernels, and what lies behind them (bytes from a 32 KB boundary of the shared window,
// so that a table address is the OR of disjoint bit fields, base | lane replica | index, and needs no addition; a launch without
// a fixed map asks for 32 KB of slack to place them)
constexpr int kSmT1p = 0;                             // 256 * 16 * 8 = 32768
constexpr int kSmT1lo = kSmT1p + 256 * 16 * 8;        // 32768
constexpr int kSmU = kSmT1lo + 256 * 16 * 8;          // 4 * 64 * 16 * 8 = 32768
constexpr int kSmBar = kSmU + 4 * 64 * 16 * 8;        // full[4], empty[4] : 64
constexpr int kSmFlags = kSmBar + 64;                 // abort flag, is_last, n_segs, first_rank : 16
constexpr int kSmSegs = kSmFlags + 16;                // Segment[32] : 768
constexpr int kSmAlign = 32768;
static_assert(kSmT1p == 0 && kSmT1lo == 32768 && kSmU == 65536, "table addresses are formed with OR");

// q (fp32) [8][128], then q' as fp16 values and as fp16 residuals.  A head's q' takes 288 bytes, its quarters (32 coordinates
// of a fragment lane c) 72 bytes each, and the residuals start 2312 bytes after the values: the 16 lanes of a half-warp
// (two heads, value or residual, four quarters) then read 16 different bank pairs.
constexpr int kQHead = 288, kQQuarter = 72, kQLo = 8 * kQHead + 8;
constexpr int kMrgStride = 136;  // floats per (warp, head) row of the merge buffer (136 = 128 + 8: heads 8 banks apart)

// ---- shared-memory map of the persistent kernel -------------------------------------------------
// Its tables have rows of 256 bytes on 64 KB boundaries of the shared window, so that one byte permute of (index bytes, table base)
// forms a lookup's address: the index byte becomes address byte 1, the base gives the others (byte 0: the lane's replica).  What
// else the kernel keeps lies around them, at fixed places of the window (dynamic shared memory starts at kWindowBase, which the
// host asks the device for):
//   ring | T [256 bytes of level-1 codes]    8 x (cos a, cos b | sin a, sin b | their residuals) in fp16 for the keys, then 16 x
//        |                                   (cos a, cos b | sin a, sin b) for the values
//        | U [256 half-block codes]          8 x (values, residuals) of half 0, then 8 x of half 1
//        | barriers, segments, q', places of a paged segment's stages
constexpr uint32_t kWindowBase = 1024;
constexpr uint32_t kFsRing = kWindowBase, kFsT = 0x10000, kFsU = 0x20000, kFsBar = 0x30000;
constexpr uint32_t kFsFlags = kFsBar + 64, kFsSegs = kFsFlags + 16, kFsQ = kFsSegs + 768;
constexpr uint32_t kFsPlaces = kFsQ + 4096 + kQLo + 8 * kQHead;
constexpr int kFsPlaceCap = 1024;                   // stages that are listed at a time
constexpr uint32_t kFsEnd = kFsPlaces + 4 * kFsPlaceCap;
constexpr int kPlaceUnit = 256;                     // a token-block's keys and values are 31 of them
constexpr int kFsTotal = (int)(kFsEnd - kWindowBase);
// after the main loop the ring is reused for the merge across the warps, four heads at a time: their accumulators, then (m, l)
constexpr int kFsMergeMl = kFastConsumerWarps * 4 * kMrgStride * 4;
static_assert(kFsRing + kStages * kStageBytes <= kFsT && kFsMergeMl + kFastConsumerWarps * 8 * 8 <= kStages * kStageBytes, "ring");
static_assert(2 * kBlockBytes128 % kPlaceUnit == 0, "places of stages");
static_assert(kFsTotal <= 227 * 1024, "shared memory of one CTA");

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait: gives up after kSpinLimit polls (or as soon as another warp gave up) and raises
// the CTA's abort flag, so that a lost copy can never hang the GPU.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  for (int i = 0; i < kSpinLimit; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if (i > 64) {
      __nanosleep(64);
      if (*abort_flag) return false;
    }
  }
  *abort_flag = 1;
  return false;
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ uint2 lds64(uint32_t addr) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr));
  return v;
}
template <int kOff>
__device__ __forceinline__ uint32_t lds32i(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(addr), "n"(kOff));
  return v;
}
template <int kOff>
__device__ __forceinline__ uint2 lds64i(uint32_t addr) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2+%3];" : "=r"(v.x), "=r"(v.y) : "r"(addr), "n"(kOff));
  return v;
}
template <int kOff>
__device__ __forceinline__ uint4 lds128i(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4+%5];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr), "n"(kOff));
  return v;
}
template <int kOff>
__device__ __forceinline__ uint32_t lds16i(uint32_t addr) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1+%2];" : "=h"(v) : "r"(addr), "n"(kOff));
  return v;
}
template <int kOff>
__device__ __forceinline__ uint32_t lds8i(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u8 %0, [%1+%2];" : "=r"(v) : "r"(addr), "n"(kOff));
  return v;
}
__device__ __forceinline__ uint32_t lds16(uint32_t addr) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ uint32_t lds8(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}

// 2^x, x <= 0 or slightly above (ex2.approx: relative error 2^-22; 2^-inf = 0)
__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
constexpr float kLazyMax = 8.f;

__device__ __forceinline__ __half2 as_h2(uint32_t v) { return *reinterpret_cast<__half2*>(&v); }
__device__ __forceinline__ uint32_t as_u32(__half2 v) { return *reinterpret_cast<uint32_t*>(&v); }

// D(16x8, f32) += A(16x16, f16, row) * B(16x8, f16, col)
__device__ __forceinline__ void mma_16816(float* d, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                          uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// Codes of one 16-coordinate block of one token, prepared for the table lookups.  Entry idx of the
// replicated u table of sub-block s sits at s * 8192 + idx * 128 with idx = c2_s | c3 << 2 | c4 << 4, i.e.
// c2_s -> address bits 7..8, c3 -> bits 9..10, c4 -> bits 11..12; `ub` = table base | lane replica has
// none of these bits set, so the address is an OR (the loads add s * 8192 as an immediate).
struct BlockRef {
  uint32_t l1;        // 8 level-1 codes, code j at bits [4j, 4j+4)
  uint32_t c2;        // 4 level-2 codes in bits 0..7 (higher bits are ignored)
  uint32_t hi0, hi1;  // ub | c4 | level-3 code of sub-blocks 0-1 / 2-3, in address position
  __half2 r2;         // the block radius in both halves
};
__device__ __forceinline__ BlockRef make_block_ref(uint32_t l1, uint32_t c2, uint32_t c3n, uint32_t c4_clean, __half2 r2,
                                                   uint32_t ub) {
  BlockRef b;
  const uint32_t a4 = c4_clean * 2048u + ub;
  b.l1 = l1;
  b.c2 = c2;
  b.hi0 = ((c3n << 9) & 0x600u) | a4;
  b.hi1 = ((c3n << 7) & 0x600u) | a4;
  b.r2 = r2;
  return b;
}
template <int kS>
__device__ __forceinline__ uint32_t u_address(const BlockRef& b) {
  return ((kS == 3 ? (b.c2 << 1) : (b.c2 << (7 - 2 * kS))) & 0x180u) | (kS < 2 ? b.hi0 : b.hi1);
}
template <int kS>
__device__ __forceinline__ uint32_t t1_address(uint32_t l1, uint32_t t1) {  // byte kS of l1 -> bits 7..14
  return ((kS == 0 ? (l1 << 7) : (l1 >> (8 * kS - 7))) & 0x7F80u) | t1;
}

// DeQuant (Algorithm 1) of sub-block kS (coordinates 4 kS .. 4 kS + 3, level-1 pairs a = 2 kS and
// b = 2 kS + 1) of a block in the rotated basis, fp16:  x = (x_a, x_b) = coordinates (4 kS, 4 kS + 2),
// y = (y_a, y_b) = coordinates (4 kS + 1, 4 kS + 3).  `t1` = level-1 table base | lane replica.
template <int kS>
__device__ __forceinline__ void sub_block_h2(const BlockRef& b, uint32_t t1, __half2& x, __half2& y) {
  const __half2 u = __hmul2(b.r2, as_h2(lds32i<kS * 8192>(u_address<kS>(b))));
  const uint2 e = lds64i<0>(t1_address<kS>(b.l1, t1));
  x = __hmul2(u, as_h2(e.x));
  y = __hmul2(u, as_h2(e.y));
}
// The same sub-block as an unevaluated sum hi + lo of fp16 values (about 21 significant bits):
//   u = r * (Uhi + Ulo)            u_hi = rn(r Uhi),  u_lo = fma(r, Uhi, -u_hi) + r Ulo
//   k = (u_hi + u_lo)(thi + tlo)   k_hi = rn(u_hi thi), k_lo = fma(u_hi, thi, -k_hi) + u_lo thi + u_hi tlo
// (fp16 fused multiply-adds return the exact rounding residual of a product).
template <int kS>
__device__ __forceinline__ void sub_block_hilo(const BlockRef& b, uint32_t t1, __half2& xh, __half2& yh, __half2& xl,
                                               __half2& yl) {
  const uint2 uu = lds64i<kS * 8192>(u_address<kS>(b));
  const __half2 u_hi = __hmul2(b.r2, as_h2(uu.x));
  const __half2 u_lo = __hfma2(b.r2, as_h2(uu.y), __hfma2(b.r2, as_h2(uu.x), __hneg2(u_hi)));
  const uint32_t ta = t1_address<kS>(b.l1, t1);
  const uint2 th = lds64i<0>(ta), tl = lds64i<kSmT1lo - kSmT1p>(ta);
  xh = __hmul2(u_hi, as_h2(th.x));
  yh = __hmul2(u_hi, as_h2(th.y));
  xl = __hfma2(u_hi, as_h2(tl.x), __hfma2(u_lo, as_h2(th.x), __hfma2(u_hi, as_h2(th.x), __hneg2(xh))));
  yl = __hfma2(u_hi, as_h2(tl.y), __hfma2(u_lo, as_h2(th.y), __hfma2(u_hi, as_h2(th.y), __hneg2(yh))));
}

// ---- lookups in tables with 256-byte rows (the persistent kernel's map) --------------------------
// Byte kByte of `index` as the row of the table with base `base` (a multiple of 64 KB | offset inside a row).
template <int kByte>
__device__ __forceinline__ uint32_t row_address(uint32_t index, uint32_t base) {
  return __byte_perm(index, base, 0x7604 | (kByte << 4));
}
// Half-block indices, four to a word: byte = the half's two level-2 codes | level-3 code << 4 | level-4 code << 6.  Each field of a byte is spread by a
// shift or a multiplication that leaves garbage in the other fields only, and two bitwise selects put the three together.
// Two blocks of one token -> (block 0: half 0, half 1; block 1: half 0, half 1).  c2: the blocks' level-2 bytes; n3: their level-3
// nibbles; c4: their level-4 codes in bits 0..3 (garbage above).
__device__ __forceinline__ uint32_t half_indices_of_blocks(uint32_t c2, uint32_t n3, uint32_t c4) {
  const uint32_t f2 = __byte_perm(c2, c2 >> 4, 0x5140);
  // even fields to bytes 0 and 2, odd ones to bytes 1 and 3; bits 6, 7 of a byte stay clear
  const uint32_t f3 = (n3 & 0x33u) * 0x10010u + (n3 & 0xCCu) * 0x400400u;
  const uint32_t f4 = (c4 & 0xFu) * 0x10104040u;
  const uint32_t w = (f2 & 0x0F0F0F0Fu) | (f3 & 0xF0F0F0F0u);
  return w ^ (f4 & 0xC0C0C0C0u);
}
// One block of two tokens -> (token A: half 0, half 1; token B: half 0, half 1).  Bits 0..15 of each argument belong to token A, the
// others to token B; c2: level-2 byte, n3: level-3 nibble, c4: level-4 code in bits 0..1 (garbage above, but n3 and c4 may be garbage).
__device__ __forceinline__ uint32_t half_indices_of_tokens(uint32_t c2, uint32_t n3, uint32_t c4) {
  const uint32_t f2 = (c2 & 0x000F000Fu) | ((c2 << 4) & 0x0F000F00u);
  const uint32_t f3 = (n3 & 0x000F000Fu) * 0x410u;
  const uint32_t f4 = (c4 & 0x00030003u) * (64u + 16384u);
  const uint32_t w = f2 | (f3 & 0x30303030u);
  return w | f4;
}
// Half kByte & 1 of a key block (byte kByte of `index`; level-1 bytes kL1, kL1 + 1 of `l1`) as unevaluated sums hi + lo, see
// sub_block_hilo.
struct KeyHalf {
  __half2 xh[2], yh[2], xl[2], yl[2];
};
template <int kByte, int kL1>
__device__ __forceinline__ void decode_key_half(uint32_t index, uint32_t l1, __half2 r2, uint32_t uk, uint32_t t, KeyHalf& k) {
  const uint4 uu = lds128i<(kByte & 1) * 128>(row_address<kByte>(index, uk));
  const uint32_t ta[2] = {row_address<kL1>(l1, t), row_address<kL1 + 1>(l1, t)};
  const uint32_t uh[2] = {uu.x, uu.y}, ul[2] = {uu.z, uu.w};
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const uint4 e = lds128i<0>(ta[i]);
    const uint2 th = make_uint2(e.x, e.y), tl = make_uint2(e.z, e.w);
    const __half2 u_hi = __hmul2(r2, as_h2(uh[i]));
    const __half2 u_lo = __hfma2(r2, as_h2(ul[i]), __hfma2(r2, as_h2(uh[i]), __hneg2(u_hi)));
    k.xh[i] = __hmul2(u_hi, as_h2(th.x));
    k.yh[i] = __hmul2(u_hi, as_h2(th.y));
    k.xl[i] = __hfma2(u_hi, as_h2(tl.x), __hfma2(u_lo, as_h2(th.x), __hfma2(u_hi, as_h2(th.x), __hneg2(k.xh[i]))));
    k.yl[i] = __hfma2(u_hi, as_h2(tl.y), __hfma2(u_lo, as_h2(th.y), __hfma2(u_hi, as_h2(th.y), __hneg2(k.yh[i]))));
  }
}
// The multipliers u = r U of half kByte & 1 of a value block.
template <int kByte>
__device__ __forceinline__ void value_half(uint32_t index, __half2 r2, uint32_t uv, __half2* u) {
  const uint2 uu = lds64i<(kByte & 1) * 128>(row_address<kByte>(index, uv));
  u[0] = __hmul2(r2, as_h2(uu.x));
  u[1] = __hmul2(r2, as_h2(uu.y));
}
template <int kByte>
__device__ __forceinline__ void value_sub_block(__half2 u, uint32_t l1, uint32_t t, __half2& x, __half2& y) {
  const uint2 e = lds64i<0>(row_address<kByte>(l1, t));
  x = __hmul2(u, as_h2(e.x));
  y = __hmul2(u, as_h2(e.y));
}
// Two 8 x 8 matrices of 16-bit elements, transposed: lane (g, c) gets element g of rows 2c and 2c + 1 of each; lanes 0..7
// and 8..15 give the rows' addresses.
__device__ __forceinline__ uint2 ldmatrix2_trans(uint32_t row) {
  uint2 v;
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(row));
  return v;
}

// plane offsets of a d = 128 token-block
constexpr int kO2 = 32 * kTokenBlock, kO3 = kO2 + 8 * kTokenBlock, kO4 = kO3 + 4 * kTokenBlock,
              kORad = kO4 + 2 * kTokenBlock;

// Build the replicated shared-memory tables from `Tables`: entry e goes to 16 consecutive slots.
// All loads are issued before the stores so that their latencies overlap.
template <int kThreads>
__device__ __forceinline__ void build_fast_tables(uint8_t* smem, const Tables* tb) {
  const int tid = threadIdx.x;
  constexpr int kPer = 256 * 16 / kThreads;
  uint2 v[3 * kPer];
#pragma unroll
  for (int r = 0; r < kPer; ++r) {
    const int e = (tid + r * kThreads) >> 4;  // 0..255
    v[r] = tb->t1p_hi[e];
    v[kPer + r] = tb->t1p_lo[e];
    v[2 * kPer + r] = tb->u_tab[e >> 6][e & 63];
  }
  uint2* t1hi = reinterpret_cast<uint2*>(smem + kSmT1p);
  uint2* t1lo = reinterpret_cast<uint2*>(smem + kSmT1lo);
  uint2* u = reinterpret_cast<uint2*>(smem + kSmU);
#pragma unroll
  for (int r = 0; r < kPer; ++r) {
    const int i = tid + r * kThreads;
    t1hi[i] = v[r];
    t1lo[i] = v[kPer + r];
    u[i] = v[2 * kPer + r];
  }
}

// The same for the map with 256-byte rows (`window`: start of the shared window).  All that a thread reads is on its way before it writes:
// with one table after the other a call took 1.5 us longer.
template <int kThreads>
__device__ __forceinline__ void build_row_tables(uint8_t* window, const Tables* tb) {
  const int row0 = threadIdx.x >> 4, rep = threadIdx.x & 15;   // 16 threads per row
  constexpr int kPer = 256 * 16 / kThreads, kStep = kThreads / 16;
  // entry i of half h: sub-blocks 2h and 2h + 1 at their level-2 codes (bits 0..1 and 2..3 of i) and the codes above, common to both
  const int h = rep >> 3;
  uint2 th[kPer], tl[kPer], ul[kPer], uh[kPer];
#pragma unroll
  for (int r = 0; r < kPer; ++r) {
    const int i = row0 + r * kStep;
    th[r] = tb->t1p_hi[i];
    tl[r] = tb->t1p_lo[i];
    ul[r] = tb->u_tab[2 * h][(i & 3) | (i >> 2 & ~3)];
    uh[r] = tb->u_tab[2 * h + 1][i >> 2];
  }
  uint8_t* t = window + kFsT + row0 * 256;
  uint8_t* u = window + kFsU + row0 * 256;
#pragma unroll
  for (int r = 0; r < kPer; ++r) {
    uint8_t* tr = t + r * kStep * 256;
    *reinterpret_cast<uint2*>(tr + 128 + rep * 8) = th[r];
    if (rep < 8) *reinterpret_cast<uint4*>(tr + rep * 16) = make_uint4(th[r].x, th[r].y, tl[r].x, tl[r].y);
    *reinterpret_cast<uint4*>(u + r * kStep * 256 + rep * 16) = make_uint4(ul[r].x, uh[r].x, ul[r].y, uh[r].y);
  }
}

// Slots of split partials for the persistent kernel: every unit (sequence, kv head) has one slot
// per CTA that works on it; the slots of all units sum to at most units + grid size.
constexpr int kFastMaxGrid = 160;
constexpr int kFastMaxUnits = 2048;  // (sequence, kv head) units the persistent schedule handles
constexpr int kSegmentCost = 7;     // stages' worth of time a CTA spends on starting and finishing a unit
constexpr int kFastMaxSegs = 16;     // units of one CTA that are listed at a time
struct Segment {
  int unit, st0, st1, part, n_parts, slot0;
};

// Persistent work split: the 128-token stages of all units, in unit order, are cut into
// gridDim.x contiguous ranges of equal cost; a CTA's range may cover the end of one unit and the
// start of the next, and a unit may be shared by several CTAs (its "parts").  Starting on another
// unit costs a CTA about kSegmentCost stages (query rotation, refilling the ring, the merge), so
// every unit is preceded by that many empty positions on the line that is cut.  A thread works out up to four
// consecutive units (positions, ranks and partial slots by block-wide scans); the units this CTA takes
// part in are consecutive among the non-empty ones and are listed kFastMaxSegs at a time (a ragged batch -- one very
// long sequence and many short ones -- can give a CTA more than that; the split is then worked out again for the next
// batch of the list, because its scratch lies in the ring).
// Fills `segs` with the CTA's units number kFastMaxSegs * batch_no .. (counted among the CTA's own) and returns how many
// units the CTA has in all.  Called by all threads; `scratch`: 16 bytes per warp.  stages_of(u): stages of unit u (0 past the last
// one); empty_unit(u) is called once for every unit without any.  The loops over a thread's units are kept rolled here and
// in the other parts that run once: at the start of a launch every instruction is fetched through cold instruction
// caches, and a short call takes longer to fetch straight-line code than to run it.
template <int kThreads, class StagesOf, class EmptyUnit>
__device__ __forceinline__ int list_segments(int batch_no, int n_units, uint8_t* scratch, Segment* segs, int* n_segs, int* first_rank,
                                             StagesOf stages_of, EmptyUnit empty_unit) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, G = gridDim.x, cta = blockIdx.x;
  long long* scan_w = reinterpret_cast<long long*>(scratch);   // [warps]
  int* scan_r = reinterpret_cast<int*>(scan_w + kThreads / 32);
  int* scan_p = scan_r + kThreads / 32;
  if (tid == 0) {
    *n_segs = 0;
    *first_rank = 0x7fffffff;
  }
  const int per = (n_units + kThreads - 1) / kThreads, u0 = tid * per;   // this thread's units u0 .. u0 + per - 1
  long long w_mine = 0;
  int r_mine = 0;
#pragma unroll 1
  for (int i = 0; i < per; ++i) {
    const int nst = stages_of(u0 + i);
    w_mine += nst > 0 ? nst + kSegmentCost : 0;
    r_mine += nst > 0;
  }
  long long w_pos = w_mine;   // inclusive scans over the warp, then over the warps
  int r_pos = r_mine;
#pragma unroll 1
  for (int o = 1; o < 32; o <<= 1) {
    const long long w = __shfl_up_sync(0xffffffffu, w_pos, o);
    const int r = __shfl_up_sync(0xffffffffu, r_pos, o);
    if (lane >= o) {
      w_pos += w;
      r_pos += r;
    }
  }
  if (lane == 31) {
    scan_w[warp] = w_pos;
    scan_r[warp] = r_pos;
  }
  __syncthreads();
  long long w_total = 0;
  w_pos -= w_mine;   // start of this thread's first unit
  r_pos -= r_mine;
#pragma unroll 4
  for (int w = 0; w < kThreads / 32; ++w) {
    w_pos += w < warp ? scan_w[w] : 0;
    r_pos += w < warp ? scan_r[w] : 0;
    w_total += scan_w[w];
  }
  // positions times G fit 32 bits for all but enormous calls: a 64-bit division costs several times a 32-bit one
  const bool small = w_total * G < (1ll << 31);
  auto ratio = [&](long long x, long long y) -> long long { return small ? (long long)((uint32_t)x / (uint32_t)y) : x / y; };
  // the CTAs c_first .. c_first + parts - 1 share a unit whose first stage has position `start`
  auto shared_by = [&](long long start, int nst, int* c_first) -> int {
    *c_first = (int)ratio((start + 1) * G + w_total - 1, w_total) - 1;                 // CTA whose range holds stage `start`
    return (int)ratio((start + nst) * G + w_total - 1, w_total) - *c_first;            // ... and the one of its last stage
  };
  int p_mine = 0, rank = r_pos;
  long long w_at = w_pos;
#pragma unroll 1
  for (int i = 0; i < per; ++i) {
    const int u = u0 + i, nst = stages_of(u);
    if (nst > 0) {
      int c_first;
      const int parts = shared_by(w_at + kSegmentCost, nst, &c_first);
      p_mine += parts;
      if (cta >= c_first && cta < c_first + parts) {
        atomicAdd(n_segs, 1);
        atomicMin(first_rank, rank);
      }
      w_at += kSegmentCost + nst;
      ++rank;
    } else if (cta == 0 && batch_no == 0 && u < n_units) {
      empty_unit(u);
    }
  }
  int p_pos = p_mine;
#pragma unroll 1
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, p_pos, o);
    if (lane >= o) p_pos += v;
  }
  if (lane == 31) scan_p[warp] = p_pos;
  __syncthreads();
  const int r0 = *first_rank + batch_no * kFastMaxSegs;  // this batch: ranks r0 .. r0 + kFastMaxSegs - 1
  p_pos -= p_mine;
#pragma unroll 4
  for (int w = 0; w < kThreads / 32; ++w) p_pos += w < warp ? scan_p[w] : 0;
  w_at = w_pos;
  rank = r_pos;
#pragma unroll 1
  for (int i = 0; i < per; ++i) {
    const int nst = stages_of(u0 + i);
    if (nst == 0) continue;
    const long long start = w_at + kSegmentCost, end = start + nst;
    int c_first;
    const int parts = shared_by(start, nst, &c_first);
    if (cta >= c_first && cta < c_first + parts && rank >= r0 && rank < r0 + kFastMaxSegs) {
      const long long lo = ratio(cta * w_total, G), hi = ratio((cta + 1) * w_total, G);
      Segment& sgm = segs[rank - r0];
      sgm.unit = u0 + i;
      sgm.st0 = (int)((lo > start ? lo : start) - start);
      sgm.st1 = (int)((hi < end ? hi : end) - start);  // > st0: the CTA's range holds a stage of the unit
      sgm.part = cta - c_first;
      sgm.n_parts = parts;
      sgm.slot0 = p_pos;  // first partial slot of the unit
    }
    p_pos += parts;
    w_at = end;
    ++rank;
  }
  __syncthreads();
  return *n_segs;
}

// Sums over the 32 lanes of eight values per lane: three halving exchanges leave lane L with row L >> 2 (summed over eight
// lanes), two more finish it.  9 shuffles instead of 40; the order is fixed.  The four lanes 4 r .. 4 r + 3 return row r.
__device__ __forceinline__ float sum_eight_rows(const float* v, int lane) {
  float w4[4], w2[2];
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
#pragma unroll
  for (int k = 0; k < 4; ++k) w4[k] = (b4 ? v[k + 4] : v[k]) + __shfl_xor_sync(0xffffffffu, b4 ? v[k] : v[k + 4], 16);
#pragma unroll
  for (int k = 0; k < 2; ++k) w2[k] = (b3 ? w4[k + 2] : w4[k]) + __shfl_xor_sync(0xffffffffu, b3 ? w4[k] : w4[k + 2], 8);
  float t = (b2 ? w2[1] : w2[0]) + __shfl_xor_sync(0xffffffffu, b2 ? w2[0] : w2[1], 4);
  t += __shfl_xor_sync(0xffffffffu, t, 2);
  return t + __shfl_xor_sync(0xffffffffu, t, 1);
}

// Merge the `ns` partials (slots slot0 .. slot0 + ns - 1) of the `g` query heads of (b, kv head) in slot order, normalise,
// rotate back by S^T and store.  Runs in the last CTA that finishes for this unit, so it is a chain of round trips to L2:
// the rows of S, the first partial outputs of a thread's coordinates and the (m, l) pairs are all requested before
// anything waits.  `sm`: kCombineFloats floats.
constexpr int kCombineFloats = 8 * kFastMaxGrid + 8 + 8 * 128;
static_assert(kCombineFloats * 4 <= kStages * kStageBytes, "the combine uses the ring");
template <int kHG>
__device__ __forceinline__ void combine_and_store(const DecodeArgs& a, int b, int hk, int g, int slot0, int ns, float* sm) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float* w_sm = sm;                          // [g][ns] weights
  float* linv_sm = w_sm + 8 * kFastMaxGrid;  // [g]
  float* o_sm = linv_sm + 8;                 // [g][128]
  const int64_t h0 = (int64_t)b * a.n_q_heads + hk * g;
  // x_hat_i = sum_j y_hat_j S[i][j]: a warp takes eight rows i, lanes over j
  constexpr int kRows = 8;
  const int i0 = warp * kRows;
  float sv[kRows][4];
#pragma unroll
  for (int r = 0; r < kRows; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) sv[r][q] = __ldg(a.S + (i0 + r) * 128 + lane + 32 * q);
  constexpr int kAhead = 16 / kHG;
  float part[kHG][kAhead];
#pragma unroll
  for (int r = 0; r < kHG; ++r) {
    const int h = (tid >> 7) + 4 * r;
    const float* op = a.ws.o + ((int64_t)slot0 * g + h) * 128 + (tid & 127);
#pragma unroll
    for (int s = 0; s < kAhead; ++s) part[r][s] = h < g && s < ns ? __ldcg(op + (int64_t)s * g * 128) : 0.f;
  }
  if (warp < g) {   // a warp per head: weights of the parts
    const float2* mlp = reinterpret_cast<const float2*>(a.ws.ml) + (int64_t)slot0 * g + warp;
    float2 ml[(kFastMaxGrid + 31) / 32];
    float M = -CUDART_INF_F;
#pragma unroll
    for (int i = 0; i < (kFastMaxGrid + 31) / 32; ++i) {
      ml[i] = make_float2(-CUDART_INF_F, 0.f);
      if (lane + 32 * i < ns) ml[i] = __ldcg(mlp + (int64_t)(lane + 32 * i) * g);
      M = fmaxf(M, ml[i].x);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
    float L = 0.f;
#pragma unroll
    for (int i = 0; i < (kFastMaxGrid + 31) / 32; ++i) {
      const float w = ml[i].x == -CUDART_INF_F ? 0.f : fast_exp2(ml[i].x - M);
      if (lane + 32 * i < ns) w_sm[warp * kFastMaxGrid + lane + 32 * i] = w;
      L = fmaf(ml[i].y, w, L);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
    if (lane == 0) {
      linv_sm[warp] = L > 0.f ? 1.f / L : 0.f;
      // scores are kept in the log2 domain: sum_t exp(s_t) = 2^M * L
      if (a.lse != nullptr) a.lse[h0 + warp] = L > 0.f ? (M + log2f(L)) * 0.693147180559945309f : -CUDART_INF_F;
    }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kHG; ++r) {
    const int h = (tid >> 7) + 4 * r, j = tid & 127;
    if (h < g) {
      float acc = 0.f;
#pragma unroll
      for (int s = 0; s < kAhead; ++s)
        if (s < ns) acc = fmaf(part[r][s], w_sm[h * kFastMaxGrid + s], acc);
      const float* op = a.ws.o + ((int64_t)slot0 * g + h) * 128 + j;
#pragma unroll 4
      for (int s = kAhead; s < ns; ++s) acc = fmaf(__ldcg(op + (int64_t)s * g * 128), w_sm[h * kFastMaxGrid + s], acc);
      o_sm[h * 128 + j] = acc * linv_sm[h];
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int h = 0; h < g; ++h) {
    float ov[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) ov[q] = o_sm[h * 128 + lane + 32 * q];
    float v[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) v[r] = fmaf(ov[3], sv[r][3], fmaf(ov[2], sv[r][2], fmaf(ov[1], sv[r][1], ov[0] * sv[r][0])));
    const float t = sum_eight_rows(v, lane);
    if ((lane & 3) == 0) {
      const int64_t oidx = (h0 + h) * 128 + i0 + (lane >> 2);
      if (a.io_dtype == PQ_DTYPE_BF16) reinterpret_cast<__nv_bfloat16*>(a.out)[oidx] = __float2bfloat16(t);
      else reinterpret_cast<float*>(a.out)[oidx] = t;
    }
  }
}

// Called by one warp of every part of unit `u` when the part's partial result is written (and a barrier has ordered the
// block's writes before this).
// Every part raises a flag of its own -- the call's epoch, so nothing in the workspace has to be cleared before the call -- and
// then looks at all flags of the unit.  The last one to raise its flag sees them all; if several do, the first to put the
// epoch into the unit's election word combines.  (One counter per unit, taken by compare-and-swap, makes the parts retry on
// one another: 20 us for the 49 parts of a short two-head call.)  The part that combines takes flags and election word
// back, so that a replayed graph, whose calls keep their epochs, starts without them; a part that meets the word in
// between combines once more, to the same result.
__device__ __forceinline__ void elect_combiner(const DecodeArgs& a, int u, int unit_slot, int part, int n_parts, int lane, int* is_last) {
  bool last = true;
  if (n_parts > 1) {
    __threadfence();   // the block's partial result before its flag
    volatile uint32_t* flags = a.ws.flags + unit_slot;
    if (lane == 0) flags[part] = a.epoch;
    __syncwarp();
    __threadfence();   // the flag before the look at the others
    for (int p0 = 0; p0 < n_parts; p0 += 32) last = last && (p0 + lane >= n_parts || flags[p0 + lane] == a.epoch);
    __threadfence();   // every lane: the flags that it has seen before the partial results that the block then reads
    last = __all_sync(0xffffffffu, last);
    if (last && lane == 0) last = atomicExch(a.ws.elected + u, a.epoch) != a.epoch;
    last = __shfl_sync(0xffffffffu, last, 0);
    if (last)   // all parts have raised theirs
      for (int p0 = lane; p0 < n_parts; p0 += 32) flags[p0] = 0u;
  }
  if (lane == 0) *is_last = last;
}

// kHG: groups of four query heads per kv head (1 or 2).
// kPaged: the cache lies behind a block table (the contiguous instantiation carries none of that code: the kernel
// sits at its register limit).
template <int kHG, bool kPaged>
__global__ void __launch_bounds__(kFastThreads, 1) decode_attention_fast_kernel(DecodeArgs a) {
  extern __shared__ __align__(128) uint8_t smem_raw[];
  uint8_t* smem = smem_raw - kWindowBase;   // the shared window; see the map
  const int g_heads = a.n_q_heads / a.n_kv_heads;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t sm_base = smem_u32(smem_raw) - kWindowBase;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kFsFlags);
  int* is_last = reinterpret_cast<int*>(smem + kFsFlags) + 1;
  const int64_t head_bytes = make_layout(128, a.pg.page_tokens).head_bytes;

  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(sm_base + kFsBar + 8 * s, 1);                                  // full: producer + tx bytes
      mbar_init(sm_base + kFsBar + 8 * (kStages + s), kFastConsumerWarps / 2);  // empty: one arrive per warp of the group
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // Launched as a programmatic dependent of the kernel before it in the stream: everything up to here may run
  // while that kernel finishes; its results (lengths, cache, queries, workspace) are read only after this wait.
  // The kernel after this one may be set up as soon as this grid has started.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  build_row_tables<kFastThreads>(smem, a.tables);   // from the caller's tables, which no kernel writes
  // What this thread needs of S (constant too) to rotate the queries: column warp * 8 + lane / 4, rows 16 i + 4 (lane & 3)
  // + 0..3 -- a warp's load covers whole 32-byte sectors, and four lanes share a column's sum.
  const int rot_j = warp * 8 + (lane >> 2), rot_k = (lane & 3) * 4;
  float s_col[32];
  auto load_s_col = [&]() {
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) s_col[4 * i + e] = ld_const_now(a.S + (16 * i + rot_k + e) * 128 + rot_j);
  };
  if (kHG == 1) load_s_col();   // two groups: held through the work split, the 32 registers spill
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __syncthreads();

  const int n_units = a.batch * a.n_kv_heads, cta = blockIdx.x;   // the work split: see list_segments
  Segment* segs = reinterpret_cast<Segment*>(smem + kFsSegs);
  int* n_segs = reinterpret_cast<int*>(smem + kFsFlags) + 2;   // units of this CTA (all batches of the list)
  int* first_rank = reinterpret_cast<int*>(smem + kFsFlags) + 3;
  // Stages of unit u (0 past the last one).
  auto stages_of = [&](int u) -> int {
    const int len_u = u < n_units ? a.visible_len(u / a.n_kv_heads) : 0;
    return len_u > 0 ? (len_u + kStageTokens - 1) / kStageTokens : 0;
  };
  auto empty_unit = [&](int u) {   // empty sequence: zeros, and the status says so
    const int b = u / a.n_kv_heads, hk = u - b * a.n_kv_heads;
#pragma unroll 1
    for (int e = 0; e < g_heads * 128; ++e) {
      const int64_t idx = ((int64_t)b * a.n_q_heads + hk * g_heads) * 128 + e;
      if (a.io_dtype == PQ_DTYPE_BF16) reinterpret_cast<__nv_bfloat16*>(a.out)[idx] = __float2bfloat16(0.f);
      else reinterpret_cast<float*>(a.out)[idx] = 0.f;
    }
    if (a.lse != nullptr)
      for (int h = 0; h < g_heads; ++h) a.lse[(int64_t)b * a.n_q_heads + hk * g_heads + h] = -CUDART_INF_F;
    else
      set_status(a.status, PQ_ERR_EMPTY);
  };
  auto build_segments = [&](int batch_no) -> int {
    return list_segments<kFastThreads>(batch_no, n_units, smem + kFsRing, segs, n_segs, first_rank, stages_of, empty_unit);
  };
  const int g = lane >> 2, c = lane & 3;
  // table base | lane replica; the value multipliers are the high parts of the keys' entries
  const uint32_t tk = sm_base + kFsT + (lane & 7) * 16, tv = sm_base + kFsT + 128 + (lane & 15) * 8, tu = sm_base + kFsU + (lane & 7) * 16;
  const int wg = warp >> 3;  // group of 8 warps
  // Offsets, inside a token-block, of what this thread reads of its tile (16 tokens from token (warp & 3) * 16).
  // Keys: tokens g and g + 8, blocks 2c and 2c + 1.  Values: block g of tokens c, c + 4, c + 8, c + 12 (these are
  // rows 2c, 2c + 1, 2c + 8, 2c + 9 of the value MMA: with this order the four lanes of a quad read four
  // consecutive tokens and the loads are free of bank conflicts).
  const int tk_k = (warp & 3) * 16 + (lane >> 2), tk_v = (warp & 3) * 16 + (lane & 3);
  const uint32_t ok_l1 = tk_k * 32 + (lane & 3) * 8, ok_r = kORad + tk_k * 16 + (lane & 3) * 4;
  const uint32_t ok_c2 = kO2 + tk_k * 8 + (lane & 3) * 2, ok_c3 = kO3 + tk_k * 4 + (lane & 3), ok_c4 = kO4 + tk_k * 2;
  const uint32_t ov_l1 = tk_v * 32 + (lane >> 2) * 4, ov_r = kORad + ((warp & 3) * 16 + ((lane >> 1) & 3) + 4 * (lane & 1) + (lane & 8)) * 16;   // rows for ldmatrix2_trans
  const uint32_t ov_c2 = kO2 + tk_v * 8 + (lane >> 2), ov_c3 = kO3 + tk_v * 4 + (lane >> 3), ov_c4 = kO4 + tk_v * 2;
  int gl0 = 0;               // stages this group has streamed so far (ring slot and barrier phase bookkeeping)

  int my_units = build_segments(0);
  for (int batch_no = 0; batch_no * kFastMaxSegs < my_units; ++batch_no) {
  if (batch_no > 0) my_units = build_segments(batch_no);
  const int my_segs = min(kFastMaxSegs, my_units - batch_no * kFastMaxSegs);
  for (int sg = 0; sg < my_segs; ++sg) {
    const int u = segs[sg].unit, st0 = segs[sg].st0, st1 = segs[sg].st1;
    const int n_parts = segs[sg].n_parts, unit_slot = segs[sg].slot0, c_first = cta - segs[sg].part;
    const int b = u / a.n_kv_heads, hk = u - b * a.n_kv_heads;
    const int len = a.visible_len(b);   // b counts (sequence, query) pairs: see DecodeArgs
    const int nblk_total = (len + kTokenBlock - 1) / kTokenBlock;
    const int seq = a.seq_of(b);
    const uint8_t* head_base = a.cache + ((int64_t)seq * a.n_kv_heads + hk) * head_bytes;  // of a contiguous cache

    // per-thread attention state
    // o_acc[hg][S][.]: head c + 4 hg, block g, coordinates 4S, 4S + 2, 4S + 1, 4S + 3 (see the value MMAs)
    float o_acc[kHG][4][4];
#pragma unroll
    for (int hg = 0; hg < kHG; ++hg)
#pragma unroll
      for (int i = 0; i < 4; ++i) o_acc[hg][i][0] = o_acc[hg][i][1] = o_acc[hg][i][2] = o_acc[hg][i][3] = 0.f;
    float m_run[kHG], l_run[kHG];  // of head c + 4 hg: reference (the same in the 8 lanes with this c), own share of the sum
#pragma unroll
    for (int hg = 0; hg < kHG; ++hg) {
      m_run[hg] = -CUDART_INF_F;
      l_run[hg] = 0.f;
    }

    // The two groups of 8 warps take alternate stages: group wg handles stages st0 + wg + 2 li and owns
    // ring slots 2 wg and 2 wg + 1.  Lane 0 of the group's first warp issues the group's copies, one
    // stage of its own ahead; it waits (bounded) until the group's 8 warps have released the slot.
    const int n_li = st1 - st0 > wg ? (st1 - st0 - wg + 1) >> 1 : 0;
    int issued = 0;
    auto stage_place = [&](int st) -> int64_t {
      Layout Lp;  // the two fields the offset needs
      Lp.block_bytes = kBlockBytes128;
      Lp.head_bytes = head_bytes;
      return kv_block_pair_offset(Lp, a.pg, a.n_kv_heads, seq, hk, 2 * st, a.status);
    };
    auto issue_copy = [&](int li, auto listed, uint32_t at) -> bool {   // at: where the place of a paged cache's stage stands, if it is listed
      const int gl = gl0 + li, s = 2 * wg + (gl & 1);
      if (gl >= 2 && !mbar_wait(sm_base + kFsBar + 8 * (kStages + s), ((gl >> 1) - 1) & 1, abort_flag)) return false;
      const int st = st0 + wg + 2 * li;
      const int nblk = min(2, nblk_total - 2 * st);
      const uint32_t bytes = nblk * 2 * kBlockBytes128;
      mbar_expect_tx(sm_base + kFsBar + 8 * s, bytes);
      // a stage is two token-blocks, K | V | K | V, of one page (page_tokens is a multiple of 128)
      const uint8_t* src = head_base + (int64_t)st * kStageBytes;
      if constexpr (kPaged) {
        if constexpr (decltype(listed)::value) src = a.cache + lds32i<0>(at) * (int64_t)kPlaceUnit;
        else src = a.cache + stage_place(st);
      }
      bulk_load(sm_base + kFsRing + s * kStageBytes, src, bytes, sm_base + kFsBar + 8 * s);
      issued = li + 1;
      return true;
    };
    // Where a paged segment's stages begin is listed in shared memory, kFsPlaceCap of them at a time and the first ones before the second
    // copy is requested (a barrier of the rotation below lies between), so that the copying thread, whose warp has a tile of its own to
    // work on, needs no division and waits for no table.  Looked up per stage they cost the whole kernel a tenth (before the keys' level-1
    // residuals were back): 8 x 32768 tokens, 32/8 heads, pages of 256 131.9 us against 122.6 (contiguous 119.4; now 132.6 and 129.3); 16 x 20000 160.6 -> 148.0, 28/4 heads 88.1 -> 84.5.  Looked up
    // inside the loop for stages beyond a longer list, the unused branch alone took 125.2: a list is made again instead.
    auto list_places = [&](int first) {
      for (int i = tid; i < min(kFsPlaceCap, st1 - st0 - first); i += kFastThreads)
        reinterpret_cast<uint32_t*>(smem + kFsPlaces)[i] = (uint32_t)(stage_place(st0 + first + i) / kPlaceUnit);
    };
    constexpr int kWindow = kFsPlaceCap / 2 - 1;   // steps of the groups that a list is enough for, with the copies one step ahead
    if (kPaged) list_places(0);
    const bool hook = !kPaged && (a.debug & 1u) && unit_slot == 0 && cta == c_first;
    const bool producer = (tid & 255) == 0;
    if (producer && n_li > 0) {
      // what list_segments, the merge or the combine left in the ring by ordinary accesses (a barrier has ordered them before this)
      // comes before the copies into it
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      issue_copy(0, std::false_type{}, 0);
    }
    __syncwarp();
    // q' = (q S) * scale * log2(e) for the unit's query heads, as an fp16 value plus an fp16 residual.
    // The first stages of the segment are already on their way while this runs.
    {
      float* q_in = reinterpret_cast<float*>(smem + kFsQ);
      __half* q_hi = reinterpret_cast<__half*>(smem + kFsQ + 4096) + (rot_j >> 5) * (kQQuarter / 2) + (rot_j & 31);
      const int64_t q0 = ((int64_t)b * a.n_q_heads + hk * g_heads) * 128;
      for (int i = tid; i < g_heads * 128; i += kFastThreads)
        q_in[i] = a.io_dtype == PQ_DTYPE_BF16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(a.q)[q0 + i])
                                              : reinterpret_cast<const float*>(a.q)[q0 + i];
      if (kHG > 1 || batch_no + sg > 0) load_s_col();
      __syncthreads();
#pragma unroll 1
      for (int h = 0; h < g_heads; ++h) {
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float4 qv = *reinterpret_cast<const float4*>(q_in + h * 128 + 16 * i + rot_k);
          acc[0] = fmaf(qv.x, s_col[4 * i], acc[0]);
          acc[1] = fmaf(qv.y, s_col[4 * i + 1], acc[1]);
          acc[2] = fmaf(qv.z, s_col[4 * i + 2], acc[2]);
          acc[3] = fmaf(qv.w, s_col[4 * i + 3], acc[3]);
        }
        float v = (acc[0] + acc[1]) + (acc[2] + acc[3]);
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        v *= a.scale * 1.4426950408889634f;
        if ((lane & 3) == (h & 3)) {
          const __half qh = __float2half_rn(v);
          q_hi[h * (kQHead / 2)] = qh;
          q_hi[h * (kQHead / 2) + kQLo / 2] = __float2half_rn(v - __half2float(qh));
        }
      }
      __syncthreads();
    }
    // q' fragments, B operand (16 coords x 8 columns per k-step): column n = 2 h + part holds the fp16 value
    // (part 0) or the fp16 residual (part 1) of head h (+ 4 hg).  k-step ks covers, for thread c, sub-block
    // (ks & 3) of block 2c + (ks >> 2).
    // With one group of heads they stay in registers (read again for every tile: 119.5 -> 122.2 us for 8 x 32768 tokens, 32/8 heads); with
    // two the 32 registers spill, and they lie in shared memory in fragment order (28/4 heads 84.9 -> 83.4 us, 16/2 55.8 -> 54.0).
    constexpr bool kQInRegs = kHG == 1;
    uint2 qb[kQInRegs ? 8 : 1];
    const uint32_t qf = sm_base + kFsQ + lane * 8;   // [hg][ks][lane], where the queries were before their rotation
    auto q_fragment = [&](int hg, int ks) {
      const int h = (g >> 1) + 4 * hg;
      uint2 v = make_uint2(0u, 0u);
      if (h < g_heads) v = reinterpret_cast<const uint2*>(smem + kFsQ + 4096 + (g & 1) * kQLo + h * kQHead + c * kQQuarter)[ks];
      // decoded keys come as (coord 0, coord 2), (coord 1, coord 3) of each sub-block: permute q' to match
      return make_uint2(__byte_perm(v.x, v.y, 0x5410), __byte_perm(v.x, v.y, 0x7632));
    };
    if constexpr (kQInRegs) {
#pragma unroll
      for (int ks = 0; ks < 8; ++ks) qb[ks] = q_fragment(0, ks);
    } else {
      const int hg = warp >> 3, ks = warp & 7;   // sixteen warps, a fragment each
      *reinterpret_cast<uint2*>(smem + kFsQ + hg * 2048 + ks * 256 + lane * 8) = q_fragment(hg, ks);
      __syncthreads();
    }
    for (int first = 0;;) {
    const int last = kPaged ? min(n_li, first + kWindow) : n_li;
    for (int li = first; li < last; ++li) {
      const int gl = gl0 + li, s = 2 * wg + (gl & 1);
      const int st = st0 + wg + 2 * li;
      if (producer && li + 1 < n_li) issue_copy(li + 1, std::true_type{}, kPaged ? sm_base + kFsPlaces + 4 * wg + 8 * (li + 1 - first) : 0);
      __syncwarp();
      if (!mbar_wait(sm_base + kFsBar + 8 * s, (gl >> 1) & 1, abort_flag)) break;
      if ((kPaged ? (a.debug & 1u) && unit_slot == 0 && cta == c_first : hook) && li == 0 && warp == 0) {  // test hook: the first wait of the CTA
        // that starts the first non-empty unit is reported as failed
        *abort_flag = 1;
        break;
      }
      const int tile_tok0 = st * kStageTokens + (warp & 7) * 16;  // first token of this warp's 16-token tile
      if (tile_tok0 < len) {
        const uint32_t kblk = sm_base + kFsRing + s * kStageBytes + ((warp >> 2) & 1) * 2 * kBlockBytes128;
        const uint32_t vblk = kblk + kBlockBytes128;
        // ---- scores S (tokens x columns): A operand = keys of tokens g (rows 0..7) and g + 8 (rows 8..15),
        // decoded as hi + lo; one MMA with the hi parts and one with the lo parts per k-step.  Column 2c is
        // q_hi of head c, column 2c+1 its q_lo, so all four products of a (token, head) land in this thread.
        float sc[kHG][4], scl[kHG][4];
#pragma unroll
        for (int hg = 0; hg < kHG; ++hg)
#pragma unroll
          for (int i = 0; i < 4; ++i) sc[hg][i] = scl[hg][i] = 0.f;
        {
          const uint2 l1pA = lds64i<0>(kblk + ok_l1), l1pB = lds64i<8 * 32>(kblk + ok_l1);
          const uint32_t rrA = lds32i<0>(kblk + ok_r), rrB = lds32i<8 * 16>(kblk + ok_r);
          const uint32_t c2A = lds16i<0>(kblk + ok_c2), c2B = lds16i<8 * 8>(kblk + ok_c2);
          const uint32_t c3A = lds8i<0>(kblk + ok_c3), c3B = lds8i<8 * 4>(kblk + ok_c3);
          const uint32_t c4A = lds16i<0>(kblk + ok_c4) >> (4 * c), c4B = lds16i<8 * 2>(kblk + ok_c4) >> (4 * c);
#define PQ_KHALF(INDEX, L1, R2, H, HALF)                                                                      \
  {                                                                                                           \
    KeyHalf kA, kB;                                                                                           \
    decode_key_half<2 * (H) + (HALF), 2 * (HALF)>(INDEX##A, L1##A, R2(as_h2(rrA)), tu, tk, kA);               \
    decode_key_half<2 * (H) + (HALF), 2 * (HALF)>(INDEX##B, L1##B, R2(as_h2(rrB)), tu, tk, kB);               \
    _Pragma("unroll") for (int i = 0; i < 2; ++i) _Pragma("unroll") for (int hg = 0; hg < kHG; ++hg) {        \
      constexpr int kKs0 = 4 * (H) + 2 * (HALF);                                                              \
      const uint2 qv = kQInRegs ? qb[kQInRegs ? kKs0 + i : 0] : lds64(qf + hg * 2048 + (kKs0 + i) * 256);     \
      mma_16816(scl[hg], as_u32(kA.xl[i]), as_u32(kB.xl[i]), as_u32(kA.yl[i]), as_u32(kB.yl[i]), qv.x, qv.y); \
      mma_16816(sc[hg], as_u32(kA.xh[i]), as_u32(kB.xh[i]), as_u32(kA.yh[i]), as_u32(kB.yh[i]), qv.x, qv.y);  \
    }                                                                                                         \
  }
          const uint32_t ixA = half_indices_of_blocks(c2A, c3A, c4A), ixB = half_indices_of_blocks(c2B, c3B, c4B);
          const uint32_t l1A = l1pA.x, l1B = l1pB.x, l1hA = l1pA.y, l1hB = l1pB.y;
          PQ_KHALF(ix, l1, __low2half2, 0, 0)
          PQ_KHALF(ix, l1, __low2half2, 0, 1)
          PQ_KHALF(ix, l1h, __high2half2, 1, 0)
          PQ_KHALF(ix, l1h, __high2half2, 1, 1)
#undef PQ_KHALF
        }
        // ---- online softmax: this thread holds head c (+ 4 hg) of tokens g and g + 8.  The reference m_run of a
        // head moves only when a score exceeds it by more than kLazyMax (log2 units), so p = 2^(s - m_run) stays
        // below 2^kLazyMax (fp16 holds it with its full relative precision) and the common tile needs neither
        // the reductions over tokens nor a rescaling; l_run is this thread's share of the denominator (its own
        // tokens), summed over the eight lanes of the head when the segment ends.
        const bool whole = tile_tok0 + 16 <= len;
        float s0[kHG], s1[kHG];
        bool over = false;
#pragma unroll
        for (int hg = 0; hg < kHG; ++hg) {
          s0[hg] = (scl[hg][0] + scl[hg][1]) + sc[hg][1] + sc[hg][0];  // small terms first
          s1[hg] = (scl[hg][2] + scl[hg][3]) + sc[hg][3] + sc[hg][2];
          if (!whole) {   // the last tile of the sequence: what lies past its end may be anything
            if (tile_tok0 + g >= len) s0[hg] = -CUDART_INF_F;
            if (tile_tok0 + g + 8 >= len) s1[hg] = -CUDART_INF_F;
          }
          over = over || fmaxf(s0[hg], s1[hg]) > m_run[hg] + kLazyMax;  // always on the first tile (m_run = -inf)
        }
        if (__any_sync(0xffffffffu, over)) {
          float corr[kHG];
#pragma unroll
          for (int hg = 0; hg < kHG; ++hg) {
            float mx = fmaxf(s0[hg], s1[hg]);
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
            const float m_new = fmaxf(m_run[hg], mx);  // finite: token 0 of the tile is inside the sequence
            corr[hg] = fast_exp2(m_run[hg] - m_new);   // 0 on the first tile
            l_run[hg] *= corr[hg];
            m_run[hg] = m_new;
          }
#pragma unroll
          for (int hg = 0; hg < kHG; ++hg)  // the accumulators of this thread belong to its own head
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              o_acc[hg][i][0] *= corr[hg];
              o_acc[hg][i][1] *= corr[hg];
              o_acc[hg][i][2] *= corr[hg];
              o_acc[hg][i][3] *= corr[hg];
            }
        }
        uint32_t ph[kHG];   // (p of token g, p of token g + 8) in fp16
#pragma unroll
        for (int hg = 0; hg < kHG; ++hg) {
          const float p0 = fast_exp2(s0[hg] - m_run[hg]), p1 = fast_exp2(s1[hg] - m_run[hg]);
          l_run[hg] += p0 + p1;
          ph[hg] = as_u32(__floats2half2_rn(p0, p1));
        }
        // B operand of the value MMAs.  The contraction index is (token, which element of a decoded half2): rows
        // 2c, 2c+1 = token c (first MMA) or c + 8 (second), rows 2c+8, 2c+9 = token c + 4 or c + 12.  Column
        // n = 2h + e is head h restricted to element e: its entry is p in half e and zero in the other, so a
        // decoded half2 is an A register as it is and no column of the MMA is idle (4 heads x 2 elements).
        uint32_t pb[kHG][2][2];
#pragma unroll
        for (int hg = 0; hg < kHG; ++hg) {
          const int srcA = c * 4 + (g >> 1);  // lane that holds tokens c and c + 8 of head g >> 1
          const uint32_t uA = __shfl_sync(0xffffffffu, ph[hg], srcA), uB = __shfl_sync(0xffffffffu, ph[hg], srcA + 16);
          const uint32_t sel_lo = (g & 1) ? 0x1044u : 0x4410u, sel_hi = (g & 1) ? 0x3244u : 0x4432u;
          pb[hg][0][0] = __byte_perm(uA, 0u, sel_lo);
          pb[hg][0][1] = __byte_perm(uB, 0u, sel_lo);
          pb[hg][1][0] = __byte_perm(uA, 0u, sel_hi);
          pb[hg][1][1] = __byte_perm(uB, 0u, sel_hi);
        }
        // ---- values: block g of tokens c, c+4, c+8, c+12 -> O^T (coordinates x (head, element)) += V_hat^T P
        {
          const uint32_t l1v[4] = {lds32i<0>(vblk + ov_l1), lds32i<4 * 32>(vblk + ov_l1), lds32i<8 * 32>(vblk + ov_l1), lds32i<12 * 32>(vblk + ov_l1)};
          uint2 rr = ldmatrix2_trans(vblk + ov_r);   // radii of tokens c | c + 4 and c + 8 | c + 12
          // codes of two tokens in one word
          const uint32_t c2v[2] = {lds8i<0>(vblk + ov_c2) | lds8i<4 * 8>(vblk + ov_c2) << 16, lds8i<8 * 8>(vblk + ov_c2) | lds8i<12 * 8>(vblk + ov_c2) << 16};
          const uint32_t c3v[2] = {lds8i<0>(vblk + ov_c3) | lds8i<4 * 4>(vblk + ov_c3) << 16, lds8i<8 * 4>(vblk + ov_c3) | lds8i<12 * 4>(vblk + ov_c3) << 16};
          const uint32_t c4v[2] = {lds16i<0>(vblk + ov_c4) | lds16i<4 * 2>(vblk + ov_c4) << 16, lds16i<8 * 2>(vblk + ov_c4) | lds16i<12 * 2>(vblk + ov_c4) << 16};
          if (!whole) {   // stale bytes past the sequence end stay out of the sums
            const int left = len - tile_tok0 - c;   // token c + 4 j is inside if 4 j < left
            rr.x = left > 4 ? rr.x : left > 0 ? rr.x & 0xFFFFu : 0u;
            rr.y = left > 12 ? rr.y : left > 8 ? rr.y & 0xFFFFu : 0u;
          }
          uint32_t ixv[2];
#pragma unroll
          for (int j = 0; j < 2; ++j) ixv[j] = half_indices_of_tokens(c2v[j], c3v[j] >> (4 * (g & 1)), c4v[j] >> (2 * g));
#define PQ_VHALF(HALF)                                                 \
  {                                                                    \
    __half2 u0[2], u1[2], u2[2], u3[2];                                \
    value_half<(HALF)>(ixv[0], __low2half2(as_h2(rr.x)), tu, u0);      \
    value_half<2 + (HALF)>(ixv[0], __high2half2(as_h2(rr.x)), tu, u1); \
    value_half<(HALF)>(ixv[1], __low2half2(as_h2(rr.y)), tu, u2);      \
    value_half<2 + (HALF)>(ixv[1], __high2half2(as_h2(rr.y)), tu, u3); \
    PQ_VSTEP(2 * (HALF), 0) PQ_VSTEP(2 * (HALF) + 1, 1)                \
  }
#define PQ_VSTEP(S, I)                                                                                     \
  {                                                                                                        \
    __half2 x0, y0, x1, y1, x2, y2, x3, y3;                                                                \
    value_sub_block<S>(u0[I], l1v[0], tv, x0, y0);                                                         \
    value_sub_block<S>(u1[I], l1v[1], tv, x1, y1);                                                         \
    value_sub_block<S>(u2[I], l1v[2], tv, x2, y2);                                                         \
    value_sub_block<S>(u3[I], l1v[3], tv, x3, y3);                                                         \
    _Pragma("unroll") for (int hg = 0; hg < kHG; ++hg) {                                                   \
      mma_16816(o_acc[hg][S], as_u32(x0), as_u32(y0), as_u32(x1), as_u32(y1), pb[hg][0][0], pb[hg][0][1]); \
      mma_16816(o_acc[hg][S], as_u32(x2), as_u32(y2), as_u32(x3), as_u32(y3), pb[hg][1][0], pb[hg][1][1]); \
    }                                                                                                      \
  }
          PQ_VHALF(0) PQ_VHALF(1)
#undef PQ_VHALF
#undef PQ_VSTEP
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(sm_base + kFsBar + 8 * (kStages + s));
    }
      first += kWindow;
      if (!kPaged || 2 * first >= st1 - st0) break;
      __syncthreads();   // nothing reads the list any more
      if (*abort_flag) break;
      list_places(2 * first);
      __syncthreads();
    }
    gl0 += n_li;
    __syncthreads();  // every copy that was consumed is done with; the rest is waited for below
    if (*abort_flag) {
      // gave up: let the copies still in flight land (bounded) before the ring is reused
      if (producer)
        for (int li = max(0, issued - 2); li < issued; ++li) {
          const int gl = gl0 - n_li + li;
          for (int i = 0; i < kSpinLimit && !mbar_try_wait(sm_base + kFsBar + 8 * (2 * wg + (gl & 1)), (gl >> 1) & 1); ++i)
            __nanosleep(64);
        }
      __syncthreads();
    }

    // ---- merge the 16 warps (fixed order), write this part's partial, last part combines the unit
    // Coordinate j of head h (of four) of warp w sits at (w * 4 + h) * kMrgStride + (j & 15) * 8 + (j >> 4): for a fixed
    // accumulator register the 32 lanes (block g, head c) then hit 32 different banks.
    float* mrg_o = reinterpret_cast<float*>(smem + kFsRing);                  // [16 warps][4 heads][kMrgStride]
    float* mrg_ml = reinterpret_cast<float*>(smem + kFsRing + kFsMergeMl);    // [16 warps][8 heads][2]
#pragma unroll
    for (int hg = 0; hg < kHG; ++hg) {  // the head's denominator: sum of the shares of its eight lanes
      l_run[hg] += __shfl_xor_sync(0xffffffffu, l_run[hg], 4);
      l_run[hg] += __shfl_xor_sync(0xffffffffu, l_run[hg], 8);
      l_run[hg] += __shfl_xor_sync(0xffffffffu, l_run[hg], 16);
    }
    if (g == 0) {
#pragma unroll
      for (int hg = 0; hg < kHG; ++hg)
        *reinterpret_cast<float2*>(mrg_ml + (warp * 8 + c + 4 * hg) * 2) = make_float2(m_run[hg], l_run[hg]);
    }
    __syncthreads();
    // In the contiguous instantiation the segment is read again (and through volatile, so that it really is): the registers that its
    // fields would hold through the tile loop cost that loop 2 % (8 x 131072 tokens: 516 -> 507 us).  In the paged one it is
    // the other way round (16 ragged sequences of up to 65536 tokens, four steps: 1313 us, 1365 with the fields read again).  That is
    // the register allocation of nvcc 12.9, not a property of paging.
    struct {
      int unit, b, hk, part, n_parts, slot0;
    } done;
    if constexpr (kPaged) {
      done = {u, b, hk, cta - c_first, n_parts, unit_slot};
    } else {
      const volatile Segment* sv = segs + sg;
      const int du = sv->unit;
      done = {du, du / a.n_kv_heads, du % a.n_kv_heads, sv->part, sv->n_parts, sv->slot0};
    }
    const int slot = done.slot0 + done.part;
    if (tid < g_heads * 16) {   // denominators: 16 lanes per head
      const int h = tid >> 4;
      const unsigned half = 0xFFFFu << (lane & 16);
      const float2 ml = *reinterpret_cast<const float2*>(mrg_ml + ((tid & 15) * 8 + h) * 2);
      float M = ml.x;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(half, M, o));
      float l = ml.x == -CUDART_INF_F ? 0.f : ml.y * fast_exp2(ml.x - M);
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) l += __shfl_xor_sync(half, l, o);
      if ((tid & 15) == 0) __stcg(reinterpret_cast<float2*>(a.ws.ml) + (int64_t)slot * g_heads + h, make_float2(M, l));
    }
    // every warp brings its accumulators to the common reference before it hands them over
#pragma unroll
    for (int hg = 0; hg < kHG; ++hg) {
      if (hg > 0) __syncthreads();   // the four heads before these have been read
      if (c + 4 * hg < g_heads) {
        float M = -CUDART_INF_F;
#pragma unroll
        for (int w = 0; w < kFastConsumerWarps; ++w) M = fmaxf(M, mrg_ml[(w * 8 + c + 4 * hg) * 2]);
        const float wgt = m_run[hg] == -CUDART_INF_F ? 0.f : fast_exp2(m_run[hg] - M);
        float* o0 = mrg_o + (warp * 4 + c) * kMrgStride + g;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          o0[(4 * i) * 8] = o_acc[hg][i][0] * wgt;
          o0[(4 * i + 2) * 8] = o_acc[hg][i][1] * wgt;
          o0[(4 * i + 1) * 8] = o_acc[hg][i][2] * wgt;
          o0[(4 * i + 3) * 8] = o_acc[hg][i][3] * wgt;
        }
      }
      __syncthreads();
      const int h = (tid >> 7) + 4 * hg, j = tid & 127;
      if (h < g_heads) {
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int w = 0; w < kFastConsumerWarps; ++w) acc[w & 3] += mrg_o[(w * 4 + (tid >> 7)) * kMrgStride + (j & 15) * 8 + (j >> 4)];
        __stcg(a.ws.o + ((int64_t)slot * g_heads + h) * 128 + j, (acc[0] + acc[1]) + (acc[2] + acc[3]));
      }
    }
    __syncthreads();
    if (warp == 0) elect_combiner(a, done.unit, done.slot0, done.part, done.n_parts, lane, is_last);
    __syncthreads();
    if (*is_last) {
      combine_and_store<kHG>(a, done.b, done.hk, g_heads, done.slot0, done.n_parts, reinterpret_cast<float*>(smem + kFsRing));
      if (tid == 0 && done.n_parts > 1) *reinterpret_cast<volatile uint32_t*>(a.ws.elected + done.unit) = 0u;
    }
    __syncthreads();  // the ring is free again for the next unit
  }
  }
  if (tid == 0 && *abort_flag) set_status(a.status, PQ_ERR_TIMEOUT);
}

}  // namespace pq
