// Quantize-pack, dequantize and append kernels of the HeadGuard KV cache.
//
// Quantize (Sec. 3 "Applying protection" over the Sec. 1 / Sec. 4 bases).
// A CTA is one warp: it stages the K rows or the V rows of a 32-token tile of
// one (layer, batch row, KV head) in shared memory with coalesced asynchronous
// copies and then works one lane per vector: per-token min-max rows (Sec. 1),
// AKVQ-style rows (Sec. 4: keys rotated by the Hadamard-128 in registers
// first, a row over a lane pair), KIVI-style value rows (four 32-channel
// groups) and KIVI-style key groups (one lane per channel pair over the 32
// image tokens of the tile).  The head's class and the image span are
// resolved once per CTA, so protected heads and text tokens take a uniform
// BF16 copy path.  Codes, scales and zeros follow the group quantizer exactly
// (round half to even of the IEEE quotient, no contraction).
#include <algorithm>
#include <atomic>
#include <climits>
#include <cmath>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "hg_common.cuh"
#include "hg_internal.h"
#include "hg_mma.cuh"

namespace hg {

namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ void bf16x4_to_f32(uint2 w, float (&x)[4]) {
  bf16x2_to_f32(w.x, x[0], x[1]);
  bf16x2_to_f32(w.y, x[2], x[3]);
}

// ---------------------------------------------------------------------------
// Per-token min-max base: one thread per (token, K or V) vector.
//
// A CTA takes the K rows or the V rows of 32 tokens of one (layer, row, KV
// head), staged in shared memory with coalesced loads (272-byte row pitch, so
// that a lane's 16-byte reads of its own row are conflict free); lane i owns
// row i.  A coded vector is quantized by its lane alone -- min / max over
// bf16x2 pairs (exact), then at 2 bits three comparisons with the BF16 values
// where the code changes (bf16_thresholds), else per element
//   T = RN(d * r + 192), d = fl(x - min), r = RN(1 / scale):
// T lies in [128, 256), so its low 16 mantissa bits hold d * r to 2^-16 and
// bits 16.. hold floor(d * r + 0.5) once 0x8000 is added.  Within 2^-16 of
// a half-integer the exact rule (round-half-even of fl(d / scale)) may differ,
// so such an element takes one IEEE division (BF16 inputs make exact
// half-integer quotients common, so this is per element, not per vector).  The
// bound: |d r - d / scale| <= 16 * 2^-24 and the FMA and the reference
// quotient each round by at most 2^-17, so any element whose low bits are not
// within one unit of 0x8000 rounds the same way as the reference.
// Uncoded vectors (text, protected heads, keys of keys-only heads) are copied.
// ---------------------------------------------------------------------------
constexpr int kQTok = 32;
constexpr int kQPitch = 272;

// Round-half-even of fl(d / scale), clamped to the levels (IEEE division).
__device__ __noinline__ uint32_t exact_code(float d, float scale, float levels) {
  return (uint32_t)fminf(fmaxf(rintf(__fdiv_rn(d, scale)), 0.0f), levels);
}

// The packed bits of one 8-channel chunk: `lo` its 32 (4-bit) or 16 (2- and
// 3-bit) low code bits in channel order, `hb` its 8 bit-2 bits (3-bit).
template <int BITS>
__device__ __forceinline__ void chunk_bits(const uint32_t (&c)[8], uint32_t& lo, uint32_t& hb) {
  lo = 0u;
  hb = 0u;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    lo |= (BITS == 4) ? (c[i] << (4 * i)) : ((c[i] & 3u) << (2 * i));
    if (BITS == 3) hb |= ((c[i] >> 2) & 1u) << i;
  }
}

// The same from the eight T' words of the fast rule (code in bits 16..): each
// code is shifted straight into its packed position (one shift and one
// and-or per element instead of extracting it first).
template <int BITS>
__device__ __forceinline__ void chunk_bits_T(const uint32_t (&a)[8], uint32_t& lo, uint32_t& hb) {
  lo = 0u;
  hb = 0u;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    if (BITS == 4) {
      const uint32_t x = (4 * i >= 16) ? (a[i] << (4 * i - 16)) : (a[i] >> (16 - 4 * i));
      lo |= x & (15u << (4 * i));
    } else {
      lo |= (a[i] >> (16 - 2 * i)) & (3u << (2 * i));
      if (BITS == 3) hb |= (a[i] >> (18 - i)) & (1u << i);
    }
  }
}

// Chunks kg..kg+3 (kg a multiple of 4) into the packed row, one vector store
// per word run: 4 bits -> words kg..kg+3 (16 bytes); 2 and 3 bits -> words
// kg/2, kg/2 + 1 (8 bytes, chunk k in half k % 2 of word k / 2); 3 bits also
// plane word 8 + kg/4, chunk k's bit-2 byte at ((k >> 1) & 1) | ((k & 1) << 1)
// (channel index bits 3 and 4 exchanged).  A packed row is 16 x bits bytes on
// a 16-byte boundary.
template <int BITS>
__device__ __forceinline__ void store_group(int kg, const uint32_t (&lo)[4], const uint32_t (&hb)[4],
                                            uint32_t* codes) {
  if (BITS == 4) {
    *reinterpret_cast<uint4*>(codes + kg) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    return;
  }
  *reinterpret_cast<uint2*>(codes + (kg >> 1)) = make_uint2(lo[0] | (lo[1] << 16), lo[2] | (lo[3] << 16));
  if (BITS == 3) codes[8 + (kg >> 2)] = hb[0] | (hb[2] << 8) | (hb[1] << 16) | (hb[3] << 24);
}

// T' = RN(fl(x - min) r + C) for the four channel pairs of a chunk (the fast
// rule of chunk_codes), element 2i + j from half j of pair i.  Returns true
// when no element has T' low bits in [0, 7] (then every code is bits 16.. of
// T'); false when some element is near a tie and must take the exact rule.
__device__ __forceinline__ bool chunk_T(const uint64_t (&x2)[4], uint64_t mn2, uint64_t r2, uint64_t c2,
                                        uint32_t (&a)[8]) {
  uint32_t low = 0xffffffffu;  // per 16-bit half: the smallest low bits seen
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint64_t t2 = f32x2_fma(f32x2_sub(x2[i], mn2), r2, c2);
    a[2 * i] = (uint32_t)t2;
    a[2 * i + 1] = (uint32_t)(t2 >> 32);
    low = __vminu2(low, __byte_perm(a[2 * i], a[2 * i + 1], 0x5410));
  }
  return __vcmpleu2(low, 0x00070007u) == 0u;
}

// max(|a|, |b|, |c|); NaN if one of them is.
__device__ __forceinline__ float abs_max3(float a, float b, float c) {
  float d;
  asm("max.NaN.abs.f32 %0, %1, %2, %3;\n" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// 4-bit codes of a chunk's four channel pairs, packed in channel order, on the
// fp32 pipe: t = RN(d r + 2^23) holds the rounded quotient f in its low bits, and
// four of them become a 16-bit word by one packed FMA (f_i + 256 f_{i+2}) and one
// integer multiply-add.  Returns true when no quotient is near a tie: e = d r - f
// is within 2e-6 of the exact quotient's distance from f (1 / scale and the
// reference division round by 2^-24 each, quotients below 16), so below 0.499995
// the code is f.  A NaN (an element's, or infinity times a step of infinity) spoils
// the word's other codes too: `top` keeps it, and the chunk counts as near a tie.
// (chunk_T and chunk_bits_T take four integer operations per
// element, and the integer pipe bound these rows: InternVL2.5-8B-shaped prefill with
// salient tokens, 4 layers one by one, 692 us with them, 657 so.)
__device__ __forceinline__ bool chunk_codes4(const uint64_t (&x2)[4], uint64_t mn2, uint64_t r2, uint32_t& lo) {
  const uint64_t m2 = f32x2(0x4B000000u, 0x4B000000u), c256 = f32x2(0xC3800000u, 0xC3800000u);  // 2^23, -256
  uint64_t t[4], g[4];
  float top = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint64_t d = f32x2_sub(x2[i], mn2);
    t[i] = f32x2_fma(d, r2, m2);
    g[i] = f32x2_sub(m2, t[i]);  // -f
    const uint64_t e = f32x2_fma(d, r2, g[i]);
    top = abs_max3(__uint_as_float((uint32_t)e), __uint_as_float((uint32_t)(e >> 32)), top);
  }
  const uint64_t u = f32x2_fma(g[1], c256, t[0]), v = f32x2_fma(g[3], c256, t[2]);
  lo = prmt((uint32_t)u + 16u * (uint32_t)(u >> 32), (uint32_t)v + 16u * (uint32_t)(v >> 32), 0x5410);
  return top < 0.499995f;
}

// Code e (0..31, token order) of one KIVI-style key group row into its packed
// words: 2 / 4 bits at word e / (32 / bits), bit bits * (e mod 32 / bits); 3
// bits: bits 0-1 at word e / 16, bit 2 e mod 16, and bit 2 into plane word 2 at
// bit e with index bits 3 and 4 exchanged.  e is a compile-time constant after
// unrolling, so each is one shift and one or.
template <int BITS>
__device__ __forceinline__ void add_key_code(uint32_t (&wd)[BITS], int e, uint32_t c) {
  if (BITS == 3) {
    wd[e / 16] |= (c & 3u) << (2 * (e % 16));
    wd[2] |= ((c >> 2) & 1u) << ((e & 7) | (((e >> 4) & 1) << 3) | (((e >> 3) & 1) << 4));
  } else {
    constexpr int per = 32 / (BITS == 3 ? 2 : BITS);
    wd[e / per] |= c << (BITS * (e % per));
  }
}

// Min and max of BF16 values held as 16-bit words, by integer maxima that take
// two new words per instruction: of values of both signs the largest is the
// largest signed word, the smallest the largest unsigned one.  (Groups of one
// sign, or with a NaN, which is the largest word of either kind, do not pass
// the test of mixed_signs or of threshold_scale.)
struct PairMinMax {
  uint32_t s, u;
};
__device__ __forceinline__ void minmax2(PairMinMax& m, uint32_t a, uint32_t b) {
  m.s = __vimax3_s16x2(m.s, a, b);
  m.u = __vimax3_u16x2(m.u, a, b);
}
// Both maxima over chunks [k0, k0 + nk) of a row, over both halves (low half).
__device__ __forceinline__ PairMinMax chunk_maxima(const uint4* r4, int k0, int nk) {
  const uint4 f = r4[k0];
  PairMinMax m = {f.x, f.x};
#pragma unroll 4
  for (int k = k0; k < k0 + nk; ++k) {
    const uint4 v = r4[k];
    minmax2(m, v.x, v.y);
    minmax2(m, v.z, v.w);
  }
  return {__vmaxs2(m.s, __byte_perm(m.s, 0u, 0x1032)), __vmaxu2(m.u, __byte_perm(m.u, 0u, 0x1032))};
}

// Min and max (signed zeros folded to +0) of chunks [k0, k0 + nk) of a row.
template <bool MAXIMA>
__device__ __forceinline__ void row_minmax(const uint4* r4, int k0, int nk, float& mn, float& mx) {
  if (MAXIMA && nk > 4) {  // (no gain over a 32-channel group)
    const PairMinMax m = chunk_maxima(r4, k0, nk);
    // values of both signs, all finite; else value by value
    if (((m.u & ~m.s) & 0x8000u) && (m.s & 0x7f80u) != 0x7f80u && (m.u & 0x7f80u) != 0x7f80u) {
      mn = __fadd_rn(__uint_as_float(m.u << 16), 0.0f);
      mx = __fadd_rn(__uint_as_float(m.s << 16), 0.0f);
      return;
    }
  }
  __nv_bfloat162 mn2, mx2;
  {
    const uint4 v = r4[k0];
    mn2 = mx2 = *reinterpret_cast<const __nv_bfloat162*>(&v.x);
  }
#pragma unroll 4
  for (int k = k0; k < k0 + nk; ++k) {
    const uint4 v = r4[k];
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(&w[i]);
      mn2 = __hmin2(mn2, h);
      mx2 = __hmax2(mx2, h);
    }
  }
  mn = __fadd_rn(fminf(__low2float(mn2), __high2float(mn2)), 0.0f);  // -0 -> +0
  mx = __fadd_rn(fmaxf(__low2float(mx2), __high2float(mx2)), 0.0f);
}

// ---------------------------------------------------------------------------
// 2-bit codes by comparison.  The code of x -- the clamped round-half-even of
// fl(fl(x - min) / scale) -- never falls as x grows, and x is a BF16 value, so a
// group's codes are given by three BF16 thresholds: t_k the smallest value
// whose code is above k.  A pair of elements then takes three packed compares
// and three logic operations, against about sixteen instructions for widening,
// scaling, rounding, the near-tie test and packing (chunk_T), and no element
// is ever near a tie: only the thresholds are found by the exact rule, tried on
// the BF16 value nearest min + (k + 1/2) scale and its two neighbours.  Should
// they not bracket t_k (a boundary within the rounding of x - min around zero),
// the group takes the rule of the other widths.
//   The exact rule without a division: with h = k + 1/2 and y = d / scale, the
// rounded quotient is at or over h when y >= h less half the spacing of floats
// below h (the tie goes to h, whose last bit is even), and over h when y > h
// plus half the spacing above; code k + 1 needs the first for k = 1 (3/2 rounds
// up to 2) and the second for k = 0 and 2.  d - h scale is exact in one FMA
// where it is small enough for this to matter.
//   KIVI-style, 16 rows, 32 heads and 3,120 tokens, 4 layers one by one: 715 us, 805
// by the rule of the other widths.  Min-max, 28 layers of 4 heads and 1,460 tokens:
// 22 us by either (not coding-bound).  With __hmin2 / __hmax2 and three candidates
// tried per threshold it was no better than the rule of the other widths.
// ---------------------------------------------------------------------------
// Steps the comparisons serve: scale 2^-25 stays normal, 1 / scale finite.
__device__ __forceinline__ bool threshold_scale(float scale) {
  return scale >= 7.8886090522101181e-31f && scale <= 8.5070591730234616e37f;  // 2^-100, 2^126
}

// The thresholds of a group with extremes mn_x < 0 <= mx and stored pair
// (scale, mn).  Each is the BF16 value c nearest v = fl(h scale + mn) or the
// next one: v is within 2^-22 (|mn| + 3 scale) of the boundary, which is less
// than half the spacing at c unless c is far smaller than the group (false is
// returned then).
__device__ __forceinline__ bool bf16_thresholds(float mn, float scale, uint32_t (&t)[3]) {
  const float small = fmaf(3.0f, scale, fabsf(mn)) * 1.220703125e-4f;  // 2^-13
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float h = (float)k + 0.5f;
    const float edge = scale * (k == 0 ? 2.98023223876953125e-8f       // 2^-25
                                       : (k == 1 ? -5.9604644775390625e-8f   // -2^-24
                                                 : 1.1920928955078125e-7f));  // 2^-23
    const uint32_t c = (__float_as_uint(__fmaf_rn(h, scale, mn)) + 0x8000u) & 0xffff0000u;
    const float e = __fmaf_rn(-h, scale, __fsub_rn(__uint_as_float(c), mn));
    const bool above = k == 1 ? e >= edge : e > edge;
    ok = ok && fabsf(__uint_as_float(c)) >= small;
    t[k] = (above ? c : c + (((int)c < 0) ? 0xffff0000u : 0x10000u)) >> 16;  // the next value up
  }
  return ok;
}

// A pair's code bits as masks over its halves: bit 0 in b0, bit 1 in b1 (t2[k]:
// threshold k of each half; a NaN is above all of them).
__device__ __forceinline__ void code_masks(uint32_t x, const uint32_t (&t2)[3], uint32_t& b0, uint32_t& b1) {
  uint32_t m[3];
#pragma unroll
  for (int k = 0; k < 3; ++k)
    m[k] = __hgeu2_mask(*reinterpret_cast<const __nv_bfloat162*>(&x), *reinterpret_cast<const __nv_bfloat162*>(&t2[k]));
  b0 = m[0] ^ m[1] ^ m[2];
  b1 = m[1];
}

// Two adjacent channels (2c, 2c + 1) of one KIVI-style key group: the 32
// bf16x2 words of the group's tokens at `col` (the group's first staged row,
// then a row pitch apart).  min / max of both channels at once over bf16x2
// pairs (exact); with fp32 metadata and both steps at least 2^-125, the codes
// of both channels come from the paired rule of the token rows (per-lane
// minimum and reciprocal), otherwise each channel takes the scalar group
// quantizer.  Codes and metadata as for one channel.
template <int BITS, bool M16>
__device__ __forceinline__ void quantize_key_pair_any(const char* col, uint32_t* dst0, uint32_t* dst1, char* meta,
                                                  size_t mi) {
  uint32_t w[kKiviGroup];
#pragma unroll
  for (int e = 0; e < kKiviGroup; ++e) w[e] = *reinterpret_cast<const uint32_t*>(col + (size_t)e * kQPitch);
  __nv_bfloat162 mn2 = *reinterpret_cast<const __nv_bfloat162*>(&w[0]), mx2 = mn2;
#pragma unroll
  for (int e = 1; e < kKiviGroup; ++e) {
    const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(&w[e]);
    mn2 = __hmin2(mn2, h);
    mx2 = __hmax2(mx2, h);
  }
  constexpr uint32_t L = (1u << BITS) - 1u;
  const float levels = (float)L;
  float mn[2] = {__fadd_rn(__low2float(mn2), 0.0f), __fadd_rn(__high2float(mn2), 0.0f)};
  const float mx[2] = {__fadd_rn(__low2float(mx2), 0.0f), __fadd_rn(__high2float(mx2), 0.0f)};
  float sc[2];
  bool fast = true;  // both channels: the fast rule applies (see quantize_row_group)
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    sc[j] = __fdiv_rn(__fsub_rn(mx[j], mn[j]), levels);
    const float mn_x = mn[j];
    if (M16) {
      sc[j] = half_sat(sc[j]);
      mn[j] = half_sat(mn[j]);
      if (sc[j] > 0.0f) {
        const float rj = __frcp_rn(sc[j]);
        const float qlo = __fmul_rn(__fsub_rn(mn_x, mn[j]), rj), qhi = __fmul_rn(__fsub_rn(mx[j], mn[j]), rj);
        fast = fast && qlo > -0.25f && qhi < levels + 0.25f;
      } else {
        fast = false;
      }
    } else {
      fast = fast && sc[j] >= 2.3509887e-38f;
    }
    store_meta(meta, mi + j, sc[j], mn[j], M16);
  }
  uint32_t wd0[BITS], wd1[BITS];  // the two channels' packed words, filled code by code
#pragma unroll
  for (int i = 0; i < BITS; ++i) wd0[i] = wd1[i] = 0u;
  uint32_t tie0 = 0u, tie1 = 0u;  // tokens whose code is near a tie
  if (fast) {
    const float r0 = __frcp_rn(sc[0]), r1 = __frcp_rn(sc[1]);
    const uint64_t mn2p = f32x2(__float_as_uint(mn[0]), __float_as_uint(mn[1]));
    const uint64_t r2 = f32x2(__float_as_uint(r0), __float_as_uint(r1));
    const uint32_t cbits = __float_as_uint(192.50006103515625f);  // 192.5 + 4 * 2^-16 (see chunk_codes)
    const uint64_t c2 = f32x2(cbits, cbits);
#pragma unroll
    for (int e = 0; e < kKiviGroup; ++e) {
      const uint64_t t2 = f32x2_fma(f32x2_sub(f32x2(w[e] << 16, w[e] & 0xffff0000u), mn2p), r2, c2);
      const uint32_t a0 = (uint32_t)t2, a1 = (uint32_t)(t2 >> 32);
      add_key_code<BITS>(wd0, e, (a0 >> 16) & L);
      add_key_code<BITS>(wd1, e, (a1 >> 16) & L);
      if (!(a0 & 0xfff8u)) tie0 |= 1u << e;
      if (!(a1 & 0xfff8u)) tie1 |= 1u << e;
    }
  } else {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const bool fast = sc[j] >= 2.3509887e-38f;  // 2^-125
      const float r = __frcp_rn(fast ? sc[j] : 1.0f);
#pragma unroll
      for (int e = 0; e < kKiviGroup; ++e) {
        const float x = __uint_as_float(j ? (w[e] & 0xffff0000u) : (w[e] << 16));
        const uint32_t c = (sc[j] == 0.0f) ? 0u : code_of(__fsub_rn(x, mn[j]), sc[j], r, levels, fast);
        if (j) add_key_code<BITS>(wd1, e, c);
        else add_key_code<BITS>(wd0, e, c);
      }
    }
  }
  // both channels' rows are contiguous (dst1 = dst0 + BITS) and start on a
  // 16-byte (2, 4 bits) or 8-byte (3 bits) boundary: vector stores
  if (BITS == 3) {
    uint2* d2 = reinterpret_cast<uint2*>(dst0);
    d2[0] = make_uint2(wd0[0], wd0[1]);
    d2[1] = make_uint2(wd0[2 % BITS], wd1[0]);
    d2[2] = make_uint2(wd1[1], wd1[2 % BITS]);
  } else {
    uint4* d4 = reinterpret_cast<uint4*>(dst0);
    if (BITS == 2) {
      d4[0] = make_uint4(wd0[0], wd0[1 % BITS], wd1[0], wd1[1 % BITS]);
    } else {
      d4[0] = make_uint4(wd0[0], wd0[1 % BITS], wd0[2 % BITS], wd0[3 % BITS]);
      d4[1] = make_uint4(wd1[0], wd1[1 % BITS], wd1[2 % BITS], wd1[3 % BITS]);
    }
  }
  // near ties by the exact rule, each code written over its stored bits (the
  // positions of add_key_code); side by side in the warp's threads.  (A branch at
  // each element of the loop above was slower: 5% on 14 layers of 14 rows, 16 heads
  // and 856 tokens at 4 bits, 16% on a 3-bit layer of 6 rows; at 2 bits, where the
  // few groups that come here hold up their warps, 4% on LLaVA-NeXT-7B-shaped layers.)
  while (tie0 | tie1) {
    const bool j = tie0 == 0u;
    const int e = __ffs(j ? tie1 : tie0) - 1;
    if (j) tie1 &= tie1 - 1;
    else tie0 &= tie0 - 1;
    const float x = __uint_as_float((uint32_t)reinterpret_cast<const uint16_t*>(col + (size_t)e * kQPitch)[j] << 16);
    const uint32_t c = exact_code(__fsub_rn(x, j ? mn[1] : mn[0]), j ? sc[1] : sc[0], levels);
    uint32_t* dst = j ? dst1 : dst0;
    constexpr int LB = BITS == 4 ? 4 : 2, per = 32 / LB;
    constexpr uint32_t M = (1u << LB) - 1u;
    const int sh = LB * (e % per);
    dst[e / per] = (dst[e / per] & ~(M << sh)) | ((c & M) << sh);
    if (BITS == 3) {
      const int b = (e & 7) | (((e >> 4) & 1) << 3) | (((e >> 3) & 1) << 4);
      dst[2] = (dst[2] & ~(1u << b)) | ((c >> 2) << b);
    }
  }
}

template <int BITS, bool M16>
__device__ __noinline__ void quantize_key_pair_rare(const char* col, uint32_t* dst0, uint32_t* dst1, char* meta, size_t mi) {
  quantize_key_pair_any<BITS, M16>(col, dst0, dst1, meta, mi);
}

// The same; 2 bits by comparison where the group allows it.
template <int BITS, bool M16>
__device__ __forceinline__ void quantize_key_pair(const char* col, uint32_t* dst0, uint32_t* dst1, char* meta,
                                                  size_t mi) {
  if constexpr (BITS != 2) {
    quantize_key_pair_any<BITS, M16>(col, dst0, dst1, meta, mi);
  } else {
    uint32_t w[kKiviGroup];
#pragma unroll
    for (int e = 0; e < kKiviGroup; ++e) w[e] = *reinterpret_cast<const uint32_t*>(col + (size_t)e * kQPitch);
    PairMinMax m = {w[0], w[0]};
#pragma unroll
    for (int e = 1; e + 1 < kKiviGroup; e += 2) minmax2(m, w[e], w[e + 1]);
    minmax2(m, w[kKiviGroup - 1], w[kKiviGroup - 1]);
    uint32_t t[2][3];
    float sc[2], mn[2];
    // both signs in both channels: signed maxima >= 0, unsigned ones with the top bit
    bool ok = ((m.u & ~m.s) & 0x80008000u) == 0x80008000u;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      mn[j] = __fadd_rn(__uint_as_float(j ? m.u & 0xffff0000u : m.u << 16), 0.0f);
      const float mx = __uint_as_float(j ? m.s & 0xffff0000u : m.s << 16);
      sc[j] = __fdiv_rn(__fsub_rn(mx, mn[j]), 3.0f);
      if (M16) {
        sc[j] = half_sat(sc[j]);
        mn[j] = half_sat(mn[j]);
      }
      ok = ok && threshold_scale(sc[j]);
      ok = bf16_thresholds(mn[j], sc[j], t[j]) && ok;
    }
    if (!ok) {
      quantize_key_pair_rare<BITS, M16>(col, dst0, dst1, meta, mi);
      return;
    }
    if (M16)
      *reinterpret_cast<uint2*>(meta + mi * 4) = make_uint2(pack_half2(sc[0], mn[0]), pack_half2(sc[1], mn[1]));
    else
      *reinterpret_cast<float4*>(meta + mi * 8) = make_float4(sc[0], mn[0], sc[1], mn[1]);
    const uint32_t t2[3] = {t[0][0] | (t[1][0] << 16), t[0][1] | (t[1][1] << 16), t[0][2] | (t[1][2] << 16)};
    uint32_t acc[4] = {0u, 0u, 0u, 0u};  // tokens 8i..8i+7 of both channels, one per half
#pragma unroll
    for (int e = 0; e < kKiviGroup; ++e) {
      uint32_t b0, b1;
      code_masks(w[e], t2, b0, b1);
      acc[e / 8] |= b0 & (0x00010001u << (2 * (e % 8)));
      acc[e / 8] |= b1 & (0x00020002u << (2 * (e % 8)));
    }
    *reinterpret_cast<uint4*>(dst0) = make_uint4(prmt(acc[0], acc[1], 0x5410), prmt(acc[2], acc[3], 0x5410),
                                                 prmt(acc[0], acc[1], 0x7632), prmt(acc[2], acc[3], 0x7632));
  }
}

// Codes of the 8 channels of one chunk (four BF16 pairs w[0..3]) in a group
// with minimum mn and step scale > 0, r = RN(1 / scale):
//   M16 (binary16 metadata, always a normal r): a binary16 scale is at least
//     2^-24, so r is finite.  The rounded zero and scale can put a quotient
//     outside [0, levels]: q = d r is clamped to [-1, levels + 1] (which
//     decides no code differently), then T = RN(q + 192) lies in
//     [191, 193 + levels] and bits 16.. of T + 0x8001, less 0x4340, are the
//     unclamped code.  The two roundings (q, then T) keep T within 2^-16 of
//     fl(d / scale) + 192 for quotients that can decide a code, so an element
//     whose low bits are not within one unit of 0x8000 rounds as the exact
//     rule does; the others take it.
//   fast (scale >= 2^-125, 1 / scale finite): two channels per paired
//     operation, d = fl(x - min), then T' = RN(d r + C) with
//     C = 192.5 + 4 * 2^-16.  In [128, 256) the grid is 2^-16, so T' is
//     T = RN(d r + 192) moved by 0x8004 units (one unit more or less when
//     d r + 192 falls exactly between two grid points, where the shift by an
//     even count flips the tie-break).  Bits 16.. of T' are then
//     floor(d r + 0.5) away from ties, and the error of T' against the exact
//     quotient is below two units (0.5 FMA rounding, 1/16 for r, 1/16 for the
//     reference division, 1 for the tie-break), so every element within two
//     units of the half-integer boundary -- T' low bits in [2, 6] -- is among
//     those with low bits in [0, 7], which take the exact rule (chunk_T,
//     chunk_bits_T; a chunk with such an element goes through chunk_near_tie).
//   otherwise (tiny scale): the exact rule for every element.
template <int BITS, bool M16>
__device__ __forceinline__ void chunk_codes(const uint32_t (&w)[4], float mn, float scale, float r,
                                            uint32_t (&c8)[8]) {
  constexpr uint32_t L = (1u << BITS) - 1u;
  const float levels = (float)L;
  if constexpr (M16) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t hw = w[i >> 1];
      const float d = __fsub_rn(__uint_as_float((i & 1) ? (hw & 0xffff0000u) : (hw << 16)), mn);
      const float q = fminf(fmaxf(__fmul_rn(d, r), -1.0f), levels + 1.0f);
      const uint32_t a = __float_as_uint(__fadd_rn(q, 192.0f)) + 0x8001u;
      const int cu = min(max((int)(a >> 16) - 0x4340, 0), (int)L);
      c8[i] = ((a & 0xffffu) < 3u) ? exact_code(d, scale, levels) : (uint32_t)cu;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t hw = w[i >> 1];
      const float x = __uint_as_float((i & 1) ? (hw & 0xffff0000u) : (hw << 16));
      c8[i] = exact_code(__fsub_rn(x, mn), scale, levels);
    }
  }
}

// Codes of a chunk that has an element near a tie: bits 16.. of T' for the
// others, the exact rule for the elements with T' low bits in [0, 7].
// x(i) gives element i's value.
template <int BITS, class X>
__device__ __forceinline__ void chunk_near_tie(const uint32_t (&a)[8], X x, float mn, float scale,
                                               uint32_t (&c8)[8]) {
  constexpr uint32_t L = (1u << BITS) - 1u;
#pragma unroll
  for (int i = 0; i < 8; ++i)
    c8[i] = (a[i] & 0xfff8u) ? ((a[i] >> 16) & L) : exact_code(__fsub_rn(x(i), mn), scale, (float)L);
}

// Elements near a tie of chunk k of a packed row that this thread has already
// stored, coded again by the exact rule, each written over its bits: word k (4
// bits), or half k % 2 of word k / 2 (2 and 3 bits) and, at 3 bits, byte
// ((k >> 1) & 1) | ((k & 1) << 1) of plane word 8 + k / 4 (the layout of
// store_group).  The other elements' codes, which the fast rule decided, are read
// back and kept, or (4 bits, where a NaN would have spoiled them) taken from T'
// again.  The loop runs over a thread's own elements near a
// tie (mostly one), so the threads of a warp divide side by side; with the eight
// elements in turn a warp went through nearly all eight for its threads'
// different ones: 15% slower on 4-bit layers of 862 to 1,560 tokens, 10% on 3-bit
// ones of 7,415.
template <int BITS>
__device__ __forceinline__ void recode_near_ties(const uint4* r4, int k, uint64_t mn2, uint64_t r2, uint64_t c2, float mn,
                                                 float scale, uint32_t* codes) {
  const uint4 v = r4[k];
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  uint64_t x2[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) x2[i] = f32x2(w[i] << 16, w[i] & 0xffff0000u);
  uint32_t a[8], el = 0u;  // bit i: T' low bits of element i in [0, 7]
  chunk_T(x2, mn2, r2, c2, a);
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (!(a[i] & 0xfff8u)) el |= 1u << i;
  uint32_t* lw = codes + (BITS == 4 ? k : k >> 1);
  uint32_t* hw = codes + 8 + (k >> 2);
  const int ls = BITS == 4 ? 0 : 16 * (k & 1), hs = 8 * (((k >> 1) & 1) | ((k & 1) << 1));
  uint32_t lo, hb;
  if (BITS == 4) {
    chunk_bits_T<4>(a, lo, hb);
  } else {
    lo = *lw;
    hb = BITS == 3 ? *hw : 0u;
  }
  while (el) {
    const int i = __ffs(el) - 1;
    el &= el - 1;
    const float x = __uint_as_float((uint32_t)reinterpret_cast<const uint16_t*>(r4 + k)[i] << 16);
    const uint32_t c = exact_code(__fsub_rn(x, mn), scale, (float)((1u << BITS) - 1u));
    constexpr int LB = BITS == 4 ? 4 : 2;
    constexpr uint32_t M = (1u << LB) - 1u;
    lo = (lo & ~(M << (ls + LB * i))) | ((c & M) << (ls + LB * i));
    if (BITS == 3) hb = (hb & ~(1u << (hs + i))) | ((c >> 2) << (hs + i));
  }
  *lw = lo;
  if (BITS == 3) *hw = hb;
}

// One group of a BF16 row: chunks [k0, k0 + nk) (8 channels each) with their
// min / max over bf16x2 pairs (exact), signed zeros folded to +0,
// scale = fl((max - min) / levels), metadata stored at index mi (binary16
// pair with M16: codes against the rounded pair), codes 0 when scale == 0.
// The chunks go in groups of four (a KIVI-style value group whole), each
// group's packed words written by one vector store (store_group); the group
// loop stays rolled so that the code stays small in the instruction cache
// (eight chunks per step measured slower on the per-token rows).
// A chunk with an element near a tie (fast rule) is emitted with its fast
// codes and flagged; after the loop each thread codes the elements of its flagged
// chunks that are near a tie again (recode_near_ties).  The threads of a warp do
// this side by side, so a warp pays for the largest number of one thread
// instead of running every thread's near ties one after another inside the
// loop.
template <int BITS, bool M16>
__device__ __forceinline__ void quantize_row_group_any(const uint4* r4, int k0, int nk, uint32_t* codes, char* meta,
                                                   size_t mi) {
  float mn, mx;
  row_minmax<BITS != 2>(r4, k0, nk, mn, mx);  // (2 bits: the groups that bf16_thresholds left)
  const float levels = (float)((1u << BITS) - 1u);
  float scale = __fdiv_rn(__fsub_rn(mx, mn), levels);
  const float mn_x = mn;  // the group's own minimum
  if (M16) {  // binary16 metadata: codes against the stored pair
    scale = half_sat(scale);
    mn = half_sat(mn);
  }
  store_meta(meta, mi, scale, mn, M16);
  bool fast = !M16 && scale >= 2.3509887e-38f;  // 2^-125: 1 / scale is finite
  const float r = (M16 || fast) ? __frcp_rn(scale) : 1.0f;
  if (M16 && scale > 0.0f) {
    // With the rounded pair the quotients fl(fl(x - min16) r) of the group run
    // monotonically from the group minimum's to the maximum's.  When both lie
    // well inside (-1/2, levels + 1/2), every code is in [0, levels] without a
    // clamp, and the fast rule of the fp32 pairs (exact against the IEEE
    // quotient, with the same near-tie window) applies to the stored pair.
    const float qlo = __fmul_rn(__fsub_rn(mn_x, mn), r), qhi = __fmul_rn(__fsub_rn(mx, mn), r);
    fast = qlo > -0.25f && qhi < levels + 0.25f;
  }
  const uint64_t mnp = f32x2(__float_as_uint(mn), __float_as_uint(mn));
  const uint64_t r2 = f32x2(__float_as_uint(r), __float_as_uint(r));
  const uint32_t cbits = __float_as_uint(192.50006103515625f);  // C = 192.5 + 4 * 2^-16
  const uint64_t c2 = f32x2(cbits, cbits);
  uint32_t ties = 0u;  // bit k - k0: chunk k has an element near a tie
#pragma unroll 1
  for (int kg = k0; kg < k0 + nk; kg += 4) {
    uint32_t lo[4], hb[4];
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      const int k = kg + kk;
      const uint4 v = r4[k];
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
      if (fast) {
        uint64_t x2[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) x2[i] = f32x2(w[i] << 16, w[i] & 0xffff0000u);  // channels 2i, 2i + 1
        if constexpr (BITS == 4) {
          if (!chunk_codes4(x2, mnp, r2, lo[kk])) ties |= 1u << (k - k0);
        } else {
          uint32_t a[8];
          if (!chunk_T(x2, mnp, r2, c2, a)) ties |= 1u << (k - k0);  // about one chunk in 100
          chunk_bits_T<BITS>(a, lo[kk], hb[kk]);
        }
      } else {
        uint32_t c8[8];
        if (scale == 0.0f) {  // constant group (or a step below binary16 range): every code 0
#pragma unroll
          for (int i = 0; i < 8; ++i) c8[i] = 0u;
        } else {
          chunk_codes<BITS, M16>(w, mn, scale, r, c8);
        }
        chunk_bits<BITS>(c8, lo[kk], hb[kk]);
      }
    }
    store_group<BITS>(kg, lo, hb, codes);
  }
  while (ties) {
    const int k = k0 + (__ffs(ties) - 1);
    ties &= ties - 1;
    recode_near_ties<BITS>(r4, k, mnp, r2, c2, mn, scale, codes);
  }
}

template <int BITS, bool M16>
__device__ __noinline__ void quantize_row_group_rare(const uint4* r4, int k0, int nk, uint32_t* codes, char* meta,
                                                     size_t mi) {
  quantize_row_group_any<BITS, M16>(r4, k0, nk, codes, meta, mi);
}

// The same; 2 bits by comparison where the group allows it.
template <int BITS, bool M16>
__device__ __forceinline__ void quantize_row_group(const uint4* r4, int k0, int nk, uint32_t* codes, char* meta,
                                                   size_t mi) {
  if constexpr (BITS != 2) {
    quantize_row_group_any<BITS, M16>(r4, k0, nk, codes, meta, mi);
  } else {
    PairMinMax m;
    {
      const uint4 v = r4[k0];
      m = {v.x, v.x};
    }
#pragma unroll 4
    for (int k = k0; k < k0 + nk; ++k) {
      const uint4 v = r4[k];
      minmax2(m, v.x, v.y);
      minmax2(m, v.z, v.w);
    }
    const uint32_t ms = __vmaxs2(m.s, __byte_perm(m.s, 0u, 0x1032)), mu = __vmaxu2(m.u, __byte_perm(m.u, 0u, 0x1032));
    float mn = __fadd_rn(__uint_as_float(mu << 16), 0.0f);  // -0 -> +0
    const float mx = __uint_as_float(ms << 16);
    float scale = __fdiv_rn(__fsub_rn(mx, mn), 3.0f);
    if (M16) {
      scale = half_sat(scale);
      mn = half_sat(mn);
    }
    uint32_t t[3];
    if (!bf16_thresholds(mn, scale, t) || !threshold_scale(scale) || !((mu & ~ms) & 0x8000u)) {
      quantize_row_group_rare<BITS, M16>(r4, k0, nk, codes, meta, mi);
      return;
    }
    store_meta(meta, mi, scale, mn, M16);
    const uint32_t t2[3] = {t[0] * 0x10001u, t[1] * 0x10001u, t[2] * 0x10001u};
#pragma unroll 1
    for (int kg = k0; kg < k0 + nk; kg += 4) {
      uint32_t acc[4];  // a chunk's even channels in the low half, odd ones in the high half, in place
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        const uint4 v = r4[kg + kk];
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        acc[kk] = 0u;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          uint32_t b0, b1;
          code_masks(w[i], t2, b0, b1);
          acc[kk] |= b0 & (0x00040001u << (4 * i));
          acc[kk] |= b1 & (0x00080002u << (4 * i));
        }
      }
      *reinterpret_cast<uint2*>(codes + (kg >> 1)) =
          make_uint2(prmt(acc[0], acc[1], 0x5410) | prmt(acc[0], acc[1], 0x7632),
                     prmt(acc[2], acc[3], 0x5410) | prmt(acc[2], acc[3], 0x7632));
    }
  }
}

// Per-token min-max over the whole 128-channel row (Sec. 1), one group.
template <int BITS, bool M16>
__device__ __forceinline__ void quantize_row_token(const char* row_s, uint32_t* codes, char* meta, size_t mi) {
  quantize_row_group<BITS, M16>(reinterpret_cast<const uint4*>(row_s), 0, 16, codes, meta, mi);
}

// KIVI-style values (Sec. 4): four groups of 32 channels per token
// (metadata mi .. mi + 3); the packing is the per-token one (channel order).
template <int BITS, bool M16>
__device__ __forceinline__ void quantize_row_kivi_v(const char* row_s, uint32_t* codes, char* meta, size_t mi) {
#pragma unroll 1
  for (int j = 0; j < 4; ++j)
    quantize_row_group<BITS, M16>(reinterpret_cast<const uint4*>(row_s), 4 * j, 4, codes, meta, mi + j);
}

// ---------------------------------------------------------------------------
// AKVQ-style keys (Sec. 4): the BF16 row is widened into 64 packed fp32 pairs
// (channels 2m, 2m + 1), rotated by the normalised Hadamard-128 in registers
// -- stage h = 1 inside each pair, stages h = 2..64 on whole pairs (both
// halves of a pair meet the same partner offset), the 1/sqrt(128) factor once
// at the end, the same butterflies in the same order as the warp-wide
// transform -- and quantized per token like the min-max rows above, with the
// same exact code rule.  SPLIT = 2 spreads a row over the lanes hh = 0, 1 of
// a lane pair (pmask): lane hh holds pairs 32 hh .. 32 hh + 31 (channels
// 64 hh ..), runs stages 2..32 alone, meets its partner for stage 64 and for
// the row's min / max by shuffles, and codes chunks 8 hh .. 8 hh + 7 into its
// own words of the packed row (lane 0 stores the metadata).  Half the pairs
// per thread: twice the rows resident.  Bound by instruction issue: stage 64 as
// one FMA by +-1, not a sum, a difference and a selection, is 5% of an
// InternVL2.5-8B-shaped prefill with salient tokens (657 us for 4 layers one by one).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float pair_lo(uint64_t x) { return __uint_as_float((uint32_t)x); }
__device__ __forceinline__ float pair_hi(uint64_t x) { return __uint_as_float((uint32_t)(x >> 32)); }

__device__ __forceinline__ uint64_t shfl_xor_pair(unsigned mask, uint64_t x, int m) {
  const uint32_t lo = __shfl_xor_sync(mask, (uint32_t)x, m), hi = __shfl_xor_sync(mask, (uint32_t)(x >> 32), m);
  return ((uint64_t)hi << 32) | lo;
}

template <int BITS, bool M16, int SPLIT>
__device__ __forceinline__ void quantize_row_rotated(const char* row_s, int hh, unsigned pmask, uint64_t nz,
                                                     uint32_t* codes, char* meta, size_t mi) {
  constexpr int NP = 64 / SPLIT;  // pairs per thread
  constexpr int NK = 16 / SPLIT;  // chunks per thread
  const uint32_t* r32 = reinterpret_cast<const uint32_t*>(row_s) + NP * hh;
  const int k0 = NK * hh;
  uint64_t xp[NP];
#pragma unroll
  for (int m = 0; m < NP; ++m) {
    const uint32_t w = r32[m];
    const float a = __uint_as_float(w << 16), b = __uint_as_float(w & 0xffff0000u);
    xp[m] = f32x2(__float_as_uint(__fadd_rn(a, b)), __float_as_uint(__fsub_rn(a, b)));  // stage h = 1
  }
#pragma unroll
  for (int hp = 1; hp < NP; hp <<= 1) {  // stage h = 2 hp
#pragma unroll
    for (int m = 0; m < NP; ++m) {
      if (m & hp) continue;
      const uint64_t a = xp[m], b = xp[m + hp];
      xp[m] = f32x2_add(a, b);
      xp[m + hp] = f32x2_sub(a, b);
    }
  }
  if (SPLIT == 2) {  // stage h = 64: pair m of lane 0 with pair m of lane 1, o + x or o - x (a product by 1 is exact)
    const uint32_t sb = hh ? 0xBF800000u : 0x3F800000u;
    const uint64_t s2 = f32x2(sb, sb);
#pragma unroll
    for (int m = 0; m < NP; ++m) {
      const uint64_t o = shfl_xor_pair(pmask, xp[m], 1);
      xp[m] = f32x2_fma(xp[m], s2, o);
    }
  }
  {
    const uint32_t cb = __float_as_uint(hadamard_c());
    const uint64_t c2 = f32x2(cb, cb);
#pragma unroll
    for (int m = 0; m < NP; ++m) xp[m] = f32x2_product(xp[m], c2, nz);
  }
  // min / max of the rotated vector (exact; signed zeros folded to +0)
  float mn = fminf(pair_lo(xp[0]), pair_hi(xp[0])), mx = fmaxf(pair_lo(xp[0]), pair_hi(xp[0]));
  {
    float mn1 = fminf(pair_lo(xp[1]), pair_hi(xp[1])), mx1 = fmaxf(pair_lo(xp[1]), pair_hi(xp[1]));
#pragma unroll
    for (int m = 2; m < NP; m += 2) {
      mn = fminf(mn, fminf(pair_lo(xp[m]), pair_hi(xp[m])));
      mx = fmaxf(mx, fmaxf(pair_lo(xp[m]), pair_hi(xp[m])));
      mn1 = fminf(mn1, fminf(pair_lo(xp[m + 1]), pair_hi(xp[m + 1])));
      mx1 = fmaxf(mx1, fmaxf(pair_lo(xp[m + 1]), pair_hi(xp[m + 1])));
    }
    mn = fminf(mn, mn1);
    mx = fmaxf(mx, mx1);
  }
  if (SPLIT == 2) {
    mn = fminf(mn, __shfl_xor_sync(pmask, mn, 1));
    mx = fmaxf(mx, __shfl_xor_sync(pmask, mx, 1));
  }
  mn = __fadd_rn(mn, 0.0f);
  mx = __fadd_rn(mx, 0.0f);
  constexpr uint32_t L = (1u << BITS) - 1u;
  const float levels = (float)L;
  float scale = __fdiv_rn(__fsub_rn(mx, mn), levels);
  const float mn_x = mn;
  if (M16) {
    scale = half_sat(scale);
    mn = half_sat(mn);
  }
  if (hh == 0) store_meta(meta, mi, scale, mn, M16);
  uint32_t lo[NK], hb[NK];  // this thread's chunks k0..k0+NK-1, stored four at a time at the end
  auto store_all = [&]() {
#pragma unroll
    for (int g = 0; g < NK / 4; ++g) {
      const uint32_t l4[4] = {lo[4 * g], lo[4 * g + 1], lo[4 * g + 2], lo[4 * g + 3]};
      const uint32_t h4[4] = {hb[4 * g], hb[4 * g + 1], hb[4 * g + 2], hb[4 * g + 3]};
      store_group<BITS>(k0 + 4 * g, l4, h4, codes);
    }
  };
  if (scale == 0.0f) {
#pragma unroll
    for (int k = 0; k < NK; ++k) lo[k] = hb[k] = 0u;
    store_all();
    return;
  }
  bool fast = scale >= 2.3509887e-38f;  // the fast rule of the min-max rows (chunk_T)
  if (M16) {  // with the stored pair: when every quotient is well inside the levels (quantize_row_group)
    const float r = __frcp_rn(scale);
    const float qlo = __fmul_rn(__fsub_rn(mn_x, mn), r), qhi = __fmul_rn(__fsub_rn(mx, mn), r);
    fast = qlo > -0.25f && qhi < levels + 0.25f;
  }
  if (M16 && !fast) {  // as the min-max rows: the quotient clamped, then the same near-tie rule
    const float r = __frcp_rn(scale);
#pragma unroll
    for (int k = 0; k < NK; ++k) {
      uint32_t c8[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const uint64_t x2 = xp[4 * k + (i >> 1)];
        const float d = __fsub_rn((i & 1) ? pair_hi(x2) : pair_lo(x2), mn);
        const float q = fminf(fmaxf(__fmul_rn(d, r), -1.0f), levels + 1.0f);
        const uint32_t a = __float_as_uint(__fadd_rn(q, 192.0f)) + 0x8001u;
        const int cu = min(max((int)(a >> 16) - 0x4340, 0), (int)L);
        c8[i] = ((a & 0xffffu) < 3u) ? exact_code(d, scale, levels) : (uint32_t)cu;
      }
      chunk_bits<BITS>(c8, lo[k], hb[k]);
    }
    store_all();
    return;
  }
  if (fast) {  // the fast rule of the min-max rows (chunk_T)
    const float r = __frcp_rn(scale);
    const uint64_t mn2 = f32x2(__float_as_uint(mn), __float_as_uint(mn));
    const uint64_t r2 = f32x2(__float_as_uint(r), __float_as_uint(r));
    const uint32_t cbits = __float_as_uint(192.50006103515625f);  // 192.5 + 4 * 2^-16
    const uint64_t c2 = f32x2(cbits, cbits);
#pragma unroll
    for (int k = 0; k < NK; ++k) {
      const uint64_t x2[4] = {xp[4 * k], xp[4 * k + 1], xp[4 * k + 2], xp[4 * k + 3]};
      uint32_t a[8];
      if (BITS == 4 ? chunk_codes4(x2, mn2, r2, lo[k]) : chunk_T(x2, mn2, r2, c2, a)) {
        if (BITS != 4) chunk_bits_T<BITS>(a, lo[k], hb[k]);
      } else {
        if (BITS == 4) chunk_T(x2, mn2, r2, c2, a);
        uint32_t c8[8];
        chunk_near_tie<BITS>(a, [&](int i) { return (i & 1) ? pair_hi(x2[i >> 1]) : pair_lo(x2[i >> 1]); }, mn,
                             scale, c8);
        chunk_bits<BITS>(c8, lo[k], hb[k]);
      }
    }
    store_all();
    return;
  }
#pragma unroll
  for (int k = 0; k < NK; ++k) {  // tiny scale: the exact rule throughout
    uint32_t c8[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint64_t x2 = xp[4 * k + (i >> 1)];
      c8[i] = exact_code(__fsub_rn((i & 1) ? pair_hi(x2) : pair_lo(x2), mn), scale, levels);
    }
    chunk_bits<BITS>(c8, lo[k], hb[k]);
  }
  store_all();
}

// A BF16 row copied as it is (SPLIT = 2: lane hh of a pair copies its half).
template <int SPLIT = 1>
__device__ __forceinline__ void copy_row(char* dst, const char* row_s, int hh = 0) {
#pragma unroll
  for (int k = 0; k < 16 / SPLIT; ++k) {
    const int c = (16 / SPLIT) * hh + k;
    reinterpret_cast<uint4*>(dst)[c] = reinterpret_cast<const uint4*>(row_s)[c];
  }
}

// Staged rows of one warp tile: row r < n holds token t0 + r, 272-byte pitch.
using StagedRows = char[kQTok][kQPitch];

// Rows 0..n-1 of a tile to n consecutive BF16 rows at dst, by the whole warp:
// lane l stores chunk l % 16 of rows l / 16, l / 16 + 2, ... (512 contiguous
// bytes per store instruction).
__device__ __forceinline__ void copy_rows_warp(char* dst, const StagedRows& rows, int n) {
  const int col = threadIdx.x & 15;
#pragma unroll
  for (int i = 0; i < kQTok / 2; ++i) {
    const int r = (threadIdx.x >> 4) + 2 * i;
    if (r < n)
      *reinterpret_cast<uint4*>(dst + (size_t)r * 256 + col * 16) = *reinterpret_cast<const uint4*>(&rows[r][col * 16]);
  }
}

// Region map of KV head h of the launch's layer li.
__device__ __forceinline__ HeadGeom quantize_head(const QuantizeParams& p, int li, int h) {
  return head_geom_at(p.d, p.gt.gc, p.gt.off[li], p.lt.mask[li], h);
}

// Token span of a tile: rows r < n hold tokens t0 + r.
struct TileSpan {
  int t0, n, tlo;  // tlo: the unclipped tile start (KIVI-style tiles)
};

// Coalesced staging of one part (K or V rows) of a tile by the CTA's warp:
// lane l copies 16-byte chunks l, l + 32, ... of the tile's contiguous rows
// (every chunk in flight at once); the caller commits the group.
__device__ __forceinline__ void stage_rows(const QuantizeParams& p, int li, int b, int h, int kv, const TileSpan& sp,
                                           StagedRows& rows) {
  const Dims& d = p.d;
  const size_t row0 = ((size_t)b * d.H + h) * (size_t)d.T + sp.t0;
  const int col = threadIdx.x & 15;  // lane l: chunk l % 16 of rows l / 16, l / 16 + 2, ...
  const char* src = reinterpret_cast<const char*>((kv ? p.v[li] : p.k[li]) + row0 * kD) + col * 16;
#pragma unroll
  for (int i = 0; i < kQTok / 2; ++i) {
    const int r = (threadIdx.x >> 4) + 2 * i;
    if (r < sp.n) cp_async16(smem_u32(&rows[r][col * 16]), src + (size_t)r * 256, 16);
  }
}

// A tile whose rows all go, as they are, to consecutive BF16 rows -- a
// protected K+V head, a tile inside one text run, or the image keys of a
// keys-only head -- copied by the whole warp, two rows per store instruction,
// instead of each lane storing its own row in sixteen pieces.  Returns false
// for any other tile (the rows' own paths then run).  Salient tokens sit in
// coded image spans only, so a text run keeps consecutive positions.  (The
// per-token tiles use it; in the KIVI-style kernels, whose code is longer,
// the extra copy path measured 8% slower.)
__device__ __forceinline__ bool copy_tile_whole(const QuantizeParams& p, int li, int b, int kv, const TileSpan& sp,
                                                const StagedRows& rows, const HeadGeom& hd) {
  const Dims& d = p.d;
  const int qs = d.s, qe = d.s + d.nq, t0 = sp.t0, t1 = sp.t0 + sp.n;
  char* Lb = p.arena + p.lt.base[li];
  const char* dst;
  if (hd.cls == kProtected || t1 <= qs || t0 >= qe)
    dst = Lb + (kv ? hd.vb : hd.kb) + b * hd.kb_bs + (size_t)bf16_pos(d, hd.cls, t0) * 256;
  else if (kv == 0 && hd.cls == kKeysOnly && t0 >= qs && t1 <= qe && d.ns == 0)
    dst = Lb + hd.kimg + b * hd.kimg_bs + (size_t)(t0 - qs) * 256;
  else
    return false;
  copy_rows_warp(const_cast<char*>(dst), rows, sp.n);
  return true;
}

// The per-token bases, one thread per vector: min-max rows (Sec. 1) and
// AKVQ-style rows (Sec. 4: keys rotated first; values per token, unrotated).
// Tiles of 32 tokens from token 0; a CTA (one warp) takes the K rows or the V
// rows of a tile.  With salient tokens (AKVQ-style, Sec. 4) a thread finds its
// token in the head's map: a salient token's K and V rows go to the BF16 region
// at position s + (its rank), every other image token to coded slot ti - (the
// salient tokens before it).
template <int BITS, bool M16, int BASE>
struct TokenTiles {
  static constexpr bool kKeysFirst = BASE == kAkvq;
  // 96: 20 warps per SM, where the rotated rows and the value rows of one kernel come
  // to 99 and 16 (InternVL2.5-8B-shaped prefill with salient tokens, 4 layers one by
  // one, 657 and 692 us; at most two registers spilled); 80: what the rows take anyway.
  static constexpr int kRegisters = BASE == kAkvq ? 96 : 80;
  static __device__ __forceinline__ TileSpan span(const QuantizeParams& p, int tx) {
    TileSpan sp;
    sp.t0 = sp.tlo = tx * kQTok;
    sp.n = min(kQTok, p.d.T - sp.t0);
    return sp;
  }
  // Row r of the tile; SPLIT = 2: lane hh of the row's lane pair (pmask).
  template <int SPLIT>
  static __device__ __forceinline__ void row(const QuantizeParams& p, int li, int b, int kv, const TileSpan& sp,
                                             const StagedRows& rows, const HeadGeom& hd, int r, int hh,
                                             unsigned pmask) {
    const Dims& d = p.d;
    char* Lb = p.arena + p.lt.base[li];
    const int t = sp.t0 + r;
    const bool coded = t >= d.s && t < d.s + d.nq;
    const int ti = t - d.s;
    int ci = ti, pos = bf16_pos(d, hd.cls, t);
    bool sal = false;
    if (BASE == kAkvq && coded && d.ns > 0 && hd.cls != kProtected) {
      const char* sm = Lb + hd.sal + b * hd.sal_bs;
      const int w = ti >> 5, e = ti & 31;
      const uint32_t sb = reinterpret_cast<const uint32_t*>(sm)[w];
      const int rank = reinterpret_cast<const int*>(sm + (size_t)sal_blocks(d) * 4)[w] +
                       __popc(sb & ((1u << e) - 1u));
      sal = (sb >> e) & 1u;
      ci = ti - rank;
      if (sal) pos = d.s + rank;
    }
    const char* row_s = rows[r];
    constexpr int W = 4 * BITS;
    if (kv == 0) {
      if (coded && hd.cls == kQuantized && !sal) {
        uint32_t* crow = reinterpret_cast<uint32_t*>(Lb + hd.kq + b * hd.kq_bs) + (size_t)ci * W;
        if constexpr (SPLIT == 2)
          quantize_row_rotated<BITS, M16, SPLIT>(row_s, hh, pmask, p.neg_zero2, crow, Lb + hd.kqm + b * hd.kqm_bs,
                                                 ci);
        else if constexpr (BASE != kAkvq)
          quantize_row_token<BITS, M16>(row_s, crow, Lb + hd.kqm + b * hd.kqm_bs, ci);
        return;
      }
      char* dst = (coded && hd.cls == kKeysOnly && !sal) ? Lb + hd.kimg + b * hd.kimg_bs + (size_t)ci * 256
                                                         : Lb + hd.kb + b * hd.kb_bs + (size_t)pos * 256;
      copy_row<SPLIT>(dst, row_s, hh);
    } else if constexpr (SPLIT == 1) {
      if (coded && hd.cls != kProtected && !sal) {
        quantize_row_token<BITS, M16>(row_s, reinterpret_cast<uint32_t*>(Lb + hd.vq + b * hd.vq_bs) + (size_t)ci * W,
                                      Lb + hd.vqm + b * hd.vqm_bs, ci);
        return;
      }
      copy_row<1>(Lb + hd.vb + b * hd.kb_bs + (size_t)pos * 256, row_s, 0);
    }
  }
  static __device__ __forceinline__ void process(const QuantizeParams& p, int li, int b, int kv, const TileSpan& sp,
                                                 const StagedRows& rows, const HeadGeom& hd) {
    if (copy_tile_whole(p, li, b, kv, sp, rows, hd)) return;
    if constexpr (BASE == kAkvq) {
      if (kv == 0) {
        // rotated key rows: two lanes per row, rows lane / 2 and 16 + lane / 2
        // (both lanes of a pair take the same path, so the pair's shuffles meet)
        const int hh = threadIdx.x & 1;
        const unsigned pmask = 3u << (threadIdx.x & 30);
#pragma unroll 1
        for (int r = threadIdx.x >> 1; r < sp.n; r += 16) row<2>(p, li, b, 0, sp, rows, hd, r, hh, pmask);
        return;
      }
    }
    if ((int)threadIdx.x < sp.n) row<1>(p, li, b, kv, sp, rows, hd, threadIdx.x, 0, 0u);
  }
};

// ---------------------------------------------------------------------------
// KIVI-style base (Sec. 4), on staged rows as above: one CTA (one warp) per
// (32-token tile, K or V rows, batch row, KV head, layer), tiles aligned so
// that each of the image's 32-token key groups (anchored at the image start)
// is one whole tile.  Values of every head whose image values are coded: one
// thread per token row, four 32-channel groups.  Keys of a quantized head:
// lane c quantizes channel pairs c and c + 32 over the tile's key group (32
// consecutive image tokens, packed in token order).  Every other row (text,
// the BF16 residual window and a trailing partial group, protected heads,
// keys of keys-only heads) is copied.
// ---------------------------------------------------------------------------
template <int BITS, bool M16>
struct KiviTiles {
  static constexpr bool kKeysFirst = true;
  static constexpr int kRegisters = 80;  // what the rows take anyway
  // tile x: [origin - 32 + 32 x, + 32) clipped to [0, T), origin = s mod 32
  static __device__ __forceinline__ TileSpan span(const QuantizeParams& p, int tx) {
    TileSpan sp;
    sp.tlo = p.tile_origin - kKiviGroup + kQTok * tx;
    sp.t0 = max(sp.tlo, 0);
    sp.n = min(sp.tlo + kQTok, p.d.T) - sp.t0;
    return sp;
  }
  static __device__ __forceinline__ void process(const QuantizeParams& p, int li, int b, int kv, const TileSpan& sp,
                                                 const StagedRows& rows, const HeadGeom& hd) {
    const Dims& d = p.d;
    const int lane = threadIdx.x;
    char* Lb = p.arena + p.lt.base[li];
    const int qs = d.s, qe = d.s + d.nq;
    const int t0 = sp.t0, tlo = sp.tlo;
    constexpr int W = 4 * BITS;
    if (kv == 1) {
      if (lane >= sp.n) return;
      const int t = t0 + lane;
      const bool coded = t >= qs && t < qe;
      const int ti = t - qs;
      if (coded && hd.cls != kProtected)
        quantize_row_kivi_v<BITS, M16>(rows[lane], reinterpret_cast<uint32_t*>(Lb + hd.vq + b * hd.vq_bs) + (size_t)ti * W,
                                       Lb + hd.vqm + b * hd.vqm_bs, (size_t)ti * 4);
      else
        copy_row(Lb + hd.vb + b * hd.kb_bs + (size_t)bf16_pos(d, hd.cls, t) * 256, rows[lane]);
      return;
    }
    // keys: a whole image key group of a quantized head, by channel pairs
    // (uniform over the warp), else the rows are copied
    if (hd.cls == kQuantized && tlo >= qs && tlo + kKiviGroup <= qe && tlo == t0 && sp.n == kKiviGroup) {
      const int grp = (tlo - qs) / kKiviGroup;
#pragma unroll 1
      for (int c2 = lane; c2 < 64; c2 += 32) {
        uint32_t* dst = reinterpret_cast<uint32_t*>(Lb + hd.kq + b * hd.kq_bs) + ((size_t)grp * kD + 2 * c2) * BITS;
        quantize_key_pair<BITS, M16>(&rows[0][4 * c2], dst, dst + BITS, Lb + hd.kqm + b * hd.kqm_bs,
                                     (size_t)grp * kD + 2 * c2);
      }
      return;
    }
    if (lane >= sp.n) return;
    const int t = t0 + lane;
    const bool coded = t >= qs && t < qe;
    if (coded && hd.cls == kQuantized) return;  // unreachable: coded key groups are whole tiles
    copy_row((coded && hd.cls == kKeysOnly) ? Lb + hd.kimg + b * hd.kimg_bs + (size_t)(t - qs) * 256
                                            : Lb + hd.kb + b * hd.kb_bs + (size_t)bf16_pos(d, hd.cls, t) * 256,
             rows[lane]);
  }
};

// The quantizer kernel: one CTA of one warp per (tile, part); grid x = tile,
// y = batch row x KV head, z = layer, and part: the lowest digit of x (min-max),
// or (kKeysFirst) the highest of z, all keys of the launch before all values,
// so that the warps of an SM share one of two unlike code paths at a time.  A
// warp stages its 32 rows, waits for its own copies and codes them; no CTA-wide
// barrier, so the warps of an SM (20 to 23 resident) run out of step and one
// warp's loads overlap another's coding.
// A programmatic dependent launch: its CTAs may come to the SMs while the
// kernels before it still run, and wait for them before their first load (no
// other grid's wait orders this one's reads).  Keys and values are one launch
// because neither needs the other: LLaVA-NeXT-7B-shaped, 4 layers one by one, 712
// us, against 740 with the values in a launch that waits for the keys'.
template <class TP>
__global__ void __maxnreg__(TP::kRegisters) quantize_tiles_kernel(const __grid_constant__ QuantizeParams p) {
  __shared__ __align__(16) StagedRows rows;
  int tx = blockIdx.x, li = blockIdx.z, kv;
  if (TP::kKeysFirst) {
    kv = li >= p.n_layers;
    li -= kv ? p.n_layers : 0;
  } else {
    kv = tx & 1;
    tx >>= 1;
  }
  const int b = blockIdx.y / p.d.H, h = blockIdx.y % p.d.H;
  const TileSpan sp = TP::span(p, tx);
  grid_dependency_wait();
  grid_launch_dependents();
  if (sp.n <= 0) return;
  stage_rows(p, li, b, h, kv, sp, rows);
  cp_async_commit();
  const HeadGeom hd = quantize_head(p, li, h);
  cp_async_wait<0>();
  __syncwarp();
  TP::process(p, li, b, kv, sp, rows, hd);
}

// ---------------------------------------------------------------------------
// AKVQ-style salient tokens (Sec. 4), two launches; protected K+V heads (no
// coded image entries) are left out.  First the squared key norms of the image
// tokens in the fixed binary32 order (32 partial sums of channels 4l..4l+3, then
// five butterfly rounds): a half-warp per row, eight rows per warp in flight,
// CTAs of 64 tokens over the whole GPU; the scores go to the head's own code
// (or BF16) rows, which the quantizer fills after the selection.  Then one CTA
// per (batch row, KV head, layer) selects the ns largest scores (ties to the
// lower index) and writes the map: a bit per image token and the salient count
// before each 32-token block.
//
// A layer of 32 rows, 8 KV heads and 3,328 image tokens (191 MB of keys read, 28 us
// at the measured copy rate): 33 us and 8 us; one CTA per head for both has too
// little in flight (8 KB, 88 us).
// ---------------------------------------------------------------------------
constexpr int kNormThreads = 256, kNormRows = 8, kNormTokens = kNormThreads / 32 * kNormRows;
constexpr int kSalThreads = 512;
// Spans up to this length: the selection's CTA sums the norms itself, one
// launch (a layer of 8 heads in 4 rows, prefill in a stream with one and two
// launches before the quantizer's: 14.4 and 14.0 us with 512 image tokens, 20.6 and
// 17.3 with 1,024; 32 rows: 38.7 and 38.6, 63.2 and 61.8.  Small layers wait for the
// host, whose time a call is that of the launches).
constexpr int kSalOneLaunch = 512;

// Where the scores of one row of a head with coded values wait for the
// selection: its value codes, or its BF16 rows when nearly every token is
// salient (nc tokens of 16 BITS bytes, ns of 256, for nc + ns scores of 4).
__device__ __forceinline__ float* salient_scores(const Dims& d, const HeadGeom& hd, char* Lb, int b) {
  const bool codes = (long long)ncoded(d) * 16 * d.bits >= (long long)d.nq * 4;
  return reinterpret_cast<float*>(codes ? Lb + hd.vq + b * hd.vq_bs : Lb + hd.kb + b * hd.kb_bs);
}

// Squared norm of the key whose channels 8j..8j+7 lane j of a half-warp holds
// (in its lane 0), in the fixed order: partial sums 2j and 2j + 1, round m of
// the butterfly with lane j ^ (m / 2), the last one inside the lane.
__device__ __forceinline__ float key_norm2(const uint4& w) {
  float a[2];
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    float x[4];
    bf16x4_to_f32(e ? make_uint2(w.z, w.w) : make_uint2(w.x, w.y), x);
    a[e] = __fmul_rn(x[0], x[0]);
    a[e] = __fadd_rn(a[e], __fmul_rn(x[1], x[1]));
    a[e] = __fadd_rn(a[e], __fmul_rn(x[2], x[2]));
    a[e] = __fadd_rn(a[e], __fmul_rn(x[3], x[3]));
  }
#pragma unroll
  for (int m = 8; m >= 1; m >>= 1) {
    a[0] = __fadd_rn(a[0], __shfl_xor_sync(kFull, a[0], m));
    a[1] = __fadd_rn(a[1], __shfl_xor_sync(kFull, a[1], m));
  }
  return __fadd_rn(a[0], a[1]);
}

__global__ void __launch_bounds__(kNormThreads) salient_norm_kernel(const __grid_constant__ QuantizeParams p) {
  const Dims& d = p.d;
  grid_dependency_wait();
  grid_launch_dependents();
  const int li = blockIdx.z, b = blockIdx.y / d.H, h = blockIdx.y % d.H;
  if (head_class(d, p.lt.mask[li], h) == kProtected) return;
  const int lane = threadIdx.x & 31, j = lane & 15;
  const int r0 = blockIdx.x * kNormTokens + (threadIdx.x >> 5) * kNormRows + (lane >> 4);
  const uint16_t* K = p.k[li] + (((size_t)b * d.H + h) * d.T + d.s) * kD + 8 * j;
  uint4 w[kNormRows / 2];
#pragma unroll
  for (int i = 0; i < kNormRows / 2; ++i) {
    const int r = r0 + 2 * i;
    w[i] = r < d.nq ? ldg16(K + (size_t)r * kD) : make_uint4(0u, 0u, 0u, 0u);
  }
  float* out = salient_scores(d, quantize_head(p, li, h), p.arena + p.lt.base[li], b);
#pragma unroll
  for (int i = 0; i < kNormRows / 2; ++i) {
    const float norm = key_norm2(w[i]);
    const int r = r0 + 2 * i;
    if (j == 0 && r < d.nq) out[r] = norm;
  }
}

template <bool NORMS>
__global__ void __launch_bounds__(kSalThreads) salient_select_kernel(const __grid_constant__ QuantizeParams p) {
  const Dims& d = p.d;
  const int bh = blockIdx.x, li = blockIdx.y;
  const int b = bh / d.H, h = bh % d.H;
  grid_dependency_wait();
  grid_launch_dependents();
  if (head_class(d, p.lt.mask[li], h) == kProtected) return;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nq = d.nq, nblk = sal_blocks(d);
  extern __shared__ __align__(16) float sal_smem[];
  float* score = sal_smem;                                     // [nq]
  uint32_t* bits = reinterpret_cast<uint32_t*>(sal_smem + nq);  // [nblk]
  const HeadGeom hd = quantize_head(p, li, h);
  if (NORMS) {
    const uint16_t* K = p.k[li] + (((size_t)b * d.H + h) * d.T + d.s) * kD + 8 * (lane & 15);
    constexpr int kStep = kSalThreads / 16;  // rows of one sweep, four sweeps in flight
    for (int r0 = tid >> 4; r0 - (lane >> 4) < nq; r0 += 4 * kStep) {  // whole warps
      uint4 w[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = r0 + i * kStep;
        w[i] = r < nq ? ldg16(K + (size_t)r * kD) : make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = r0 + i * kStep;
        const float norm = key_norm2(w[i]);
        if ((lane & 15) == 0 && r < nq) score[r] = norm;
      }
    }
  } else {
    const float* src = salient_scores(d, hd, p.arena + p.lt.base[li], b);
    for (int i = tid; i < nq; i += kSalThreads) score[i] = src[i];
  }
  __shared__ uint32_t hist[256];
  __shared__ uint32_t s_prefix, s_need, s_eq, s_diff;
  if (tid == 0) {
    s_eq = (uint32_t)nq;
    s_diff = 0u;
  }
  __syncthreads();

  // The ns largest scores, ties to the lower index -- the set that ns rounds
  // of arg-max (taken tokens dropping out) would pick -- by a radix select on
  // the scores' bit patterns (non-negative floats order as their bits): 8-bit
  // digits from the highest bit in which two keys differ, each pass a histogram
  // of the candidates that match the digits chosen so far and the digit where
  // the count of larger keys reaches ns.  When all candidates with that digit are
  // taken, no lower digit matters.  Then every key above the final threshold T is
  // taken, and of the keys equal to T the first `need` by index.  A pass is
  // three barriers, a histogram and a scan, about 2 us: usually two of them, where
  // four fixed digits spent the first on a byte that two values share.  Spread
  // digits make plain atomics the better histogram (one per distinct digit of a
  // warp, found by a match: 2 us more).  A layer of 32 rows, 8 KV heads and 3,328
  // image tokens 8 us, 12 in four fixed passes; with one key far above the others,
  // or all equal, the same.
  static_assert(kSalThreads >= 256, "a thread per histogram bin");
  uint32_t diff = 0u;
  const uint32_t key0 = __float_as_uint(score[0]);
  for (int i = tid; i < nq; i += kSalThreads) diff |= __float_as_uint(score[i]) ^ key0;
  diff = __reduce_or_sync(kFull, diff);
  if (lane == 0 && diff) atomicOr(&s_diff, diff);
  __syncthreads();
  int left_bits = 32 - __clz(s_diff);  // the low bits not decided yet
  uint32_t pmask = left_bits == 32 ? 0u : ~0u << left_bits, prefix = key0 & pmask, need = (uint32_t)d.ns;
#pragma unroll 1
  while (left_bits > 0 && s_eq != need) {
    const int shift = max(left_bits - 8, 0);
    const uint32_t dmask = (1u << (left_bits - shift)) - 1u;
    if (tid < 256) hist[tid] = 0u;
    __syncthreads();
    for (int i0 = warp * 32; i0 < nq; i0 += kSalThreads) {  // warp-uniform: lane i0 + lane
      const int i = i0 + lane;
      const uint32_t key = i < nq ? __float_as_uint(score[i]) : 0u;
      const bool cand = i < nq && (key & pmask) == prefix;
      const uint32_t dg = (key >> shift) & dmask;
      if (cand) atomicAdd(&hist[dg], 1u);
    }
    __syncthreads();
    if (warp == 0) {
      // lane l holds bins 255 - 8l .. 248 - 8l (largest digits first)
      uint32_t c[8], tot = 0u;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        c[j] = hist[255 - 8 * lane - j];
        tot += c[j];
      }
      uint32_t incl = tot;  // keys in this lane's bins and all larger digits
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += v;
      }
      const uint32_t excl = incl - tot;
      if (excl < need && need <= incl) {  // exactly one lane
        uint32_t above = excl;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (above + c[j] >= need) {
            const uint32_t dg = 255u - 8u * lane - j;
            s_prefix = prefix | (dg << shift);
            s_need = need - above;
            s_eq = c[j];
            break;
          }
          above += c[j];
        }
      }
    }
    __syncthreads();
    prefix = s_prefix;
    need = s_need;
    pmask |= dmask << shift;
    left_bits = shift;
  }
  // T = prefix: `need` of the s_eq keys equal to T are taken, by index
  const uint32_t T = prefix;
  if (s_eq == need) {
    for (int w = warp; w < nblk; w += kSalThreads / 32) {
      const int i = w * 32 + lane;
      const bool take = i < nq && __float_as_uint(score[i]) >= T;
      const uint32_t word = __ballot_sync(kFull, take);
      if (lane == 0) bits[w] = word;
    }
  } else if (warp == 0) {
    uint32_t left = need;  // equal keys still to take, in index order
    for (int w = 0; w < nblk; ++w) {
      const int i = w * 32 + lane;
      const uint32_t key = i < nq ? __float_as_uint(score[i]) : 0u;
      const bool eq = i < nq && key == T;
      const uint32_t eqm = __ballot_sync(kFull, eq);
      const uint32_t before = __popc(eqm & ((1u << lane) - 1u));
      const bool take = i < nq && (key > T || (eq && before < left));
      const uint32_t word = __ballot_sync(kFull, take);
      const uint32_t ne = __popc(eqm);
      left = left > ne ? left - ne : 0u;
      if (lane == 0) bits[w] = word;
    }
  }
  __syncthreads();

  char* dst = p.arena + p.lt.base[li] + hd.sal + b * hd.sal_bs;
  uint32_t* out_bits = reinterpret_cast<uint32_t*>(dst);
  int* out_rank = reinterpret_cast<int*>(dst + (size_t)nblk * 4);
  for (int w = tid; w < nblk; w += kSalThreads) out_bits[w] = bits[w];
  if (warp == 0) {
    int before = 0;
    for (int w0 = 0; w0 < nblk; w0 += 32) {
      const int c = w0 + lane < nblk ? __popc(bits[w0 + lane]) : 0;
      int incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += v;
      }
      if (w0 + lane < nblk) out_rank[w0 + lane] = before + incl - c;
      before += __shfl_sync(kFull, incl, 31);
    }
  }
}

// ---------------------------------------------------------------------------
// Reconstruction (Sec. 4: codes to floats, code * scale + zero; AKVQ-style keys
// rotated back; BF16 entries copied), every layer of the launch in original
// token order followed by the appended tokens.  One CTA per span of 32-token
// tiles of a (batch row, KV head, layer), tiles aligned with the image start;
// warps 0-3 take eight rows each of K, warps 4-7 of V.  Almost every such run
// of eight rows is of one kind -- coded tokens, or BF16 rows that lie one after
// the other -- and is found so once per warp: its loads and stores are then at
// constant strides from one address.  The rest (a run across a span's end, or
// with a salient token) resolve each row.
//   Rows: a half-warp per row, lane j channels 8j..8j+7, the warp's eight rows
// in flight together; a BF16 entry written as BF16 is copied as it is.
//   KIVI-style keys: lane l has channels 4l..4l+3 of the group, reads their
// words and metadata once and writes the warp's eight tokens from registers (a
// half-warp per token instead read every word and pair of the group sixteen
// times).
// The AKVQ-style inverse rotation runs its first three butterfly stages inside
// a lane and the last four across the half-warp, in the same order as the
// forward transform.
//
// Bound by DRAM on large caches (four LLaVA-NeXT-7B-shaped layers of 16 rows, BF16
// output: 658 us, 0.99 of the measured copy rate; with every row finding its own
// place, 146 warp instructions per pair of rows, 1,510 us), by the ramp and the tail
// on small ones (Qwen2.5-VL-7B-shaped, 28 layers: 19.8 us; 30.8).
// ---------------------------------------------------------------------------
constexpr int kDqThreads = 256;
constexpr int kDqTile = 32;
constexpr int kDqRows = 8;   // rows of one warp in a tile
// First token of the first tile (0 or less).
HG_HD int dq_origin(const Dims& d) { return d.s % kDqTile ? d.s % kDqTile - kDqTile : 0; }

// Two floats to BF16 bits (round to nearest even, low half first): one cvt.
__device__ __forceinline__ uint32_t pack_bf16x2_rn(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

__device__ __forceinline__ void bf16x8_to_f32(const uint4& w, float (&x)[8]) {
  bf16x2_to_f32(w.x, x[0], x[1]);
  bf16x2_to_f32(w.y, x[2], x[3]);
  bf16x2_to_f32(w.z, x[4], x[5]);
  bf16x2_to_f32(w.w, x[6], x[7]);
}

// Codes of channels 8c..8c+7 of a per-token packed row: `lo` their 32 (4-bit)
// or 16 (2- and 3-bit) low bits in channel order, `hi` (3 bits) the plane byte
// of channels 8c..8c+7, which holds them in order at byte
// ((c >> 1) & 1) | ((c & 1) << 1) of plane word c / 4.
struct Codes8 {
  uint32_t lo, hi;
};
template <int BITS>
__device__ __forceinline__ Codes8 load_codes8(const char* row, int c) {
  Codes8 r = {0u, 0u};
  if (BITS == 4) {
    r.lo = reinterpret_cast<const uint32_t*>(row)[c];
  } else {
    r.lo = reinterpret_cast<const uint16_t*>(row)[c];
    if (BITS == 3)
      r.hi = reinterpret_cast<const uint8_t*>(row)[32 + 4 * (c >> 2) + (((c >> 1) & 1) | ((c & 1) << 1))];
  }
  return r;
}

// The integer c < 2^23 as a float: 2^23 + c in the mantissa, less 2^23 (exact).
__device__ __forceinline__ uint32_t int_magic(uint32_t c) { return c | 0x4B000000u; }
__device__ __forceinline__ uint64_t magic_pair() { return f32x2(0x4B000000u, 0x4B000000u); }

// fl(fl(x s) + z) of two elements.
__device__ __forceinline__ uint64_t scale_add(uint64_t x, uint64_t s, uint64_t z, uint64_t nz) {
  return f32x2_add(f32x2_product(x, s, nz), z);
}

// fl(fl(code * scale) + zero) of eight codes.
template <int BITS>
__device__ __forceinline__ void dequant8(const Codes8& k, float scale, float zero, uint64_t nz, float (&x)[8]) {
  const uint64_t s2 = f32x2(__float_as_uint(scale), __float_as_uint(scale));
  const uint64_t z2 = f32x2(__float_as_uint(zero), __float_as_uint(zero));
#pragma unroll
  for (int i = 0; i < 8; i += 2) {
    uint32_t c[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      c[e] = (k.lo >> ((BITS == 4 ? 4 : 2) * (i + e))) & (BITS == 4 ? 15u : 3u);
      if (BITS == 3) c[e] |= ((k.hi >> (i + e)) & 1u) << 2;
    }
    const uint64_t v = f32x2_sub(f32x2(int_magic(c[0]), int_magic(c[1])), magic_pair());
    const uint64_t r = scale_add(v, s2, z2, nz);
    x[i] = __uint_as_float((uint32_t)r);
    x[i + 1] = __uint_as_float((uint32_t)(r >> 32));
  }
}

// Normalised Hadamard-128 of a vector spread over a half-warp, lane j holding
// channels 8j..8j+7: stages h = 1, 2, 4 in the lane, h = 8..64 with lane
// j ^ (h / 8); butterflies (a, b) -> (a + b, a - b), one multiply at the end.
// (fma(x, +-1, p) is p + x or p - x, rounded once.)
__device__ __forceinline__ void fwht128_half(float (&x)[8], int j) {
#pragma unroll
  for (int h = 1; h < 8; h <<= 1) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (i & h) continue;
      const float a = x[i], b = x[i + h];
      x[i] = __fadd_rn(a, b);
      x[i + h] = __fsub_rn(a, b);
    }
  }
#pragma unroll
  for (int m = 1; m < 16; m <<= 1) {
    const float sgn = (j & m) ? -1.f : 1.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = __fmaf_rn(x[i], sgn, __shfl_xor_sync(kFull, x[i], m));
  }
  const float c = hadamard_c();
#pragma unroll
  for (int i = 0; i < 8; ++i) x[i] = __fmul_rn(x[i], c);
}

// Eight reconstructed channels, or the BF16 entry w (raw), to row element o
// (this lane's first channel) of an output, where ok; called by whole warps.
// fp32: lanes 2i and 2i + 1 exchange halves, so that each of the two stores
// writes whole 32-byte sectors.
__device__ __forceinline__ void store8(const DequantParams& p, void* dst, size_t o, bool raw, uint4 w, float (&x)[8],
                                       bool ok = true) {
  if (p.out_fp32) {
    if (raw) bf16x8_to_f32(w, x);
    const bool odd = threadIdx.x & 1;
    float r[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) r[i] = __shfl_xor_sync(kFull, odd ? x[i] : x[4 + i], 1);
    float4* f = reinterpret_cast<float4*>(static_cast<float*>(dst) + (odd ? o - 4 : o));
    if (ok) {
      f[0] = odd ? make_float4(r[0], r[1], r[2], r[3]) : make_float4(x[0], x[1], x[2], x[3]);
      f[2] = odd ? make_float4(x[4], x[5], x[6], x[7]) : make_float4(r[0], r[1], r[2], r[3]);
    }
  } else {
    if (!raw)
      w = make_uint4(pack_bf16x2_rn(x[0], x[1]), pack_bf16x2_rn(x[2], x[3]), pack_bf16x2_rn(x[4], x[5]),
                     pack_bf16x2_rn(x[6], x[7]));
    if (ok) *reinterpret_cast<uint4*>(static_cast<uint16_t*>(dst) + o) = w;
  }
}

// Tokens 8u..8u+7 (u = 0..3, the warp's) of one KIVI-style key group: codes and
// metadata of its 128 channels, first output element o (lane l: channels
// 4l..4l+3 of each token).
template <int BITS, bool M16>
__device__ __forceinline__ void dequant_key_group(const DequantParams& p, const char* codes, const char* meta, int u,
                                                  int lane, size_t o) {
  // each channel's BITS words; the eight tokens' codes are in one half of a
  // 2-bit word, or one 4-bit word, and at bits plane_bit + i of the 3-bit plane
  const uint4* cw = reinterpret_cast<const uint4*>(codes) + lane * BITS;
  uint32_t w[4 * BITS];
#pragma unroll
  for (int v = 0; v < BITS; ++v) {
    const uint4 q = cw[v];
    w[4 * v] = q.x;
    w[4 * v + 1] = q.y;
    w[4 * v + 2] = q.z;
    w[4 * v + 3] = q.w;
  }
  float2 m[4];
  if (M16) {
    const uint4 q = reinterpret_cast<const uint4*>(meta)[lane];
    m[0] = half2_bits_to_float2(q.x);
    m[1] = half2_bits_to_float2(q.y);
    m[2] = half2_bits_to_float2(q.z);
    m[3] = half2_bits_to_float2(q.w);
  } else {
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const float4 q = reinterpret_cast<const float4*>(meta)[2 * lane + v];
      m[2 * v] = make_float2(q.x, q.y);
      m[2 * v + 1] = make_float2(q.z, q.w);
    }
  }
  Codes8 k[4];  // eight tokens of each channel, in the layout of a row's eight channels
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const uint32_t* x = w + c * BITS;
    if (BITS == 4) {
      k[c].lo = (u & 2) ? ((u & 1) ? x[3 % BITS] : x[2 % BITS]) : ((u & 1) ? x[1] : x[0]);
    } else {
      k[c].lo = ((u & 2) ? x[1] : x[0]) >> (16 * (u & 1));
      // token 8u + i: index bits 3 and 4 (of u) exchanged
      if (BITS == 3) k[c].hi = x[2 % BITS] >> (8 * ((u >> 1) | ((u & 1) << 1)));
    }
  }
  const uint64_t s01 = f32x2(__float_as_uint(m[0].x), __float_as_uint(m[1].x));
  const uint64_t s23 = f32x2(__float_as_uint(m[2].x), __float_as_uint(m[3].x));
  const uint64_t z01 = f32x2(__float_as_uint(m[0].y), __float_as_uint(m[1].y));
  const uint64_t z23 = f32x2(__float_as_uint(m[2].y), __float_as_uint(m[3].y));
#pragma unroll
  for (int i = 0; i < kDqRows; ++i) {
    uint32_t c[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      c[e] = (k[e].lo >> ((BITS == 4 ? 4 : 2) * i)) & (BITS == 4 ? 15u : 3u);
      if (BITS == 3) c[e] |= ((k[e].hi >> i) & 1u) << 2;
    }
    const uint64_t a = scale_add(f32x2_sub(f32x2(int_magic(c[0]), int_magic(c[1])), magic_pair()), s01, z01, p.neg_zero2);
    const uint64_t b = scale_add(f32x2_sub(f32x2(int_magic(c[2]), int_magic(c[3])), magic_pair()), s23, z23, p.neg_zero2);
    const size_t e0 = o + (size_t)i * kD + 4 * lane;
    if (p.out_fp32)
      *reinterpret_cast<float4*>(static_cast<float*>(p.k_out) + e0) =
          make_float4(pair_lo(a), pair_hi(a), pair_lo(b), pair_hi(b));
    else
      *reinterpret_cast<uint2*>(static_cast<uint16_t*>(p.k_out) + e0) =
          make_uint2(pack_bf16x2_rn(pair_lo(a), pair_hi(a)), pack_bf16x2_rn(pair_lo(b), pair_hi(b)));
  }
}

// BITS, BASE and M16 are compile-time, so each (code width, base, metadata
// width) runs code of its own.
template <int BITS, int BASE, bool M16>
__global__ void __launch_bounds__(kDqThreads, 6) dequantize_kernel(const __grid_constant__ DequantParams p) {
  const Dims& d = p.d;
  const int li = blockIdx.z, bh = blockIdx.y;
  const int b = bh / d.H, h = bh % d.H;
  const int Tt = d.T + p.appended;
  // the head's region map, computed once for the CTA (64-bit arithmetic)
  __shared__ HeadGeom s_hd;
  grid_launch_dependents();
  if (threadIdx.x == 0) s_hd = head_geom(d, layer_geom(d, p.lt.mask[li]), h);
  grid_dependency_wait();
  __syncthreads();
  const HeadGeom& hd = s_hd;
  const int cls = hd.cls;
  const int warp = __shfl_sync(kFull, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const bool is_k = warp < 4;
  const int j = lane & 15, hw = lane >> 4;  // a half-warp's row: channels 8j..8j+7
  const char* Lb = p.arena + p.lt.base[li];
  const int qs = d.s, qe = d.s + d.nq;
  constexpr int CB = kD * BITS / 8;  // code bytes of a token
  constexpr int MB = M16 ? 4 : 8;
  constexpr int VG = BASE == kKivi ? 4 : 1;
  const bool has_salient = BASE == kAkvq && d.ns > 0 && cls != kProtected;
  // this warp's operand: BF16 rows, and codes + metadata (or the keys-only
  // head's BF16 image keys) of the coded tokens
  const char* rows = Lb + (is_k ? hd.kb : hd.vb) + b * hd.kb_bs;
  const bool coded_here = cls != kProtected && !(is_k && cls == kKeysOnly);
  const char* img = Lb + hd.kimg + b * hd.kimg_bs;  // keys-only heads
  const char* codes = Lb + (is_k ? hd.kq : hd.vq) + b * (is_k ? hd.kq_bs : hd.vq_bs);
  const char* meta = Lb + (is_k ? hd.kqm : hd.vqm) + b * (is_k ? hd.kqm_bs : hd.vqm_bs);
  void* out = is_k ? p.k_out : p.v_out;
  const size_t out0 = (((size_t)li * d.B + b) * d.H + h) * (size_t)Tt * kD;
  const int shift = cls == kProtected ? 0 : d.nq - d.ns;  // token - position of the rows past the image
  const int origin = dq_origin(d);
  const int ntiles = (Tt - origin + kDqTile - 1) / kDqTile;
  const int span = (ntiles + (int)gridDim.x - 1) / (int)gridDim.x;
  const int x1 = min(((int)blockIdx.x + 1) * span, ntiles);

#pragma unroll 1
  for (int x = blockIdx.x * span; x < x1; ++x) {
    const int a = origin + x * kDqTile + (warp & 3) * kDqRows, e = a + kDqRows;  // the warp's tokens [a, e)
    if (e <= 0 || a >= Tt) continue;
    const bool whole = a >= 0 && e <= Tt;
    const bool in_image = a >= qs && e <= qe, outside = cls == kProtected || e <= qs || a >= qe;
    // Salient tokens: a run without one (eight tokens of one map word; most runs)
    // is of one kind as well, moved down by the salient ones before it
    // (InternVL2.5-8B-shaped, 2% salient, 32 layers, BF16: 5.84 TB/s; 4.55 with
    // every row resolved).
    bool plain = whole && in_image && !has_salient;
    int ti = a - qs;
    if (whole && in_image && has_salient) {
      const char* sm = Lb + hd.sal + b * hd.sal_bs;
      const uint32_t sb = reinterpret_cast<const uint32_t*>(sm)[ti >> 5];
      plain = ((sb >> (ti & 31)) & 255u) == 0u;
      ti -= reinterpret_cast<const int*>(sm + (size_t)sal_blocks(d) * 4)[ti >> 5] + __popc(sb & ((1u << (ti & 31)) - 1u));
    }
    // ---- eight BF16 rows one after the other ----
    if ((whole && outside) || (plain && !coded_here)) {
      const char* src = (outside ? rows + (size_t)(a >= qe ? a - shift : a) * 256 : img + (size_t)ti * 256) +
                        hw * 256 + j * 16;
      uint4 w[kDqRows / 2];
#pragma unroll
      for (int i = 0; i < kDqRows / 2; ++i) w[i] = ldg16(src + i * 512);
      const size_t o = out0 + (size_t)(a + hw) * kD + 8 * j;
#pragma unroll
      for (int i = 0; i < kDqRows / 2; ++i) {
        float x8[8];
        store8(p, out, o + i * 2 * kD, true, w[i], x8);
      }
      continue;
    }
    // ---- eight coded tokens ----
    if (plain && coded_here) {
      if (BASE == kKivi && is_k) {
        const int grp = ti / kKiviGroup;
        dequant_key_group<BITS, M16>(p, codes + (size_t)grp * (kD * BITS * 4), meta + (size_t)grp * (kD * MB),
                                     (ti >> 3) & 3, lane, out0 + (size_t)a * kD);
        continue;
      }
      Codes8 c[kDqRows / 2];
      float2 m[kDqRows / 2];
      const char* cr = codes + (size_t)(ti + hw) * CB;
      const char* mr = meta + ((size_t)(ti + hw) * VG + (BASE == kKivi ? (j >> 2) : 0)) * MB;
#pragma unroll
      for (int i = 0; i < kDqRows / 2; ++i) {
        c[i] = load_codes8<BITS>(cr + i * 2 * CB, j);
        m[i] = load_meta(mr + i * 2 * VG * MB, 0, M16);
      }
      const size_t o = out0 + (size_t)(a + hw) * kD + 8 * j;
#pragma unroll
      for (int i = 0; i < kDqRows / 2; ++i) {
        float x8[8];
        dequant8<BITS>(c[i], m[i].x, m[i].y, p.neg_zero2, x8);
        if (BASE == kAkvq && is_k) fwht128_half(x8, j);  // inverse rotation (H is self-inverse)
        store8(p, out, o + i * 2 * kD, false, make_uint4(0u, 0u, 0u, 0u), x8);
      }
      continue;
    }
    // ---- each row for itself, two pairs of rows at a time (loads, then stores) ----
    constexpr int kPairs = 2;
#pragma unroll 1
    for (int i = 0; i < kDqRows / 2; i += kPairs) {
      uint4 w[kPairs];
      Codes8 c[kPairs];
      float2 m[kPairs];
      bool ok[kPairs], code[kPairs];
#pragma unroll
      for (int u = 0; u < kPairs; ++u) {
        const int t = a + 2 * (i + u) + hw;
        ok[u] = t >= 0 && t < Tt;
        bool coded = t >= qs && t < qe;  // an image token: code, BF16 image key, or salient
        int ci = t - qs, pos = (t < qs || cls == kProtected) ? t : t - shift;
        if (has_salient && ok[u] && coded) {
          const char* sm = Lb + hd.sal + b * hd.sal_bs;
          const int word = ci >> 5, k = ci & 31;
          const uint32_t sb = reinterpret_cast<const uint32_t*>(sm)[word];
          const int rank = reinterpret_cast<const int*>(sm + (size_t)sal_blocks(d) * 4)[word] +
                           __popc(sb & ((1u << k) - 1u));
          if ((sb >> k) & 1u) {
            coded = false;
            pos = qs + rank;
          }
          ci -= rank;
        }
        code[u] = coded && coded_here;
        w[u] = make_uint4(0u, 0u, 0u, 0u);
        c[u] = {0u, 0u};
        m[u] = make_float2(0.f, 0.f);
        if (ok[u]) {
          if (!code[u]) {
            w[u] = ldg16(((coded && cls == kKeysOnly) ? img + (size_t)ci * 256 : rows + (size_t)pos * 256) + j * 16);
          } else if (!(BASE == kKivi && is_k)) {
            c[u] = load_codes8<BITS>(codes + (size_t)ci * CB, j);
            m[u] = load_meta(meta, (size_t)ci * VG + (BASE == kKivi ? (j >> 2) : 0), M16);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < kPairs; ++u) {
        float x8[8];
        dequant8<BITS>(c[u], m[u].x, m[u].y, p.neg_zero2, x8);
        if (BASE == kAkvq && is_k) fwht128_half(x8, j);  // by every lane: rows that are not coded drop it
        store8(p, out, out0 + (size_t)(a + 2 * (i + u) + hw) * kD + 8 * j, !code[u], w[u], x8, ok[u]);
      }
    }
  }
}

// One decode token per (layer, row, head) into the head's BF16 region.  Part of
// the programmatic dependent launches of a decode loop: the next launch may be
// scheduled at once, and everything before the first store comes from the
// launch parameters.  Appending and attending without a workspace, layer by
// layer (append, clear, decode: 6 layers of 5 KV heads, 2 tokens): 184 us with the
// three overlapping, 246 with an append and a memset that each run alone.
__global__ void __launch_bounds__(64) append_kernel(const __grid_constant__ AppendParams p) {
  grid_launch_dependents();
  const Dims& d = p.d;
  const int li = blockIdx.x, bh = blockIdx.y;
  const int b = bh / d.H, h = bh % d.H;
  const LayerGeom g = layer_geom(d, p.lt.mask[li]);
  const HeadGeom hd = head_geom(d, g, h);
  char* Lb = p.arena + p.lt.base[li];
  const int pos = hd.bf16_prefill + p.appended[li];
  const size_t src = (((size_t)li * d.B + b) * d.H + h) * kD;
  const int lane = threadIdx.x & 31;
  const bool is_k = threadIdx.x < 32;
  char* dst = Lb + (is_k ? hd.kb : hd.vb) + b * hd.kb_bs + ((size_t)pos * kD + lane * 4) * 2;
  grid_dependency_wait();
  *reinterpret_cast<uint2*>(dst) = ldg8((is_k ? p.k_new : p.v_new) + src + lane * 4);
}

// Zeroes n 16-byte words between two decode launches of the same chain.
__global__ void __launch_bounds__(256) clear_kernel(uint4* words, int n) {
  grid_launch_dependents();
  grid_dependency_wait();
  for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) words[i] = make_uint4(0u, 0u, 0u, 0u);
}

}  // namespace

// A launch that may be scheduled while the kernel before it still runs.
template <class... P, class... A>
cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s,
                             const A&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// Launch of the quantizer kernel over every tile of the launch's layers, keys and values.
template <class TP>
cudaError_t launch_tiles(const QuantizeParams& p, int tiles_x, cudaStream_t s) {
  const dim3 grid((unsigned)(tiles_x * (TP::kKeysFirst ? 1 : 2)), (unsigned)(p.d.B * p.d.H),
                  (unsigned)(p.n_layers * (TP::kKeysFirst ? 2 : 1)));
  return launch_dependent(quantize_tiles_kernel<TP>, grid, 32, 0, s, p);
}

template <int BITS, bool M16>
cudaError_t launch_quantize_bits(const QuantizeParams& p, cudaStream_t s) {
  const Dims& d = p.d;
  if (d.base == kKivi)
    return launch_tiles<KiviTiles<BITS, M16>>(p, (d.T - p.tile_origin + kKiviGroup + kQTok - 1) / kQTok, s);
  const int tx = (d.T + kQTok - 1) / kQTok;
  if (d.base == kAkvq) return launch_tiles<TokenTiles<BITS, M16, kAkvq>>(p, tx, s);
  return launch_tiles<TokenTiles<BITS, M16, kMinMax>>(p, tx, s);
}

cudaError_t launch_quantize(const QuantizeParams& p, cudaStream_t s) {
  const bool m16 = p.d.meta16 != 0;
  if (p.d.bits == 2) return m16 ? launch_quantize_bits<2, true>(p, s) : launch_quantize_bits<2, false>(p, s);
  if (p.d.bits == 3) return m16 ? launch_quantize_bits<3, true>(p, s) : launch_quantize_bits<3, false>(p, s);
  return m16 ? launch_quantize_bits<4, true>(p, s) : launch_quantize_bits<4, false>(p, s);
}

template <bool NORMS>
cudaError_t launch_salient_select(const QuantizeParams& p, cudaStream_t s) {
  return launch_dependent(salient_select_kernel<NORMS>, dim3((unsigned)(p.d.B * p.d.H), (unsigned)p.n_layers, 1),
                          kSalThreads, salient_smem_bytes(p.d), s, p);
}

// Lets the selection have the shared memory of the longest span, once per device:
// the same value whatever the call's span, so host threads with different ones
// cannot take it from each other.  (The default 48 KB also hold the kernel's own
// arrays, so spans of less than that need it too.)
cudaError_t allow_salient_smem() {
  static std::atomic<bool> configured[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < 64 && configured[dev].load(std::memory_order_acquire)) return cudaSuccess;
  e = cudaFuncSetAttribute(salient_select_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kMaxSalientSmem);
  if (e == cudaSuccess && dev >= 0 && dev < 64) configured[dev].store(true, std::memory_order_release);
  return e;
}

cudaError_t launch_salient(const QuantizeParams& p, cudaStream_t s) {
  if (p.d.nq <= kSalOneLaunch) return launch_salient_select<true>(p, s);
  cudaError_t e = allow_salient_smem();  // before anything is enqueued
  if (e != cudaSuccess) return e;
  e = launch_dependent(
      salient_norm_kernel,
      dim3((p.d.nq + kNormTokens - 1) / kNormTokens, (unsigned)(p.d.B * p.d.H), (unsigned)p.n_layers), kNormThreads, 0, s, p);
  if (e != cudaSuccess) return e;
  return launch_salient_select<false>(p, s);
}

template <int BITS, int BASE, bool M16>
cudaError_t launch_dequantize_t(const DequantParams& p, dim3 grid, cudaStream_t s) {
  return launch_dependent(dequantize_kernel<BITS, BASE, M16>, grid, kDqThreads, 0, s, p);
}

template <int BITS>
cudaError_t launch_dequantize_bits(const DequantParams& p, dim3 grid, cudaStream_t s) {
  const bool m16 = p.d.meta16 != 0;
  if (p.d.base == kKivi)
    return m16 ? launch_dequantize_t<BITS, kKivi, true>(p, grid, s) : launch_dequantize_t<BITS, kKivi, false>(p, grid, s);
  if (p.d.base == kAkvq)
    return m16 ? launch_dequantize_t<BITS, kAkvq, true>(p, grid, s) : launch_dequantize_t<BITS, kAkvq, false>(p, grid, s);
  return m16 ? launch_dequantize_t<BITS, kMinMax, true>(p, grid, s)
             : launch_dequantize_t<BITS, kMinMax, false>(p, grid, s);
}

cudaError_t launch_dequantize(const DequantParams& p, int sm_count, cudaStream_t s) {
  const int Tt = p.d.T + p.appended;
  const int ntiles = (Tt - dq_origin(p.d) + kDqTile - 1) / kDqTile;
  // Tiles per CTA (1 to 4): whole waves of 6 CTAs per SM, each as long as its
  // tiles and a start worth 0.4 of one.  (Qwen2.5-VL-7B-shaped, 28 layers: 21.2
  // us with one tile per CTA, 19.5 with two, 20.4 with four, 23.6 with eight; four
  // LLaVA-NeXT-7B-shaped layers of 16 rows one by one 786, 664, 661 and 676 us.)
  const double groups = (double)p.d.B * p.d.H * p.n_layers, wave = 6.0 * (sm_count > 0 ? sm_count : 1);
  int span = 1;
  double best = 0.0;
  for (int n = 1; n <= 4; ++n) {
    const double t = std::ceil(groups * ((ntiles + n - 1) / n) / wave) * (n + 0.4);
    if (n == 1 || t < best) {
      best = t;
      span = n;
    }
  }
  dim3 grid((ntiles + span - 1) / span, p.d.B * p.d.H, p.n_layers);
  if (p.d.bits == 2) return launch_dequantize_bits<2>(p, grid, s);
  if (p.d.bits == 3) return launch_dequantize_bits<3>(p, grid, s);
  return launch_dequantize_bits<4>(p, grid, s);
}

cudaError_t launch_append(const AppendParams& p, cudaStream_t s) {
  return launch_dependent(append_kernel, dim3(p.n_layers, p.d.B * p.d.H, 1), 64, 0, s, p);
}

cudaError_t launch_clear(void* words, size_t bytes, cudaStream_t s) {
  const int n = (int)(bytes / 16);
  return launch_dependent(clear_kernel, dim3(std::max(1, std::min(64, (n + 255) / 256)), 1, 1), 256, 0, s,
                          static_cast<uint4*>(words), n);
}

}  // namespace hg
