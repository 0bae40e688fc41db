// Split-K decode attention over the mixed-precision cache (tensor cores).
//
// One CTA per work item = one chunk of one (layer, batch row, KV head).  A
// chunk is uniform: a run of BF16 tokens (text, uncoded image tokens,
// protected heads, appended tokens), a run of coded image tokens (packed
// codes + fp32 scale/zero for K and V), or, for keys-only protected heads, BF16
// keys with coded values.  The only branch on the mask or the image span is
// therefore taken once per CTA.
//
// Each of the CTA's four warps takes a quarter of the chunk's tokens and
// streams it through a TMA pipeline of its own (12 KB, two to four slots with
// an mbarrier each, copies issued by its lane 0): BF16 rows arrive as
// tensor-map boxes with the 128-byte swizzle, packed codes and metadata as
// one bulk copy per array.  The warps meet only before their first tile and
// after their last one.  A warp works on 16-token slices and computes, with
// mma.sync m16n8k16 (BF16 in, fp32 accumulate):
//   S^T[token][query] = K . q     A = keys (BF16 via ldmatrix, or codes masked
//                                 in registers),
//                                 B = the G queries of the KV head (padded to 8)
//   O^T[chan][query] += V^T . P^T A = values (ldmatrix.trans, or codes),
//                                 B = P^T, transposed from the score fragment
//                                 with movmatrix.
// Codes enter the MMAs as FP16 bit patterns: an integer i < 2^11 in the low
// bits is exactly i 2^-24 (a subnormal, or the binade above them, which
// continues the same steps), so a masked word is an operand as it is -- no
// offset to add and remove again, no subtraction -- and a code may sit at any of
// the low bit positions, where it counts 2^position times.  The position's
// factor is taken out of the other operand or of the result; 2^24 of the result.
// Coded keys are contracted in the code domain: with per-token groups
// k^_d = s c_d + z, so q.k^ = s (q.c) + z sum(q), with the query row scaled by
// a power of two into FP16's range (exact).  KIVI-style per-channel groups fold
// the channel scale into the query (q~_d = q_d s_d, split into a hi + lo pair)
// and add sum_d q_d z_d.  Values fold the token scale into P (p s) and add
// sum_t p_t z_t.  (KIVI-style codes with more than two queries per KV head are
// converted to BF16 keys and FP16 values instead: their pairs sit at bit
// positions that differ between lanes.)  AKVQ-style keys are coded in the
// rotated domain; since the normalised Hadamard matrix is symmetric and
// orthonormal, <q, H k'> = <H q, k'>, so the query is rotated once per CTA (hi +
// lo split).
//
// The online softmax rescales its accumulators only when a running maximum
// grows by more than 2^8 (probabilities stay <= 256 before normalisation).
// Warps are combined in shared memory; a CTA that is not alone on its head
// writes an (m, l, o) partial to the workspace and the last CTA to arrive
// (atomic ticket, no waiting) merges them and writes the BF16 output.
//
// The kernel templates live in this header; hg_decode.cu instantiates them
// for fp32 metadata pairs and hg_decode_m16.cu for binary16 pairs, so the two
// sets compile in parallel.
#pragma once
#include <cuda_runtime.h>

#include <atomic>

#include "hg_common.cuh"
#include "hg_internal.h"
#include "hg_mma.cuh"

namespace hg {

namespace {

constexpr int kThreads = 128;
constexpr int kWarps = 4;
constexpr int kBufBytes = 49152;   // pipeline buffers of the four warps
constexpr int kWarpBuf = kBufBytes / kWarps;
constexpr int kPartialStride = kD + 4;  // m, l, 2 pad, o[128]: rows of 528 bytes (16-byte multiple)
// Shared memory, from a 1024-byte aligned base (swizzled TMA boxes need it).
constexpr int kStageOff = 0;                    // pipeline buffer
// Four CTAs per SM for up to 8 queries per KV head (NT = 1), two above.
// Staged queries: row r (query r of the KV head), channel c at r * kQRow + c.
// The row stride of 36 16-byte units (4 mod 8) spreads the 16-byte reads of
// one warp in the KIVI-style key path (8 rows x 4 consecutive channel
// quads) over all banks.
constexpr int kQRow = 144;
__device__ __forceinline__ int qidx(int r, int c) { return r * kQRow + c; }

template <int NT>
struct SmemLayout {
  static constexpr int q = kStageOff + kBufBytes;  // float q[NT * 8][kQRow] (qidx)
  static constexpr int bar = q + NT * 8 * kQRow * 4;  // mbarrier per warp and slot (4 x 4), abort flag
  static constexpr int qn = bar + 192;              // float qn[NT * 8]: scale of each staged query row
  static constexpr int bytes = qn + 64 + 1024;     // + alignment slack
};
constexpr int kMaxSlots = 4;  // per warp
constexpr unsigned kFull = 0xffffffffu;
// A wait for a tile is declared stuck after kWaitRounds suspensions of up to
// kWaitSleepNs each (about a second); a healthy wait ends within microseconds.
constexpr uint32_t kWaitRounds = 20000;
constexpr uint32_t kWaitSleepNs = 50000;

enum KMode { K_BF16 = 0, K_TOKEN = 1, K_KIVI = 2 };
enum VMode { V_BF16 = 0, V_TOKEN = 1, V_KIVI = 2 };

template <int VM>
struct NZOf {
  static constexpr int value = VM == V_TOKEN ? 1 : (VM == V_KIVI ? 4 : 1);
};

// Where the operands of an item's chunk lie.
struct Seg {
  int k_row0;      // arena tensor-map row of key token 0 (K_BF16)
  int v_row0;      // arena tensor-map row of value token 0 (V_BF16)
  const char* kc;  // key codes
  const char* km;  // key metadata
  const char* vc;  // value codes
  const char* vm;  // value metadata
};

// Mask of a code pair at bits [0, b) and [16, 16 + b).
template <int BITS>
__host__ __device__ constexpr uint32_t pair_mask() { return ((1u << BITS) - 1u) * 0x00010001u; }

// Result of an MMA over codes, in units of 2^-24 (see the file comment).
constexpr float kCodeUnit = 16777216.f;

// A word (half) of packed codes holds pairs (j, j + half a word) 16 bits apart.
// Pair j as an MMA operand register: masked at bit code_pos(j) and 16 above,
// after one of three shifts (2-bit codes, and the 2-bit part of 3-bit codes) or
// two (4 bits).  The values are 2^code_pos(j) times the codes.  The positions
// are the high ones of the 11 bits: the tensor cores line an operand's products
// up by its exponent field, so a code in the lowest bits would lose as many
// bits of the sum as it has leading zeros (with positions 0..8 in one shift per
// five pairs, KIVI-style values moved 1% away from the 64-bit result).
template <int BITS>
__host__ __device__ constexpr int code_pos(int j) {
  return BITS == 4 ? 4 * (j % 2) : (j < 2 ? 2 * j + 6 : (j < 5 ? 2 * j : 2 * j - 6));
}
template <int BITS>
__device__ __forceinline__ uint32_t code_pair(uint32_t w, int j) {
  const uint32_t x = BITS == 4 ? w >> (8 * (j / 2)) : (j < 2 ? w << 6 : (j < 5 ? w : w >> 6));
  return x & (pair_mask<BITS == 4 ? 4 : 2>() << code_pos<BITS>(j));
}
template <int BITS>
__host__ __device__ constexpr float code_unit(int j) { return 1.0f / (float)(1 << code_pos<BITS>(j)); }

__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
  return y;
}

template <int NT, int NZ>
struct WarpState {
  float o[NT][8][4];
  float vb;           // coded values: power-of-two bound of the value scales seen so far
  float m[NT][2];
  float l[NT][2];
  float z[NT][2][NZ];
};

// 1 / x for a power of two x in [2^-126, 2^126], exactly (exponent arithmetic).
__device__ __forceinline__ float pow2_inv(float x) { return __uint_as_float(0x7F000000u - __float_as_uint(x)); }

// 3-bit codes keep bits 0-1 in the 2-bit packing and bit 2 in a plane word
// per 32 codes (element e at bit e mod 32 with index bits 3 and 4 exchanged),
// so the bit-2 pair of two codes 8 apart in one 2-bit word sits 16 bits apart
// too.  plane_pair moves such a pair from bits (i, i + 16) of a plane-derived
// register to bits (p + 2, p + 18), on top of the 2-bit pair extracted at
// bits (p, p + 16); i and p are compile-time after unrolling.
__device__ __forceinline__ uint32_t plane_pair(uint32_t pl, int i, int p) {
  const int d = i - (p + 2);
  const uint32_t x = d >= 0 ? (pl >> d) : (pl << (-d));
  return x & (0x00010001u << (p + 2));
}
// prmt selector: byte bs of a into bytes 0-1 of the result, byte bs of b into
// bytes 2-3 (the plane bytes of two tokens or two channels, side by side).
__device__ __forceinline__ uint32_t plane_sel(int bs) {
  return (uint32_t)(bs | (bs << 4) | ((4 + bs) << 8) | ((4 + bs) << 12));
}

// Bounds of the power-of-two scales: their products and inverses stay finite.
constexpr float kScaleLow = 7.8886090522101181e-31f;  // 2^-100
constexpr float kScaleTop = 8.5070591730234616e37f;   // 2^126

// Smallest power of two >= m (m > 0, finite).
__device__ __forceinline__ float pow2_ceil(float m) {
  return __uint_as_float((__float_as_uint(m) + 0x007FFFFFu) & 0xFF800000u);
}

// Metadata pairs {scale, zero} in a stage: MB = 8 for two fp32, MB = 4 for
// two binary16 (scale in the low half).  meta_quad reads pairs i..i+3 (i a
// multiple of 4: one 16-byte load at MB = 4, two at MB = 8).
template <int MB>
__device__ __forceinline__ float2 meta_pair(const char* base, int i) {
  if (MB == 4) return half2_bits_to_float2(reinterpret_cast<const uint32_t*>(base)[i]);
  return reinterpret_cast<const float2*>(base)[i];
}
template <int MB>
__device__ __forceinline__ void meta_quad(const char* base, int i, float2 (&m)[4]) {
  if (MB == 4) {
    const uint4 w = *reinterpret_cast<const uint4*>(base + i * 4);
    m[0] = half2_bits_to_float2(w.x);
    m[1] = half2_bits_to_float2(w.y);
    m[2] = half2_bits_to_float2(w.z);
    m[3] = half2_bits_to_float2(w.w);
  } else {
    const float4 a = *reinterpret_cast<const float4*>(base + i * 8);
    const float4 b = *reinterpret_cast<const float4*>(base + i * 8 + 16);
    m[0] = make_float2(a.x, a.y);
    m[1] = make_float2(a.z, a.w);
    m[2] = make_float2(b.x, b.y);
    m[3] = make_float2(b.z, b.w);
  }
}

// One warp's pipeline.  A tile is the tokens between two refills.  SPLIT (BF16
// rows for K and V): a 16-token tile's K and V rows land in slots of their
// own, so a K slot is refilled while the tile's values are still at work --
// three 4 KB slots where two 8 KB ones would not fit.  Else a slot holds a
// whole tile, as large as fits twice, since a wait and a refill cost a warp
// as much as a third of a slice: 64 tokens of per-token 2-bit codes (5 KB; 32
// and 48 measured 4% and 1.5% slower on one layer of 32 rows, 8 KV heads and
// 8,576 tokens), 32 at 3 and 4 bits (16: 3% slower with rotated 4-bit keys; the
// value offsets are folded once per tile, and over 48 or 64 tokens of wider
// codes the fp32 accumulators lose bits that the output shows), a KIVI-style
// group of 32, 16 tokens of BF16 keys and coded values.
//
// (One ring of tiles for all four warps, filled by one thread with a CTA barrier
// per tile, leaves a warp one or two 16-token slices between barriers: 7% slower on
// that layer and on 3,520 tokens of 4-bit rotated keys, 13% on 32 KV heads of KIVI-
// style codes in 16 rows and on one row of 4 KV heads and 1,460 tokens.  The gain
// needs every address known to be the same in the warp's lanes, so that the refill
// runs on the uniform path.)
//
// COLS (run_item_cols): SPLIT as well, two KIVI-style groups per tile (K and V
// 4 KB each at 2 bits), or 16 tokens of BF16 keys and KIVI-style values.
template <int BITS, int KM, int VM, int MB, bool COLS = false>
struct Tile {
  static constexpr bool SPLIT = COLS || (KM == K_BF16 && VM == V_BF16);
  static constexpr int tokens = (KM == K_BF16) ? 16
                                : (KM == K_KIVI ? (COLS ? 2 : 1) * kKiviGroup : (BITS == 2 ? 64 : 32));
  static constexpr int kc_bytes = (KM == K_BF16) ? tokens * 256 : tokens * 16 * BITS;
  static constexpr int km_bytes = (KM == K_TOKEN) ? tokens * MB : (KM == K_KIVI ? tokens * 4 * MB : 0);
  static constexpr int vc_bytes = (VM == V_BF16) ? tokens * 256 : tokens * 16 * BITS;
  static constexpr int vm_bytes = (VM == V_TOKEN) ? tokens * MB : (VM == V_KIVI ? tokens * 4 * MB : 0);
  static constexpr int km_off = kc_bytes;  // from the tile's K base
  static constexpr int vc_off = SPLIT ? 0 : km_off + km_bytes;  // from its V base (not SPLIT: the slot)
  static constexpr int vm_off = vc_off + vc_bytes;
  // slots that hold BF16 rows start on 1024-byte boundaries (swizzled boxes)
  static constexpr int align = (KM == K_BF16) ? 1024 : 128;
  static constexpr int k_end = kc_bytes + km_bytes, v_end = vm_off + vm_bytes;
  static constexpr int slot_bytes = ((k_end > v_end ? k_end : v_end) + align - 1) / align * align;
  static constexpr int slots = (kWarpBuf / slot_bytes) > kMaxSlots ? kMaxSlots : (kWarpBuf / slot_bytes);
  static_assert(slots >= 2, "a tile must fit twice in a warp's buffer");
  static_assert(KM != K_BF16 || tokens == kArenaBoxRows, "a BF16 tile is one TMA box high");
  static_assert(kWarpBuf % 1024 == 0, "the warps' buffers keep the slots' alignment");
};

// BF16 rows [row0, +16) of the arena into shared memory at dst: two column
// halves of 16 x 128 bytes (channels 0-63, 64-127), each a TMA box with the
// 128-byte swizzle (16-byte chunk c of row r at chunk c ^ (r % 8)).  Rows past
// the segment's end are loaded too and ignored or zeroed by the consumer.
__device__ __forceinline__ void issue_rows(uint32_t dst, const CUtensorMap* map, int row0, uint32_t bar) {
  tma_load_2d(dst, map, 0, row0, bar);
  tma_load_2d(dst + kArenaBoxRows * 128, map, 64, row0, bar);
}

// Fill i of a warp's pipeline into its slot, issued by a single thread: the
// expected byte count on the slot's mbarrier, then the copies.  SPLIT: fill 2t
// is the K rows of the warp's tile t, fill 2t + 1 its V rows; else fill t is
// tile t.  Packed codes and metadata arrive as one bulk copy per array
// (metadata rounded up to 16 bytes: the arena pads every metadata row to 16
// bytes); bytes past the range [wb, we) are left stale.
template <int BITS, int KM, int VM, int MB, bool COLS>
__device__ __forceinline__ void issue_fill(uint32_t slot, uint32_t bar, const Seg& sg, int i, int wb, int we,
                                           const CUtensorMap* map) {
  using TL = Tile<BITS, KM, VM, MB, COLS>;
  const int t0 = wb + (TL::SPLIT ? i >> 1 : i) * TL::tokens;
  if (KM == K_BF16 && VM == V_BF16) {
    mbar_arrive_expect_tx(bar, TL::kc_bytes);
    issue_rows(slot, map, ((i & 1) ? sg.v_row0 : sg.k_row0) + t0, bar);
    return;
  }
  const bool do_k = !TL::SPLIT || !(i & 1), do_v = !TL::SPLIT || (i & 1);
  constexpr int kmb = (KM == K_TOKEN) ? MB : 4 * MB;  // metadata bytes per token
  constexpr int vmb = (VM == V_TOKEN) ? MB : 4 * MB;
  const int n = min(TL::tokens, we - t0);
  const uint32_t kc_bytes = (KM == K_BF16) ? TL::kc_bytes : n * 16 * BITS;
  const uint32_t km_bytes = (KM == K_BF16) ? 0u : (uint32_t)((n * kmb + 15) & ~15);
  const uint32_t vc_bytes = n * 16 * BITS;
  const uint32_t vm_bytes = (uint32_t)((n * vmb + 15) & ~15);
  mbar_arrive_expect_tx(bar, (do_k ? kc_bytes + km_bytes : 0u) + (do_v ? vc_bytes + vm_bytes : 0u));
  if (do_k) {
    if (KM == K_BF16) {
      issue_rows(slot, map, sg.k_row0 + t0, bar);
    } else {
      bulk_g2s(slot, sg.kc + (size_t)t0 * 16 * BITS, kc_bytes, bar);
      bulk_g2s(slot + TL::km_off, sg.km + (size_t)t0 * kmb, km_bytes, bar);
    }
  }
  if (do_v) {
    bulk_g2s(slot + TL::vc_off, sg.vc + (size_t)t0 * 16 * BITS, vc_bytes, bar);
    bulk_g2s(slot + TL::vm_off, sg.vm + (size_t)t0 * vmb, vm_bytes, bar);
  }
}

// Bounded wait for a phase of a slot's mbarrier.  On timeout, or once another
// warp gave up, marks the CTA aborted, records the failure in the workspace
// status word and returns false (the caller skips the tile's work).
__device__ __forceinline__ bool wait_tile(uint32_t bar, uint32_t parity, volatile int* abort, uint32_t* status,
                                          uint32_t rounds = kWaitRounds) {
  for (uint32_t i = 0; i < rounds; ++i) {
    if (mbar_try_wait_sleep(bar, parity, kWaitSleepNs)) return true;
    if (*abort) return false;
  }
  *abort = 1;
  atomicOr(status, kStatusWaitTimeout);
  return false;
}

// A warp's pipeline over its token range [wb, we): fill i uses slot i % SLOTS
// and phase i / SLOTS of that slot's mbarrier; fills are consumed in order.  The
// CTA's chunk is divided in units of GRAN tokens.
template <int BITS, int NT, int KM, int VM, int MB, bool COLS, int GRAN>
struct WarpPipe {
  using TL = Tile<BITS, KM, VM, MB, COLS>;
  static constexpr int SLOTS = TL::slots, FPT = TL::SPLIT ? 2 : 1;  // fills per tile
  // A tile of KIVI-style keys is a whole group, of which only one half may be the
  // warp's: tiles then start at multiples of ALIGN.
  static constexpr int ALIGN = KM == K_KIVI && GRAN < kKiviGroup ? kKiviGroup : 1;
  const Seg& sg;
  const DecodeParams& p;
  int wb, we;  // the warp's tokens; wb of its first tile
  int skip;    // tokens of the first tile that are another warp's
  int n_tiles, n_fills, issued;
  int fs, fp;  // slot and phase parity of the next fill to consume
  char* buf;
  uint32_t buf0, bars;
  volatile int* abort;

  // The warp's quarter of the chunk [tb, te).
  // Only the first tile goes in flight now: with every CTA of the launch
  // starting at once, first tiles alone make a burst the memory system serves
  // quickly, so compute starts early; the other slots are filled once the
  // first tile has landed.  (Filling them all at once measured the same, also
  // in launches of a few dozen CTAs.)
  __device__ __forceinline__ WarpPipe(char* smem, int warp, const Seg& s, const DecodeParams& dp, int tb, int te)
      : sg(s), p(dp), fs(0), fp(0) {
    const int span = (max(te - tb, 0) + kWarps * GRAN - 1) / (kWarps * GRAN) * GRAN;
    wb = min(tb + warp * span, te);
    we = min(wb + span, te);
    skip = wb < we ? wb % ALIGN : 0;
    wb -= skip;
    n_tiles = (max(we - wb, 0) + TL::tokens - 1) / TL::tokens;
    n_fills = n_tiles * FPT;
    buf = smem + kStageOff + warp * kWarpBuf;
    buf0 = smem_u32(buf);
    bars = smem_u32(smem + SmemLayout<NT>::bar) + warp * (8 * kMaxSlots);
    abort = reinterpret_cast<volatile int*>(smem + SmemLayout<NT>::bar + 8 * kMaxSlots * kWarps);
    issued = min(n_fills, FPT);
    if (elect_one())
      for (int i = 0; i < issued; ++i) issue(i, i);
  }
  __device__ __forceinline__ void issue(int slot, int i) {
    issue_fill<BITS, KM, VM, MB, COLS>(buf0 + slot * TL::slot_bytes, bars + 8 * slot, sg, i, wb,
                                       (we + ALIGN - 1) / ALIGN * ALIGN, &p.arena_map);
  }
  __device__ __forceinline__ int tile_tokens(int it) const { return min(TL::tokens, we - wb - it * TL::tokens); }
  __device__ __forceinline__ const char* slot() const { return buf + fs * TL::slot_bytes; }
  __device__ __forceinline__ const char* next_slot() const {
    return buf + (fs + 1 == SLOTS ? 0 : fs + 1) * TL::slot_bytes;
  }
  // Wait for the next fill; false when a wait of the CTA ran out.
  __device__ __forceinline__ bool landed() {
    if (__all_sync(kFull, mbar_try_wait(bars + 8 * fs, fp))) return true;
    return (bool)__all_sync(kFull, wait_tile(bars + 8 * fs, fp, abort, p.status));
  }
  // The first tile landed: fill the other slots.
  __device__ __forceinline__ void fill_rest() {
    const int upto = min(n_fills, SLOTS);
    if (elect_one())
      for (int i = issued; i < upto; ++i) issue(i, i);
    issued = upto;
  }
  // Every lane has read the consumed fill: refill its slot and move on.
  __device__ __forceinline__ void refill() {
    __syncwarp();
    if (issued < n_fills) {
      if (elect_one()) {
        fence_proxy_async_shared();
        issue(fs, issued);
      }
      ++issued;
    }
    if (++fs == SLOTS) {
      fs = 0;
      fp ^= 1;
    }
  }
  // After a wait ran out: a slot is refilled only after its previous fill
  // landed, so only the last SLOTS fills can still be in flight; let them land
  // (bounded) before the buffer is reused or the CTA exits.
  __device__ __forceinline__ void drain(int lane) {
    if (*abort && lane == 0) {
      for (int t = (issued > SLOTS ? issued - SLOTS : 0); t < issued; ++t)
        for (uint32_t i = 0; i < kWaitRounds && !mbar_try_wait_sleep(bars + 8 * (t % SLOTS), (t / SLOTS) & 1,
                                                                      kWaitSleepNs);
             ++i) {
        }
    }
  }
};

// ---------------------------------------------------------------------------
// Query fragments
// ---------------------------------------------------------------------------
// hi + lo FP16 split of an fp32 pair below FP16's largest value (x = hi + lo to
// 22 significant bits, 2^-25 at least)
__device__ __forceinline__ void split_pair16(float x0, float x1, uint32_t& hi, uint32_t& lo) {
  hi = pack_half2(x0, x1);
  const float2 h = half2_bits_to_float2(hi);
  lo = pack_half2(x0 - h.x, x1 - h.y);
}

// hi + lo BF16 split of an fp32 pair (x = hi + lo to ~16 significant bits)
__device__ __forceinline__ void split_pair(float x0, float x1, uint32_t& hi, uint32_t& lo) {
  hi = pack_bf16x2(x0, x1);
  const float h0 = __uint_as_float(hi << 16), h1 = __uint_as_float(hi & 0xffff0000u);
  lo = pack_bf16x2(x0 - h0, x1 - h1);
}

// Natural channel order (BF16 keys): k-step j covers channels 16j..16j+15.
template <int NT>
__device__ __forceinline__ void qfrag_natural(uint32_t (&qb)[NT][8][2], const float* q_s, int g, int tq) {
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    const int r = nt * 8 + g;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int c = 16 * j + 2 * tq;
      qb[nt][j][0] = pack_bf16x2(q_s[qidx(r, c)], q_s[qidx(r, c + 1)]);
      qb[nt][j][1] = pack_bf16x2(q_s[qidx(r, c + 8)], q_s[qidx(r, c + 9)]);
    }
  }
}

// Channels matching the in-register expansion of a packed token row.
// 2-bit: thread tq reads words 2tq and 2tq+1; k-step j takes code pair
// (j, j+8) of each.  4-bit: thread tq reads words 4tq..4tq+3; k-step j takes
// pairs (i, i+4) and (i+1, i+5), i = 2 (j & 1), of word 4tq + j/2.
template <int BITS>
__device__ __forceinline__ void token_channels(int tq, int j, int (&c)[4]) {
  if (BITS != 4) {  // 2 bits, and the 2-bit part of 3-bit codes
    c[0] = 32 * tq + j;
    c[1] = 32 * tq + j + 8;
    c[2] = 32 * tq + 16 + j;
    c[3] = 32 * tq + 24 + j;
  } else {
    const int w = 4 * tq + (j >> 1), i = 2 * (j & 1);
    c[0] = 8 * w + i;
    c[1] = 8 * w + i + 4;
    c[2] = 8 * w + i + 1;
    c[3] = 8 * w + i + 5;
  }
}

// Query fragments (FP16) for coded per-token keys from the staged, scaled rows:
// k-step j's k-slots carry q times the unit of the codes they meet.  Rotated
// queries are not BF16 values any more and take a hi + lo pair; the others are
// exact in one.  s0 = sum of the (scaled) query of this thread's columns.
template <int BITS, int NT, bool ROT>
__device__ __forceinline__ void qfrag_token(uint32_t (&qb)[NT][8][2], uint32_t (&ql)[NT][8][2],
                                            float (&s0)[NT][2], const float* q_s, int g, int tq) {
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    const int r = nt * 8 + g;
    float a0 = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      int c[4];
      token_channels<BITS>(tq, j, c);
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        const float f = code_unit<BITS>(BITS == 4 ? hh : j);
        const float x0 = q_s[qidx(r, c[2 * hh])], x1 = q_s[qidx(r, c[2 * hh + 1])];
        a0 += x0 + x1;
        if (ROT) {
          split_pair16(x0 * f, x1 * f, qb[nt][j][hh], ql[nt][j][hh]);
        } else {
          qb[nt][j][hh] = pack_half2(x0 * f, x1 * f);
        }
      }
    }
    // the total for query g, then the values of this thread's columns 2tq, 2tq+1
    a0 += __shfl_xor_sync(kFull, a0, 1);
    a0 += __shfl_xor_sync(kFull, a0, 2);
#pragma unroll
    for (int e = 0; e < 2; ++e) s0[nt][e] = __shfl_sync(kFull, a0, (2 * tq + e) << 2);
  }
}

// ---------------------------------------------------------------------------
// Softmax update of one 16-token slice
// ---------------------------------------------------------------------------
template <int NT, int NZ>
__device__ __forceinline__ void softmax_update(WarpState<NT, NZ>& ws, float (&sc)[NT][4], float (&p)[NT][4]) {
  // The running maxima are only moved when a score exceeds them by 2^8, so the
  // exact column maxima are needed only when some lane sees such a score.
  bool need = false;
#pragma unroll
  for (int nt = 0; nt < NT; ++nt)
#pragma unroll
    for (int e = 0; e < 2; ++e) need |= fmaxf(sc[nt][e], sc[nt][2 + e]) > ws.m[nt][e] + 8.0f;
  if (__any_sync(kFull, need)) {
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        float v = fmaxf(sc[nt][e], sc[nt][2 + e]);
        v = fmaxf(v, __shfl_xor_sync(kFull, v, 4));
        v = fmaxf(v, __shfl_xor_sync(kFull, v, 8));
        v = fmaxf(v, __shfl_xor_sync(kFull, v, 16));
        const float mn = fmaxf(ws.m[nt][e], v);
        const float a = (ws.m[nt][e] == -INFINITY) ? 0.f : fast_exp2(ws.m[nt][e] - mn);
        ws.m[nt][e] = mn;
        ws.l[nt][e] *= a;
#pragma unroll
        for (int zz = 0; zz < NZ; ++zz) ws.z[nt][e][zz] *= a;
#pragma unroll
        for (int mt = 0; mt < 8; ++mt) {
          ws.o[nt][mt][e] *= a;
          ws.o[nt][mt][2 + e] *= a;
        }
      }
    }
  }
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
    for (int i = 0; i < 4; ++i) p[nt][i] = fast_exp2(sc[nt][i] - ws.m[nt][i & 1]);
#pragma unroll
    for (int e = 0; e < 2; ++e) ws.l[nt][e] += p[nt][e] + p[nt][2 + e];
  }
}

// B fragments of P^T (rows scaled by fg for token g, fg8 for token g+8), as a
// BF16 hi + lo pair: b[0..1] hi, b[2..3] lo, so that P is carried to ~16 bits.
__device__ __forceinline__ void pfrag(const float (&p)[4], float fg, float fg8, uint32_t (&b)[4]) {
  uint32_t h0, l0, h1, l1;
  split_pair(p[0] * fg, p[1] * fg, h0, l0);
  split_pair(p[2] * fg8, p[3] * fg8, h1, l1);
  b[0] = movtrans(h0);
  b[1] = movtrans(h1);
  b[2] = movtrans(l0);
  b[3] = movtrans(l1);
}

// O^T m-tile += A * P^T (hi and lo parts)
__device__ __forceinline__ void mma_pv(float (&o)[4], const uint32_t (&a)[4], const uint32_t (&b)[4]) {
  mma_bf16(o, a, b[0], b[1]);
  mma_bf16(o, a, b[2], b[3]);
}

// Coded values multiply exact FP16 codes by P' = p * s / vb in FP16 (one MMA;
// about 11 significant bits, so each product carries at most 2^-12 relative
// error, far inside the tolerance).  vb is a power of two bounding every value
// scale s seen so far, so P' <= p <= 256 never overflows, and only weights
// below ~1e-4 of the largest reach FP16's subnormal range; when a larger
// scale arrives, vb grows and the accumulators are rescaled exactly.  The
// accumulators are in units of vb.
__device__ __forceinline__ void pfrag16(const float (&p)[4], float fg, float fg8, uint32_t (&b)[2]) {
  b[0] = movtrans(pack_half2(p[0] * fg, p[1] * fg));
  b[1] = movtrans(pack_half2(p[2] * fg8, p[3] * fg8));
}

// O^T += V^T . P^T over one slice of coded values in channel order: tokens ta,
// tb (k-slots 2tq, 2tq + 1) and tc, td (2tq + 8, 2tq + 9) of this lane.  M-tile
// mt's rows g and g + 8 are channels 16g + mt and 16g + 8 + mt, in units of
// code_unit(mt) 2^24 (4 bits: of m-tile mt % 4).
template <int BITS, int NT>
__device__ __forceinline__ void pv_codes(float (&o)[NT][8][4], const uint32_t* vc32, int ta, int tb, int tc, int td,
                                         int g, const uint32_t (&b)[NT][2]) {
  const int t[4] = {ta, tb, tc, td};
  if (BITS != 4) {
    // word g of a token row holds channels 16g..16g+15
    constexpr int RW = 4 * BITS;  // words per token row
    const uint32_t w0 = vc32[t[0] * RW + g], w1 = vc32[t[1] * RW + g];
    const uint32_t w8 = vc32[t[2] * RW + g], w9 = vc32[t[3] * RW + g];
    const uint32_t x[4] = {prmt(w0, w1, 0x5410), prmt(w0, w1, 0x7632), prmt(w8, w9, 0x5410),
                           prmt(w8, w9, 0x7632)};
    // 3 bits: bit 2 of word g's codes 0-7 is byte g % 2 of plane word
    // 8 + g / 2, codes 8-15 byte 2 + g % 2; two tokens side by side
    uint32_t hp[4] = {0u, 0u, 0u, 0u};
    if (BITS == 3) {
      const int pw = 8 + (g >> 1), bs = g & 1;
      const uint32_t p0 = vc32[t[0] * RW + pw], p1 = vc32[t[1] * RW + pw];
      const uint32_t p8 = vc32[t[2] * RW + pw], p9 = vc32[t[3] * RW + pw];
      hp[0] = prmt(p0, p1, plane_sel(bs));
      hp[1] = prmt(p0, p1, plane_sel(2 + bs));
      hp[2] = prmt(p8, p9, plane_sel(bs));
      hp[3] = prmt(p8, p9, plane_sel(2 + bs));
    }
#pragma unroll
    for (int mt = 0; mt < 8; ++mt) {
      uint32_t a[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        a[k] = code_pair<BITS>(x[k], mt);
        if (BITS == 3) a[k] |= plane_pair(hp[k], mt, code_pos<BITS>(mt));
      }
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) mma_f16(o[nt][mt], a, b[nt][0], b[nt][1]);
    }
  } else {
    // word 2g holds channels 16g..16g+7 (codes 0-3 low half, 4-7 high), 2g+1 the next 8
    const uint2 v0 = *reinterpret_cast<const uint2*>(vc32 + t[0] * 16 + 2 * g);
    const uint2 v1 = *reinterpret_cast<const uint2*>(vc32 + t[1] * 16 + 2 * g);
    const uint2 v8 = *reinterpret_cast<const uint2*>(vc32 + t[2] * 16 + 2 * g);
    const uint2 v9 = *reinterpret_cast<const uint2*>(vc32 + t[3] * 16 + 2 * g);
    const uint32_t xa = prmt(v0.x, v1.x, 0x5410), ya = prmt(v0.x, v1.x, 0x7632);
    const uint32_t xb = prmt(v0.y, v1.y, 0x5410), yb = prmt(v0.y, v1.y, 0x7632);
    const uint32_t xc = prmt(v8.x, v9.x, 0x5410), yc = prmt(v8.x, v9.x, 0x7632);
    const uint32_t xd = prmt(v8.y, v9.y, 0x5410), yd = prmt(v8.y, v9.y, 0x7632);
#pragma unroll
    for (int mt = 0; mt < 8; ++mt) {
      uint32_t a[4];
      a[0] = code_pair<4>(mt < 4 ? xa : ya, mt & 3);
      a[1] = code_pair<4>(mt < 4 ? xb : yb, mt & 3);
      a[2] = code_pair<4>(mt < 4 ? xc : yc, mt & 3);
      a[3] = code_pair<4>(mt < 4 ? xd : yd, mt & 3);
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) mma_f16(o[nt][mt], a, b[nt][0], b[nt][1]);
    }
  }
}

template <int NT, int NZ>
__device__ __forceinline__ void vscale_update(WarpState<NT, NZ>& ws, float smax) {
  if (__any_sync(kFull, smax > ws.vb)) {
    const float nb = pow2_ceil(warp_max(smax));
    const float a = ws.vb * pow2_inv(nb);  // a power of two: exact
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
      for (int mt = 0; mt < 8; ++mt)
#pragma unroll
        for (int i = 0; i < 4; ++i) ws.o[nt][mt][i] *= a;
    }
    ws.vb = nb;
  }
}

// ---------------------------------------------------------------------------
// One tile of a warp: kst / vst its K and V in shared memory, of which the tokens
// [skip, nvalid) are the warp's (skip: KIVI-style keys, 0 or 16).  between() runs
// after the last read of kst by a SPLIT tile (one slice) and returns false
// when the values did not arrive; the tile's probabilities are then dropped.
// ---------------------------------------------------------------------------
template <int BITS, int NT, int KM, int VM, bool ROT, int MB, class F>
__device__ __forceinline__ void compute_tile(WarpState<NT, NZOf<VM>::value>& ws, const char* kst, const char* vst,
                                             int skip, int nvalid, const uint32_t (&qb)[NT][8][2],
                                             const uint32_t (&ql)[NT][8][2], const float* q_s,
                                             const float (&kq)[NT][2], const float (&s0)[NT][2],
                                             float scale_log2, int lane, F&& between) {
  using TL = Tile<BITS, KM, VM, MB>;
  constexpr int NZ = NZOf<VM>::value;
  const int g = lane >> 2, tq = lane & 3;
  const uint32_t k_u32 = smem_u32(kst), v_u32 = smem_u32(vst) + TL::vc_off;
  const uint32_t* kc32 = reinterpret_cast<const uint32_t*>(kst);
  const char* kmp = kst + TL::km_off;
  const uint32_t* vc32 = reinterpret_cast<const uint32_t*>(vst + TL::vc_off);
  const char* vmp = vst + TL::vm_off;

  // KIVI-style keys: a warp takes whole 32-token groups (two slices) so the
  // group's scaled query fragments are built once.
  constexpr int SPU = (KM == K_KIVI) ? 2 : 1;  // slices per unit
  constexpr int UNITS = TL::tokens / (16 * SPU);
#pragma unroll 1
  for (int u = 0; u < UNITS; ++u) {
    if (u * 16 * SPU >= nvalid) break;
    float acc[SPU][NT][4];
#pragma unroll
    for (int s = 0; s < SPU; ++s)
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[s][nt][i] = 0.f;
    float zk[NT][2];  // KIVI-style: sum_c q_c z_c of the group, per query column
    uint32_t qh[NT][8][2], qlo[NT][8][2];  // KIVI-style: the group's scaled queries (hi + lo)
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) zk[nt][0] = zk[nt][1] = 0.f;

    // ---------------- scores ----------------
    if (KM == K_BF16) {
      const int tok0 = u * 16;
      const int row = tok0 + (lane & 7) + 8 * ((lane >> 3) & 1);
      const uint32_t rbase = k_u32 + row * 128;
      const int rsw = lane & 7, ch = lane >> 4;  // row % 8; second 8 channels of the k-step
      float acc2[NT][4];
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc2[nt][i] = 0.f;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        uint32_t a[4];
        ldsm_x4(a, rbase + (j >> 2) * (TL::tokens * 128) + (((2 * (j & 3) + ch) ^ rsw) << 4));
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
          mma_bf16((j & 1) ? acc2[nt] : acc[0][nt], a, qb[nt][j][0], qb[nt][j][1]);
      }
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[0][nt][i] += acc2[nt][i];
      if (TL::SPLIT && !between()) return;
    } else if (KM == K_TOKEN) {
      const int tok0 = u * 16;
      float acc2[NT][4];
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc2[nt][i] = 0.f;
      if (BITS != 4) {
        constexpr int RW = 4 * BITS;  // words per token row
        const uint2 ka = *reinterpret_cast<const uint2*>(kc32 + (tok0 + g) * RW + 2 * tq);
        const uint2 kb = *reinterpret_cast<const uint2*>(kc32 + (tok0 + g + 8) * RW + 2 * tq);
        const uint32_t w[4] = {ka.x, kb.x, ka.y, kb.y};
        // 3 bits: plane word tq holds bit 2 of words 2tq (pairs at j, j + 16)
        // and 2tq + 1 (at j + 8, j + 24)
        uint32_t pl[4] = {0u, 0u, 0u, 0u};
        if (BITS == 3) {
          const uint32_t pa = kc32[(tok0 + g) * RW + 8 + tq], pb = kc32[(tok0 + g + 8) * RW + 8 + tq];
          pl[0] = pa;
          pl[1] = pb;
          pl[2] = pa >> 8;
          pl[3] = pb >> 8;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          uint32_t a[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            a[k] = code_pair<BITS>(w[k], j);
            if (BITS == 3) a[k] |= plane_pair(pl[k], j, code_pos<BITS>(j));
          }
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) {
            float (&dst)[4] = (j & 1) ? acc2[nt] : acc[0][nt];
            mma_f16(dst, a, qb[nt][j][0], qb[nt][j][1]);
            if (ROT) mma_f16(dst, a, ql[nt][j][0], ql[nt][j][1]);
          }
        }
      } else {
        const uint4 ka = *reinterpret_cast<const uint4*>(kc32 + (tok0 + g) * 16 + 4 * tq);
        const uint4 kb = *reinterpret_cast<const uint4*>(kc32 + (tok0 + g + 8) * 16 + 4 * tq);
        const uint32_t wa[4] = {ka.x, ka.y, ka.z, ka.w};
        const uint32_t wb[4] = {kb.x, kb.y, kb.z, kb.w};
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int wi = j >> 1, i = 2 * (j & 1);
          uint32_t a[4];
          a[0] = code_pair<4>(wa[wi], i);
          a[1] = code_pair<4>(wb[wi], i);
          a[2] = code_pair<4>(wa[wi], i + 1);
          a[3] = code_pair<4>(wb[wi], i + 1);
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) {
            float (&dst)[4] = (j & 1) ? acc2[nt] : acc[0][nt];
            mma_f16(dst, a, qb[nt][j][0], qb[nt][j][1]);
            if (ROT) mma_f16(dst, a, ql[nt][j][0], ql[nt][j][1]);
          }
        }
      }
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[0][nt][i] += acc2[nt][i];
    } else {  // K_KIVI: group u of the tile; channel c has (scale, zero) = meta[u][c]
      const int gm = u * kD;  // first metadata pair of the group
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        const float* qr = q_s + (nt * 8 + g) * kQRow;
        float zpart = 0.f;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          // k-slots 2tq, 2tq+1, 2tq+8, 2tq+9 of k-step j <-> channels 16j + 4tq + 0..3
          // (the four tq lanes read four different banks of codes and metadata)
          const int c0 = 16 * j + 4 * tq;
          float2 m[4];
          meta_quad<MB>(kmp, gm + c0, m);
          const float4 qv = *reinterpret_cast<const float4*>(qr + c0);
          split_pair(qv.x * m[0].x, qv.y * m[1].x, qh[nt][j][0], qlo[nt][j][0]);
          split_pair(qv.z * m[2].x, qv.w * m[3].x, qh[nt][j][1], qlo[nt][j][1]);
          zpart = fmaf(qv.x, m[0].y, zpart);
          zpart = fmaf(qv.y, m[1].y, zpart);
          zpart = fmaf(qv.z, m[2].y, zpart);
          zpart = fmaf(qv.w, m[3].y, zpart);
        }
        // sum over the four tq lanes of query g, then fetch the columns' values
        zpart += __shfl_xor_sync(kFull, zpart, 1);
        zpart += __shfl_xor_sync(kFull, zpart, 2);
        zk[nt][0] = __shfl_sync(kFull, zpart, (2 * tq) << 2);
        zk[nt][1] = __shfl_sync(kFull, zpart, (2 * tq + 1) << 2);
      }
    }

    // ---------------- per slice: (KIVI-style keys: scores), softmax, then P.V ----------------
    // The loop stays rolled: for KIVI-style keys (two slices per unit) an
    // unrolled copy doubles the longest code path of the kernel.
#pragma unroll 1
    for (int s = 0; s < SPU; ++s) {
      const int tok0 = (u * SPU + s) * 16;
      if (tok0 >= nvalid) break;
      if (SPU > 1 && tok0 < skip) continue;
      float ks[NT][4];  // KIVI-style: this slice's scores against the scaled queries
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) ks[nt][i] = 0.f;
      if (KM == K_KIVI) {
        const uint32_t* gc = kc32 + u * kD * BITS;  // [128 channels][BITS words], token order
        // byte selector: byte (g/2) of a -> byte 0, byte (g/2) of b -> byte 2
        const uint32_t sel4 = (uint32_t)(g >> 1) | ((uint32_t)(4 + (g >> 1)) << 8);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int c0 = 16 * j + 4 * tq;
          // per channel: the word(s) of tokens 16s..16s+15 (3 bits: and the bit-2 plane)
          uint32_t w[4][2];
#pragma unroll
          for (int cc = 0; cc < 4; ++cc) {
            if (BITS == 2) {
              w[cc][0] = gc[(c0 + cc) * 2 + s];
              w[cc][1] = 0u;
            } else if (BITS == 3) {
              w[cc][0] = gc[(c0 + cc) * 3 + s];
              w[cc][1] = gc[(c0 + cc) * 3 + 2];
            } else {
              const uint2 t2 = *reinterpret_cast<const uint2*>(gc + (c0 + cc) * 4 + 2 * s);
              w[cc][0] = t2.x;
              w[cc][1] = t2.y;
            }
          }
          uint32_t a[4];
          if (BITS == 2) {
            // the word's low half holds tokens 16s..16s+7, its high half the next 8
            a[0] = codes_bf16x2((prmt(w[0][0], w[1][0], 0x5410) >> (2 * g)) & pair_mask<2>());
            a[1] = codes_bf16x2((prmt(w[0][0], w[1][0], 0x7632) >> (2 * g)) & pair_mask<2>());
            a[2] = codes_bf16x2((prmt(w[2][0], w[3][0], 0x5410) >> (2 * g)) & pair_mask<2>());
            a[3] = codes_bf16x2((prmt(w[2][0], w[3][0], 0x7632) >> (2 * g)) & pair_mask<2>());
          } else if (BITS == 3) {
            // bit 2 of token 16s + i: plane byte s (i < 8) or 2 + s (i >= 8), bit i % 8
            const uint32_t lo0 = prmt(w[0][0], w[1][0], 0x5410) >> (2 * g);
            const uint32_t lo1 = prmt(w[0][0], w[1][0], 0x7632) >> (2 * g);
            const uint32_t lo2 = prmt(w[2][0], w[3][0], 0x5410) >> (2 * g);
            const uint32_t lo3 = prmt(w[2][0], w[3][0], 0x7632) >> (2 * g);
            const uint32_t h0 = prmt(w[0][1], w[1][1], plane_sel(s)) >> g;
            const uint32_t h1 = prmt(w[0][1], w[1][1], plane_sel(2 + s)) >> g;
            const uint32_t h2 = prmt(w[2][1], w[3][1], plane_sel(s)) >> g;
            const uint32_t h3 = prmt(w[2][1], w[3][1], plane_sel(2 + s)) >> g;
            a[0] = codes_bf16x2((lo0 & 0x00030003u) | ((h0 & 0x00010001u) << 2));
            a[1] = codes_bf16x2((lo1 & 0x00030003u) | ((h1 & 0x00010001u) << 2));
            a[2] = codes_bf16x2((lo2 & 0x00030003u) | ((h2 & 0x00010001u) << 2));
            a[3] = codes_bf16x2((lo3 & 0x00030003u) | ((h3 & 0x00010001u) << 2));
          } else {
            // words 2s, 2s+1 of a channel: tokens 16s..16s+7 and 16s+8..16s+15
            const int sh = 4 * (g & 1);
            a[0] = codes_bf16x2((prmt(w[0][0], w[1][0], sel4) >> sh) & pair_mask<4>());
            a[1] = codes_bf16x2((prmt(w[0][1], w[1][1], sel4) >> sh) & pair_mask<4>());
            a[2] = codes_bf16x2((prmt(w[2][0], w[3][0], sel4) >> sh) & pair_mask<4>());
            a[3] = codes_bf16x2((prmt(w[2][1], w[3][1], sel4) >> sh) & pair_mask<4>());
          }
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) {
            mma_bf16(ks[nt], a, qh[nt][j][0], qh[nt][j][1]);
            mma_bf16(ks[nt], a, qlo[nt][j][0], qlo[nt][j][1]);
          }
        }
      }
      float sc[NT][4];
      if (KM == K_TOKEN) {
        // score = s (q.c) + z sum(q), kq and s0 with the units and the softmax scale
        const float2 mg = meta_pair<MB>(kmp, tok0 + g), mg8 = meta_pair<MB>(kmp, tok0 + g + 8);
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            sc[nt][e] = fmaf(mg.x, acc[s][nt][e] * kq[nt][e], mg.y * s0[nt][e]);
            sc[nt][2 + e] = fmaf(mg8.x, acc[s][nt][2 + e] * kq[nt][e], mg8.y * s0[nt][e]);
          }
        }
      } else if (KM == K_KIVI) {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
          for (int i = 0; i < 4; ++i) sc[nt][i] = (ks[nt][i] + zk[nt][i & 1]) * scale_log2;
      } else {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
          for (int i = 0; i < 4; ++i) sc[nt][i] = acc[s][nt][i] * scale_log2;
      }
      if (tok0 + 16 > nvalid) {
        const bool vg0 = tok0 + g < nvalid, vg8 = tok0 + g + 8 < nvalid;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          if (!vg0) sc[nt][0] = sc[nt][1] = -INFINITY;
          if (!vg8) sc[nt][2] = sc[nt][3] = -INFINITY;
        }
      }
      float p[NT][4];
      softmax_update<NT, NZ>(ws, sc, p);

      if (VM == V_BF16) {
        uint32_t b[NT][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) pfrag(p[nt], 1.f, 1.f, b[nt]);
        if (tok0 + 16 > nvalid) {
          // rows past the end hold whatever follows in the arena: zero them so
          // that 0 * (non-finite) cannot reach the accumulators
          for (int i = lane; i < (tok0 + 16 - nvalid) * 16; i += 32) {
            const int rr = nvalid + (i >> 4), c = i & 15;
            *reinterpret_cast<uint4*>(const_cast<char*>(vst) + TL::vc_off + (c >> 3) * (TL::tokens * 128) +
                                      rr * 128 + (c & 7) * 16) = make_uint4(0u, 0u, 0u, 0u);
          }
          fence_proxy_async_shared();  // the slot is refilled by TMA later
          __syncwarp();
        }
        const int row = tok0 + (lane & 7) + 8 * (lane >> 4);
        const uint32_t rbase = v_u32 + row * 128;
        const int rsw = lane & 7, ch = (lane >> 3) & 1;
#pragma unroll
        for (int mt = 0; mt < 8; ++mt) {
          uint32_t a[4];
          ldsm_x4_trans(a, rbase + (mt >> 2) * (TL::tokens * 128) + (((2 * (mt & 3) + ch) ^ rsw) << 4));
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) mma_pv(ws.o[nt][mt], a, b[nt]);
        }
      } else if (VM == V_TOKEN) {
        // metadata past the end of the tile is stale: its factors are zeroed
        const bool ok0 = tok0 + g < nvalid, ok8 = tok0 + g + 8 < nvalid;
        const float2 vg = ok0 ? meta_pair<MB>(vmp, tok0 + g) : make_float2(0.f, 0.f);
        const float2 vg8 = ok8 ? meta_pair<MB>(vmp, tok0 + g + 8) : make_float2(0.f, 0.f);
        vscale_update(ws, fmaxf(vg.x, vg8.x));
        const float inv = pow2_inv(ws.vb);
        uint32_t b[NT][2];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          pfrag16(p[nt], vg.x * inv, vg8.x * inv, b[nt]);
#pragma unroll
          for (int e = 0; e < 2; ++e) ws.z[nt][e][0] += p[nt][e] * vg.y + p[nt][2 + e] * vg8.y;
        }
        const int t0 = tok0 + 2 * tq;
        pv_codes<BITS, NT>(ws.o, vc32, t0, t0 + 1, t0 + 8, t0 + 9, g, b);
      } else {  // V_KIVI: 4 value groups of 32 channels; m-tile mt = channels 16mt..16mt+15
        float sv_g[4], zv_g[4], sv_g8[4], zv_g8[4];
        {
          // the four (scale, zero) pairs of a token; stale metadata past the end is zeroed
          const bool ok0 = tok0 + g < nvalid, ok8 = tok0 + g + 8 < nvalid;
          float2 a[4], c[4];
          meta_quad<MB>(vmp, (tok0 + g) * 4, a);
          meta_quad<MB>(vmp, (tok0 + g + 8) * 4, c);
#pragma unroll
          for (int jg = 0; jg < 4; ++jg) {
            sv_g[jg] = ok0 ? a[jg].x : 0.f;
            zv_g[jg] = ok0 ? a[jg].y : 0.f;
            sv_g8[jg] = ok8 ? c[jg].x : 0.f;
            zv_g8[jg] = ok8 ? c[jg].y : 0.f;
          }
        }
        vscale_update(ws, fmaxf(fmaxf(fmaxf(sv_g[0], sv_g[1]), fmaxf(sv_g[2], sv_g[3])),
                                fmaxf(fmaxf(sv_g8[0], sv_g8[1]), fmaxf(sv_g8[2], sv_g8[3]))));
        const float inv = pow2_inv(ws.vb);
        uint32_t b[NT][4][2];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
          for (int jg = 0; jg < 4; ++jg) {
            pfrag16(p[nt], sv_g[jg] * inv, sv_g8[jg] * inv, b[nt][jg]);
#pragma unroll
            for (int e = 0; e < 2; ++e)
              ws.z[nt][e][jg % NZ] += p[nt][e] * zv_g[jg] + p[nt][2 + e] * zv_g8[jg];
          }
        }
        const int t0 = tok0 + 2 * tq;
        constexpr int W = 4 * BITS;  // words per token
        const uint32_t sel4 = (uint32_t)(g >> 1) | ((uint32_t)(4 + (g >> 1)) << 8);
#pragma unroll
        for (int mt = 0; mt < 8; ++mt) {
          uint32_t a[4];
          if (BITS == 2) {
            const uint32_t w0 = vc32[t0 * W + mt], w1 = vc32[(t0 + 1) * W + mt];
            const uint32_t w8 = vc32[(t0 + 8) * W + mt], w9 = vc32[(t0 + 9) * W + mt];
            a[0] = codes_f16x2((prmt(w0, w1, 0x5410) >> (2 * g)) & pair_mask<2>());
            a[1] = codes_f16x2((prmt(w0, w1, 0x7632) >> (2 * g)) & pair_mask<2>());
            a[2] = codes_f16x2((prmt(w8, w9, 0x5410) >> (2 * g)) & pair_mask<2>());
            a[3] = codes_f16x2((prmt(w8, w9, 0x7632) >> (2 * g)) & pair_mask<2>());
          } else if (BITS == 3) {
            // channels 16mt + g and 16mt + 8 + g: bit 2 in byte mt % 2 and
            // 2 + mt % 2 of plane word 8 + mt / 2, bit g
            const uint32_t w0 = vc32[t0 * W + mt], w1 = vc32[(t0 + 1) * W + mt];
            const uint32_t w8 = vc32[(t0 + 8) * W + mt], w9 = vc32[(t0 + 9) * W + mt];
            const int pw = 8 + (mt >> 1), bs = mt & 1;
            const uint32_t p0 = vc32[t0 * W + pw], p1 = vc32[(t0 + 1) * W + pw];
            const uint32_t p8 = vc32[(t0 + 8) * W + pw], p9 = vc32[(t0 + 9) * W + pw];
            const uint32_t h0 = prmt(p0, p1, plane_sel(bs)) >> g, h1 = prmt(p0, p1, plane_sel(2 + bs)) >> g;
            const uint32_t h2 = prmt(p8, p9, plane_sel(bs)) >> g, h3 = prmt(p8, p9, plane_sel(2 + bs)) >> g;
            a[0] = codes_f16x2(((prmt(w0, w1, 0x5410) >> (2 * g)) & 0x00030003u) | ((h0 & 0x00010001u) << 2));
            a[1] = codes_f16x2(((prmt(w0, w1, 0x7632) >> (2 * g)) & 0x00030003u) | ((h1 & 0x00010001u) << 2));
            a[2] = codes_f16x2(((prmt(w8, w9, 0x5410) >> (2 * g)) & 0x00030003u) | ((h2 & 0x00010001u) << 2));
            a[3] = codes_f16x2(((prmt(w8, w9, 0x7632) >> (2 * g)) & 0x00030003u) | ((h3 & 0x00010001u) << 2));
          } else {
            const uint2 u0 = *reinterpret_cast<const uint2*>(vc32 + t0 * W + 2 * mt);
            const uint2 u1 = *reinterpret_cast<const uint2*>(vc32 + (t0 + 1) * W + 2 * mt);
            const uint2 u8 = *reinterpret_cast<const uint2*>(vc32 + (t0 + 8) * W + 2 * mt);
            const uint2 u9 = *reinterpret_cast<const uint2*>(vc32 + (t0 + 9) * W + 2 * mt);
            const int sh = 4 * (g & 1);
            a[0] = codes_f16x2((prmt(u0.x, u1.x, sel4) >> sh) & pair_mask<4>());
            a[1] = codes_f16x2((prmt(u0.y, u1.y, sel4) >> sh) & pair_mask<4>());
            a[2] = codes_f16x2((prmt(u8.x, u9.x, sel4) >> sh) & pair_mask<4>());
            a[3] = codes_f16x2((prmt(u8.y, u9.y, sel4) >> sh) & pair_mask<4>());
          }
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) mma_f16(ws.o[nt][mt], a, b[nt][mt >> 1][0], b[nt][mt >> 1][1]);
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Combine of (m, l, o) partials of the same queries (the four warps of a CTA,
// or the splits of a head): part s, query j at parts + s * sstride + j * 132
// (m at +0, l at +1, o at +4).  With M = max_s m_s and f_s = 2^(m_s - M):
// o = sum_s f_s o_s / L, L = sum_s f_s l_s.  combine_weights leaves f_s in
// fw[s][j] (s < 16), L in fw[kFwL][j], M in fw[kFwM][j] and 1 / L in
// fw[kFwR][j] (rows of kMaxG).  Both steps are short dependency chains: eight
// threads per query reduce the weights with shuffles, and each thread then
// accumulates one channel of every query at once.
// ---------------------------------------------------------------------------
constexpr int kFwL = 16, kFwM = 17, kFwR = 18;
static_assert(kThreads == 8 * kMaxG, "eight combine threads per query");

__device__ __forceinline__ void combine_weights(const float* parts, int n, int sstride, int G, float* fw,
                                                int tid) {
  // thread t: query t / 8, parts t % 8 and t % 8 + 8
  const int j = tid >> 3, sl = tid & 7;
  const bool h0 = j < G && sl < n, h1 = j < G && sl + 8 < n;
  const float* pj = parts + j * kPartialStride;
  const float m0 = h0 ? pj[sl * sstride] : -INFINITY;
  const float l0 = h0 ? pj[sl * sstride + 1] : 0.f;
  const float m1 = h1 ? pj[(sl + 8) * sstride] : -INFINITY;
  const float l1 = h1 ? pj[(sl + 8) * sstride + 1] : 0.f;
  float M = fmaxf(m0, m1);
  M = fmaxf(M, __shfl_xor_sync(kFull, M, 1));
  M = fmaxf(M, __shfl_xor_sync(kFull, M, 2));
  M = fmaxf(M, __shfl_xor_sync(kFull, M, 4));
  const float f0 = (m0 == -INFINITY) ? 0.f : fast_exp2(m0 - M);
  const float f1 = (m1 == -INFINITY) ? 0.f : fast_exp2(m1 - M);
  float Ls = fmaf(f0, l0, f1 * l1);
  Ls += __shfl_xor_sync(kFull, Ls, 1);
  Ls += __shfl_xor_sync(kFull, Ls, 2);
  Ls += __shfl_xor_sync(kFull, Ls, 4);
  if (h0) fw[sl * kMaxG + j] = f0;
  if (h1) fw[(sl + 8) * kMaxG + j] = f1;
  if (j < G && sl == 0) {
    fw[kFwL * kMaxG + j] = Ls;
    fw[kFwM * kMaxG + j] = M;
    fw[kFwR * kMaxG + j] = 1.0f / Ls;
  }
  __syncthreads();
}

// Channel c of queries 0..JM-1 (those below G): acc[j] = sum_s f_s o_s[j][c].
template <int JM>
__device__ __forceinline__ void combine_out(const float* parts, int n, int sstride, const float* fw, int G, int c,
                                            float (&acc)[JM]) {
#pragma unroll
  for (int j = 0; j < JM; ++j) acc[j] = 0.f;
#pragma unroll 1
  for (int s = 0; s < n; ++s) {
    const float* ps = parts + s * sstride + 4 + c;
    const float* fs = fw + s * kMaxG;
#pragma unroll
    for (int j = 0; j < JM; ++j)
      if (j < G) acc[j] = fmaf(fs[j], ps[j * kPartialStride], acc[j]);
  }
}

// One combine pass: the weights, then channel `tid` of every query, written
// as the final BF16 output rows (out: row 0 of this head's queries) or as this
// split's partial (mine).  Not inlined: the warp combine and the split merge
// run the same instructions, so the merge -- once per head, at the end of the
// launch -- executes from cached code.
template <int JM>
__device__ __noinline__ void combine_pass(const float* src, int n, int sstride, float* fw, int G, int tid,
                                          bool final, uint16_t* out, float* mine) {
  combine_weights(src, n, sstride, G, fw, tid);
  float acc[JM];
  combine_out<JM>(src, n, sstride, fw, G, tid, acc);
#pragma unroll
  for (int j = 0; j < JM; ++j) {
    if (j >= G) break;
    if (final) {
      out[(size_t)j * kD + tid] = (uint16_t)f32_to_bf16_rn(acc[j] * fw[kFwR * kMaxG + j]);
    } else {
      mine[j * kPartialStride + 4 + tid] = acc[j];
      if (tid == 0) {
        mine[j * kPartialStride + 0] = fw[kFwM * kMaxG + j];
        mine[j * kPartialStride + 1] = fw[kFwL * kMaxG + j];
      }
    }
  }
}

// ---------------------------------------------------------------------------
// One work item with a given key / value mode: pipeline, then per-warp results
// into shared memory (m, l, o[q][channel]).
// ---------------------------------------------------------------------------
// 16-byte pieces of the staged queries per thread (piece i: query row i / 16,
// channels 8 (i % 16) .. + 7).
template <int NT>
struct QPieces {
  static constexpr int n = (NT * 8 * 16 + kThreads - 1) / kThreads;
};

// The queries as fp32 rows in shared memory (rows >= G zero).  TOP >= 0: each
// row divided by a power of two (exact) that brings its largest element to
// 2^TOP at most, kept in qn[row].
template <int NT, int TOP>
__device__ __forceinline__ void stage_queries(float* q_s, float* qn, const uint4 (&qv)[QPieces<NT>::n], int tid) {
#pragma unroll
  for (int k = 0; k < QPieces<NT>::n; ++k) {
    const int i = tid + k * kThreads;
    if (i < NT * 8 * 16) {  // whole warps
      // piece i: row i / 16, channels 8 (i % 16) .. + 7
      float4* dst = reinterpret_cast<float4*>(q_s + qidx(i >> 4, 8 * (i & 15)));
      float f[8];
      bf16x2_to_f32(qv[k].x, f[0], f[1]);
      bf16x2_to_f32(qv[k].y, f[2], f[3]);
      bf16x2_to_f32(qv[k].z, f[4], f[5]);
      bf16x2_to_f32(qv[k].w, f[6], f[7]);
      if (TOP >= 0) {
        float m = 0.f;
#pragma unroll
        for (int e = 0; e < 8; ++e) m = fmaxf(m, fabsf(f[e]));
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, o));  // the row's 16 threads
        const float n = pow2_ceil(fminf(fmaxf(m, kScaleLow), kScaleTop)) * (1.0f / (float)(1 << (TOP < 0 ? 0 : TOP)));
        const float inv = pow2_inv(n);
#pragma unroll
        for (int e = 0; e < 8; ++e) f[e] *= inv;
        if ((i & 15) == 0) qn[i >> 4] = n;
      }
      dst[0] = make_float4(f[0], f[1], f[2], f[3]);
      dst[1] = make_float4(f[4], f[5], f[6], f[7]);
    }
  }
}

template <int BITS, int NT, int KM, int VM, bool ROT, int MB, int GRAN = 16>
__device__ __forceinline__ void run_item(char* smem, const Seg& sg, int tb, int te, const DecodeParams& p,
                                         const uint4 (&qv)[QPieces<NT>::n], int G, float* parts) {
  using TL = Tile<BITS, KM, VM, MB>;
  constexpr int NZ = NZOf<VM>::value;
  const int tid = threadIdx.x, lane = tid & 31;
  // the same in every lane, and known to be: the pipeline's addresses and
  // branches below are uniform
  const int warp = __shfl_sync(kFull, tid >> 5, 0);
  const int g = lane >> 2, tq = lane & 3;
  float* q_s = reinterpret_cast<float*>(smem + SmemLayout<NT>::q);
  const float scale_log2 = p.scale_log2;

  WarpPipe<BITS, NT, KM, VM, MB, false, GRAN> pipe(smem, warp, sg, p, tb, te);

  // Queries of this KV head's group (fp32, rows >= G zero), rotated for
  // AKVQ-style coded keys.
  // Per-token coded keys: rows scaled so that every staged and rotated element (at most
  // sqrt(128) times the row's largest) is below FP16's 65504.
  constexpr int TOP = KM == K_TOKEN ? (ROT ? 11 : 15) : -1;
  float* qn = reinterpret_cast<float*>(smem + SmemLayout<NT>::qn);
  stage_queries<NT, TOP>(q_s, qn, qv, tid);
  __syncthreads();
  if (ROT) {
    for (int j = warp; j < G; j += kWarps) {
      float x[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) x[i] = q_s[qidx(j, lane * 4 + i)];
      fwht128_warp(x, lane);
#pragma unroll
      for (int i = 0; i < 4; ++i) q_s[qidx(j, lane * 4 + i)] = x[i];
    }
    __syncthreads();
  }
  uint32_t qb[NT][8][2], ql[NT][8][2];
#pragma unroll
  for (int nt = 0; nt < NT; ++nt)
#pragma unroll
    for (int j = 0; j < 8; ++j) qb[nt][j][0] = qb[nt][j][1] = ql[nt][j][0] = ql[nt][j][1] = 0u;
  // per-token coded keys, per column: unit of the key MMAs' results and sum of
  // the query, both with the softmax scale
  float kq[NT][2], s0[NT][2];
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) kq[nt][0] = kq[nt][1] = s0[nt][0] = s0[nt][1] = 0.f;
  if (KM == K_BF16) qfrag_natural<NT>(qb, q_s, g, tq);
  if (KM == K_TOKEN) {
    qfrag_token<BITS, NT, ROT>(qb, ql, s0, q_s, g, tq);
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float n = qn[nt * 8 + 2 * tq + e] * scale_log2;
        s0[nt][e] *= n;
        kq[nt][e] = n * kCodeUnit;
      }
  }

  WarpState<NT, NZ> ws;
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      ws.m[nt][e] = -INFINITY;
      ws.l[nt][e] = 0.f;
#pragma unroll
      for (int zz = 0; zz < NZ; ++zz) ws.z[nt][e][zz] = 0.f;
    }
#pragma unroll
    for (int mt = 0; mt < 8; ++mt)
#pragma unroll
      for (int i = 0; i < 4; ++i) ws.o[nt][mt][i] = 0.f;
  }
  ws.vb = __uint_as_float(0x00800000u);  // 2^-126: no value scale seen yet

#pragma unroll 1
  for (int it = 0; it < pipe.n_tiles; ++it) {
    if (!pipe.landed()) break;
    if (it == 0) pipe.fill_rest();
    const char* kst = pipe.slot();
    const char* vst = TL::SPLIT ? pipe.next_slot() : kst;
    bool ok = true;
    compute_tile<BITS, NT, KM, VM, ROT, MB>(ws, kst, vst, it == 0 ? pipe.skip : 0, pipe.tile_tokens(it), qb, ql, q_s, kq,
                                            s0, scale_log2, lane, [&]() {
                                              pipe.refill();
                                              return ok = pipe.landed();
                                            });
    if (TL::SPLIT && !ok) break;
    pipe.refill();
  }
  pipe.drain(lane);
  __syncthreads();  // the warps' buffers are reused for the reduction below

  // ---- per-warp results: reduce l and the value-zero terms over the 8 rows g ----
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      float l = ws.l[nt][e];
      l += __shfl_xor_sync(kFull, l, 4);
      l += __shfl_xor_sync(kFull, l, 8);
      l += __shfl_xor_sync(kFull, l, 16);
#pragma unroll
      for (int zz = 0; zz < NZ; ++zz) {
        float z = ws.z[nt][e][zz];
        z += __shfl_xor_sync(kFull, z, 4);
        z += __shfl_xor_sync(kFull, z, 8);
        z += __shfl_xor_sync(kFull, z, 16);
        ws.z[nt][e][zz] = z;
      }
      const int q = nt * 8 + 2 * tq + e;
      float* prow = parts + (warp * kMaxG + q) * kPartialStride;  // (m, l, -, -, o[128])
      if (g == 0) {
        prow[0] = ws.m[nt][e];
        prow[1] = l;
      }
      float* orow = prow + 4;
#pragma unroll
      for (int mt = 0; mt < 8; ++mt) {
        int c_lo, c_hi;  // channels of rows g and g+8 of m-tile mt
        if (VM == V_TOKEN) {
          c_lo = 16 * g + mt;
          c_hi = 16 * g + 8 + mt;
          // units of the codes (a position's factor, 2^24), then of the scales (vb)
          const float f = code_unit<BITS>(BITS == 4 ? mt % 4 : mt) * kCodeUnit;
          orow[c_lo] = fmaf(ws.o[nt][mt][e] * f, ws.vb, ws.z[nt][e][0]);
          orow[c_hi] = fmaf(ws.o[nt][mt][2 + e] * f, ws.vb, ws.z[nt][e][0]);
        } else {
          c_lo = 16 * mt + g;
          c_hi = 16 * mt + 8 + g;
          const float z = (VM == V_KIVI) ? ws.z[nt][e][(mt >> 1) % NZ] : 0.f;
          if (VM == V_KIVI) {
            orow[c_lo] = fmaf(ws.o[nt][mt][e], ws.vb, z);
            orow[c_hi] = fmaf(ws.o[nt][mt][2 + e], ws.vb, z);
          } else {
            orow[c_lo] = ws.o[nt][mt][e];
            orow[c_hi] = ws.o[nt][mt][2 + e];
          }
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// KIVI-style items with QC = 1 or 2 queries per KV head (multi-head attention):
// the eight MMA columns hold what run_item leaves to lane-dependent shifts.
//
// Keys, 64 tokens (two 32-token groups) at a time.  Row g of every m-tile is
// half g / 4 of code word g % 4 (16 tokens: word s of group r is 2r + s), and
// the m-tile picks the position inside the half, so a lane expands its words
// at fixed bit positions (three shifts for eight of them, see code_pair) instead
// of shifting every pair by its own amount.  The rows of one m-tile then belong to both groups, whose scaled queries q_c s_c differ: column
// 4r + 2k + h holds group r's, h the FP16 hi or lo part, k the query (QC = 2)
// or the parity of the k-steps the lane scales (QC = 1: each lane builds half
// of them, the other columns see zeros).  Row g reads columns 4r .. 4r + 3 of
// its group r = (g / 2) % 2.
// The 64 scores pass through shared memory, so the softmax works on two tokens
// per lane instead of four columns of which one or two are real.
//
// Values: column 4q + j holds p_t s_tj of value group j, so every row takes the
// channel-order expansion of per-token codes (pv_codes) and reads the column of
// its own group (channels 16g .. 16g + 15: group g / 2).  Tokens tq, tq + 4,
// tq + 8, tq + 12 of a slice sit in one lane's k-slots (codes and metadata of
// the four tq lanes on different banks).
//
// 278 warp instructions per 16-token slice; 32 KV heads of 3,120 tokens in 16 rows
// 55 us a layer, 0.77 of the measured copy rate.  (run_item, with one query in eight
// columns, takes 772 and is bound by issue: 105 us.)  Error against 64 bits 1.7e-3,
// as run_item's (with BF16 128 + c and FP16 1024 + c operands, the offsets removed by
// MMAs over constant tiles, 2.1e-3).
// ---------------------------------------------------------------------------
template <int QC>
struct ColState {
  float o[1][8][4];   // as WarpState, in units of vb
  float vb;
  float kb;      // power-of-two bound of the key channel scales seen so far
  float z;       // column g: sum_t p_t z_t of value group g % 4, query g / 4
  float m[QC], l[QC];  // running maxima (the warp's), sums of this lane's tokens
};

// Scores of the tile's tokens 2 lane, 2 lane + 1 (x[q][i], log2 units, -inf past
// the end) -> probabilities into ps[q][token], a slice's 16 tokens permuted so
// that lane tq's four are contiguous (token t of a slice at 4 (t % 4) + t / 4).
template <int QC>
__device__ __forceinline__ void cols_softmax(ColState<QC>& ws, const float (&x)[QC][2], float* ps, int lane) {
  bool need = false;
#pragma unroll
  for (int q = 0; q < QC; ++q) need |= fmaxf(x[q][0], x[q][1]) > ws.m[q] + 8.0f;
  if (__any_sync(kFull, need)) {
    float a[QC];
#pragma unroll
    for (int q = 0; q < QC; ++q) {
      const float mn = fmaxf(ws.m[q], warp_max(fmaxf(x[q][0], x[q][1])));
      a[q] = (ws.m[q] == -INFINITY) ? 0.f : fast_exp2(ws.m[q] - mn);
      ws.m[q] = mn;
      ws.l[q] *= a[q];
    }
    const float az = (QC == 2 && (lane & 16)) ? a[QC - 1] : a[0];  // this lane's column g: query g / 4
    const float ao = (QC == 2 && (lane & 2)) ? a[QC - 1] : a[0];   // its accumulator columns 2tq, 2tq + 1
    ws.z *= az;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int mt = 0; mt < 8; ++mt) ws.o[0][mt][i] *= ao;
  }
  __syncwarp();  // the scores have been read
  const int t = 2 * lane;
  float* dst = ps + (t & ~15) + 4 * (t & 3) + ((t >> 2) & 3);
#pragma unroll
  for (int q = 0; q < QC; ++q) {
    const float p0 = fast_exp2(x[q][0] - ws.m[q]), p1 = fast_exp2(x[q][1] - ws.m[q]);
    ws.l[q] += p0 + p1;
    dst[64 * q] = p0;
    dst[64 * q + 4] = p1;
  }
  __syncwarp();
}

// The query rows of run_item_cols are staged with their largest element at 1 at
// most, so that no sum over them overflows where the scores would not; times a
// channel scale over kb it is brought to 2^kColsTop, near the top of FP16's range.
constexpr int kColsTop = 15;

// Raw scores of a 64-token tile of KIVI-style keys: kst its codes and metadata,
// x[q][i] the scores of tokens 2 lane + i, in units of the staged query rows
// and without the softmax scale.
template <int BITS, int QC, int MB>
__device__ __forceinline__ void cols_scores(const char* kst, const char* kmeta, const float* q_s, float* ps, float& kb,
                                            bool two_groups, int lane, float (&x)[QC][2]) {
  const int g = lane >> 2, tq = lane & 3;
  const int sel = (g >> 1) & 1, lo = g & 1;  // this lane's column: k-step parity or query; hi or lo part
  // scaled queries of group g / 4, this lane's column
  constexpr int NB = QC == 1 ? 4 : 8;
  uint32_t own[NB][2];
  float zk = 0.f;
  {
    // in units of kb, a power of two no smaller than any channel scale so far
    float top = 0.f;
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      float2 m[4];
      meta_quad<MB>(kmeta, (g >> 2) * kD + 16 * (QC == 1 ? 2 * i + sel : i) + 4 * tq, m);
      top = fmaxf(top, fmaxf(fmaxf(m[0].x, m[1].x), fmaxf(m[2].x, m[3].x)));
    }
    if (!two_groups && lane >= 16) top = 0.f;  // stale metadata of an absent second group
    if (__any_sync(kFull, top > kb)) kb = pow2_ceil(fminf(warp_max(top), kScaleTop));
  }
  const float inv = pow2_inv(kb) * (float)(1 << kColsTop);
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    const int c0 = 16 * (QC == 1 ? 2 * i + sel : i) + 4 * tq;
    float2 m[4];
    meta_quad<MB>(kmeta, (g >> 2) * kD + c0, m);
    const float4 qv = *reinterpret_cast<const float4*>(q_s + (QC == 1 ? 0 : sel) * kQRow + c0);
    uint32_t hi, rest;
    split_pair16(qv.x * (m[0].x * inv), qv.y * (m[1].x * inv), hi, rest);
    own[i][0] = lo ? rest : hi;
    split_pair16(qv.z * (m[2].x * inv), qv.w * (m[3].x * inv), hi, rest);
    own[i][1] = lo ? rest : hi;
    zk = fmaf(qv.x, m[0].y, zk);
    zk = fmaf(qv.y, m[1].y, zk);
    zk = fmaf(qv.z, m[2].y, zk);
    zk = fmaf(qv.w, m[3].y, zk);
  }
  zk += __shfl_xor_sync(kFull, zk, 1);
  zk += __shfl_xor_sync(kFull, zk, 2);
  const float zo = __shfl_xor_sync(kFull, zk, 8);  // the other parity's part, or the other query's term

  const int r = (g >> 1) & 1, s = g & 1;  // group and word of this lane's rows
  const bool upper = g >= 4;              // half of the word
  const uint32_t half = upper ? 0x7632u : 0x5410u;
  const uint32_t* gc = reinterpret_cast<const uint32_t*>(kst) + r * (kD * BITS);
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int mt = 0; mt < 4; ++mt) acc[mt][i] = 0.f;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    // k-slots 2tq, 2tq + 1, 2tq + 8, 2tq + 9 of k-step j <-> channels 16j + 4tq + 0..3
    const int c0 = 16 * j + 4 * tq;
    uint32_t b0 = own[QC == 1 ? j >> 1 : j][0], b1 = own[QC == 1 ? j >> 1 : j][1];
    if (QC == 1 && sel != (j & 1)) b0 = b1 = 0u;
    uint32_t y[2][2], hp[2] = {0u, 0u};  // per channel pair: codes of its half word(s), bit-2 planes
#pragma unroll
    for (int cp = 0; cp < 2; ++cp) {
      const uint32_t* w = gc + (c0 + 2 * cp) * BITS;
      if (BITS == 4) {
        const int i = 2 * s + (upper ? 1 : 0);
        y[cp][0] = prmt(w[i], w[4 + i], 0x5410);
        y[cp][1] = prmt(w[i], w[4 + i], 0x7632);
      } else {
        y[cp][0] = y[cp][1] = prmt(w[s], w[BITS + s], half);
        if (BITS == 3) hp[cp] = prmt(w[2], w[BITS + 2], plane_sel(0) + 0x1111u * (s + (upper ? 2 : 0)));
      }
    }
#pragma unroll
    for (int mt = 0; mt < 4; ++mt) {
      uint32_t a[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int pos = mt + 4 * (k & 1);  // rows g: positions 0..3, rows g + 8: 4..7
        a[k] = code_pair<BITS>(y[k >> 1][BITS == 4 ? k & 1 : 0], BITS == 4 ? mt : pos);
        if (BITS == 3) a[k] |= plane_pair(hp[k >> 1], pos, code_pos<BITS>(pos));
      }
      mma_f16(acc[mt], a, b0, b1);
    }
  }
  // rows g and g + 8 of m-tile mt: tokens 16 (g % 4) + 8 (g / 4) + mt and + 4
  if ((tq >> 1) == r) {
    float v[8];
#pragma unroll
    for (int mt = 0; mt < 4; ++mt) {
      constexpr float unit = kCodeUnit / (float)(1 << kColsTop);
      v[mt] = (acc[mt][0] + acc[mt][1]) * (code_unit<BITS>(mt) * unit) * kb;
      v[4 + mt] = (acc[mt][2] + acc[mt][3]) * (code_unit<BITS>(BITS == 4 ? mt : mt + 4) * unit) * kb;
    }
    float4* dst = reinterpret_cast<float4*>(ps + 64 * (tq & 1) + 16 * (g & 3) + 8 * (g >> 2));
    dst[0] = make_float4(v[0], v[1], v[2], v[3]);
    dst[1] = make_float4(v[4], v[5], v[6], v[7]);
  }
  __syncwarp();
  // tokens 2 lane, 2 lane + 1 are of group lane / 16, as is this lane's zk
  const float2 u0 = *reinterpret_cast<const float2*>(ps + 2 * lane);
  const float2 u1 = *reinterpret_cast<const float2*>(ps + 64 + 2 * lane);
  if (QC == 1) {
    x[0][0] = (u0.x + u1.x) + (zk + zo);
    x[0][1] = (u0.y + u1.y) + (zk + zo);
  } else {
    const float z0 = sel ? zo : zk, z1 = sel ? zk : zo;
    x[0][0] = u0.x + z0;
    x[0][1] = u0.y + z0;
    x[QC - 1][0] = u1.x + z1;
    x[QC - 1][1] = u1.y + z1;
  }
}

// KM: K_KIVI (quantized heads) or K_BF16 (image keys of keys-only heads).
template <int BITS, int QC, int KM, int MB>
__device__ __forceinline__ void run_item_cols(char* smem, const Seg& sg, int tb, int te, const DecodeParams& p,
                                              const uint4 (&qv)[QPieces<1>::n], float* parts) {
  using TL = Tile<BITS, KM, V_KIVI, MB, true>;
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(kFull, tid >> 5, 0);
  const int g = lane >> 2, tq = lane & 3;
  float* q_s = reinterpret_cast<float*>(smem + SmemLayout<1>::q);
  // scores and probabilities of the warp's tile, [2][64], behind the QC query rows
  static_assert((2 * kQRow + kWarps * 128) * 4 <= 8 * kQRow * 4, "the query rows above the first two hold the scores");
  float* ps = q_s + 2 * kQRow + warp * 128;
  WarpPipe<BITS, 1, KM, V_KIVI, MB, true, KM == K_KIVI ? kKiviGroup : 16> pipe(smem, warp, sg, p, tb, te);

  float* qn = reinterpret_cast<float*>(smem + SmemLayout<1>::qn);
  stage_queries<1, KM == K_BF16 ? -1 : 0>(q_s, qn, qv, tid);
  __syncthreads();
  float unit[QC];  // of the scores: the staged rows' and the softmax scale
#pragma unroll
  for (int q = 0; q < QC; ++q) unit[q] = (KM == K_BF16 ? 1.f : qn[q]) * p.scale_log2;
  uint32_t qb[1][8][2];
  if (KM == K_BF16) {
    qfrag_natural<1>(qb, q_s, g, tq);
    __syncthreads();  // rows 2.. hold the scores from here on
  }
  ColState<QC> ws;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int mt = 0; mt < 8; ++mt) ws.o[0][mt][i] = 0.f;
#pragma unroll
  for (int q = 0; q < QC; ++q) {
    ws.m[q] = -INFINITY;
    ws.l[q] = 0.f;
  }
  ws.z = 0.f;
  ws.vb = __uint_as_float(0x00800000u);  // 2^-126: no value scale seen yet
  ws.kb = kScaleLow;

#pragma unroll 1
  for (int it = 0; it < pipe.n_tiles; ++it) {
    if (!pipe.landed()) break;
    if (it == 0) pipe.fill_rest();
    const char* kst = pipe.slot();
    const char* vst = pipe.next_slot();
    const int nvalid = pipe.tile_tokens(it);  // whole slices: coded tokens come in groups of 32
    float x[QC][2];
    if constexpr (KM == K_KIVI) {
      cols_scores<BITS, QC, MB>(kst, kst + TL::km_off, q_s, ps, ws.kb, nvalid > kKiviGroup, lane, x);
    } else {
      const uint32_t rbase = smem_u32(kst) + ((lane & 7) + 8 * ((lane >> 3) & 1)) * 128;
      const int rsw = lane & 7, ch = lane >> 4;
      float acc[2][4];
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[0][i] = acc[1][i] = 0.f;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        uint32_t a[4];
        ldsm_x4(a, rbase + (j >> 2) * (TL::tokens * 128) + (((2 * (j & 3) + ch) ^ rsw) << 4));
        mma_bf16(acc[j & 1], a, qb[0][j][0], qb[0][j][1]);
      }
      if (tq == 0) {  // columns 0, 1: the queries
        ps[g] = acc[0][0] + acc[1][0];
        ps[g + 8] = acc[0][2] + acc[1][2];
        if (QC == 2) {
          ps[64 + g] = acc[0][1] + acc[1][1];
          ps[64 + g + 8] = acc[0][3] + acc[1][3];
        }
      }
      __syncwarp();
#pragma unroll
      for (int q = 0; q < QC; ++q) {
        const float2 u = *reinterpret_cast<const float2*>(ps + 64 * q + (2 * lane & 15));
        x[q][0] = u.x;
        x[q][1] = u.y;
      }
    }
    pipe.refill();
    const bool in = 2 * lane < nvalid;
#pragma unroll
    for (int q = 0; q < QC; ++q)
#pragma unroll
      for (int i = 0; i < 2; ++i) x[q][i] = in ? x[q][i] * unit[q] : -INFINITY;
    cols_softmax<QC>(ws, x, ps, lane);
    if (!pipe.landed()) break;

    const uint32_t* vc32 = reinterpret_cast<const uint32_t*>(vst);
    const char* vmp = vst + TL::vm_off;
#pragma unroll 1
    for (int t0 = 0; t0 < nvalid; t0 += 16) {
      const float4 pt = *reinterpret_cast<const float4*>(ps + (QC == 2 ? 64 * (g >> 2) : 0) + t0 + 4 * tq);
      const int t = t0 + tq;  // and t + 4, + 8, + 12
      float2 vm[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) vm[i] = meta_pair<MB>(vmp, (t + 4 * i) * 4 + (g & 3));
      const float smax = fmaxf(fmaxf(vm[0].x, vm[1].x), fmaxf(vm[2].x, vm[3].x));
      if (__any_sync(kFull, smax > ws.vb)) {
        const float nb = pow2_ceil(warp_max(smax));
        const float a = ws.vb * pow2_inv(nb);  // a power of two: exact
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int mt = 0; mt < 8; ++mt) ws.o[0][mt][i] *= a;
        ws.vb = nb;
      }
      const float inv = pow2_inv(ws.vb);
      uint32_t b[1][2];
      b[0][0] = pack_half2(pt.x * (vm[0].x * inv), pt.y * (vm[1].x * inv));
      b[0][1] = pack_half2(pt.z * (vm[2].x * inv), pt.w * (vm[3].x * inv));
      ws.z = fmaf(pt.x, vm[0].y, ws.z);
      ws.z = fmaf(pt.y, vm[1].y, ws.z);
      ws.z = fmaf(pt.z, vm[2].y, ws.z);
      ws.z = fmaf(pt.w, vm[3].y, ws.z);
      pv_codes<BITS, 1>(ws.o, vc32, t, t + 4, t + 8, t + 12, g, b);
    }
    pipe.refill();
  }
  pipe.drain(lane);
  __syncthreads();  // the warps' buffers are reused for the reduction below

  ws.z += __shfl_xor_sync(kFull, ws.z, 1);
  ws.z += __shfl_xor_sync(kFull, ws.z, 2);
#pragma unroll
  for (int q = 0; q < QC; ++q) {
    const float l = warp_sum(ws.l[q]);
    float* prow = parts + (warp * kMaxG + q) * kPartialStride;  // (m, l, -, -, o[128])
    if (lane == 0) {
      prow[0] = ws.m[q];
      prow[1] = l;
    }
    // rows g, g + 8 of m-tile mt: channels 16g + mt, 16g + 8 + mt, value group g / 2
    const int col = 4 * q + (g >> 1);
    const float z = __shfl_sync(kFull, ws.z, col << 2);
    if (tq == (col >> 1)) {
      float v[16];
#pragma unroll
      for (int mt = 0; mt < 8; ++mt) {
        const float f = code_unit<BITS>(BITS == 4 ? mt % 4 : mt) * kCodeUnit;
        v[mt] = fmaf(((col & 1) ? ws.o[0][mt][1] : ws.o[0][mt][0]) * f, ws.vb, z);
        v[8 + mt] = fmaf(((col & 1) ? ws.o[0][mt][3] : ws.o[0][mt][2]) * f, ws.vb, z);
      }
      float4* dst = reinterpret_cast<float4*>(prow + 4 + 16 * g);
#pragma unroll
      for (int i = 0; i < 4; ++i) dst[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    }
  }
}

// (layer in the launch, batch row, KV head, chunk of the head) of CTA x's item.
// Runs of items and, in a run, chunks, heads and rows are found by arithmetic
// on the launch parameters, the layer by a warp-wide comparison with the
// per-layer counts, the head by its rank among the layer's mask bits, so the
// order of items -- costliest first, dealt out over the SMs -- needs no table
// and holds for any number of items.
__device__ __forceinline__ void locate_item(const DecodeParams& p, int x, int& li, int& b, int& h, int& r) {
  const Dims& d = p.d;
  const int round = x / p.deal;
  int item = x;
  if ((round & 1) && (round + 1) * p.deal <= p.total_items) item = (2 * round + 1) * p.deal - 1 - x;
  int k = 0, start = 0;
  while (k + 1 < kWorkRuns && item >= p.run[k].end) start = p.run[k++].end;
  const int kind = p.run[k].kind;
  const int rows = p.run[k].heads * d.B;
  const int in_run = item - start;
  const int chunk = in_run / rows, in_chunk = in_run - chunk * rows;
  const int rank = in_chunk / d.B;  // of the (layer, head) among the run's
  b = in_chunk - rank * d.B;
  r = (kind == kWorkBf16 || kind == kWorkProtected) ? chunk : p.counts.nbU + chunk;
  // heads of this kind in the layers before layer l
  const bool all = kind == kWorkBf16 && d.keys_only, prot = kind == kWorkKeysOnly || kind == kWorkProtected;
  auto before = [&](int l) { return all ? l * d.H : (prot ? l * d.H - p.unprot_before[l] : p.unprot_before[l]); };
  li = 0;
  if (p.n_layers > 1) {
    const int l0 = threadIdx.x & 31, l1 = l0 + 32;
    const bool in0 = l0 < p.n_layers && before(l0) <= rank, in1 = l1 < p.n_layers && before(l1) <= rank;
    li = __popc(__ballot_sync(kFull, in0)) + __popc(__ballot_sync(kFull, in1)) - 1;
  }
  const int n = rank - before(li);
  const uint64_t mask = p.lt.mask[li];
  h = all ? n : nth_bit(prot ? mask : ~mask, n);
}

// Tokens in which the warps of a CTA divide a chunk of KIVI-style codes (run_item).
// Half groups keep the four warps' shares within 16 tokens of each other; the two
// warps that share a group both scale its queries.  In whole groups a chunk of 160
// tokens was 64, 64, 32 and none.  One layer or a few in one call: 9 rows of 5 KV
// heads, G = 12, 2,112 tokens at 4 bits 52.0 -> 49.7 us; 10 rows of 8, G = 8, 1,024
// tokens at 3 bits 58.7 -> 55.7 us; small launches up to 15% (11.8 -> 10.1 us), no
// change to -2% where the shares were even.  3-bit codes with four CTAs per SM, which
// are short of registers, stay with whole groups (44.5 us, 48.6 in halves).
template <int BITS, int NT, int QC>
__host__ __device__ constexpr int kivi_unit() { return BITS == 3 && NT == 1 && QC == 0 ? kKiviGroup : 16; }

// NT: 8-query column tiles of the MMAs.  QC: queries per KV head where
// run_item_cols serves the KIVI-style items (1 or 2), else 0; -1: the same with
// registers for three CTAs per SM instead of four.
template <int BITS, int NT, int BASE, int MB, int QC>
__global__ void __launch_bounds__(kThreads, NT == 1 ? (QC < 0 ? 3 : 4) : 2)
decode_kernel(const __grid_constant__ DecodeParams p) {
  extern __shared__ __align__(1024) char smem_raw[];
  // swizzled TMA boxes need 1024-byte aligned shared addresses
  char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const Dims& d = p.d;
  // Programmatic dependent launch: the next launch on the stream (the next
  // layer's or step's decode) may be scheduled as soon as every CTA of this
  // one runs; it builds its prologue from its parameters and waits (below)
  // before it touches memory that earlier kernels write.
  grid_launch_dependents();
  if ((int)blockIdx.x >= p.total_items) return;
  if (threadIdx.x == 0) {
    const uint32_t bars = smem_u32(smem + SmemLayout<NT>::bar);
    for (int s = 0; s < kMaxSlots * kWarps; ++s) mbar_init(bars + 8 * s, 1);
    mbar_init_fence();
    *reinterpret_cast<volatile int*>(smem + SmemLayout<NT>::bar + 8 * kMaxSlots * kWarps) = 0;  // abort flag
    prefetch_tensormap(&p.arena_map);
  }
  int li, b, h, r;
  locate_item(p, (int)blockIdx.x, li, b, h, r);
  const int G = d.G;
  const uint64_t mask = p.lt.mask[li];
  const int cls = head_class(d, mask, h);
  int nb;
  const int ni = head_chunks(cls, p.counts, &nb);
  const LayerGeom lg = layer_geom(d, mask);
  const HeadGeom hd = head_geom(d, lg, h);
  const char* Lb = p.arena + p.lt.base[li];
  // Everything above comes from the launch parameters.  From here on the CTA
  // reads the queries, the new K/V, the arena and the workspace, which the
  // kernels before this one on the stream write.
  grid_dependency_wait();
  // The queries are requested first: they gate every warp's first tile, and
  // their latency overlaps the first tile's copy.
  const uint16_t* qg = p.q + (((size_t)li * d.B + b) * d.Hq + (size_t)h * G) * kD;
  uint4 qv[QPieces<NT>::n];
#pragma unroll
  for (int k = 0; k < QPieces<NT>::n; ++k) {
    const int i = threadIdx.x + k * kThreads;
    qv[k] = (i < G * 16) ? ldg16(qg + i * 8) : make_uint4(0u, 0u, 0u, 0u);
  }
  const bool coded = r >= nb;
  int tb, te;
  if (!coded) {
    const int c = (cls == kProtected) ? p.plan.cbP : p.plan.cbU;
    tb = r * c;
    te = min(tb + c, hd.bf16_prefill + p.appended[li]);
  } else {
    const int c = (cls == kKeysOnly) ? p.plan.cqK : p.plan.cqU;
    tb = (r - nb) * c;
    te = min(tb + c, ncoded(d));
  }
  const int tid = threadIdx.x;

  // the warps' (m, l, o) partials [warp][16][132], in the stage buffer once the
  // tiles are consumed (the same row layout as the split partials)
  float* parts = reinterpret_cast<float*>(smem + kStageOff);
  Seg sg;
  sg.kc = sg.km = sg.vc = sg.vm = nullptr;
  sg.k_row0 = sg.v_row0 = 0;
  if (!coded) {
    sg.k_row0 = (int)((p.lt.base[li] + hd.kb + b * hd.kb_bs) >> 8);
    sg.v_row0 = (int)((p.lt.base[li] + hd.vb + b * hd.kb_bs) >> 8);
    const int pos = hd.bf16_prefill + p.appended[li] - 1;  // the step's new token
    if (p.k_new && pos >= tb && pos < te) {
      const size_t row = (((size_t)li * d.B + b) * d.H + h) * kD;
      // this CTA alone owns the position in this launch: store it in the
      // arena, ordered before the TMA reads of its tile
      if (threadIdx.x < 32) {
        const int c = threadIdx.x & 15;
        const char* src = reinterpret_cast<const char*>(((threadIdx.x < 16) ? p.k_new : p.v_new) + row);
        char* dst = const_cast<char*>(Lb) + ((threadIdx.x < 16) ? hd.kb : hd.vb) + b * hd.kb_bs + (size_t)pos * 256;
        *reinterpret_cast<uint4*>(dst + c * 16) = ldg16(src + c * 16);
        fence_proxy_async_global();
      }
    }
    __syncthreads();  // barriers initialised, new row stored
    run_item<BITS, NT, K_BF16, V_BF16, false, MB>(smem, sg, tb, te, p, qv, G, parts);
  } else if (hd.cls == kKeysOnly) {
    __syncthreads();  // barriers initialised
    sg.k_row0 = (int)((p.lt.base[li] + hd.kimg + b * hd.kimg_bs) >> 8);
    sg.vc = Lb + hd.vq + b * hd.vq_bs;
    sg.vm = Lb + hd.vqm + b * hd.vqm_bs;
    if constexpr (QC > 0)
      run_item_cols<BITS, QC, K_BF16, MB>(smem, sg, tb, te, p, qv, parts);
    else if constexpr (BASE == kKivi)
      run_item<BITS, NT, K_BF16, V_KIVI, false, MB>(smem, sg, tb, te, p, qv, G, parts);
    else
      run_item<BITS, NT, K_BF16, V_TOKEN, false, MB>(smem, sg, tb, te, p, qv, G, parts);
  } else {
    __syncthreads();  // barriers initialised
    sg.kc = Lb + hd.kq + b * hd.kq_bs;
    sg.km = Lb + hd.kqm + b * hd.kqm_bs;
    sg.vc = Lb + hd.vq + b * hd.vq_bs;
    sg.vm = Lb + hd.vqm + b * hd.vqm_bs;
    if constexpr (QC > 0)
      run_item_cols<BITS, QC, K_KIVI, MB>(smem, sg, tb, te, p, qv, parts);
    else if constexpr (BASE == kKivi)
      run_item<BITS, NT, K_KIVI, V_KIVI, false, MB, kivi_unit<BITS, NT, QC>()>(smem, sg, tb, te, p, qv, G, parts);
    else if constexpr (BASE == kAkvq)
      run_item<BITS, NT, K_TOKEN, V_TOKEN, true, MB>(smem, sg, tb, te, p, qv, G, parts);
    else
      run_item<BITS, NT, K_TOKEN, V_TOKEN, false, MB>(smem, sg, tb, te, p, qv, G, parts);
  }
  __syncthreads();

  // ---- combine the warps, then write the output (a head in one chunk) or this
  // split's partial; the last split of a head to finish then runs the same
  // combine over all splits' partials ----
  float* fw = reinterpret_cast<float*>(smem + SmemLayout<NT>::q);  // weights; queries no longer needed
  const size_t out_row = ((size_t)li * d.B + b) * d.Hq + (size_t)h * G;
  const size_t head_lin = ((size_t)li * d.B + b) * d.H + h;
  float* part = p.partials + (head_lin * p.max_items) * (size_t)G * kPartialStride;
  float* mine = part + (size_t)r * G * kPartialStride;
  __shared__ int s_last;
  const float* src = parts;
  int n = kWarps, sstride = kMaxG * kPartialStride;
  bool final = ni == 1;
#pragma unroll 1
  for (;;) {
    combine_pass<NT * 8>(src, n, sstride, fw, G, tid, final, p.out + out_row * kD, mine);
    if (final) break;

    // Publish the partial and take a ticket with one acquire-release atomic:
    // the CTA barrier orders every thread's stores before thread 0's release
    // (release is cumulative); for the last CTA, the acquire side orders the
    // other CTAs' partials before its reads (extended to its threads by the
    // second barrier).  No full device fence is needed.
    __syncthreads();
    if (tid == 0) {
      unsigned prev;
      asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;\n"
                   : "=r"(prev)
                   : "l"(p.counters + head_lin)
                   : "memory");
      s_last = (prev == (unsigned)(ni - 1));
    }
    __syncthreads();
    if (!s_last) return;

    // Last CTA of the head: all ni partials in one asynchronous sweep into the
    // stage buffer (the plan keeps them within it).
    const int bytes = ni * G * kPartialStride * 4;
    const uint32_t buf_u32 = smem_u32(smem + kStageOff);
    const char* psrc = reinterpret_cast<const char*>(part);
#pragma unroll 1
    for (int off = tid * 16; off < bytes; off += kThreads * 16) cp_async16(buf_u32 + off, psrc + off, 16);
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    src = reinterpret_cast<const float*>(smem + kStageOff);  // [ni][G][132]
    n = ni;
    sstride = G * kPartialStride;
    final = true;
  }
  if (ni > 1 && tid == 0) atomicExch(p.counters + head_lin, 0u);
}

template <int BITS, int NT, int BASE, int MB, int QC>
cudaError_t launch_t(const DecodeParams& p, cudaStream_t s) {
  // set once per device; host threads that race here both set the same
  // attributes, and the flags themselves are atomic
  static std::atomic<bool> configured[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64 || !configured[dev].load(std::memory_order_acquire)) {
    e = cudaFuncSetAttribute(decode_kernel<BITS, NT, BASE, MB, QC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             SmemLayout<NT>::bytes);
    if (e != cudaSuccess) return e;
    // four CTAs of 54 KB share an SM: ask for the full shared-memory carve-out
    e = cudaFuncSetAttribute(decode_kernel<BITS, NT, BASE, MB, QC>, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) configured[dev].store(true, std::memory_order_release);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)p.total_items, 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = SmemLayout<NT>::bytes;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, decode_kernel<BITS, NT, BASE, MB, QC>, p);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

template <int BITS, int NT, int MB>
cudaError_t launch_base(const DecodeParams& p, cudaStream_t s) {
  switch (p.d.base) {
    case kKivi:
      if constexpr (NT == 1) {
        if (p.d.G == 1) return launch_t<BITS, NT, kKivi, MB, 1>(p, s);
        if (p.d.G == 2) return launch_t<BITS, NT, kKivi, MB, 2>(p, s);
        // Four CTAs per SM leave the converting path short of registers (50 to 100
        // bytes of spills).  A launch of one wave or less is better off without
        // them, even if some of its CTAs have to wait (one layer, 8 KV heads: 2 rows
        // of 2,900 tokens at 4 bits 19 us, 23 with four; 4 rows of 8,200 at 2 bits 33
        // and 41); more waves want the fourth CTA (10 rows of 3,400 tokens: 48 us with
        // three, 45 with four; of 28 other launches of 1.2 to 7 waves 24 were 1 to 17%
        // faster with four, and four, three of them of 3-bit codes, 4 to 15% slower).
        if (p.total_items <= 4 * p.deal) return launch_t<BITS, NT, kKivi, MB, -1>(p, s);
      }
      return launch_t<BITS, NT, kKivi, MB, 0>(p, s);
    case kAkvq: return launch_t<BITS, NT, kAkvq, MB, 0>(p, s);
    default: return launch_t<BITS, NT, kMinMax, MB, 0>(p, s);
  }
}

// Every kernel shape for one metadata width (MB bytes per {scale, zero} pair).
template <int MB>
cudaError_t launch_decode_mb(const DecodeParams& p, cudaStream_t s) {
  if (p.d.bits == 2)
    return p.d.G <= 8 ? launch_base<2, 1, MB>(p, s) : launch_base<2, 2, MB>(p, s);
  if (p.d.bits == 3)
    return p.d.G <= 8 ? launch_base<3, 1, MB>(p, s) : launch_base<3, 2, MB>(p, s);
  return p.d.G <= 8 ? launch_base<4, 1, MB>(p, s) : launch_base<4, 2, MB>(p, s);
}

}  // namespace
}  // namespace hg
