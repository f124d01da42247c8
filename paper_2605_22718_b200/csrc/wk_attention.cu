// Memory attention (Section 4.2): the denoising chunk's queries attend, unmasked, over
// [dense segments ..., retrieved pool slots ...] of one layer.  O = softmax(scale Q K^T) V per head.
//
// Flash-style kernel on the 5th-generation tensor cores:
//   * a work unit is (head, 256 query rows = two 128-row Q tiles).  CTAs (one per SM) take whole units, which go straight to
//     bf16 output and share a head's K/V tiles through L2 because they walk the keys in step; the units of a last, partial
//     wave are cut into ranges over all SMs where that pays (split_default): a range writes a normalised fp32 partial plus
//     its log-sum-exp per piece, and combine_kernel merges them;
//   * K/V tiles (80 rows x 128 columns of one head, bf16; or 64 rows, see kFewTiles) are fetched by TMA straight from where they lie:
//     a dense segment (2-D tensor map per segment) or a pool slot (3-D tensor map [layer*slot][row][col]; the
//     slot id is read from device memory, so the retrieval result never visits the host).  Rows past the end
//     of a segment/slot are zero-filled by TMA and masked to -inf before the exponentials;
//   * S = Q K^T and O += P V are tcgen05.mma (M = 128, N = 80 and 128, K = 16 steps) with fp32 accumulators in tensor memory.
//     O0 and O1 take half of its 512 columns; 80 keys is the widest tile whose S (80 columns) and P (bf16: 40 columns, the A
//     operand of P V) lie side by side in the other half, so that S of the next tile can be multiplied while the softmax works
//     on this one, which it has read into registers.  (With 128 keys P has to overwrite S and the two take turns: 12 heads x
//     2,640 queries x 15,840 keys 261 us back to back instead of 249, although Q K^T alone runs at its full rate only from
//     N = 128 on: shared memory gives a Q K^T step of 80 keys (4 + 2.5 KB) in 52 clk, one of 128 (4 + 4 KB) in 64.)
//   * warp roles: warps 0-3 / 4-7 = softmax of Q tile 0 / 1 (one thread per row, fp32 in the exp2
//     domain, against a reference that follows the row's maximum: see kStreamSum), warps 8 / 9 = MMA issue for Q tile 0 / 1,
//     warp 10 = TMA producer.  The producer walks the tile list, and hands each tile's height to the others beside the tile;
//   * a tile with fewer valid rows (the last one of a segment or slot: 1,320 rows are 16 tiles and 40 rows) is
//     multiplied over ceil(nv / 16) * 16 rows.
// What bounds it: the chain of a step, at the clock that the board's 1,000 W cap leaves.  2,640 queries x 15,840 keys x 12 heads is one
// unit of 201 KV tiles on each of 132 SMs: 249 us.  A tile takes 1,869 clk in a CTA that runs alone (1,965 MHz) and 1,932 to 1,995
// beside 131 others (1,570 to 1,635 MHz); 1,432 of them the tensor pipe needs (measured with nothing else running), and S ->
// registers, exponentials, P -> P V, Q K^T of one Q tile is a chain of its own under the other's.  4,680 x 32,760 x 40: 2,740 us.
// Every wait is bounded; a wait that runs out sets WK_DEV_TIMEOUT, the CTA drains and frees its tensor memory.
#include <stddef.h>

#include "ptx_sm100.cuh"
#include "wk_internal.cuh"

namespace wk {
namespace {

using namespace ptx;

// The kernel is instantiated by the rows of its KV tiles, kKv: kTileKV and kTileKVFew, and kTileKVLse in LSE-only launches.
template <int kKv> constexpr bool is_lse = kKv == kTileKVLse;
// softmax warps, then the MMA warps, then the TMA warp.  LSE-only launches have a softmax warpgroup per S buffer.
template <int kKv> constexpr int kSoftWarps = is_lse<kKv> ? 16 : 8;
template <int kKv> constexpr int kMmaWarps = is_lse<kKv> ? 1 : 2;
template <int kKv> constexpr int kThreads = 32 * (kSoftWarps<kKv> + kMmaWarps<kKv> + 1);
template <int kKv> constexpr uint32_t kHalfKvBytes = kKv * 64 * 2;   // one TMA box: 64 columns
template <int kKv> constexpr uint32_t kKvBytes = 2 * kHalfKvBytes<kKv>;
constexpr uint32_t kHalfQBytes = kTileQ * 64 * 2, kQBytes = 2 * kHalfQBytes;
// A stage holds what one step of the MMA warp consumes: V of tile j and K of tile j + 2 (LSE-only launches: K alone).
constexpr int kStages = 4;
template <int kKv> constexpr uint32_t kStageBytes = (is_lse<kKv> ? 1 : 2) * kKvBytes<kKv>;
template <int kKv> constexpr size_t kSmemBytes = 1024 + 2 * kQBytes + kStages * kStageBytes<kKv>;   // align slack + Q0, Q1 + stages
constexpr int kNvRing = 16;   // tile heights handed from the TMA warp to the others; the TMA warp is at most kStages + 2 tiles ahead
// The softmax weighs a key with P = 2^(s * scale - m), where m is a maximum that the row has reached: rounded to bf16, the
// weight of the key that set it is exactly 1, so a dominating key returns its V row unchanged.  (Against a reference that is
// no maximum, say the largest of the first 32 logits, every weight is rounded: relative error of O 2.3e-3 instead of 2.1e-3 ..
// 1.7e-3 for logits with a standard deviation of 4 to 16.)  m moves when the maximum has left it by more than kRescaleThreshold.
// Taking the maximum first costs instructions and time before the first exponential.  A piece's first tile pays for it; other tiles
// are streamed on trust.  Their sum tells whether that was right: no weight above 2^8 hides in a sum of at most kStreamSum.  A warp
// in which a row's sum is larger still has S in registers, moves its references to the maximum where that is more than 2^8 above,
// and takes the exponentials again; tiles after that are read for the maximum first, twice as many each time.  12 heads x 2,640
// queries x 15,840 keys, back to back: 253.6 us with the maximum first for all, 248.5 this way.
constexpr float kRescaleThreshold = 8.0f;           // log2 units: P stays <= 2^8 between maximum updates
constexpr float kStreamSum = 256.0f;
// Pieces of at most kFewTiles tiles move the reference to every tile's own maximum, down as well as up: beside few other keys a
// tile's largest weight counts, and it is exact this way, as if the tile were a piece of its own.  450 queries x 5 heads x 1,040
// keys (three pieces of four or five tiles), relative error of O at deviations 1 / 2 / 4: 2.11 / 1.77 / 1.68e-3, without 2.30 / 2.23 / 2.09e-3.
// Calls of at most kFewTilesOfCall tiles of kTileKVFew rows walk them in such tiles, so that no more keys share a maximum.  So do calls
// whose segments and slots fill tiles of kTileKV rows badly: a tile of 64 takes 1,713 clk where one of 80 takes 1,919, by the clocks
// that the power cap leaves 6 to 7 for 7 to 8 (16,000 rows in slots of C, 12 heads x 2,640 queries, us in tiles of 80 / 64: C = 170 358 /
// 302, 190 329 / 272, 256 279 / 235, 512 264 / 257, 448 258 / 258, 384 251 / 260, 320 235 / 256; in tiles of 128 rows, which S and P
// of their own left no room for, 306, 280, 218, 253, 262, 248 and 264).
constexpr int kFewTiles = 10, kFewTilesOfCall = 8;
constexpr float kOwnSum = 1024.0f;
constexpr int kCost64 = 7, kCost80 = 8;
// tensor-memory columns: S0, P0, S1, P1 (80 + 40 of 128 each), O0, O1; LSE-only: S0, S1 twice
constexpr uint32_t kTmemS = 0, kTmemP = kTileKV, kTmemO = 256;
static_assert(kTileKV * 3 / 2 <= 128, "S and P of a Q tile share 128 columns");
constexpr int kPairRows = 2 * kTileQ;
constexpr int kMaxPieces = 32;                      // most ranges one unit may be cut into

struct AttnParams {
  CUtensorMap tm_q;
  CUtensorMap tm_kpool, tm_vpool;
  CUtensorMap tm_kd[kMaxDenseSegs], tm_vd[kMaxDenseSegs];
  int seg_tile_prefix[kMaxDenseSegs + 1];
  int seg_rows[kMaxDenseSegs];
  int n_segs, n_dense_tiles;
  const int32_t* slots;
  const int32_t* valid;
  int n_slots, pool_slots, layer, C, tiles_per_slot;
  int tile_rows;    // rows from one KV tile to the next
  int n_tiles, n_qpairs, n_units;
  int n_full, n_ranges;
  int lq, H;
  int slot_units;   // 1: every listed slot is a problem of its own: unit = (slot ordinal, head, q-pair), n_tiles =
                    //    tiles_per_slot, lse laid out [slot ordinal][H][lq]; stale slots give -inf and are not reported (LSE-only launches)
  float scale_log2;
  __nv_bfloat16* O;
  float* lse;
  float4* opart;    // [2 * n_ranges][32 groups of 4 columns][256 rows] fp32: a warp's 32 rows are one contiguous store
  float* lsepart;   // [2 * n_ranges][256]
  uint32_t* status;
};

// Work distribution.  Units 0 .. n_full - 1 are done whole, unit u by CTA u % gridDim.x; the tiles of the remaining units
// are numbered through and cut into n_ranges equal ranges, range c done by CTA c.
__host__ __device__ __forceinline__ int64_t range_start(int64_t tail_tiles, int n_ranges, int c) {
  return static_cast<int64_t>(c) * tail_tiles / n_ranges;
}

struct TileInfo {
  int seg;    // >= 0: dense segment index; -1: pool
  int row0;
  int z;
  int nv;     // valid rows (> 0)
};

// Walks the effective KV tiles of [tb, te): dense segments first, then pool slots; stale or -1 slots are skipped.
// Two levels, so that stepping to the next tile of the same segment touches no memory: (segment, tile in segment).
struct TileIter {
  int t, te;       // flat tile position, end of the range
  int seg;         // dense segment index, or n_segs + index into the slot list
  int r, n_r;      // tile inside the current segment / slot, and how many it has
  int tail;        // valid rows of its last tile
  int z;           // pool matrix index (layer * pool_slots + slot)
  bool ok;         // false for a stale or -1 slot
  bool entered;    // n_r, tail, z and ok are those of seg
  __device__ __forceinline__ void enter(const AttnParams& p, bool report) {
    if (seg < p.n_segs) {
      n_r = p.seg_tile_prefix[seg + 1] - p.seg_tile_prefix[seg];
      tail = p.seg_rows[seg] - (n_r - 1) * p.tile_rows;
      z = 0;
      ok = true;
    } else {
      n_r = p.tiles_per_slot;
      tail = p.C - (n_r - 1) * p.tile_rows;
      const int si = seg - p.n_segs;
      ok = false;
      z = 0;
      if (si < p.n_slots) {
        const int slot = ld_dep(p.slots + si);
        ok = slot >= 0 && slot < p.pool_slots;
        if (ok) ok = ld_dep(p.valid + slot) != 0;
        if (!ok && report && slot != -1) atomicOr(p.status, WK_DEV_BAD_SLOT);   // never dereferenced
        if (ok) z = p.layer * p.pool_slots + slot;
      }
    }
  }
  // Where the walk starts, from the launch's parameters alone (the slot list may be the work of the kernel before).
  __device__ __forceinline__ void init(const AttnParams& p, int tb, int te_) {
    t = tb;
    te = te_;
    if (tb < p.n_dense_tiles) {
      seg = 0;
      while (seg + 1 < p.n_segs && tb >= p.seg_tile_prefix[seg + 1]) ++seg;
      r = tb - p.seg_tile_prefix[seg];
    } else {
      const int u = tb - p.n_dense_tiles;
      const int si = u / p.tiles_per_slot;
      seg = p.n_segs + si;
      r = u - si * p.tiles_per_slot;
    }
    entered = false;
  }
  __device__ __forceinline__ void open(const AttnParams& p, bool report) {   // looks the first segment or slot up
    if (!entered && t < te) enter(p, report);
    entered = true;
  }
  __device__ __forceinline__ bool next(const AttnParams& p, TileInfo& ti, bool report) {
    while (t < te) {
      if (!entered) {
        enter(p, report);
        entered = true;
      }
      if (r == n_r) {   // first tile of the next segment / slot
        ++seg;
        r = 0;
        entered = false;
        continue;
      }
      ti.seg = seg < p.n_segs ? seg : -1;
      ti.row0 = r * p.tile_rows;
      ti.z = z;
      ti.nv = (r == n_r - 1) ? tail : p.tile_rows;
      ++r;
      ++t;
      if (ok) return true;
    }
    return false;
  }
};

// Number of effective tiles in [tb, te), by a whole warp: the lanes look at the slot list side by side.
__device__ __forceinline__ int count_tiles(const AttnParams& p, int tb, int te) {
  const int dense = max(0, min(te, p.n_dense_tiles) - tb);
  const int ub = max(tb, p.n_dense_tiles) - p.n_dense_tiles, ue = te - p.n_dense_tiles;
  int n = 0;
  if (ue > ub) {
    const int last = (ue - 1) / p.tiles_per_slot;
    for (int si = ub / p.tiles_per_slot + static_cast<int>(threadIdx.x & 31); si <= last; si += 32) {
      const int slot = ld_dep(p.slots + si);
      if (slot >= 0 && slot < p.pool_slots && ld_dep(p.valid + slot) != 0)
        n += min(ue, (si + 1) * p.tiles_per_slot) - max(ub, si * p.tiles_per_slot);
    }
    n = __reduce_add_sync(0xffffffffu, n);
  }
  return dense + n;
}

struct __align__(8) Barriers {
  uint64_t q_full, q_empty;
  uint64_t kv_full[kStages], kv_empty[kStages];
  uint64_t s_full[4], p_full[4], turn[2], o_done[2], o_free[2], m_full[2], m_empty[2];   // index of s_full, p_full: Q tile + 2 x S buffer (LSE-only)
};

// Bounded wait that also gives up when another role has already aborted; false then.  A loop of eight instructions and
// nothing else: what follows a failed wait (the status bit, the abort flag) stands once per role, at its end (leave_role).
__device__ __forceinline__ bool wait_or_abort(uint64_t* bar, uint32_t parity, volatile uint32_t* abort_flag) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .u32 n, a;\n\t"
      "mov.u32 n, 0;\n"
      "WAIT_LOOP:\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "@p bra WAIT_DONE;\n\t"
      "ld.volatile.shared.u32 a, [%3];\n\t"
      "setp.ne.u32 q, a, 0;\n\t"
      "@q bra WAIT_DONE;\n\t"
      "add.u32 n, n, 1;\n\t"
      "setp.lt.u32 q, n, %4;\n\t"
      "@q bra WAIT_LOOP;\n"
      "WAIT_DONE:\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(smem_u32(const_cast<uint32_t*>(abort_flag))), "n"(WK_WAIT_CAP)
      : "memory");
  return ok != 0;
}
// A role that has given up tells the others and sets the status bit (unless it left because another role did).
__device__ __forceinline__ void leave_role(bool ok, volatile uint32_t* abort_flag, uint32_t* status) {
  if (!ok && *abort_flag == 0) {
    *abort_flag = 1;
    atomicOr(status, WK_DEV_TIMEOUT);
  }
}

__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ float fmax3_nan(float a, float b, float c) {   // NaN if any is
  float d;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// 2^x of a pair.  The exponentials bound LSE-only launches (16 per clock and SM on the special-function unit: 2,048 clk per tile of 128
// keys), so a share of the pairs takes 2^x from the FMA pipe instead (2,640 queries x 12 heads x 250 slots of 1,320 rows: 3,563 / 3,487 /
// 3,434 / 3,493 / 3,725 us at 0 ... 4 of 8): x = n + f with n = round(x) by the add-a-large-constant trick, 2^f on [-1/2, 1/2] by a cubic
// (relative error 7.7e-5), 2^n by adding n to the exponent field; all in packed fp32 pairs.  That path clamps at x = -120 (a weight of
// 1e-36), needs x < 127, and drops NaN: the caller looks for it in the logits (big).
template <bool kPoly>
__device__ __forceinline__ void exp2_pair(uint64_t e, float& p0, float& p1) {
  float e0, e1;
  unpack_f32x2(e, e0, e1);
  if (kPoly) {
    const uint64_t magic2 = pack_f32x2(12582912.f, 12582912.f), nmagic2 = pack_f32x2(-12582912.f, -12582912.f);
    const uint64_t mone2 = pack_f32x2(-1.f, -1.f);
    const uint64_t c0 = pack_f32x2(0.9999289512634277f, 0.9999289512634277f);
    const uint64_t c1 = pack_f32x2(0.6932762265205383f, 0.6932762265205383f);
    const uint64_t c2 = pack_f32x2(0.242604061961174f, 0.242604061961174f);
    const uint64_t c3 = pack_f32x2(0.055088773369789124f, 0.055088773369789124f);
    const uint64_t x = pack_f32x2(fmaxf(e0, -120.f), fmaxf(e1, -120.f));
    const uint64_t t = add_f32x2(x, magic2);                  // low mantissa bits = round(x)
    const uint64_t f = fma_f32x2(add_f32x2(t, nmagic2), mone2, x);   // x - round(x), in [-1/2, 1/2]
    uint64_t y = fma_f32x2(c3, f, c2);
    y = fma_f32x2(y, f, c1);
    y = fma_f32x2(y, f, c0);
    float t0, t1, y0, y1;
    unpack_f32x2(t, t0, t1);
    unpack_f32x2(y, y0, y1);
    p0 = __uint_as_float(__float_as_uint(y0) + (__float_as_uint(t0) << 23));
    p1 = __uint_as_float(__float_as_uint(y1) + (__float_as_uint(t1) << 23));
  } else {
    p0 = ex2_approx(e0);
    p1 = ex2_approx(e1);
  }
}
__device__ __forceinline__ float sum4_f32x2(const uint64_t (&acc)[4]) {
  float a, b;
  unpack_f32x2(add_f32x2(add_f32x2(acc[0], acc[1]), add_f32x2(acc[2], acc[3])), a, b);
  return a + b;
}

constexpr int kLsePoly = 2;
// Sum of 2^(s * scale - m) over 32 columns of a row, in four independent (lo, hi) accumulators.  kLsePoly of every 8 pairs take
// the FMA pipe; big = the largest of their raw values, or NaN (the caller checks that they stay below that path's limit).
__device__ __forceinline__ void exp_chunk(uint32_t (&r)[32], int rem, uint64_t scale2, uint64_t neg_m2, uint64_t (&acc)[4],
                                          float& big) {
  if (rem < 32) {   // columns past the end of the segment or slot
#pragma unroll
    for (int i = 0; i < 32; ++i) r[i] = i < rem ? r[i] : 0xff800000u;
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const float s0 = __uint_as_float(r[2 * i]), s1 = __uint_as_float(r[2 * i + 1]);
    const uint64_t e = fma_f32x2(pack_f32x2(s0, s1), scale2, neg_m2);
    float p0, p1;
    if ((i & 7) < kLsePoly) {
      exp2_pair<true>(e, p0, p1);
      big = fmax3_nan(big, s0, s1);
    } else {
      exp2_pair<false>(e, p0, p1);
    }
    acc[i & 3] = add_f32x2(acc[i & 3], pack_f32x2(p0, p1));
  }
}
// The largest of a row's first nv columns of S in tensor memory.
__device__ __forceinline__ float row_max_tmem(uint32_t tS, int nv) {
  float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll 1
  for (int c = 0; c < nv; c += 32) {
    uint32_t r[32];
    tmem_ld_x32(tS + c, r);
    tc_wait_ld(r);
    if (nv - c < 32) {
#pragma unroll
      for (int i = 0; i < 32; ++i)
        if (c + i >= nv) r[i] = 0xff800000u;
    }
#pragma unroll
    for (int i = 0; i < 32; i += 2) mx[(i >> 1) & 1] = fmax3(mx[(i >> 1) & 1], __uint_as_float(r[i]), __uint_as_float(r[i + 1]));
  }
  return fmaxf(mx[0], mx[1]);
}
// S of a tile, a row per thread, into registers.
template <int kKv>
__device__ __forceinline__ void tmem_ld_tile(uint32_t tS, uint32_t (&r)[kKv]) {
  static_assert(kKv == 64 || kKv == 80, "loads of 32 + 32 (+ 16) columns");
  tmem_ld_x32(tS, *reinterpret_cast<uint32_t(*)[32]>(&r[0]));
  tmem_ld_x32(tS + 32, *reinterpret_cast<uint32_t(*)[32]>(&r[32]));
  if constexpr (kKv == 80) tmem_ld_x16(tS + 64, *reinterpret_cast<uint32_t(*)[16]>(&r[64]));
}
template <int kKv>
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&r)[kKv]) {
  tc_wait_ld(*reinterpret_cast<uint32_t(*)[32]>(&r[0]));
  pin_x32(*reinterpret_cast<uint32_t(*)[32]>(&r[32]));
  if constexpr (kKv == 80) pin_x16(*reinterpret_cast<uint32_t(*)[16]>(&r[64]));
}
template <int kHalf>
__device__ __forceinline__ void tmem_st_half_tile(uint32_t tP, const uint32_t (&p)[kHalf]) {
  tmem_st_x32(tP, *reinterpret_cast<const uint32_t(*)[32]>(&p[0]));
  if constexpr (kHalf == 40) tmem_st_x8(tP + 32, *reinterpret_cast<const uint32_t(*)[8]>(&p[32]));
}
template <int kKv>
__device__ __forceinline__ float row_max(const uint32_t (&r)[kKv]) {
  float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
  for (int i = 0; i < kKv; i += 2) mx[(i >> 1) & 3] = fmax3(mx[(i >> 1) & 3], __uint_as_float(r[i]), __uint_as_float(r[i + 1]));
  return fmax3(fmaxf(mx[0], mx[1]), mx[2], mx[3]);
}
// P = 2^(s * scale - m) of a row, as bf16 pairs, and their sum.  (All exponentials on the special-function unit: a share of cubics as in
// exp_chunk costs time, 12 heads x 2,640 queries x 15,840 keys 253.3 us with one pair in eight and 248.8 without, and leaves the
// log-sum-exp of segments of 100 keys within 1e-5 instead of 9e-7.)
template <int kKv>
__device__ __forceinline__ float exp_tile(const uint32_t (&r)[kKv], uint64_t scale2, float m, uint32_t (&pk)[kKv / 2]) {
  const uint64_t neg_m2 = pack_f32x2(-m, -m);
  uint64_t acc[4] = {0, 0, 0, 0};
#pragma unroll
  for (int i = 0; i < kKv / 2; ++i) {
    const uint64_t e = fma_f32x2(pack_f32x2(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1])), scale2, neg_m2);
    float e0, e1;
    unpack_f32x2(e, e0, e1);
    const float p0 = ex2_approx(e0), p1 = ex2_approx(e1);
    acc[i & 3] = add_f32x2(acc[i & 3], pack_f32x2(p0, p1));
    pk[i] = pack_bf16x2(p0, p1);
  }
  return sum4_f32x2(acc);
}

// One piece of work: unit u, KV tiles [tb, te), and where its result goes.
struct Piece {
  int h, q0, tb, te, slot;   // slot < 0: the piece covers the whole unit -> direct output
  int ord;                   // slot ordinal the unit belongs to (0 unless every slot is its own problem)
  bool has_q1;
};
struct PieceWalker {
  int full;            // next whole unit
  int u, tb;           // next unit of this CTA's range and the first tile in it
  int u_last, tb_last; // a range that starts inside a unit does that unit's piece last: by then the other CTAs are about
  int len_last;        // as far into the keys, so that CTAs of a head go on sharing its tiles through L2
  int64_t left;        // tiles of the range not handed out yet (the postponed piece not counted)
  __device__ __forceinline__ void init(const AttnParams& p) {
    full = blockIdx.x;
    left = 0;
    len_last = 0;
    if (p.n_full == p.n_units || blockIdx.x >= p.n_ranges) return;
    const int64_t tail = static_cast<int64_t>(p.n_units - p.n_full) * p.n_tiles;
    const int64_t start = range_start(tail, p.n_ranges, blockIdx.x);
    left = range_start(tail, p.n_ranges, blockIdx.x + 1) - start;
    const int ur = static_cast<int>(start / p.n_tiles);
    u = p.n_full + ur;
    tb = static_cast<int>(start - static_cast<int64_t>(ur) * p.n_tiles);
    if (tb > 0) {
      u_last = u++;
      tb_last = tb;
      len_last = static_cast<int>(min(left, static_cast<int64_t>(p.n_tiles - tb)));
      left -= len_last;
      tb = 0;
    }
  }
  __device__ __forceinline__ bool next(const AttnParams& p, Piece& pc) {
    int v;
    if (full < p.n_full) {
      v = full;
      full += gridDim.x;
      pc.tb = 0;
      pc.te = p.n_tiles;
      pc.slot = -1;
    } else if (left > 0) {
      v = u++;
      pc.tb = 0;
      pc.te = static_cast<int>(min(left, static_cast<int64_t>(p.n_tiles)));
      left -= pc.te;
      // partial results: slot 2 c for the piece that range c starts with, 2 c + 1 for the one it ends with
      pc.slot = pc.te == p.n_tiles ? -1 : 2 * static_cast<int>(blockIdx.x) + (tb_first(p, v) ? 0 : 1);
    } else if (len_last > 0) {
      v = u_last;
      pc.tb = tb_last;
      pc.te = tb_last + len_last;
      len_last = 0;
      pc.slot = 2 * static_cast<int>(blockIdx.x);
    } else {
      return false;
    }
    pc.ord = 0;
    if (p.slot_units) {   // the unit's tiles are those of one slot: shift the range into that slot's part of the tile space
      const int base = p.H * p.n_qpairs;
      pc.ord = v / base;
      v -= pc.ord * base;
      pc.tb += pc.ord * p.tiles_per_slot;
      pc.te += pc.ord * p.tiles_per_slot;
    }
    pc.h = v / p.n_qpairs;
    pc.q0 = (v - pc.h * p.n_qpairs) * kPairRows;
    pc.has_q1 = pc.q0 + kTileQ < p.lq;
    return true;
  }
  // is unit v, entered at its first tile, the start of this CTA's range?
  __device__ __forceinline__ bool tb_first(const AttnParams& p, int v) const {
    const int64_t tail = static_cast<int64_t>(p.n_units - p.n_full) * p.n_tiles;
    return range_start(tail, p.n_ranges, blockIdx.x) == static_cast<int64_t>(v - p.n_full) * p.n_tiles;
  }
};

// kKv = kTileKVLse is the LSE-only instantiation (query-based retrieval): no V, no P, no O.  S has two buffers per Q tile and a
// softmax warpgroup per buffer, so the tensor pipe works ahead of the softmax, which bounds it (issue and special-function
// unit) until the board's power cap does.  2,640 queries x 12 heads x 250 slots of 1,320 rows: two warpgroups and one buffer
// per Q tile on 132 SMs 4,070 us; all SMs, two buffers, streamed sums 3,540; four warpgroups 3,070 (2,136 clk per KV tile).
// What the roles of a CTA share besides the tiles.
template <int kKv>
struct CtaShared {
  Barriers bars;
  uint32_t tmem;
  volatile uint32_t abort;
  float2 merge[is_lse<kKv> ? 2 : 1][is_lse<kKv> ? 128 : 1];   // (reference, sum) of a Q tile's odd KV tiles
  volatile int nv[kNvRing];   // valid rows of tile number t (counted over the CTA's pieces) at t % kNvRing
};

// Issues the MMAs of a CTA's tiles.  The whole warp runs the control flow and one lane's predicate issues (see mma_ss_if).
template <int kKv>
struct Mma {
  uint32_t one, bar0;
  uint64_t q_desc, k_desc, v_desc;   // descriptors of the tile bases; a K = 16 step advances the low word by a constant
  __device__ __forceinline__ Mma(uint32_t smem_base, const Barriers& bars) {
    one = elect_one() ? 1u : 0u;
    bar0 = smem_u32(&bars);
    constexpr uint64_t hi = static_cast<uint64_t>(smem_desc_hi_sw128(1024)) << 32;
    q_desc = hi | smem_desc_lo(smem_base, 16);
    k_desc = hi | smem_desc_lo(smem_base + 2 * kQBytes, 16);
    v_desc = hi | smem_desc_lo(smem_base + 2 * kQBytes + kKvBytes<kKv>, kHalfKvBytes<kKv>);
  }
  __device__ __forceinline__ void commit(size_t offset) const { mma_commit_if(one, bar0 + static_cast<uint32_t>(offset)); }
  // S = Q K^T over the first nv rows of the K tile: ceil(nv / 16) * 16 columns.  (A branch that gives full tiles a constant
  // descriptor costs more than it saves: LSE-only launches 3,413 us instead of 3,361.)
  // qt: Q tile in shared memory, d: S columns
  __device__ __forceinline__ void s(uint32_t qt, uint32_t d, uint32_t st, int nv) const {
    const uint32_t idesc = idesc_bf16_f32(128, 0, 0, 0) | (static_cast<uint32_t>((nv + 15) >> 4) << 18);
    const uint64_t a = q_desc + qt * (kQBytes >> 4), b = k_desc + st * (kStageBytes<kKv> >> 4);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const uint32_t in_row = (k & 3) * 2;   // 32 bytes per step inside a 128-byte row
      mma_ss_if(one, d, a + (k >> 2) * (kHalfQBytes >> 4) + in_row, b + (k >> 2) * (kHalfKvBytes<kKv> >> 4) + in_row, idesc, k > 0);
    }
  }
  // O_i (+)= P_i V: A = P from tensor memory (bf16 pairs, 8 columns per K = 16 step); B = V, rows = K dimension,
  // MN-major: 16 rows of 128 bytes = 2048 bytes per step
  __device__ __forceinline__ void pv(uint32_t i, uint32_t st, int nv, uint32_t accumulate) const {
    constexpr uint32_t idesc = idesc_bf16_f32(128, 128, 0, 1);
    const uint64_t b = v_desc + st * (kStageBytes<kKv> >> 4);
#pragma unroll 1
    for (int k = 0; k < (nv + 15) >> 4; ++k)
      mma_ts_if(one, kTmemO + i * 128, kTmemP + i * 128 + k * 8, b + k * 128, idesc, k > 0 ? 1u : accumulate);
  }
};

// MMA warp of Q tile kQt.  Two warps issue because a commit holds its warp until the tensor pipe has nearly caught up, and the
// waits behind it would leave the pipe idle: while one warp is held, the other has waited already and goes on.  They take turns
// (turn[]), step by step: the pipe runs a group of MMAs that accumulate into one tile slower when another tile's come between them.
template <int kKv, int kQt>
__device__ __forceinline__ void mma_role(const AttnParams& p, CtaShared<kKv>& sh, uint32_t smem_base) {
  Barriers& bars = sh.bars;
  const int lane = threadIdx.x & 31;
  const Mma<kKv> mma(smem_base, bars);
  PieceWalker walk;
  walk.init(p);
  Piece pc;
  uint32_t st = 0, ph = 0;       // stage and its parity
  uint32_t p_ph = 0;             // parity of p_full
  uint32_t n = 0, t = 0, e = 0;  // pieces, tiles, pieces with output of this Q tile so far
  uint32_t k = 0;                // steps that both Q tiles took part in so far
  bool ok = true, more = walk.next(p, pc);
  dep_wait();
  for (; ok && more; more = walk.next(p, pc)) {
    const int n_eff = count_tiles(p, pc.tb, pc.te);
    const bool both = pc.has_q1, mine = kQt == 0 || both;
    if (!(ok = wait_or_abort(&bars.q_full, n & 1, &sh.abort))) break;
    ++n;
    if (n_eff == 0) {
      if (lane == 0) mbar_arrive(&bars.q_empty);
      continue;
    }
    // Step j: once P of tile j - 2 is in tensor memory and S of tile j - 1 in registers (p_full), P V of the one and Q K^T of
    // tile j.  The softmax of tile j - 1 runs meanwhile; it stores its P when this step's commit arrives.
    if (!mine) {
      // Nothing else in this piece waits for this warp, so Q is given back by it too: otherwise q_full could complete twice before
      // it looks, and a parity wait cannot tell phase n from phase n + 2.
      if (lane == 0) mbar_arrive(&bars.q_empty);
      const uint32_t used = st + (n_eff == 1 ? 2 : n_eff + 2);
      ph ^= (used / kStages) & 1;
      st = used % kStages;
      t += n_eff;
      continue;
    }
    int nv = 0, nv_1 = 0, nv_2 = 0;   // valid rows of tiles j, j - 1, j - 2
    for (int j = 0; j < n_eff + 2; ++j, nv_2 = nv_1, nv_1 = nv) {
      nv = 0;
      if (j == 1 && n_eff == 1) continue;      // a piece of one tile has nothing to multiply in its second step
      if (!(ok = wait_or_abort(&bars.kv_full[st], ph, &sh.abort))) break;
      if (j < n_eff) nv = sh.nv[t++ % kNvRing];
      if (j > 0) {
        ok = wait_or_abort(&bars.p_full[kQt], p_ph, &sh.abort);
        p_ph ^= 1;
        // A piece's first P V overwrites O: the epilogue of the last piece that used it must have read it.  o_free
        // completes once per piece in which the warpgroup ran an epilogue, so neither side can run two phases ahead of
        // the other (a parity wait cannot tell phase n from phase n + 2).
        if (j == 2 && e++ > 0) ok = ok && wait_or_abort(&bars.o_free[kQt], e & 1, &sh.abort);
      }
      if (both && (kQt == 1 || k > 0)) ok = ok && wait_or_abort(&bars.turn[kQt], (kQt == 1 ? k : k + 1) & 1, &sh.abort);
      if (!ok) break;
      tc_fence_after();
      if (j >= 2) mma.pv(kQt, st, nv_2, j > 2);
      if (nv > 0) mma.s(kQt, kTmemS + kQt * 128, st, nv);
      if (both) {
        ++k;
        if (mma.one) mbar_arrive(&bars.turn[kQt ^ 1]);
      }
      mma.commit((j == n_eff + 1 ? offsetof(Barriers, o_done) : offsetof(Barriers, s_full)) + 8 * kQt);
      if (++st == kStages) { st = 0; ph ^= 1; }
    }
  }
  if (lane == 0) leave_role(ok, &sh.abort, p.status);
}

// LSE-only: two S buffers per Q tile, no P V; p_full says that a buffer has been read.
__device__ __forceinline__ void mma_lse_role(const AttnParams& p, CtaShared<kTileKVLse>& sh, uint32_t smem_base) {
  Barriers& bars = sh.bars;
  const int lane = threadIdx.x & 31;
  const Mma<kTileKVLse> mma(smem_base, bars);
  PieceWalker walk;
  walk.init(p);
  Piece pc;
  uint32_t st = 0, ph = 0;   // stage and its parity
  uint32_t n = 0, t = 0;     // pieces and tiles so far
  uint32_t s0 = 0, s1 = 0;   // products of Q tile 0 / 1 so far
  bool ok = true, more = walk.next(p, pc);
  for (; ok && more; more = walk.next(p, pc)) {
    const int n_eff = count_tiles(p, pc.tb, pc.te);
    if (!(ok = wait_or_abort(&bars.q_full, n & 1, &sh.abort))) break;
    ++n;
    if (n_eff == 0) {
      if (lane == 0) mbar_arrive(&bars.q_empty);
      continue;
    }
    for (int j = 0; j < n_eff; ++j) {
      if (!(ok = wait_or_abort(&bars.kv_full[st], ph, &sh.abort))) break;
      const int nv = sh.nv[t++ % kNvRing];
      const uint32_t b0 = s0 & 1, b1 = s1 & 1;
      auto issue = [&](uint32_t qt, uint32_t d) {
        tc_fence_after();
        mma.s(qt, d, st, nv);
      };
      if (s0 >= 2 && !(ok = wait_or_abort(&bars.p_full[2 * b0], ((s0 >> 1) & 1) ^ 1, &sh.abort))) break;
      ++s0;
      issue(0, b0 * 256);
      mma.commit(offsetof(Barriers, s_full) + 16 * b0);
      if (pc.has_q1) {
        if (s1 >= 2 && !(ok = wait_or_abort(&bars.p_full[2 * b1 + 1], ((s1 >> 1) & 1) ^ 1, &sh.abort))) break;
        ++s1;
        issue(1, b1 * 256 + 128);
        mma.commit(offsetof(Barriers, s_full) + 16 * b1 + 8);
      }
      if (++st == kStages) { st = 0; ph ^= 1; }
    }
  }
  if (lane == 0) leave_role(ok, &sh.abort, p.status);
}

// All of a CTA's work.
template <int kKv>
__device__ __forceinline__ void attention_roles(const AttnParams& p, CtaShared<kKv>& sh, uint8_t* smem) {
  constexpr bool kLse = is_lse<kKv>;
  const uint32_t smem_base = smem_u32(smem);
  uint8_t* sQ = smem;                 // [2 q tiles][2 halves][128 rows][128 B]
  uint8_t* sKV = sQ + 2 * kQBytes;    // [stages][K, V][2 halves][rows][128 B]; LSE-only: [stages][K]
  Barriers& bars = sh.bars;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == kSoftWarps<kKv> + kMmaWarps<kKv>) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      PieceWalker walk;
      walk.init(p);
      Piece pc;
      TileIter it;
      uint32_t st = 0, ph = 1, steps = 0, n = 0, t = 0;   // stage, its parity, stages and Q pairs armed so far, tiles so far
      bool ok = true, more = walk.next(p, pc);
      TileInfo ti, t1, t2;   // this tile and the two before it
      bool have = false;
      if (more) it.init(p, pc.tb, pc.te);
      const bool early = more && pc.tb < p.n_dense_tiles;   // the first tile is known without the slot list
      if (early) have = it.next(p, ti, false);
      if (!kLse) dep_wait();
      const bool report = !p.slot_units;
      for (; ok && more; more = walk.next(p, pc)) {
        if (n > 0) {   // the first slot is looked up under the wait for Q; the first piece has no such wait, and its Q goes first
          it.init(p, pc.tb, pc.te);
          it.open(p, report);
        }
        if (!(ok = wait_or_abort(&bars.q_empty, (n & 1) ^ 1, &sh.abort))) break;
        mbar_expect_tx(&bars.q_full, 2 * kQBytes);
        ++n;
        for (int i = 0; i < 2; ++i)
          for (int half = 0; half < 2; ++half)
            tma_load_2d(sQ + i * kQBytes + half * kHalfQBytes, &p.tm_q, &bars.q_full,
                        pc.h * kHeadDim + half * 64, pc.q0 + i * kTileQ);
        const int x = pc.h * kHeadDim;
        auto load = [&](uint8_t* dst, const TileInfo& ti, const CUtensorMap* seg_maps, const CUtensorMap* pool_map) {
          if (ti.seg >= 0) {
            tma_load_2d(dst, seg_maps + ti.seg, &bars.kv_full[st], x, ti.row0);
            tma_load_2d(dst + kHalfKvBytes<kKv>, seg_maps + ti.seg, &bars.kv_full[st], x + 64, ti.row0);
          } else {
            tma_load_3d(dst, pool_map, &bars.kv_full[st], x, ti.row0, ti.z);
            tma_load_3d(dst + kHalfKvBytes<kKv>, pool_map, &bars.kv_full[st], x + 64, ti.row0, ti.z);
          }
        };
        bool have1 = false, have2 = false;
        if (n > 1 || !early) have = it.next(p, ti, report);
        while (have || have1 || have2) {   // step: K of this tile, V of the last but one (not in LSE-only launches)
          if (have || have2) {             // (a piece of one tile has nothing in its second step)
            if (!(ok = wait_or_abort(&bars.kv_empty[st], ph, &sh.abort))) break;
            if (have) sh.nv[t++ % kNvRing] = ti.nv;   // read after kv_full
            mbar_expect_tx(&bars.kv_full[st], (have ? kKvBytes<kKv> : 0) + (have2 ? kKvBytes<kKv> : 0));
            ++steps;
            uint8_t* dst = sKV + st * kStageBytes<kKv>;
            if (have2) load(dst + kKvBytes<kKv>, t2, p.tm_vd, &p.tm_vpool);
            if (have) load(dst, ti, p.tm_kd, &p.tm_kpool);
            if (++st == kStages) { st = 0; ph ^= 1; }
          }
          t2 = t1;
          have2 = have1;
          t1 = ti;
          have1 = have && !kLse;
          if (have) have = it.next(p, ti, report);
        }
      }
      leave_role(ok, &sh.abort, p.status);
      // After an abort the consumers no longer wait for the tiles in flight, so this thread does: a CTA must not free
      // its shared memory under copies that are still landing.  Per stage, the load armed last is use u = (count - 1 -
      // stage) / stages of that stage's barrier, whose phase u has parity u & 1; a stage that was never armed is skipped.
      if (sh.abort) {
        auto drain = [](uint64_t* bar, uint32_t use) {
          for (uint32_t i = 0; i < (1u << 16); ++i)
            if (mbar_try_wait(bar, use & 1)) break;
        };
        if (n > 0) drain(&bars.q_full, n - 1);
        for (uint32_t q = 0; q < kStages; ++q)
          if (steps > q) drain(&bars.kv_full[q], (steps - 1 - q) / kStages);
      }
    }
  } else if (warp == kSoftWarps<kKv>) {
    if constexpr (kLse) mma_lse_role(p, sh, smem_base);
    else mma_role<kKv, 0>(p, sh, smem_base);
  } else if (!kLse && warp == kSoftWarps<kKv> + 1) {
    if constexpr (!kLse) mma_role<kKv, 1>(p, sh, smem_base);
  } else if constexpr (kLse) {
    // ------------------------------------------------------------------ LSE-only softmax warpgroups (one thread per row)
    // Warpgroup qt + 2 b works on S buffer b of Q tile qt, i.e. on every other KV tile of these rows: four warps per
    // scheduler instead of two, which is what hides the latencies of this issue-bound loop.  At the end of a unit the two
    // warpgroups of a Q tile merge (reference, sum) through shared memory.
    const int wg = warp >> 2, qt = wg & 1, buf = wg >> 1;
    const int row = (warp & 3) * 32 + lane;
    const uint32_t tS = (static_cast<uint32_t>((warp & 3) * 32) << 16) + buf * 256 + qt * 128;
    const uint64_t scale2 = pack_f32x2(p.scale_log2, p.scale_log2);
    PieceWalker walk;
    walk.init(p);
    Piece pc;
    uint32_t g = 0;     // KV tiles of this Q tile so far: tile number g is in buffer g & 1
    uint32_t t0 = 0;    // tiles of the CTA's pieces so far
    uint32_t n = 0;     // units of this Q tile so far
    bool ok = true;
    bool more = walk.next(p, pc);
    for (; ok && more; more = walk.next(p, pc)) {
      const int n_eff = count_tiles(p, pc.tb, pc.te);
      if (qt == 1 && !pc.has_q1) { t0 += n_eff; continue; }
      const bool releases = qt == (pc.has_q1 ? 1 : 0);   // the Q tile whose product comes last
      float m = 0.f, l = 0.f;
      bool first = true;
      for (int j = (g ^ buf) & 1; j < n_eff; j += 2) {
        if (!(ok = wait_or_abort(&bars.s_full[wg], ((g + j) >> 1) & 1, &sh.abort))) break;
        const int nv = sh.nv[(t0 + j) % kNvRing], n_ch = (nv + 31) >> 5;
        if (releases && row == 0) {   // the products that read this tile's stage (and, with the last tile, Q) are done
          mbar_arrive(&bars.kv_empty[(t0 + j) % kStages]);
          if (j + 1 == n_eff) mbar_arrive(&bars.q_empty);
        }
        tc_fence_after();
        // The row is streamed from tensor memory 32 columns at a time, without a maximum: the sum is taken against a fixed
        // reference, 0 at first (logits of a few log2 units lose nothing there).  A warp in which a row's tile sum leaves
        // [2^-12 (first tile only), 2^15] reads S again and takes the row's maximum as its reference from there on.
        float sum = 0.f;
#pragma unroll 1
        for (int attempt = 0; attempt < 2; ++attempt) {
          const uint64_t neg_m2 = pack_f32x2(-m, -m);
          uint64_t acc[4] = {0, 0, 0, 0};
          float big = -INFINITY;
#pragma unroll 1
          for (int c = 0; c < n_ch; ++c) {
            uint32_t r[32];
            tmem_ld_x32(tS + c * 32, r);
            tc_wait_ld(r);
            exp_chunk(r, nv - c * 32, scale2, neg_m2, acc, big);
          }
          sum = big != big ? big : sum4_f32x2(acc);
          const bool off = !(sum <= 32768.f) || big * p.scale_log2 - m > 100.f || (first && sum < 2.44140625e-4f);
          if (attempt > 0 || !__any_sync(0xffffffffu, off)) break;
          const float mx = row_max_tmem(tS, nv);
          if (off) {
            const float m_new = first ? mx * p.scale_log2 : fmaxf(m, mx * p.scale_log2);
            l *= ex2_approx(m - m_new);
            m = m_new;
          }
        }
        l += sum;
        first = false;
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars.p_full[wg]);   // the buffer has been read
      }
      if (!ok) break;
      g += n_eff;
      t0 += n_eff;
      if (buf == 1) {
        if (!(ok = wait_or_abort(&bars.m_empty[qt], (n & 1) ^ 1, &sh.abort))) break;
        sh.merge[qt][row] = make_float2(m, l);
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars.m_full[qt]);
      } else {
        if (!(ok = wait_or_abort(&bars.m_full[qt], n & 1, &sh.abort))) break;
        const float2 o = sh.merge[qt][row];
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars.m_empty[qt]);
        const int qrow = pc.q0 + qt * kTileQ + row;
        if (qrow < p.lq) {
          // (a warpgroup without tiles leaves a sum of 0, a stale slot two of them; a logit that is NaN leaves NaN, and the slot then
          // counts for nothing in this row)
          const float mm = l > 0.f ? (o.y > 0.f ? fmaxf(m, o.x) : m) : o.x;
          const float sum = (l != 0.f ? l * ex2_approx(m - mm) : 0.f) + (o.y != 0.f ? o.y * ex2_approx(o.x - mm) : 0.f);
          p.lse[(static_cast<int64_t>(pc.ord) * p.H + pc.h) * p.lq + qrow] =
              sum > 0.f ? (mm + log2f(sum)) * 0.6931471805599453f : -INFINITY;
        }
      }
      ++n;
    }
    if (!ok) leave_role(false, &sh.abort, p.status);
  } else {
    // ------------------------------------------------------------------ softmax warpgroups (one thread per query row)
    const int wg = warp >> 2;
    const int row = (warp & 3) * 32 + lane;
    const uint32_t lane_base = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const uint32_t tS = lane_base + kTmemS + wg * 128;
    const uint32_t tP = lane_base + kTmemP + wg * 128;
    const uint32_t tO = lane_base + kTmemO + wg * 128;
    PieceWalker walk;
    walk.init(p);
    Piece pc;
    uint32_t g = 0;       // steps of this warpgroup waited for so far
    uint32_t t0 = 0;      // tiles of the CTA's pieces so far
    uint32_t steps = 0;   // stages used by the pieces so far
    uint32_t n_out = 0;   // pieces of this warpgroup that produced output
    bool ok = true;
    const uint64_t scale2 = pack_f32x2(p.scale_log2, p.scale_log2);
    const bool wide = (reinterpret_cast<uint64_t>(p.O) & 31) == 0;
    bool more = walk.next(p, pc);
    dep_wait();
    dep_release();
    for (; ok && more; more = walk.next(p, pc)) {
      const bool active = (wg == 0) || pc.has_q1;
      const int n_eff = count_tiles(p, pc.tb, pc.te);
      float m = -INFINITY, l = 0.f;
      const bool few = n_eff <= kFewTiles;
      // Stages and Q are given back by both warpgroups, for the step whose commit they have seen: a commit of the MMA warps to these
      // barriers would hold them much longer than this.  Where there is no second Q tile, warpgroup 0 gives a stage back twice, and
      // Q is given back by warpgroup 0 and the idle MMA warp.
      auto give_back = [&](int i) {
        if (row == 0) {
          mbar_arrive(&bars.kv_empty[(steps + i) % kStages]);
          if (i + 1 == n_eff) mbar_arrive(&bars.q_empty);
          if (!pc.has_q1) mbar_arrive(&bars.kv_empty[(steps + i) % kStages]);
        }
      };
      int j = 0;
      if (active) {
        if (n_eff > 0) {
          uint32_t pk[kKv / 2] = {};   // P of tile j - 1
          float alpha = 1.f;
          bool rescale = false;
          int careful = 0, redos = 0;   // tiles whose maximum is taken first from here on; tiles streamed twice so far
          for (;; ++j) {
            // Step j is done: S of tile j is there, and P V of tile j - 2 has read its P.  (A piece of one tile has no step 1.)
            if (j != 1 || n_eff > 1) {
              ok = wait_or_abort(&bars.s_full[wg], g++ & 1, &sh.abort);
              if (!ok) break;
              tc_fence_after();
            }
            if (rescale) {
#pragma unroll 1
              for (int c = 0; c < 128; c += 32) {
                uint32_t o[32];
                tmem_ld_x32(tO + c, o);
                tc_wait_ld(o);
#pragma unroll
                for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                tmem_st_x32(tO + c, o);
              }
            }
            // (the first time there is no P to store and the last time no S to load: nobody reads what these move then)
            uint32_t r[kKv];   // S of tile j
            tmem_st_half_tile(tP, pk);
            tmem_ld_tile(tS, r);
            const int nv = sh.nv[(t0 + j) % kNvRing];
            tmem_ld_wait(r);
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            // One arrival per warp: the waits above covered all 32 lanes.  (Of a piece of one tile only P is handed over: nothing holds
            // this warp between its S and its P, and the MMA warp cannot tell two completions that it has not seen from none.)
            if (lane == 0 && (j > 0 || n_eff > 1)) mbar_arrive(&bars.p_full[wg]);
            if (j != 1 || n_eff > 1) give_back(j);
            if (j == n_eff) break;
            if (nv < kKv) {   // columns past the end of the segment or slot
#pragma unroll
              for (int i = 0; i < kKv; ++i) r[i] = i < nv ? r[i] : 0xff800000u;
            }
            // known: the row's maximum over the tile is taken before the exponentials
            bool known = few || j == 0 || careful > 0;
            if (careful > 0) --careful;
            rescale = false;
            float sum;
            for (;;) {
              if (known) {
                const float mt = row_max(r) * p.scale_log2;
                const float alpha_mt = ex2_approx(m - mt);
                const bool move = few ? mt > m || (mt < m && l * alpha_mt <= kOwnSum) : mt > m + kRescaleThreshold;   // also true on the first tile (m = -inf)
                rescale = j > 0 && __any_sync(0xffffffffu, move);
                alpha = move ? alpha_mt : 1.f;
                if (move) m = mt;
                l *= alpha;
              }
              sum = exp_tile(r, scale2, m, pk);
              if (known || !__any_sync(0xffffffffu, !(sum <= kStreamSum))) break;
              known = true;
              careful = 1 << min(++redos, 6);
            }
            l += sum;
          }
        }
        // ---------------------------------------------------------------- epilogue of this piece
        const int prow = wg * kTileQ + row;
        const int qrow = pc.q0 + prow;
        if (ok && j > 0) {
          ok = wait_or_abort(&bars.o_done[wg], n_out++ & 1, &sh.abort);   // completes once per piece
          give_back(n_eff == 1 ? 1 : n_eff + 1);
        }
        if (ok) {
          tc_fence_after();
          // without keys 0 and -inf; a sum that is NaN (a logit was) makes the row and its log-sum-exp NaN
          const float inv_l = (j > 0 && l != 0.f) ? 1.f / l : 0.f;
          const float lse = (j > 0 && l != 0.f) ? (m + log2f(l)) * 0.6931471805599453f : -INFINITY;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            uint32_t r[32];
            if (j > 0) {
              tmem_ld_x32(tO + c * 32, r);
              tc_wait_ld(r);
            } else {
#pragma unroll
              for (int i = 0; i < 32; ++i) r[i] = 0u;
            }
            if (qrow < p.lq) {
              if (pc.slot < 0) {
                // a row per lane: 32 lines per store whatever its width, so the widest that O's alignment allows
                __nv_bfloat16* dst = p.O + (static_cast<int64_t>(qrow) * p.H + pc.h) * kHeadDim + c * 32;
                uint32_t o[16];
#pragma unroll
                for (int v = 0; v < 16; ++v) o[v] = pack_bf16x2(__uint_as_float(r[2 * v]) * inv_l, __uint_as_float(r[2 * v + 1]) * inv_l);
                if (wide) {
                  st_global_x8(dst, o);
                  st_global_x8(dst + 16, o + 8);
                } else {
#pragma unroll
                  for (int v = 0; v < 4; ++v)
                    reinterpret_cast<uint4*>(dst)[v] = make_uint4(o[4 * v], o[4 * v + 1], o[4 * v + 2], o[4 * v + 3]);
                }
              } else {
                float4* dst = p.opart + (static_cast<int64_t>(pc.slot) * 32 + c * 8) * kPairRows + prow;
#pragma unroll
                for (int v = 0; v < 8; ++v)
                  dst[v * kPairRows] = make_float4(__uint_as_float(r[4 * v]) * inv_l, __uint_as_float(r[4 * v + 1]) * inv_l,
                                       __uint_as_float(r[4 * v + 2]) * inv_l, __uint_as_float(r[4 * v + 3]) * inv_l);
              }
            }
          }
          if (qrow < p.lq) {
            if (pc.slot < 0) {
              if (p.lse) p.lse[static_cast<int64_t>(pc.h) * p.lq + qrow] = lse;
            } else {
              p.lsepart[static_cast<int64_t>(pc.slot) * kPairRows + prow] = lse;
            }
          }
        }
      }
      t0 += n_eff;
      if (n_eff > 0) steps += n_eff == 1 ? 2 : n_eff + 2;
      // O of this piece has been read: the next piece that uses this accumulator may overwrite it
      if (active && j > 0) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars.o_free[wg]);
      }
    }
    if (!ok) leave_role(false, &sh.abort, p.status);
  }
}

template <int kKv>
__global__ void __launch_bounds__(kThreads<kKv>, 1)
memory_attention_kernel(const __grid_constant__ AttnParams p) {
  constexpr bool kLse = is_lse<kKv>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + (((smem_u32(smem_raw) + 1023u) & ~1023u) - smem_u32(smem_raw));
  __shared__ CtaShared<kKv> sh;
  const int tid = threadIdx.x;
  if (tid == 0) {
    mbar_init(&sh.bars.q_full, 1);
    mbar_init(&sh.bars.q_empty, kLse ? 1 : 2);
    for (int s = 0; s < kStages; ++s) { mbar_init(&sh.bars.kv_full[s], 1); mbar_init(&sh.bars.kv_empty[s], kLse ? 1 : 2); }
    for (int i = 0; i < 4; ++i) { mbar_init(&sh.bars.s_full[i], 1); mbar_init(&sh.bars.p_full[i], 4); }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sh.bars.turn[i], 1);
      mbar_init(&sh.bars.o_done[i], 1);
      mbar_init(&sh.bars.o_free[i], 4);
      mbar_init(&sh.bars.m_full[i], 4);
      mbar_init(&sh.bars.m_empty[i], 4);
    }
    fence_mbar_init();
    sh.abort = 0;
  }
  if (tid < 32) {
    tmem_alloc(&sh.tmem, 512);
    tmem_relinquish();
  }
  if (!kLse && tid >= 32 && tid < 32 + 3 + 2 * kMaxDenseSegs) {
    const int i = tid - 32;   // tm_q, tm_kpool, tm_vpool, tm_kd[], tm_vd[] lie one behind the other
    if (i < 3 || (i - 3) % kMaxDenseSegs < p.n_segs) prefetch_tensormap(&p.tm_q + i);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // Everything up to the roles' dep_wait() runs under the end of the kernel before this one, and nothing that it may write is read
  // or overwritten there: a role works out from the launch's parameters where it starts (0.7 to 2 us after the wait before).  LSE-only
  // launches follow the one-CTA ranking of the call before, under which nothing of theirs runs, and wait here (query retrieval with
  // roles that wait, tensor maps prefetched and the first slot looked up before Q is asked for, in brackets this way: 148 units of
  // one tile 17.9 us a call (17.6), of eleven 29.3 (29.0)).
  // an allocation of all 512 columns starts at column 0; addresses known at compile time keep the MMAs' operands cheap
  if (sh.tmem != 0 && tid == 0) {
    dep_wait();
    sh.abort = 1;
    atomicOr(p.status, WK_DEV_TIMEOUT);
  }

  if (kLse) {
    dep_wait();
    dep_release();
  }
  attention_roles<kKv>(p, sh, smem);
  tc_fence_before();
  __syncthreads();
  if (tid < 32) tmem_dealloc(sh.tmem, 512);
}

// Merge the pieces of every unit that was cut: O = sum_s w_s O_s / sum_s w_s with w_s = exp(lse_s - max lse).  Bound by
// reading the fp32 partials (they come from L2).  A block merges 32 rows x 32 columns of one unit: warp w holds column
// group w of the 32 rows, so that every load is one contiguous 512-byte line, and the bf16 result leaves through shared
// memory as 64 contiguous bytes per row.  Units written directly by a single CTA are left alone.
constexpr int kCombineThreads = 256;
__global__ void __launch_bounds__(kCombineThreads)
combine_kernel(const float4* __restrict__ opart, const float* __restrict__ lsepart, int G, int n_full, int n_units, int n_tiles,
               int n_qpairs, int H, int lq, __nv_bfloat16* __restrict__ O, float* __restrict__ lse_out) {
  __shared__ float s_lse[kMaxPieces][32], s_w[kMaxPieces][32];
  __shared__ __align__(16) uint2 s_out[32][8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ut = blockIdx.x >> 5, u = n_full + ut, rg = (blockIdx.x >> 2) & 7, cg = blockIdx.x & 3;   // unit, row group, column group
  const int h = u / n_qpairs, qrow0 = (u - h * n_qpairs) * kPairRows + rg * 32;
  // the CTAs whose ranges touch the unit: lane i looks at the i-th one (every range holds at least one tile)
  const int64_t W = static_cast<int64_t>(n_units - n_full) * n_tiles;
  const int64_t ustart = static_cast<int64_t>(ut) * n_tiles, uend = ustart + n_tiles;
  auto start_of = [&](int c) { return range_start(W, G, c); };
  int c0 = static_cast<int>(ustart * G / W);
  while (c0 > 0 && start_of(c0) > ustart) --c0;
  while (c0 + 1 < G && start_of(c0 + 1) <= ustart) ++c0;
  const int cc = c0 + lane;
  const int64_t sc = start_of(cc);
  const bool mine = cc < G && sc < uend;
  const int np = __popc(__ballot_sync(0xffffffffu, mine));
  const bool single = np == 1 && start_of(c0) <= ustart && start_of(c0 + 1) >= uend;   // one CTA covered the whole unit
  // the partial-result slots of range c: 2 c for the piece it starts with, 2 c + 1 for the one it ends with
  const int enters = start_of(c0) < ustart ? 1 : 0;
  auto slot_of = [&](int s) { return static_cast<int64_t>(2 * (c0 + s) + (s == 0 ? enters : 0)); };
  const int64_t at = static_cast<int64_t>(cg * 8 + warp) * kPairRows + rg * 32 + lane;
  auto load8 = [&](int s0, float4 (&o)[8]) {   // eight pieces' loads in flight
#pragma unroll
    for (int i = 0; i < 8; ++i)
      o[i] = s0 + i < np ? __ldcg(opart + slot_of(s0 + i) * 32 * kPairRows + at) : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  dep_wait();
  if (single || qrow0 >= lq) return;
  float4 o[8];
  load8(0, o);   // beside the weights, which need two trips of their own
  for (int s = warp; s < np; s += kCombineThreads / 32)
    s_lse[s][lane] = __ldcg(lsepart + slot_of(s) * kPairRows + rg * 32 + lane);
  __syncthreads();
  float mx = -INFINITY;
  for (int s = 0; s < np; ++s) mx = fmaxf(mx, s_lse[s][lane]);
  for (int s = warp; s < np; s += kCombineThreads / 32)
    s_w[s][lane] = s_lse[s][lane] == -INFINITY ? 0.f : expf(s_lse[s][lane] - mx);
  __syncthreads();
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  float wsum = 0.f;
  for (int s0 = 0; s0 < np; s0 += 8) {
    if (s0 > 0) load8(s0, o);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (s0 + i < np) {
        const float w = s_w[s0 + i][lane];
        acc.x = fmaf(w, o[i].x, acc.x); acc.y = fmaf(w, o[i].y, acc.y);
        acc.z = fmaf(w, o[i].z, acc.z); acc.w = fmaf(w, o[i].w, acc.w);
        wsum += w;
      }
    }
  }
  const float inv = wsum != 0.f ? 1.f / wsum : 0.f;   // NaN stays NaN
  s_out[lane][warp] = make_uint2(ptx::pack_bf16x2(acc.x * inv, acc.y * inv), ptx::pack_bf16x2(acc.z * inv, acc.w * inv));
  __syncthreads();
  if (tid < 128) {
    const int r = tid >> 2, v = tid & 3;
    if (qrow0 + r < lq)
      reinterpret_cast<uint4*>(O + (static_cast<int64_t>(qrow0 + r) * H + h) * kHeadDim + cg * 32)[v] =
          reinterpret_cast<const uint4*>(&s_out[r][0])[v];
  }
  if (lse_out && cg == 0 && warp == 0 && qrow0 + lane < lq)
    lse_out[static_cast<int64_t>(h) * lq + qrow0 + lane] = wsum != 0.f ? mx + logf(wsum) : -INFINITY;
}

}  // namespace

int attention_partial_slots(int n_heads, int max_lq, int max_splits) {
  const int units = n_heads * ((max_lq + kPairRows - 1) / kPairRows);
  const int by_split = units * (max_splits > 1 ? max_splits : 1);
  return 2 * (by_split > 256 ? by_split : 256);
}

// Default distribution over the SMs: whole units in full waves, then, where it pays, the units of the last, partial wave cut
// and merged.  Times in us on 148 SMs, whole / cut, back to back, one dense segment.
//   * Where every unit can be cut at least in two, it is, into equal ranges that end with their unit: no CTA gets two pieces, and
//     the idle SMs cost less than pieces that straddle units (30 units of 32 tiles: 120 ranges 28.3, 148 ranges 31.2; of 64
//     tiles 33.2 and 41.8; 66 units of 38 tiles: 132 ranges 43.5, 148 ranges 55.5).  A piece has 5 tiles or more (2 heads x
//     3,960 keys, 8 units of 50 tiles: 5 tiles 19.9, 4 19.9, 3 21.5, 10 24.8).  Else equal ranges over all SMs.
//   * A cut saves at most (sms - rest) / sms of a unit's tiles and costs about 8 tiles (the combine launch, a second prologue) and
//     up to 22 more where every CTA writes partials: 12 units of 12 tiles 17.7 / 16.3; 24 of 15 20.7 / 21.0; 30 of 16 21.7 / 21.8, of 20
//     25.6 / 23.5; 40 of 21 27.1 / 28.4; 50 of 16 22.3 / 29.7, of 24 30.0 / 30.4; 66 of 25 31.8 / 35.7, of 38 46.0 / 43.5; 88 of 38
//     52.9 / 64.4, of 57 77.8 / 81.1; 99 of 63 89.1 / 97.0; 110 of 94 136 / 142, of 150 216 / 202; 121 of 125 185 / 196, of 150 226 /
//     231; 132 of 198 253 / 266, of 282 358 / 361, of 500 638 / 605.  With full waves before it: 760 units of 410 tiles (rest 20)
//     2,953 / 2,763.
//   * Units of a little more than kFewTiles tiles are cut before that saves time, where a cut leaves pieces of few tiles, whose every
//     largest weight is exact (24 units of 1,040 keys: relative error of O at deviations 1 / 2 / 4 2.33 / 2.29 / 2.14e-3 whole at 19.1
//     us, 2.14 / 1.78 / 1.68e-3 in three pieces at 20.5; 40 of 1,520: 25.4 and 27.7 us).  The line is drawn in tiles of 128 rows, of
//     which a range of four, 512 rows, is at most eight of the kernel's: at three cuts or more it is crossed at 6 of them (10 units), 8
//     (24) and 12 (40).
static void split_default(int64_t units, int64_t tiles, int64_t tiles128, int64_t sms, int64_t* G, int64_t* n_full, int64_t* ranges) {
  const int64_t waves = units / sms, rest = units - waves * sms;
  *G = units < sms ? units : sms;
  *n_full = units;
  *ranges = 0;
  const bool faster = (sms - rest) * tiles >= 8 * sms + 22 * rest;
  const bool closer = sms >= 3 * rest && tiles > kFewTiles && (sms - rest) * tiles128 >= 4 * sms + 16 * rest;
  if (rest == 0 || !(faster || closer)) return;
  int64_t r;
  if (sms >= 2 * rest) {
    int64_t cuts = sms / rest;
    if (cuts > kMaxPieces - 2) cuts = kMaxPieces - 2;
    int64_t per = (tiles + cuts - 1) / cuts;
    if (per < 5) per = 5;
    r = rest * ((tiles + per - 1) / per);
  } else {
    r = sms;
    if (r > rest * tiles) r = rest * tiles;
  }
  *n_full = waves * sms;
  *ranges = r;
  *G = waves > 0 ? sms : r;
}

wk_status launch_attention(wk_ctx* ctx, int layer, const __nv_bfloat16* Q, int lq, const wk_dense_seg* segs, int n_segs,
                           const int32_t* slots_dev, int n_slots, __nv_bfloat16* O, float* lse, int kv_splits,
                           cudaStream_t s, bool lse_only) {
  if (!ctx->attn_attr_set) {   // the attribute belongs to the device the context lives on
    WK_CUDA_TRY(ctx, cudaFuncSetAttribute(memory_attention_kernel<kTileKV>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          static_cast<int>(kSmemBytes<kTileKV>)));
    WK_CUDA_TRY(ctx, cudaFuncSetAttribute(memory_attention_kernel<kTileKVFew>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          static_cast<int>(kSmemBytes<kTileKVFew>)));
    WK_CUDA_TRY(ctx, cudaFuncSetAttribute(memory_attention_kernel<kTileKVLse>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          static_cast<int>(kSmemBytes<kTileKVLse>)));
    ctx->attn_attr_set = true;
  }
  AttnParams p;
  wk_status st = encode_rows_map(ctx, Q, lq, kTileQ, &p.tm_q);
  if (st != WK_OK) return st;
  // Keys beside which every tile's largest weight counts are tiled in 64 rows, as are keys that fill tiles of 80 badly (see kFewTiles); all
  // others in 80, what tensor memory has room for.
  auto count = [&](int rows, int n_rows) { return (n_rows + rows - 1) / rows; };
  auto count_all = [&](int rows) {
    int n = n_slots * count(rows, ctx->C);
    for (int i = 0; i < n_segs; ++i) n += count(rows, segs[i].n_tokens);
    return n;
  };
  const int few = count_all(kTileKVFew);
  const bool in_64 = few <= kFewTilesOfCall || kCost64 * few <= kCost80 * count_all(kTileKV);
  p.tile_rows = lse_only ? kTileKVLse : in_64 ? kTileKVFew : kTileKV;
  p.tm_kpool = lse_only ? ctx->tm_kpool_lse : in_64 ? ctx->tm_kpool_few : ctx->tm_kpool;
  p.tm_vpool = in_64 ? ctx->tm_vpool_few : ctx->tm_vpool;
  const int most = count_all(128);   // as many ranges of a unit may a caller ask for
  int tiles = 0;
  for (int i = 0; i < n_segs; ++i) {
    const CUtensorMap* mk = cached_rows_map(ctx, segs[i].K, segs[i].n_tokens, p.tile_rows, &st);
    if (st != WK_OK) return st;
    p.tm_kd[i] = *mk;
    const CUtensorMap* mv = cached_rows_map(ctx, segs[i].V, segs[i].n_tokens, p.tile_rows, &st);
    if (st != WK_OK) return st;
    p.tm_vd[i] = *mv;
    p.seg_tile_prefix[i] = tiles;
    p.seg_rows[i] = segs[i].n_tokens;
    tiles += count(p.tile_rows, segs[i].n_tokens);
  }
  for (int i = n_segs; i < kMaxDenseSegs; ++i) {
    p.tm_kd[i] = p.tm_q;
    p.tm_vd[i] = p.tm_q;
    p.seg_rows[i] = 0;
  }
  for (int i = n_segs; i <= kMaxDenseSegs; ++i) p.seg_tile_prefix[i] = tiles;
  p.n_segs = n_segs;
  p.n_dense_tiles = tiles;
  p.slots = slots_dev;
  p.valid = ctx->valid_dev;
  p.n_slots = n_slots;
  p.pool_slots = ctx->cfg.pool_slots;
  p.layer = layer;
  p.C = ctx->C;
  p.tiles_per_slot = count(p.tile_rows, ctx->C);
  p.n_tiles = tiles + n_slots * p.tiles_per_slot;
  p.lq = lq;
  p.slot_units = lse_only ? 1 : 0;
  p.H = ctx->cfg.n_heads;
  p.n_qpairs = (lq + kPairRows - 1) / kPairRows;
  p.n_units = p.n_qpairs * p.H;
  p.scale_log2 = ctx->scale * 1.4426950408889634f;
  p.O = O;
  p.lse = lse;
  p.opart = reinterpret_cast<float4*>(ctx->scratch_base + ctx->sl.opart_off);
  p.lsepart = reinterpret_cast<float*>(ctx->scratch_base + ctx->sl.lsepart_off);
  p.status = ctx->status_dev;
  if (lse_only) {
    // every listed slot is scored on its own: one unit per (slot, head, q-pair), each over that slot's tiles only
    if (n_segs != 0 || n_slots < 1) return WK_ERR_ARG;
    p.n_tiles = p.tiles_per_slot;
    p.n_units *= n_slots;
  }
  const int64_t sms = ctx->sm_count;
  int64_t G, n_full = 0, ranges = 0;   // CTAs, units done whole, ranges the rest is cut into
  if (lse_only) {
    // whole units, dealt out one by one: the CTAs of one (slot, head) run side by side and share its tiles through L2
    n_full = p.n_units;
    G = sms < n_full ? sms : n_full;
  } else if (kv_splits == 0) {
    split_default(p.n_units, p.n_tiles, most, sms, &G, &n_full, &ranges);
  } else if (kv_splits > 0) {
    int sp = kv_splits < most ? kv_splits : most;
    if (sp > kMaxPieces) sp = kMaxPieces;
    if (sp == 1) n_full = G = p.n_units;
    else ranges = G = static_cast<int64_t>(p.n_units) * sp;   // every unit cut into exactly sp ranges
  } else {
    ranges = G = -static_cast<int64_t>(kv_splits);      // caller-chosen number of equal ranges
    if (G > static_cast<int64_t>(p.n_units) * (kMaxPieces - 2)) return WK_ERR_SHAPE;   // a unit would be cut into too many pieces
    if (G > static_cast<int64_t>(p.n_units) * most) ranges = G = static_cast<int64_t>(p.n_units) * most;
  }
  const int max_slots = attention_partial_slots(p.H, ctx->max_lq, ctx->max_splits);
  if (!lse_only && 2 * ranges > max_slots) return WK_ERR_SHAPE;
  p.n_full = static_cast<int>(n_full);
  p.n_ranges = static_cast<int>(ranges);
  const dim3 grid(static_cast<unsigned>(G));
  if (lse_only) launch_chained(memory_attention_kernel<kTileKVLse>, grid, dim3(kThreads<kTileKVLse>), kSmemBytes<kTileKVLse>, s, p);
  else if (in_64) launch_chained(memory_attention_kernel<kTileKVFew>, grid, dim3(kThreads<kTileKVFew>), kSmemBytes<kTileKVFew>, s, p);
  else launch_chained(memory_attention_kernel<kTileKV>, grid, dim3(kThreads<kTileKV>), kSmemBytes<kTileKV>, s, p);
  if ((st = after_launch(ctx)) != WK_OK) return st;
  if (!lse_only && n_full != p.n_units) {   // some unit was cut
    launch_chained(combine_kernel, dim3(static_cast<unsigned>(p.n_units - n_full) * 32), dim3(kCombineThreads), 0, s, p.opart,
                   p.lsepart, p.n_ranges, p.n_full, p.n_units, p.n_tiles, p.n_qpairs, p.H, lq, O, lse);
    if ((st = after_launch(ctx)) != WK_OK) return st;
  }
  return WK_OK;
}

}  // namespace wk
