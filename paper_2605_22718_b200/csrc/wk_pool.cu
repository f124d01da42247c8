// Chunk pool (Section 4.2): device side of append (row-gather compaction of K and V into a slot) and of the
// slot table (validity flag + pose).  Slot allocation and FIFO bookkeeping are host side (wk_api.cu).
#include "wk_internal.cuh"

namespace wk {
namespace {

constexpr int kAppendThreads = 256;

constexpr int kAppendRows = 32;   // stored rows per block (fewer where they are few in all)

struct Pose8 { float v[8]; };

struct AppendParams {
  const __nv_bfloat16 *Ksrc, *Vsrc;
  int64_t stride;               // elements between layers of the source chunk
  const int32_t* keep_idx;
  int hs, T, C, FT, D, n;       // index lists per layer, anchor rows, stored rows, chunk rows, row width, layers
  __nv_bfloat16 *Kdst, *Vdst;
  int64_t dst_layer_stride;
  int k_row0, v_row0;           // first row of K / V that the index list is needed for (0 or T)
  int v_anchor_blocks;          // blocks that copy V's anchor frame: they come first and do not wait for the selection
  int reverse;
  int rows;                     // stored rows per block
  int mark_slot;                // >= 0: mark this slot valid
  int32_t* valid;
  float* poses;
  Pose8 pose;
  uint32_t* status;
};

// Bound by memory (5.6-6.5 TB/s of reads and writes).  One warp per stored row, 16-byte vectors, four loads in flight per
// lane before the first store.  With per-head keep-sets (hs = n_heads index lists per layer) every 128-column block of a
// stored row has its own source token.  Behind a selection, the anchor frame needs no index list: the scoring kernels have
// stored its K rows and, where score_select runs (see AnchorStore), its V rows; where they have not (compress_fused, per-head
// keys, calls without scores), V's are copied by the first blocks, which need no index list.  The kernels in front of those
// calls do not let this one start before they end, so nothing overlaps there; the rows are contiguous on both sides.
__global__ void __launch_bounds__(kAppendThreads)
append_rows(const __grid_constant__ AppendParams p) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int vecs = p.D >> 3;
  int id = blockIdx.x;
  // Marking here is safe: a kernel behind this one on the stream sees the slot only once all of this one's rows are stored.
  if (id == 0 && p.mark_slot >= 0) {
    if (threadIdx.x < 8) p.poses[p.mark_slot * 8 + threadIdx.x] = p.pose.v[threadIdx.x];
    if (threadIdx.x == 0) p.valid[p.mark_slot] = 1;
  }
  if (id < p.v_anchor_blocks) {
    // (every earlier kernel on the stream but the selection has finished: a scoring kernel lets this one start only after
    // it has waited for them itself)
    const int per = (p.T + kAppendRows - 1) / kAppendRows;
    const int l = id / per, r0 = (id - l * per) * kAppendRows, rows = min(kAppendRows, p.T - r0);
    const uint4* src = reinterpret_cast<const uint4*>(p.Vsrc + static_cast<int64_t>(l) * p.stride) + static_cast<int64_t>(r0) * vecs;
    uint4* dst = reinterpret_cast<uint4*>(p.Vdst + static_cast<int64_t>(l) * p.dst_layer_stride) + static_cast<int64_t>(r0) * vecs;
    const int total = rows * vecs;   // the rows are contiguous on both sides
    for (int v0 = threadIdx.x; v0 < total; v0 += 4 * kAppendThreads) {
      uint4 q[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (v0 + u * kAppendThreads < total) q[u] = __ldcs(src + v0 + u * kAppendThreads);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (v0 + u * kAppendThreads < total) dst[v0 + u * kAppendThreads] = q[u];
    }
    return;
  }
  dep_wait();   // returns at once unless the launch was chained to the selection that writes keep_idx
  id -= p.v_anchor_blocks;
  const int per_k = (p.C - p.k_row0 + p.rows - 1) / p.rows, per_v = (p.C - p.v_row0 + p.rows - 1) / p.rows;
  // reverse: walk the layers last to first, so that the layers whose keys the scoring pass touched last (and L2 still
  // holds) are gathered first
  const int lb = id / (per_k + per_v);
  const int l = p.reverse ? p.n - 1 - lb : lb;
  int blk = id - lb * (per_k + per_v);
  const bool is_v = blk >= per_k;
  if (is_v) blk -= per_k;
  const __nv_bfloat16* src = (is_v ? p.Vsrc : p.Ksrc) + static_cast<int64_t>(l) * p.stride;
  __nv_bfloat16* dst = (is_v ? p.Vdst : p.Kdst) + static_cast<int64_t>(l) * p.dst_layer_stride;
  const int32_t* idx = p.keep_idx + static_cast<int64_t>(l) * p.hs * p.C;
  const int vecs_per_list = vecs / p.hs;
  const int r0 = (is_v ? p.v_row0 : p.k_row0) + blk * p.rows, r1 = min(p.C, r0 + p.rows);
  for (int r = r0 + warp; r < r1; r += kAppendThreads / 32) {
    uint4* d = reinterpret_cast<uint4*>(dst + static_cast<int64_t>(r) * p.D);
    for (int v0 = lane; v0 < vecs; v0 += 128) {
      uint4 q[4];
      bool ok[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int v = v0 + 32 * u;
        ok[u] = v < vecs;
        if (ok[u]) {
          const int j = idx[(v / vecs_per_list) * p.C + r];
          if (j < 0 || j >= p.FT) {                   // never dereference a bad index
            atomicOr(p.status, WK_DEV_BAD_SLOT);
            ok[u] = false;
          } else {
            q[u] = __ldg(reinterpret_cast<const uint4*>(src + static_cast<int64_t>(j) * p.D) + v);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (ok[u]) d[v0 + 32 * u] = q[u];
    }
  }
}

__global__ void slot_mark(int32_t* __restrict__ valid, float* __restrict__ poses, int slot, int is_valid, Pose8 pose) {
  if (threadIdx.x < 8) poses[slot * 8 + threadIdx.x] = pose.v[threadIdx.x];
  if (threadIdx.x == 0) valid[slot] = is_valid;
}

}  // namespace

__nv_bfloat16* pool_rows(wk_ctx* ctx, __nv_bfloat16* base, int layer, int slot) {
  return base + (static_cast<int64_t>(layer) * ctx->cfg.pool_slots + slot) * ctx->C * ctx->D;
}

wk_status launch_append(wk_ctx* ctx, int layer0, int n, int slot, const __nv_bfloat16* K, const __nv_bfloat16* V,
                        int64_t stride, const int32_t* keep_idx, cudaStream_t s, const AnchorStore* stored, const float* mark_pose) {
  const int T = ctx->cfg.tokens_per_frame, C = ctx->C;
  AppendParams p;
  p.Ksrc = K;
  p.Vsrc = V;
  p.stride = stride;
  p.keep_idx = keep_idx;
  p.hs = ctx->cfg.score_mode == WK_SCORE_PER_HEAD ? ctx->cfg.n_heads : 1;
  p.T = T;
  p.C = C;
  p.FT = ctx->FT;
  p.D = ctx->D;
  p.n = n;
  p.Kdst = pool_rows(ctx, ctx->Kpool, layer0, slot);
  p.Vdst = pool_rows(ctx, ctx->Vpool, layer0, slot);
  p.dst_layer_stride = static_cast<int64_t>(C) * ctx->D * ctx->cfg.pool_slots;
  p.k_row0 = stored && stored->k_done ? T : 0;
  p.v_row0 = stored ? T : 0;
  p.v_anchor_blocks = stored && !stored->v_done ? n * ((T + kAppendRows - 1) / kAppendRows) : 0;
  p.reverse = stored != nullptr;
  p.mark_slot = mark_pose ? slot : -1;
  p.valid = ctx->valid_dev;
  p.poses = ctx->poses_dev;
  for (int i = 0; i < 8; ++i) p.pose.v[i] = mark_pose ? mark_pose[i] : 0.f;
  p.status = ctx->status_dev;
  // Rows per block: every row of a warp is an index, then the row, then its stores, one after the other, so few layers are spread
  // over more blocks (one layer of 440 + 440 rows in a call of its own: 28 blocks 37.5 us, 110 blocks 32.9).
  const int64_t rows = static_cast<int64_t>(n) * (2 * C - p.k_row0 - p.v_row0);
  p.rows = rows < static_cast<int64_t>(kAppendRows) * 4 * ctx->sm_count ? kAppendThreads / 32 : kAppendRows;
  const int per_k = (C - p.k_row0 + p.rows - 1) / p.rows, per_v = (C - p.v_row0 + p.rows - 1) / p.rows;
  const dim3 grid(static_cast<unsigned>(p.v_anchor_blocks + n * (per_k + per_v)));
  if (stored) launch_chained(append_rows, grid, dim3(kAppendThreads), 0, s, p);
  else append_rows<<<grid, kAppendThreads, 0, s>>>(p);
  return after_launch(ctx);
}

wk_status launch_slot_mark(wk_ctx* ctx, int slot, int valid, const float* pose, cudaStream_t s) {
  Pose8 p;
  for (int i = 0; i < 8; ++i) p.v[i] = pose[i];
  slot_mark<<<1, 32, 0, s>>>(ctx->valid_dev, ctx->poses_dev, slot, valid, p);
  return after_launch(ctx);
}

}  // namespace wk
