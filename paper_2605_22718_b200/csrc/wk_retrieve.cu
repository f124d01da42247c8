// World Retrieval (Section 4.2, Eq. 4) with the camera distance of Section 5.1: squared-L2 translation
// distance and geodesic rotation angle to the current pose, each divided by its maximum over the stored
// chunks, summed; the k smallest win, ties to the lowest slot.  The whole pool is a few KB of poses, so one
// CTA does everything in fp64 in a single launch and the result stays in device memory for the attention call.
#include "wk_internal.cuh"

namespace wk {
namespace {

constexpr int kRetrieveThreads = 1024;

struct Pose8 { float v[8]; };

__device__ __forceinline__ double block_max(double v, double* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double r = red[0];
  for (int w = 1; w < kRetrieveThreads / 32; ++w) r = fmax(r, red[w]);
  return r;
}

__global__ void __launch_bounds__(kRetrieveThreads)
retrieve_kernel(const float* __restrict__ poses, const int32_t* __restrict__ valid, int n_slots, Pose8 cur, int k,
                int max_k, double* __restrict__ dist /*[2][n_slots]*/, int32_t* __restrict__ slots_out,
                double* __restrict__ dist_out, uint32_t* __restrict__ status /*may be null*/) {
  __shared__ double red[kRetrieveThreads / 32];
  const int tid = threadIdx.x;
  double* dt = dist;
  double* dr = dist + n_slots;
  double mt = 0.0, mr = 0.0;
  for (int s = tid; s < n_slots; s += kRetrieveThreads) {
    if (!valid[s]) { dt[s] = -1.0; continue; }     // negative marks "not a candidate"
    const float* p = poses + s * 8;
    const double dx = static_cast<double>(p[0]) - static_cast<double>(cur.v[0]);
    const double dy = static_cast<double>(p[1]) - static_cast<double>(cur.v[1]);
    const double dz = static_cast<double>(p[2]) - static_cast<double>(cur.v[2]);
    const double t = dx * dx + dy * dy + dz * dz;
    const double dot = static_cast<double>(p[4]) * cur.v[4] + static_cast<double>(p[5]) * cur.v[5] +
                       static_cast<double>(p[6]) * cur.v[6] + static_cast<double>(p[7]) * cur.v[7];
    if (!isfinite(t) || !isfinite(dot)) {          // a NaN/Inf pose (stored or current) is not a candidate
      dt[s] = -1.0;
      if (status) atomicOr(status, WK_DEV_NONFINITE);
      continue;
    }
    const double r = 2.0 * acos(fmin(1.0, fabs(dot)));    // q and -q are the same rotation
    dt[s] = t;
    dr[s] = r;
    mt = fmax(mt, t);
    mr = fmax(mr, r);
  }
  mt = block_max(mt, red);
  mr = block_max(mr, red);
  __syncthreads();
  // combined distance, each term normalised by its maximum over the candidates (a zero maximum drops the term)
  for (int s = tid; s < n_slots; s += kRetrieveThreads) {
    if (dt[s] < 0.0) continue;
    const double a = mt > 0.0 ? dt[s] / mt : 0.0;
    const double b = mr > 0.0 ? dr[s] / mr : 0.0;
    dr[s] = a + b;
  }
  for (int i = tid; i < max_k; i += kRetrieveThreads) {
    slots_out[i] = -1;
    if (dist_out) dist_out[i] = 0.0;
  }
  __syncthreads();
  // rank by counting: position of slot s = number of candidates that precede it under (distance, slot)
  for (int s = tid; s < n_slots; s += kRetrieveThreads) {
    if (dt[s] < 0.0) continue;
    const double d = dr[s];
    int rank = 0;
    for (int u = 0; u < n_slots; ++u) {
      if (dt[u] < 0.0) continue;
      const double du = dr[u];
      rank += (du < d) || (du == d && u < s);
    }
    if (rank < k) {
      slots_out[rank] = s;
      if (dist_out) dist_out[rank] = d;
    }
  }
}

// Pools of at most 1,024 slots: a thread per slot, distances in registers and shared memory, nothing goes through global
// memory but the poses and the result.  Bound by latency: launch, one trip to memory, the fp64 acos and two divisions, two
// block-wide reductions.  Non-negative doubles order like their bit patterns, so maxima and ranks are taken on integers.
// The same operations in the same order as retrieve_kernel, hence the same distances.  250 slots, back to back: 14.3 us with
// retrieve_kernel (distances through global memory, a rank loop of dependent global loads), 5.3 us here.
constexpr int kSmallSlots = 1024;

__device__ __forceinline__ unsigned long long warp_max_bits(unsigned long long v) {
  const uint32_t hi = static_cast<uint32_t>(v >> 32), mhi = __reduce_max_sync(0xffffffffu, hi);
  const uint32_t mlo = __reduce_max_sync(0xffffffffu, hi == mhi ? static_cast<uint32_t>(v) : 0u);
  return (static_cast<unsigned long long>(mhi) << 32) | mlo;
}

// The slots that may be among the k first under (key, slot), with their ranks.  A key is ascending, kNone for a slot that is no
// candidate (and for threads without one).
constexpr unsigned long long kNone = ~0ull;
struct BestSlots {
  unsigned long long group[kSmallSlots / 8], key[kSmallSlots], cut;
  int slot[kSmallSlots], rank[kSmallSlots], n;
};
// Called by the whole block (slot tid's key comes from thread tid; as many threads as slots at least), a block barrier after
// rank_begin; returns the number of entries in sh.  Ranks come from counting comparisons, which all slots against all others would make most of a kernel's time (250
// slots: 8,900 of 12,600 clocks).  So a cut first: the k-th smallest of the minima of groups of eight slots has at least k
// slots at or below it and leaves few more.  250 slots, k = 8: 6.85 -> 5.28 us per call; 1,000 slots 13.6 -> 5.2.  Where the block
// has threads enough for all comparisons at once the cut costs more (two barriers) than it saves; all slots are entries then, in place (through
// the list, query retrieval over 16 and 64 slots: 13.3 and 17.8 us a call, in place 13.1 and 17.4).
__device__ __forceinline__ void rank_begin(BestSlots& sh) {
  sh.rank[threadIdx.x] = 0;
  if (threadIdx.x == 0) { sh.cut = kNone - 1; sh.n = 0; }
}
__device__ __forceinline__ int rank_best(BestSlots& sh, unsigned long long key, int n_slots, int k) {
  const int tid = threadIdx.x;
  const bool cut = n_slots * n_slots > 16 * static_cast<int>(blockDim.x);
  if (cut) {
    unsigned long long g = key;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
      const unsigned long long v = __shfl_xor_sync(0xffffffffu, g, o);
      g = v < g ? v : g;
    }
    const int n_groups = (n_slots + 7) >> 3;
    if ((tid & 7) == 0 && (tid >> 3) < n_groups) sh.group[tid >> 3] = g;
    __syncthreads();
    if (tid < n_groups && k <= n_groups) {
      const unsigned long long kg = sh.group[tid];
      int rank = 0;
#pragma unroll 8
      for (int u = 0; u < n_groups; ++u) {
        const unsigned long long ku = sh.group[u];
        rank += static_cast<int>(ku < kg) | (static_cast<int>(ku == kg) & static_cast<int>(u < tid));
      }
      if (rank == k - 1 && kg != kNone) sh.cut = kg;
    }
    __syncthreads();
  }
  if (!cut && tid < n_slots) {   // all slots are entries, and one that is no candidate gets no rank that counts
    sh.key[tid] = key;
    sh.slot[tid] = tid;
    if (key == kNone) sh.rank[tid] = 1 << 30;
  } else if (cut && key <= sh.cut) {
    const int pos = atomicAdd(&sh.n, 1);
    sh.key[pos] = key;
    sh.slot[pos] = tid;
  }
  __syncthreads();
  // The block's threads share the comparisons: P of them per entry, each with every P-th of the others.
  const int n = cut ? sh.n : n_slots;
  int shift = 0;
  while (shift < 4 && (n << (shift + 1)) <= static_cast<int>(blockDim.x)) ++shift;
  const int P = 1 << shift, e = tid >> shift;
  if (e < n) {
    const unsigned long long ke = sh.key[e];
    const int se = sh.slot[e];
    int rank = 0;
#pragma unroll 4
    for (int u = tid & (P - 1); u < n; u += P) {
      const unsigned long long ku = sh.key[u];
      const int su = sh.slot[u];
      rank += static_cast<int>(ku < ke) | (static_cast<int>(ku == ke) & static_cast<int>(su < se));
    }
    if (rank) atomicAdd(&sh.rank[e], rank);
  }
  __syncthreads();
  return n;
}

template <bool kVec>   // kVec: poses are 16-byte aligned
__global__ void __launch_bounds__(kSmallSlots)
retrieve_small(const float* __restrict__ poses, const int32_t* __restrict__ valid, int n_slots, Pose8 cur, int k, int max_k,
               int32_t* __restrict__ slots_out, double* __restrict__ dist_out, uint32_t* __restrict__ status /*may be null*/) {
  __shared__ unsigned long long s_t[32], s_r[32];
  __shared__ BestSlots sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  rank_begin(sh);
  dep_wait();
  dep_release();
  double t = 0.0, r = 0.0;
  bool cand = false;
  if (tid < n_slots) {
    float p[8];
    if (kVec) {
      const float4 a = ld_dep(reinterpret_cast<const float4*>(poses) + 2 * tid), b = ld_dep(reinterpret_cast<const float4*>(poses) + 2 * tid + 1);
      p[0] = a.x; p[1] = a.y; p[2] = a.z; p[4] = b.x; p[5] = b.y; p[6] = b.z; p[7] = b.w;
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) p[i] = ld_dep(poses + tid * 8 + i);
    }
    if (ld_dep(valid + tid)) {
      const double dx = static_cast<double>(p[0]) - static_cast<double>(cur.v[0]);
      const double dy = static_cast<double>(p[1]) - static_cast<double>(cur.v[1]);
      const double dz = static_cast<double>(p[2]) - static_cast<double>(cur.v[2]);
      t = dx * dx + dy * dy + dz * dz;
      const double dot = static_cast<double>(p[4]) * cur.v[4] + static_cast<double>(p[5]) * cur.v[5] +
                         static_cast<double>(p[6]) * cur.v[6] + static_cast<double>(p[7]) * cur.v[7];
      cand = isfinite(t) && isfinite(dot);
      if (cand) {
        r = 2.0 * acos(fmin(1.0, fabs(dot)));    // q and -q are the same rotation
      } else {                                   // a NaN/Inf pose (stored or current) is not a candidate
        t = 0.0;
        if (status) atomicOr(status, WK_DEV_NONFINITE);
      }
    }
  }
  const unsigned long long wt = warp_max_bits(static_cast<unsigned long long>(__double_as_longlong(t)));
  const unsigned long long wr = warp_max_bits(static_cast<unsigned long long>(__double_as_longlong(r)));
  if (lane == 0) { s_t[warp] = wt; s_r[warp] = wr; }
  for (int i = tid; i < max_k; i += blockDim.x) {
    slots_out[i] = -1;
    if (dist_out) dist_out[i] = 0.0;
  }
  __syncthreads();
  const int nw = blockDim.x >> 5;
  const double mt = __longlong_as_double(static_cast<long long>(warp_max_bits(lane < nw ? s_t[lane] : 0ull)));
  const double mr = __longlong_as_double(static_cast<long long>(warp_max_bits(lane < nw ? s_r[lane] : 0ull)));
  // combined distance, each term normalised by its maximum over the candidates (a zero maximum drops the term)
  const double a = mt > 0.0 ? t / mt : 0.0;
  const double b = mr > 0.0 ? r / mr : 0.0;
  const double d = a + b;
  const int n = rank_best(sh, cand ? static_cast<unsigned long long>(__double_as_longlong(d)) : kNone, n_slots, k);
  if (tid < n && sh.rank[tid] < k) {
    slots_out[sh.rank[tid]] = sh.slot[tid];
    if (dist_out) dist_out[sh.rank[tid]] = __longlong_as_double(static_cast<long long>(sh.key[tid]));
  }
}

// ---- query-based retrieval (Appendix C) --------------------------------------------------------------------------
// lse[slot][h][r] holds, for every valid slot, the log-sum-exp of query row r of head h over that slot's stored keys.
// The softmax mass of a slot for (h, r) is exp(lse[slot] - logsumexp over slots); a slot's score is the mean mass.
// query_mass: a block takes 256 (h, r) columns, eight warps side by side; four warps share a column group's slots.  Each
// warp first takes the running maximum and sum of its slots, eight loads in flight, the four shares meet in shared memory,
// and a second walk (the values come from L2 now) turns them into masses, added over the warp's columns by shuffles and over
// the block in a fixed order: one partial per (block, slot), no floating-point atomics, so the ranking is reproducible.
// Bound by reading the LSEs twice; 250 slots x 31,680 columns: one thread per column with three serial walks 116 us.
constexpr int kMassCols = 256, kMassThreads = 1024, kMassShares = 4;

__global__ void __launch_bounds__(kMassThreads)
query_mass(const float* __restrict__ lse, const int32_t* __restrict__ valid, int n_slots, int n_hr,
           double* __restrict__ block_part /*[gridDim.x][n_slots]*/) {
  extern __shared__ float s_dyn[];                       // [8 column groups][n_slots] masses, then n_slots validity words
  __shared__ float s_mx[kMassShares][kMassCols], s_den[kMassShares][kMassCols];
  float* s_mass = s_dyn;
  int32_t* s_valid = reinterpret_cast<int32_t*>(s_dyn + 8 * n_slots);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int cg = warp & 7, share = warp >> 3, col = cg * 32 + lane;
  const int i = blockIdx.x * kMassCols + col;
  const bool live = i < n_hr;
  const float* mine = lse + (live ? i : 0);
  dep_wait();
  dep_release();
  for (int s = tid; s < n_slots; s += kMassThreads) s_valid[s] = valid[s];
  __syncthreads();
  float mx = -INFINITY, den = 0.f;
  for (int s0 = share; s0 < n_slots; s0 += 8 * kMassShares) {
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int s = s0 + k * kMassShares;
      v[k] = s < n_slots && s_valid[s] ? __ldcg(mine + static_cast<int64_t>(s) * n_hr) : -INFINITY;
    }
    float m8 = mx;
#pragma unroll
    for (int k = 0; k < 8; ++k) m8 = fmaxf(m8, v[k]);
    if (m8 > -INFINITY) {
      float add = 0.f;
#pragma unroll
      for (int k = 0; k < 8; ++k) add += expf(v[k] - m8);
      den = den * expf(mx - m8) + add;
      mx = m8;
    }
  }
  s_mx[share][col] = mx;
  s_den[share][col] = den;
  __syncthreads();
  mx = fmaxf(fmaxf(s_mx[0][col], s_mx[1][col]), fmaxf(s_mx[2][col], s_mx[3][col]));
  den = 0.f;
  if (mx > -INFINITY) {
#pragma unroll
    for (int k = 0; k < kMassShares; ++k) den += s_den[k][col] * expf(s_mx[k][col] - mx);
  }
  const float inv = (live && den > 0.f) ? 1.f / den : 0.f;
  for (int s0 = share; s0 < n_slots; s0 += 8 * kMassShares) {
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int s = s0 + k * kMassShares;
      v[k] = s < n_slots && s_valid[s] ? __ldcg(mine + static_cast<int64_t>(s) * n_hr) : -INFINITY;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int s = s0 + k * kMassShares;
      float m = inv > 0.f ? expf(v[k] - mx) * inv : 0.f;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
      if (lane == 0 && s < n_slots) s_mass[cg * n_slots + s] = m;
    }
  }
  __syncthreads();
  for (int s = tid; s < n_slots; s += kMassThreads) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += static_cast<double>(s_mass[w * n_slots + s]);
    block_part[static_cast<int64_t>(blockIdx.x) * n_slots + s] = t;
  }
}

// One CTA: adds the blocks' partials in a fixed order, ranks the valid slots by (score descending, slot ascending).  1024
// threads share the slots: P of them per slot, each with every P-th block and every P-th comparison.
__global__ void __launch_bounds__(1024)
query_topk(const double* __restrict__ block_part, int n_blocks, const int32_t* __restrict__ valid, int n_slots, int n_hr,
           int k, int max_k, int32_t* __restrict__ slots_out, float* __restrict__ score_out) {
  __shared__ double part[1024];
  __shared__ BestSlots sh;
  const int tid = threadIdx.x;
  int P = 1;
  while (P < 8 && n_slots * P * 2 <= 1024) P <<= 1;
  const int s = tid % n_slots, q = tid / n_slots;   // slot and share (threads with q >= P idle)
  rank_begin(sh);
  dep_wait();
  for (int i = tid; i < max_k; i += 1024) {
    slots_out[i] = -1;
    if (score_out) score_out[i] = 0.f;
  }
  double t = 0.0;
  if (q < P) {
#pragma unroll 8
    for (int b = q; b < n_blocks; b += P) t += __ldcg(block_part + static_cast<int64_t>(b) * n_slots + s);
  }
  part[tid] = t;
  __syncthreads();
  constexpr unsigned long long kTop = ~0ull >> 1;
  unsigned long long key = kNone;   // ascending as the scores descend
  if (q == 0) {
    for (int w = 1; w < P; ++w) t += part[w * n_slots + s];
    const double v = valid[s] ? t / static_cast<double>(n_hr) : -1.0;   // negative marks "not a candidate"
    if (v >= 0.0) key = kTop - static_cast<unsigned long long>(__double_as_longlong(v + 0.0));   // never kNone
  }
  const int n = rank_best(sh, key, n_slots, k);
  if (tid < n && sh.rank[tid] < k) {
    slots_out[sh.rank[tid]] = sh.slot[tid];
    if (score_out) score_out[sh.rank[tid]] = static_cast<float>(__longlong_as_double(static_cast<long long>(kTop - sh.key[tid])));
  }
}

// Scratch of the allocation-free entry point: two doubles per slot, held by every GPU that loads the library.
constexpr int kStaticMaxSlots = 4096;
static __device__ __align__(256) double g_retrieve_scratch[2 * kStaticMaxSlots];

}  // namespace

// threads of retrieve_small: one per slot
static unsigned small_threads(int n_slots) {
  unsigned t = 128;
  while (t < kSmallSlots && t < static_cast<unsigned>(n_slots)) t <<= 1;
  return t;
}

wk_status launch_retrieve(wk_ctx* ctx, const float* cur_pose, int k, int32_t* slots_out, double* dist_out,
                          cudaStream_t s) {
  Pose8 cur;
  for (int i = 0; i < 8; ++i) cur.v[i] = cur_pose[i];
  if (ctx->cfg.pool_slots <= kSmallSlots) {
    launch_chained(retrieve_small<true>, dim3(1), dim3(small_threads(ctx->cfg.pool_slots)), 0, s, ctx->poses_dev, ctx->valid_dev,
                   ctx->cfg.pool_slots, cur, k, ctx->cfg.max_k, slots_out, dist_out, ctx->status_dev);
    return after_launch(ctx);
  }
  double* dist = reinterpret_cast<double*>(ctx->scratch_base + ctx->sl.dist_off);
  retrieve_kernel<<<1, kRetrieveThreads, 0, s>>>(ctx->poses_dev, ctx->valid_dev, ctx->cfg.pool_slots, cur, k,
                                                 ctx->cfg.max_k, dist, slots_out, dist_out, ctx->status_dev);
  return after_launch(ctx);
}

wk_status launch_retrieve_query(wk_ctx* ctx, int layer, const __nv_bfloat16* Q, int lq, int k, int32_t* slots_out,
                                float* score_out, cudaStream_t s) {
  const int H = ctx->cfg.n_heads, S = ctx->cfg.pool_slots, n_hr = H * lq;
  float* lse = reinterpret_cast<float*>(ctx->scratch_base + ctx->sl.qr_lse_off);
  const int32_t* ids = reinterpret_cast<const int32_t*>(ctx->scratch_base + ctx->sl.qr_ids_off);
  double* part = reinterpret_cast<double*>(ctx->scratch_base + ctx->sl.qr_part_off);
  // log-sum-exp of the query over each stored chunk alone: the attention kernel in its LSE-only mode, every pool slot a
  // problem of its own in one launch (slots that hold nothing come back as -inf and are masked by the valid flags)
  wk_status st = launch_attention(ctx, layer, Q, lq, nullptr, 0, ids, S, nullptr, lse, 1, s, true);
  if (st != WK_OK) return st;
  const int blocks = (n_hr + kMassCols - 1) / kMassCols;
  launch_chained(query_mass, dim3(blocks), dim3(kMassThreads), static_cast<size_t>(9) * S * sizeof(float), s, lse, ctx->valid_dev, S,
                 n_hr, part);
  if ((st = after_launch(ctx)) != WK_OK) return st;
  launch_chained(query_topk, dim3(1), dim3(1024), 0, s, part, blocks, ctx->valid_dev, S, n_hr, k, ctx->cfg.max_k, slots_out, score_out);
  return after_launch(ctx);
}

}  // namespace wk

extern "C" wk_status wk_retrieve_noalloc(const float* poses_dev, const int32_t* valid_dev, int32_t n_slots,
                                         const float* cur_pose_host, int32_t k, int32_t max_k, int32_t* slots_out_dev,
                                         double* dist_out_dev, void* stream) {
  using namespace wk;
  if (!poses_dev || !valid_dev || !cur_pose_host || !slots_out_dev) return WK_ERR_ARG;
  if (n_slots < 0 || k < 0 || max_k < 1 || k > max_k) return WK_ERR_ARG;
  if (n_slots > kStaticMaxSlots) return WK_ERR_SHAPE;   // the built-in scratch holds 4096 slots and cannot grow
  // Set-up, once per device and with that device current: in host code the array's name is only a stand-in, the
  // device address has to be asked for.
  static double* scratch_of_device[64] = {};
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return WK_ERR_NO_DEVICE;
  if (!scratch_of_device[dev]) {
    double* ptr = nullptr;
    if (cudaGetSymbolAddress(reinterpret_cast<void**>(&ptr), g_retrieve_scratch) != cudaSuccess || !ptr) return WK_ERR_CUDA;
    scratch_of_device[dev] = ptr;
  }
  Pose8 cur;
  for (int i = 0; i < 8; ++i) cur.v[i] = cur_pose_host[i];
  if (n_slots > 0 && n_slots <= kSmallSlots) {
    const bool vec = (reinterpret_cast<uintptr_t>(poses_dev) & 15u) == 0;
    auto* kernel = vec ? retrieve_small<true> : retrieve_small<false>;
    kernel<<<1, small_threads(n_slots), 0, static_cast<cudaStream_t>(stream)>>>(poses_dev, valid_dev, n_slots, cur, k, max_k,
                                                                                slots_out_dev, dist_out_dev, nullptr);
    return cudaGetLastError() == cudaSuccess ? WK_OK : WK_ERR_CUDA;
  }
  retrieve_kernel<<<1, kRetrieveThreads, 0, static_cast<cudaStream_t>(stream)>>>(
      poses_dev, valid_dev, n_slots, cur, k, max_k, scratch_of_device[dev], slots_out_dev, dist_out_dev, nullptr);
  return cudaGetLastError() == cudaSuccess ? WK_OK : WK_ERR_CUDA;
}
