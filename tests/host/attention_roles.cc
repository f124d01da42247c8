// The roles of an attention CTA (csrc/wk_attention.cu) on the host.  roles.inc is that file up to its first kernel, with its PTX
// taken out; this file stands in for the PTX: barriers with arrivals, bytes and phases, and asynchronous copies and matrix products
// that land whenever the schedule says so.  Every warp is a fiber that computes its lane 0 (one query row of 32), and a schedule
// decides at every barrier operation who goes on.  Keys, queries and values have one component.  Reported are memory that is read
// or written while a copy or a product in flight writes or reads it, arrivals that a barrier does not expect, waits that never
// end, and outputs other than the softmax of the rows that the piece should have seen.
#include <math.h>
#include <stdio.h>
#include <string.h>
#include <ucontext.h>

#include <algorithm>
#include <deque>
#include <map>
#include <random>
#include <string>
#include <vector>

#include "wk_internal.cuh"

#define WK_ASM(...)
using std::max;
using std::min;
struct Index { unsigned x; };
static Index threadIdx, blockIdx, gridDim;
static inline float __uint_as_float(uint32_t u) { float f; memcpy(&f, &u, 4); return f; }
static inline uint32_t __float_as_uint(float f) { uint32_t u; memcpy(&u, &f, 4); return u; }
static inline void __syncwarp() {}
static inline bool __any_sync(unsigned, bool x) { return x; }
static inline int __reduce_add_sync(unsigned, int x) { return x; }
static inline void atomicOr(uint32_t* p, uint32_t v) { *p |= v; }

namespace wk {
static std::string fault;
static void fail(const std::string& what) { if (fault.empty()) fault = what; }

// ------------------------------------------------------------------ fibers and schedule
struct Bar { int count, left; long bytes; uint32_t phase; };
static std::map<const void*, Bar> bars;
static Bar& bar_at(const void* b) {
  auto it = bars.find(b);
  if (it == bars.end()) { fail("a barrier that was not initialised"); return bars[b]; }
  return it->second;
}
static void settle(Bar& b) {
  if (b.left < 0) fail("an arrival that the barrier does not expect");
  if (b.left == 0 && b.bytes == 0) { ++b.phase; b.left = b.count; }
}
struct Fiber {
  ucontext_t ctx;
  std::vector<char> stack;
  bool done;
  const void* bar;   // waits for this barrier's phase of this parity, if any
  uint32_t parity;
  unsigned thread;
};
static std::vector<Fiber> fibers;
static ucontext_t scheduler;
static int current;
static bool stuck;
static bool passes(const void* bar, uint32_t parity) { return (bar_at(bar).phase & 1) != parity; }
static void pause() {
  Fiber& f = fibers[current];
  swapcontext(&f.ctx, &scheduler);
}

// ------------------------------------------------------------------ memory
constexpr int kMaxRows = 128;
static float q_mem[2][4], k_mem[8][kMaxRows], v_mem[8][kMaxRows];   // one row per softmax warp; rows of a stage
static uint32_t tmem[4][512];
struct Use { int writes, reads; };
static Use q_use[2], k_use[8], v_use[8], t_use[512];
struct Copy { int what, at; std::vector<float> rows; uint32_t bytes; void* bar; };   // what: 0 Q, 1 K, 2 V, 3 (second half of a row) none
static std::deque<Copy> copies;
struct Product { bool pv; int qt, st, k, d, n; bool add; };
struct Commit { std::vector<Product> products; void* bar; };
static std::vector<Product> issued[2];
static std::deque<Commit> commits[2];
static int mma_warp;   // first MMA warp
static uint8_t* arena;
static uint32_t offset(const void* p) { return static_cast<uint32_t>(static_cast<const uint8_t*>(p) - arena); }
static Use& use_of(int what, int at) { return what == 0 ? q_use[at] : what == 1 ? k_use[at] : v_use[at]; }

namespace ptx {
static uint32_t smem_u32(const void* p) { return offset(p); }
static void mbar_init(uint64_t* b, int count) { bars[b] = {count, count, 0, 0}; }
static void mbar_arrive(uint64_t* b) {
  pause();
  Bar& x = bar_at(b);
  --x.left;
  settle(x);
}
static void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  pause();
  Bar& x = bar_at(b);
  x.bytes += bytes;
  --x.left;
  settle(x);
}
static bool mbar_try_wait(uint64_t*, uint32_t) { return true; }   // draining after an abort
static bool wait_or_abort(uint64_t* b, uint32_t parity, volatile uint32_t* abort) {
  Fiber& f = fibers[current];
  do {
    f.bar = b;
    f.parity = parity;
    pause();
    f.bar = nullptr;
    if (stuck || *abort) return false;
  } while (!passes(b, parity));
  return true;
}
static void fence_mbar_init() {}
static void tc_fence_before() {}
static void tc_fence_after() {}
template <class R> static void tc_wait_ld(R&) {}
template <class R> static void pin_x32(R&) {}
template <class R> static void pin_x16(R&) {}
static void tc_wait_st() {}
static bool elect_one() { return true; }
static constexpr uint32_t smem_desc_hi_sw128(uint32_t) { return 0; }
static uint32_t smem_desc_lo(uint32_t addr, uint32_t) { return addr >> 4; }
static constexpr uint32_t idesc_bf16_f32(uint32_t, uint32_t, int, int) { return 0; }
static void mma_ss_if(uint32_t, uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t add);
static void mma_ts_if(uint32_t, uint32_t d, uint32_t a, uint64_t b, uint32_t, uint32_t add);
static void mma_commit_if(uint32_t, uint32_t bar) {
  pause();
  const int w = threadIdx.x / 32 - mma_warp;
  commits[w].push_back({issued[w], arena + bar});
  issued[w].clear();
}
static void tma_load_2d(void* dst, const CUtensorMap* m, uint64_t* bar, int x, int y);
static void tma_load_3d(void* dst, const CUtensorMap* m, uint64_t* bar, int x, int y, int z);
template <int N> static void load(uint32_t addr, uint32_t* r) {
  for (int i = 0; i < N; ++i) {
    if (t_use[(addr & 0xffff) + i].writes) fail("tensor memory read before a product has written it");
    r[i] = tmem[addr >> 21][(addr & 0xffff) + i];
  }
}
template <int N> static void store(uint32_t addr, const uint32_t* r) {
  for (int i = 0; i < N; ++i) {
    const Use& u = t_use[(addr & 0xffff) + i];
    if (u.writes || u.reads) fail("tensor memory written under a product that uses it");
    tmem[addr >> 21][(addr & 0xffff) + i] = r[i];
  }
}
static void tmem_ld_x32(uint32_t a, uint32_t (&r)[32]) { load<32>(a, r); }
static void tmem_ld_x16(uint32_t a, uint32_t (&r)[16]) { load<16>(a, r); }
static void tmem_st_x32(uint32_t a, const uint32_t (&r)[32]) { store<32>(a, r); }
static void tmem_st_x8(uint32_t a, const uint32_t (&r)[8]) { store<8>(a, r); }
static float ex2_approx(float x) { return exp2f(x); }
static uint64_t pack_f32x2(float a, float b) { return static_cast<uint64_t>(__float_as_uint(b)) << 32 | __float_as_uint(a); }
static void unpack_f32x2(uint64_t v, float& a, float& b) { a = __uint_as_float(static_cast<uint32_t>(v)); b = __uint_as_float(v >> 32); }
static uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
  float x[6];
  unpack_f32x2(a, x[0], x[1]); unpack_f32x2(b, x[2], x[3]); unpack_f32x2(c, x[4], x[5]);
  return pack_f32x2(fmaf(x[0], x[2], x[4]), fmaf(x[1], x[3], x[5]));
}
static uint64_t add_f32x2(uint64_t a, uint64_t b) { return fma_f32x2(a, pack_f32x2(1.f, 1.f), b); }
static uint32_t bf16_bits(float f) { const uint32_t u = __float_as_uint(f); return (u + 0x7fff + ((u >> 16) & 1)) >> 16; }
static uint32_t pack_bf16x2(float lo, float hi) { return bf16_bits(hi) << 16 | bf16_bits(lo); }
static void st_global_x8(void* dst, const uint32_t* v) { memcpy(dst, v, 32); }
}  // namespace ptx
static void dep_wait() {}
static void dep_release() {}
template <class T> static T ld_dep(const T* p) { return *p; }
static float fmax3(float a, float b, float c) { return fmaxf(fmaxf(a, b), c); }
static float fmax3_nan(float a, float b, float c) { return a != a || b != b || c != c ? NAN : fmax3(a, b, c); }
}  // namespace wk

#include "roles.inc"   // opens namespace wk and an unnamed one and leaves them open

AttnParams par;
constexpr int kRows = WK_TEST_ROWS;   // of a KV tile: picks the instantiation
constexpr bool kL = is_lse<kRows>;
struct Arena {
  alignas(1024) uint8_t smem[kSmemBytes<kRows>];
  CtaShared<kRows> sh;
} ar;

int count_tiles(const AttnParams& p, int tb, int te) {
  TileIter it;
  TileInfo ti;
  it.init(p, tb, te);
  int n = 0;
  while (it.next(p, ti, false)) ++n;
  return n;
}

// What stands in the rows of the inputs: pseudo-random numbers of (which, segment or matrix, head, row).
float value(int which, int seg, int h, int row) {
  uint32_t x = 2654435761u * (which + 1) + 40503u * (seg + 7) + 97u * h + row * 2246822519u;
  x ^= x >> 15; x *= 2246822519u; x ^= x >> 13; x *= 3266489917u; x ^= x >> 16;
  const float u = x * 0x1p-32f;
  return which == 0 ? 0.5f + u : which == 1 ? 6.f * u - 3.f : (row / 16 % 3 - 1.f) * 2.f + u;
}
int rows_of(int seg) { return seg < par.n_segs ? par.seg_rows[seg] : par.C; }   // matrices of the pool: n_segs + z

// ------------------------------------------------------------------ copies and products
void start_copy(void* dst, uint64_t* bar, int what_in, int seg, int x, int y) {
  pause();
  const uint32_t at = offset(dst);
  Copy c;
  c.bar = bar;
  const bool is_q = at < 2 * kQBytes;
  c.bytes = is_q ? kHalfQBytes : kHalfKvBytes<kRows>;
  if (x % 128) {
    c.what = 3;
    c.at = 0;
  } else {
    const int h = x / 128, in = at - 2 * kQBytes;
    c.what = is_q ? 0 : in % kStageBytes<kRows> >= kKvBytes<kRows> ? 2 : 1;
    c.at = is_q ? at / kQBytes : in / kStageBytes<kRows>;
    if (!is_q && c.what != what_in) fail("K where V belongs");
    for (int r = 0; r < (is_q ? 4 : kRows); ++r) {
      const int row = y + (is_q ? 32 * r : r);
      c.rows.push_back(row < (is_q ? par.lq : rows_of(seg)) ? value(c.what, is_q ? 0 : seg, h, row) : 0.f);
    }
    Use& u = use_of(c.what, c.at);
    if (u.writes || u.reads) fail("a copy into memory in use");
    ++u.writes;
  }
  copies.push_back(c);
}
void end_copy(int i) {
  const Copy c = copies[i];
  copies.erase(copies.begin() + i);
  if (c.what < 3) {
    float* to = c.what == 0 ? q_mem[c.at] : c.what == 1 ? k_mem[c.at] : v_mem[c.at];
    std::copy(c.rows.begin(), c.rows.end(), to);
    --use_of(c.what, c.at).writes;
  }
  Bar& b = bar_at(c.bar);
  b.bytes -= c.bytes;
  settle(b);
}
float bf16(uint32_t bits) { return __uint_as_float(bits << 16); }
void mark(const Product& p, int by) {
  for (int i = 0; i < (p.pv ? 128 : p.n); ++i) t_use[p.d + i].writes += by;
  if (p.pv) for (int i = 0; i < 8; ++i) t_use[kTmemP + p.qt * 128 + p.k * 8 + i].reads += by;
  if (!p.pv) q_use[p.qt].reads += by;
  (p.pv ? v_use : k_use)[p.st].reads += by;
}
void issue(const Product& p) {
  if ((p.pv ? v_use : k_use)[p.st].writes || (!p.pv && q_use[p.qt].writes)) fail("a product reads what a copy still writes");
  if (p.pv) for (int i = 0; i < 8; ++i) if (t_use[kTmemP + p.qt * 128 + p.k * 8 + i].writes) fail("P is still being written");
  mark(p, 1);
  issued[threadIdx.x / 32 - mma_warp].push_back(p);
}
void end_commit(int w) {
  const Commit c = commits[w].front();
  commits[w].pop_front();
  for (const Product& p : c.products) {
    mark(p, -1);
    for (int q = 0; q < 4; ++q) {
      uint32_t* t = tmem[q] + p.d;
      if (!p.pv) {
        for (int i = 0; i < p.n; ++i) t[i] = __float_as_uint(q_mem[p.qt][q] * k_mem[p.st][i]);
      } else {
        float sum = p.add ? __uint_as_float(t[0]) : 0.f;
        for (int i = 0; i < 16; ++i) {
          const uint32_t pair = tmem[q][kTmemP + p.qt * 128 + p.k * 8 + i / 2];
          sum += bf16(i & 1 ? pair >> 16 : pair & 0xffff) * v_mem[p.st][p.k * 16 + i];
        }
        for (int i = 0; i < 128; ++i) t[i] = __float_as_uint(sum);
      }
    }
  }
  Bar& b = bar_at(c.bar);
  --b.left;
  settle(b);
}
}  // namespace
namespace ptx {
static void mma_ss_if(uint32_t, uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t add) {
  if (add) return;   // the first of the eight K = 16 steps stands for all of them
  issue({false, static_cast<int>((a << 4) / kQBytes), static_cast<int>(((b << 4) - 2 * kQBytes) / kStageBytes<kRows>), 0,
         static_cast<int>(d), static_cast<int>(idesc >> 18) * 16, false});
}
static void mma_ts_if(uint32_t, uint32_t d, uint32_t a, uint64_t b, uint32_t, uint32_t add) {
  const uint32_t at = static_cast<uint32_t>(b << 4) - 2 * kQBytes;
  issue({true, static_cast<int>((d - kTmemO) / 128), static_cast<int>(at / kStageBytes<kRows>),
         static_cast<int>((at % kStageBytes<kRows> - kKvBytes<kRows>) / 2048), static_cast<int>(d), 0, add != 0});
  if (a != kTmemP + (d - kTmemO) + (at % kStageBytes<kRows> - kKvBytes<kRows>) / 2048 * 8) fail("P of another step");
}
static void tma_load_2d(void* dst, const CUtensorMap* m, uint64_t* bar, int x, int y) {
  const int k = static_cast<int>(m - par.tm_kd), v = static_cast<int>(m - par.tm_vd);
  if (m == &par.tm_q) start_copy(dst, bar, 0, 0, x, y);
  else if (k >= 0 && k < kMaxDenseSegs) start_copy(dst, bar, 1, k, x, y);
  else start_copy(dst, bar, 2, v, x, y);
}
static void tma_load_3d(void* dst, const CUtensorMap* m, uint64_t* bar, int x, int y, int z) {
  start_copy(dst, bar, m == &par.tm_kpool ? 1 : 2, par.n_segs + z, x, y);
}
}  // namespace ptx
namespace {

void fiber_main() {
  attention_roles<kRows>(par, ar.sh, ar.smem);
  fibers[current].done = true;
  for (;;) pause();
}

// One CTA's work under one schedule.  hold: the fiber (or, from the number of fibers on: the copies, the products of MMA warp 0, 1)
// that does not move from its `from`-th turn on until nothing else can; -1: a random one each time.  Returns the held one's turns.
int run_cta(int hold, int from, unsigned seed) {
  const int n = kThreads<kRows> / 32;
  bars.clear();
  copies.clear();
  memset(q_use, 0, sizeof(q_use)); memset(k_use, 0, sizeof(k_use)); memset(v_use, 0, sizeof(v_use)); memset(t_use, 0, sizeof(t_use));
  memset(tmem, 0xff, sizeof(tmem));
  for (int w = 0; w < 2; ++w) { issued[w].clear(); commits[w].clear(); }
  memset(static_cast<void*>(&ar.sh), 0, sizeof(ar.sh));
  init_barriers<kRows>(ar.sh);
  ar.sh.abort = 0;
  stuck = false;
  fibers.resize(n);
  for (int i = 0; i < n; ++i) {
    Fiber& f = fibers[i];
    f.stack.resize(1 << 16);
    f.done = false;
    f.bar = nullptr;
    f.thread = 32 * i;
    getcontext(&f.ctx);
    f.ctx.uc_stack.ss_sp = f.stack.data();
    f.ctx.uc_stack.ss_size = f.stack.size();
    f.ctx.uc_link = nullptr;
    makecontext(&f.ctx, fiber_main, 0);
  }
  std::mt19937 rng(seed);
  int turns = 0, last = 0;
  for (int step = 0; fault.empty() && step < 1000000; ++step) {
    int can[64], m = 0;
    bool alive = false, held = false;
    for (int i = 0; i < n + 3; ++i) {
      const bool ok = i < n ? !fibers[i].done && (!fibers[i].bar || stuck || ar.sh.abort || passes(fibers[i].bar, fibers[i].parity))
                            : i == n ? !copies.empty() : !commits[i - n - 1].empty();
      alive = alive || (i < n && !fibers[i].done);
      if (!ok) continue;
      if (i == hold && turns >= from) held = true;
      else can[m++] = i;
    }
    if (!alive) break;
    int who;
    if (m == 0) {
      if (!held) {
        if (stuck) break;
        fail("a wait that never ends");
        break;
      }
      who = hold;
      from = 1 << 30;   // it has been held once
    } else if (hold < 0) {
      who = can[rng() % m];
    } else {
      who = can[0];
      for (int i = 0; i < m; ++i) if (can[i] > last) { who = can[i]; break; }   // in turns
      last = who;
    }
    if (who == hold) ++turns;
    if (who < n) {
      current = who;
      threadIdx.x = fibers[who].thread;
      swapcontext(&scheduler, &fibers[who].ctx);
    } else if (who == n) {
      end_copy(hold < 0 ? rng() % copies.size() : 0);
    } else {
      end_commit(who - n - 1);
    }
  }
  return turns;
}
}  // namespace
}  // namespace wk

using namespace wk;

// All CTAs of a call of H heads x lq queries over dense segments of seg_rows[] keys and pool slots (slot_ids[], -1 or a stale slot
// among them), C rows each; n_full units whole, the others in n_ranges ranges, on `grid` CTAs.  schedules random schedules, and, where
// hold is set, one for every turn of every role.  Returns 0, or 1 with what went wrong in `what`.
extern "C" int run_roles(int H, int lq, const int* seg_rows, int n_segs, const int* slot_ids, int n_slots, int C, int n_full, int n_ranges,
                         int grid, int schedules, int hold, char* what, int what_size) {
  memset(static_cast<void*>(&par), 0, sizeof(par));
  arena = reinterpret_cast<uint8_t*>(&ar);
  mma_warp = kSoftWarps<kRows>;
  constexpr int kPool = 8;   // slots of the pool; odd ones are stale
  std::vector<int32_t> valid(kPool), slots(slot_ids, slot_ids + n_slots);
  for (int i = 0; i < kPool; ++i) valid[i] = !(i & 1);
  par.tile_rows = kRows;
  int tiles = 0;
  for (int i = 0; i <= kMaxDenseSegs; ++i) {
    par.seg_tile_prefix[i] = tiles;
    if (i < n_segs) { par.seg_rows[i] = seg_rows[i]; tiles += (seg_rows[i] + par.tile_rows - 1) / par.tile_rows; }
  }
  par.n_segs = n_segs;
  par.n_dense_tiles = tiles;
  par.slots = slots.data();
  par.valid = valid.data();
  par.n_slots = n_slots;
  par.pool_slots = kPool;
  par.C = C;
  par.tiles_per_slot = (C + par.tile_rows - 1) / par.tile_rows;
  par.n_tiles = kL ? par.tiles_per_slot : tiles + n_slots * par.tiles_per_slot;
  par.lq = lq;
  par.slot_units = kL;
  par.H = H;
  par.n_qpairs = (lq + kPairRows - 1) / kPairRows;
  par.n_units = par.n_qpairs * H * (kL ? n_slots : 1);
  par.n_full = n_full;
  par.n_ranges = n_ranges;
  par.scale_log2 = 1.f;
  uint32_t status = 0;
  par.status = &status;
  std::vector<uint16_t> O(static_cast<size_t>(lq) * H * 128 + 32);
  std::vector<float> lse(static_cast<size_t>(H) * lq * max(1, n_slots)), lsepart(2 * n_ranges * kPairRows + 1), opart(2 * n_ranges * 32 * kPairRows * 4 + 8);
  par.O = reinterpret_cast<__nv_bfloat16*>((reinterpret_cast<uintptr_t>(O.data()) + 31) / 32 * 32);
  par.lse = lse.data();
  par.lsepart = lsepart.data();
  par.opart = reinterpret_cast<float4*>((reinterpret_cast<uintptr_t>(opart.data()) + 15) / 16 * 16);
  gridDim.x = grid;
  // the pieces' outputs, row by row: log-sum-exp and O
  auto check = [&]() {
    for (blockIdx.x = 0; blockIdx.x < static_cast<unsigned>(grid) && fault.empty(); ++blockIdx.x) {
      PieceWalker walk;
      Piece pc;
      walk.init(par);
      while (walk.next(par, pc)) {
        for (int prow = 0; prow < kPairRows && pc.q0 + prow < lq; prow += 32) {
          double sum = 0, acc = 0;
          TileIter it;
          TileInfo ti;
          it.init(par, pc.tb, pc.te);
          while (it.next(par, ti, false))
            for (int r = ti.row0; r < ti.row0 + ti.nv; ++r) {
              const int seg = ti.seg >= 0 ? ti.seg : n_segs + ti.z;
              const double w = exp2(static_cast<double>(value(0, 0, pc.h, pc.q0 + prow)) * value(1, seg, pc.h, r));
              sum += w;
              acc += w * value(2, seg, pc.h, r);
            }
          const int row = pc.q0 + prow;
          const double l = pc.slot < 0 ? lse[(static_cast<size_t>(pc.ord) * H + pc.h) * lq + row] : lsepart[pc.slot * kPairRows + prow];
          const double want = sum > 0 ? log(sum) : -INFINITY;
          if (!(l == want || fabs(l - want) < 1e-3)) fail("a log-sum-exp is wrong");
          for (int col = 0; col < (kL ? 0 : 128); col += 37) {
            const double o = pc.slot < 0 ? bf16(reinterpret_cast<uint16_t*>(par.O)[(static_cast<size_t>(row) * H + pc.h) * 128 + col])
                                         : reinterpret_cast<float*>(par.opart)[((static_cast<size_t>(pc.slot) * 32 + col / 4) * kPairRows + prow) * 4 + col % 4];
            if (!(fabs(o - (sum > 0 ? acc / sum : 0.0)) < 0.02)) fail("an output row is wrong");   // values up to 3, weights and result in bf16
          }
        }
      }
    }
  };
  auto all = [&](int h, int from, unsigned seed) {
    std::fill(O.begin(), O.end(), 0x7fc0);
    std::fill(lse.begin(), lse.end(), NAN);
    std::fill(lsepart.begin(), lsepart.end(), NAN);
    int turns = 0;
    for (unsigned b = 0; b < static_cast<unsigned>(grid) && fault.empty(); ++b) {
      blockIdx.x = b;
      turns = max(turns, run_cta(h, from, seed + b));
    }
    if (fault.empty() && (status & ~WK_DEV_BAD_SLOT)) fail("status " + std::to_string(status));
    if (fault.empty()) check();
    return turns;
  };
  fault.clear();
  for (int s = 0; s < schedules && fault.empty(); ++s) all(-1, 0, s);
  for (int h = 0; hold && h < kThreads<kRows> / 32 + 3 && fault.empty(); ++h) {
    const int turns = all(h, 1 << 30, 0);
    for (int from = 0; from < turns && fault.empty(); ++from) {
      all(h, from, 0);
      if (!fault.empty()) fault += " (role " + std::to_string(h) + " held at its turn " + std::to_string(from) + " of " + std::to_string(turns) + ")";
    }
  }
  snprintf(what, what_size, "%s", fault.c_str());
  return fault.empty() ? 0 : 1;
}
