// nw_host.h -- host-side internals of libnw shared by its translation units:
// the context and dictionary objects, device buffers with budget accounting,
// the pair planner, kernel launching and error handling.  Everything except
// the two object definitions sits in an anonymous namespace (one copy per
// translation unit).
#pragma once

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <atomic>
#include <climits>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <set>
#include <string>
#include <utility>
#include <vector>

#include "nw.h"
#include "nw_proposal.h"
#include "nw_internal.cuh"
#include "nw_launch.h"
#include "nw_spare.h"

using namespace nw;

namespace {

thread_local std::string g_create_error;

struct DevBuf {
  void* p = nullptr;
  size_t bytes = 0;
  template <class T>
  T* as() const { return static_cast<T*>(p); }
};

// A word set on the device (see nw_internal.cuh for the layout).
struct WordSet {
  uint32_t n = 0;
  uint32_t min_len = 0, max_len = 0;
  Buckets bk{};
  DevBuf perm, rank, slen, aoff, brec_w, a_enc, b_rec;
};

// One alignment launch: a range of longer lengths of the DPX kernel, or the
// bit-parallel kernel's length pairs of one step class.
struct Launch {
  int range = 0;            // DPX kernel: dp_range_of the longer length; -1: bit-parallel
  int m = 0, x = 0;         // bit-parallel: the reduced steps
  uint32_t alphabet = 0;    // bit-parallel: the largest of the launch's sets
  uint32_t ta = 0;          // A words per task
  uint32_t bps = 0;         // resident blocks per SM at most (0: as many as fit)
  uint32_t seg_first = 0, nsegs = 0;
  uint64_t ntasks = 0;
  uint32_t max_la = 0;      // longest A word
};

struct Plan {
  std::vector<Seg> segs;
  std::vector<Launch> launches;
  uint64_t pairs = 0, cells = 0;
};

}  // namespace

struct nw_ctx {
  int device = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  size_t budget = 0, used = 0;
  uint32_t fail_countdown = 0;
  // debug bounds (nw_debug_set_bounds): list-insertion retries (-1 = the
  // kernel's own bound), pipeline wait cycles (-1 = the kernel's own bound),
  // and a column tile the candidate kernel's producer never issues (UINT32_MAX
  // = none)
  int32_t dbg_insert_iters = -1;
  int64_t dbg_wait_cycles = -1;
  uint32_t dbg_withhold_tile = UINT32_MAX;
  std::string err;
  bool profiling = false;
  nw_profile prof{};
  int sm_count = 0;
  std::set<nw_dict*> dicts;
  std::set<nw_model*> models;
  std::atomic<int> busy{0};
  // grow-only workspace
  DevBuf ws_slots, ws_thr, ws_hist, ws_small, ws_out_idx, ws_out_score, ws_mat, ws_pairs, ws_segs, ws_norm;
  std::vector<cudaEvent_t> events;
};

struct nw_dict {
  nw_ctx* ctx = nullptr;
  WordSet ws;
  nw_scoring sc{};
  ShiftedScoring ss{};
  uint32_t alphabet = 0;
  int32_t score_lo = 0, score_hi = 0;
  Plan plan;
  DevBuf d_segs;       // the plan's segments
  bool subst = false;  // scored with a full similarity matrix (d_tab)
  DevBuf d_tab;        // kTabDim x kTabDim s'+ table
  uint64_t serial = 0;  // unique per loaded dictionary (caches keyed on it)
  DevBuf rec;           // the words' 16-byte records, once they repay their making (pair_records)
  uint64_t pairs_scored = 0;  // by the calls that could have read them
};

namespace {

nw_status set_err(nw_ctx* c, nw_status st, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  if (c) c->err = buf; else g_create_error = buf;
  return st;
}

nw_status cuda_fail(nw_ctx* c, cudaError_t e, const char* what) {
  cudaGetLastError();  // clear a non-sticky error
  return set_err(c, NW_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

#define NW_CK(call)                                                 \
  do {                                                              \
    cudaError_t e_ = (call);                                        \
    if (e_ != cudaSuccess) return cuda_fail(c, e_, #call);          \
  } while (0)

#define NW_TRY(expr)                        \
  do {                                      \
    nw_status s_ = (expr);                  \
    if (s_ != NW_OK) return s_;             \
  } while (0)

bool ctx_drop_records(nw_ctx* c);

// give_up: what is kept only for speed (spare blocks, word records) is released
// before the allocation is refused.
nw_status ctx_alloc(nw_ctx* c, DevBuf& b, size_t bytes, const char* what, bool give_up = true) {
  if (bytes == 0) bytes = 16;
  if (c->fail_countdown) {
    if (--c->fail_countdown == 0)
      return set_err(c, NW_ENOMEM, "injected allocation failure for %s (%zu bytes)", what, bytes);
  }
  if (c->budget && c->used + bytes > c->budget && give_up) ctx_drop_records(c);
  if (c->budget && c->used + bytes > c->budget)
    return set_err(c, NW_ENOMEM, "memory budget exceeded: %s needs %zu bytes, %zu of %zu in use", what,
                   bytes, c->used, c->budget);
  // a spare block that is not much larger (under a budget only an own one of the
  // same size: what fitted it before still fits)
  size_t have = 0;
  if (void* p = spare_take(c->budget ? c : nullptr, c->device, bytes, c->budget ? bytes : bytes + bytes / 4 + 4096,
                           &have)) {
    b.p = p;
    b.bytes = have;
    c->used += have;
    return NW_OK;
  }
  while (c->budget && c->used + spare_held(c) + bytes > c->budget && spare_drop_oldest(c)) {
  }
  void* p = nullptr;
  cudaError_t e = cudaMalloc(&p, bytes);
  if (e != cudaSuccess && spare_drop_device(c->device)) {
    cudaGetLastError();
    e = cudaMalloc(&p, bytes);
  }
  if (e != cudaSuccess && give_up && ctx_drop_records(c)) {
    cudaGetLastError();
    e = cudaMalloc(&p, bytes);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    return set_err(c, NW_ENOMEM, "cudaMalloc(%zu) for %s failed: %s", bytes, what, cudaGetErrorString(e));
  }
  b.p = p;
  b.bytes = bytes;
  c->used += bytes;
  return NW_OK;
}

void ctx_free(nw_ctx* c, DevBuf& b) {
  if (b.p) {
    cudaFree(b.p);
    c->used -= b.bytes;
  }
  b = DevBuf{};
}

// Frees the word records of the context's dictionaries; they are made again once
// as many pairs have been scored as the first time.  A call takes its records after
// its last allocation.
bool ctx_drop_records(nw_ctx* c) {
  bool any = false;
  for (nw_dict* d : c->dicts) {
    if (!d->rec.p) continue;
    if (!any) cudaStreamSynchronize(c->stream);  // an asynchronous call may still read them
    ctx_free(c, d->rec);
    d->pairs_scored = 0;
    any = true;
  }
  return any;
}

// For a buffer that no work in flight uses: kept for the next call (nw_spare.h).
void ctx_release(nw_ctx* c, DevBuf& b) {
  if (b.p) {
    c->used -= b.bytes;
    spare_give(c, c->device, b.p, b.bytes);
  }
  b = DevBuf{};
}

// RAII: a call's own buffers; `done` once the call has synchronised its stream
// (a call that fails frees them: its stream may still be using them).
struct CallBufs {
  nw_ctx* c;
  std::vector<DevBuf*> bufs;
  bool done = false;
  ~CallBufs() {
    for (DevBuf* b : bufs) done ? ctx_release(c, *b) : ctx_free(c, *b);
  }
};

nw_status ctx_ensure(nw_ctx* c, DevBuf& b, size_t bytes, const char* what) {
  if (b.p && b.bytes >= bytes) return NW_OK;
  ctx_free(c, b);
  return ctx_alloc(c, b, bytes, what);
}

// RAII: one call at a time per context, on the context's device.
struct CallGuard {
  nw_ctx* c;
  bool ok = false;
  explicit CallGuard(nw_ctx* ctx) : c(ctx) {
    int expected = 0;
    ok = c->busy.compare_exchange_strong(expected, 1);
  }
  ~CallGuard() {
    if (ok) c->busy.store(0);
  }
};

// RAII: an NVTX range named after the entry point, so a timeline profiler
// (Nsight Systems) shows each library call around its copies and launches.
// Without a profiler attached the push and pop cost a few nanoseconds.
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
};

#define NW_ENTER(ctxp)                                                              \
  if (!(ctxp)) return NW_EINVAL;                                                    \
  NvtxRange nvtx_(__func__);                                                        \
  CallGuard guard_(ctxp);                                                           \
  if (!guard_.ok) return set_err(ctxp, NW_EBUSY, "context in use by another call"); \
  (ctxp)->err.clear();                                                              \
  {                                                                                 \
    cudaError_t e_ = cudaSetDevice((ctxp)->device);                                 \
    if (e_ != cudaSuccess) return cuda_fail(ctxp, e_, "cudaSetDevice");             \
  }

uint32_t pack16(int32_t v) {
  const uint32_t h = (uint32_t)v & 0xffffu;
  return h | (h << 16);
}

// The reduced steps of the bit-parallel kernel: s'_m and max(s'_x, 0) over
// their gcd.  match == mismatch (every cell gains the same) and s'_m = 0 keep
// the DPX kernel, as do steps above kBitMaxStep: a row takes about m^2 logic
// operations for 64 columns against 2 m for 2 cells there.
void bit_steps(ShiftedScoring& s) {
  const int m = s.sm, x = std::max(s.sx, 0);
  s.bit_m = s.bit_x = s.bit_coef = 0;
  if (m <= 0 || x >= m) return;
  int g = m, h = x;
  while (h) { const int r = g % h; g = h; h = r; }
  if (m / g > kBitMaxStep) return;
  s.bit_m = m / g;
  s.bit_x = x / g;
  s.bit_coef = g;
}

nw_status make_shifted(nw_ctx* c, const nw_scoring& s, uint32_t alphabet, ShiftedScoring& out) {
  if (std::abs(s.match) > 1024 || std::abs(s.mismatch) > 1024 || std::abs(s.gap) > 1024)
    return set_err(c, NW_EINVAL, "scoring values must lie in [-1024, 1024]");
  if (s.mismatch > s.match) return set_err(c, NW_EINVAL, "mismatch (%d) must not exceed match (%d)", s.mismatch, s.match);
  const int32_t sm = s.match - 2 * s.gap, sx = s.mismatch - 2 * s.gap;
  if (sm < 0) return set_err(c, NW_EINVAL, "2*gap (%d) must not exceed match (%d)", 2 * s.gap, s.match);
  if ((int64_t)sm * kMaxLen > 32767)
    return set_err(c, NW_ERANGE, "match - 2*gap = %d is too large for 16-bit cells at length %d", sm, kMaxLen);
  const int32_t delta = s.match - s.mismatch;
  uint32_t shift = 0;
  while ((1 << shift) < delta) ++shift;
  if (((alphabet - 1u) << shift) >= 32768u)
    return set_err(c, NW_EINVAL, "alphabet %u with match - mismatch = %d does not fit the 15-bit code encoding", alphabet, delta);
  out.sm = sm;
  out.sx = sx;
  out.shift = shift;
  out.C1 = pack16(sm + 1);
  out.C2 = pack16(std::max(sx, 0));  // a negative mismatch term never wins (see nw_dp.cuh)
  bit_steps(out);
  return NW_OK;
}

const uint16_t* dict_tab(const nw_dict* d) { return d->subst ? d->d_tab.as<uint16_t>() : nullptr; }

void pair_bounds(const nw_scoring& s, int la, int lb, int& lo, int& hi) {
  const int mn = std::min(la, lb), d = std::abs(la - lb);
  const int allgap = (la + lb) * s.gap;
  lo = std::max(allgap, mn * std::min(s.match, s.mismatch) + d * s.gap);
  hi = std::max(allgap, mn * std::max(s.match, s.mismatch) + d * s.gap);
}

// Buckets with every base filled from the counts.
void fill_buckets(Buckets& bk) {
  uint64_t pos = 0, aenc = 0, brec = 0;
  for (int L = 0; L < kBuckets; ++L) {
    bk.start[L] = (uint32_t)pos;
    bk.aenc_base[L] = (uint32_t)aenc;
    bk.brec_word_base[L] = (uint32_t)brec;
    pos += bk.count[L];
    aenc += (uint64_t)bk.count[L] * L;
    brec += (uint64_t)((bk.count[L] + 1) / 2) * (uint64_t)ceil4(L);
  }
  bk.start[kBuckets] = (uint32_t)pos;
}

uint64_t aenc_words(const Buckets& bk) {
  uint64_t s = 0;
  for (int L = 0; L < kBuckets; ++L) s += (uint64_t)bk.count[L] * L;
  return s;
}
uint64_t brec_words(const Buckets& bk) {
  uint64_t s = 0;
  for (int L = 0; L < kBuckets; ++L) s += (uint64_t)((bk.count[L] + 1) / 2) * (uint64_t)ceil4(L);
  return s;
}

uint64_t cdiv(uint64_t a, uint64_t b) { return (a + b - 1) / b; }

// ---------------------------------------------------------------------------
// plans.  A call's pairs are listed as rectangles of buckets, the shorter
// words on the A side; the kernel that scores them cuts them into segments and
// tasks.

// Words [a0, a1) of bucket La of set A against words [b0, b1) of bucket LB of
// set B (relative to the buckets), La <= LB; tri: the same bucket, only pairs
// a < b.  `dict` names the terms, dict_swapped those with the sides exchanged.
struct Rect {
  const Buckets* A;
  const Buckets* B;
  int La, LB;
  uint32_t a0, a1, b0, b1;
  bool tri;
  uint32_t dict, dict_swapped;
};
using Rects = std::vector<Rect>;

// Every unordered pair of one set, once.
void rects_all(const Buckets& bk, uint32_t dict, Rects& out) {
  for (int L = 0; L < kBuckets; ++L)
    for (int s = 0; s <= L; ++s)
      if (bk.count[s] && bk.count[L] && (s < L || bk.count[L] > 1))
        out.push_back({&bk, &bk, s, L, 0, bk.count[s], 0, bk.count[L], s == L, dict, dict});
}

// Every (query, dictionary word) pair, once: terms dict where the queries are
// the A words, dict + 1 where they are the B words.
void rects_queries(const Buckets& qb, const Buckets& db, uint32_t dict, Rects& out) {
  for (int lq = 0; lq < kBuckets; ++lq)
    for (int ld = 0; ld < kBuckets; ++ld) {
      if (!qb.count[lq] || !db.count[ld]) continue;
      if (lq <= ld) out.push_back({&qb, &db, lq, ld, 0, qb.count[lq], 0, db.count[ld], false, dict, dict + 1});
      else out.push_back({&db, &qb, ld, lq, 0, db.count[ld], 0, qb.count[lq], false, dict + 1, dict});
    }
}

// Shard `shard` of `nshards` of one set's pairs.  The partition: per longer
// length LB a task list (same-length strips of 256 words first, then shorter
// lengths in falling order; tasks of 256 A words by 64 B words, A chunks
// fastest), each list cut into nshards contiguous ranges.  It is fixed,
// whatever kernel scores the pairs and however it cuts them, so that shards
// saved by one build combine with another's.
constexpr uint32_t kShardTA = 256;
void rects_shard(const Buckets& bk, uint32_t shard, uint32_t nshards, Rects& out) {
  struct Block {
    int La;
    uint32_t a0, a1, b0, b1;
    uint32_t nca, ncb;
  };
  for (int LB = 0; LB < kBuckets; ++LB) {
    const uint32_t nB = bk.count[LB];
    std::vector<Block> blocks;
    uint64_t total = 0;
    auto add = [&](int La, uint32_t a0, uint32_t a1, uint32_t b0) {
      blocks.push_back({La, a0, a1, b0, nB, (uint32_t)cdiv(a1 - a0, kShardTA), (uint32_t)cdiv(nB - b0, kWarpB)});
      total += (uint64_t)blocks.back().nca * blocks.back().ncb;
    };
    if (nB == 0) continue;
    for (uint32_t a = 0; a + 1 < nB; a += kShardTA) add(LB, a, std::min(nB, a + kShardTA), a);
    for (int La = LB - 1; La >= 0; --La)
      if (bk.count[La]) add(La, 0, bk.count[La], 0);
    const uint64_t lo = total * shard / nshards, hi = total * (shard + 1) / nshards;
    uint64_t t0 = 0;
    for (const Block& k : blocks) {
      const uint64_t t1 = t0 + (uint64_t)k.nca * k.ncb, a = std::max(lo, t0), b = std::min(hi, t1);
      if (a < b) {
        // tasks [a, b): whole rows of B chunks, and parts of the first and last
        auto rect = [&](uint32_t ca0, uint32_t ca1, uint32_t cb0, uint32_t cb1) {
          if (ca0 >= ca1 || cb0 >= cb1) return;
          out.push_back({&bk, &bk, k.La, LB, std::min(k.a1, k.a0 + ca0 * kShardTA), std::min(k.a1, k.a0 + ca1 * kShardTA),
                         std::min(k.b1, k.b0 + cb0 * (uint32_t)kWarpB), std::min(k.b1, k.b0 + cb1 * (uint32_t)kWarpB),
                         k.La == LB, 0u, 0u});
        };
        const uint32_t l0 = (uint32_t)((a - t0) / k.nca), c0 = (uint32_t)((a - t0) % k.nca);
        const uint32_t l1 = (uint32_t)((b - t0) / k.nca), c1 = (uint32_t)((b - t0) % k.nca);
        if (l0 == l1) {
          rect(c0, c1, l0, l0 + 1);
        } else {
          rect(c0, k.nca, l0, l0 + 1);
          rect(0, k.nca, l0 + 1, l1);
          rect(0, c1, l1, l1 + 1);
        }
      }
      t0 = t1;
    }
  }
}

// Pairs and cells of whole-bucket rectangles.
void count_rects(const Rects& rects, uint64_t& pairs, uint64_t& cells) {
  for (const Rect& r : rects) {
    const uint64_t na = r.a1 - r.a0, nb = r.b1 - r.b0, n = r.tri ? na * (na - 1) / 2 : na * nb;
    pairs += n;
    cells += n * (uint64_t)(r.La * r.LB);
  }
}

// Smallest length difference first: a word's best neighbours mostly have
// nearly its length, so its list bound rises before the many low-scoring pairs
// arrive.  Within a difference the long words (the long tasks) come first.
void order_rects(Rects& rects) {
  std::stable_sort(rects.begin(), rects.end(), [](const Rect& x, const Rect& y) {
    const int dx = x.LB - x.La, dy = y.LB - y.La;
    return dx != dy ? dx < dy : x.LB > y.LB;
  });
}

// Appends a rectangle to the launch's segments.  Same-bucket rectangles are
// cut into strips of ta A words, each against the B words from its start on.
void add_rect(Plan& p, Launch& l, const Rect& r) {
  const bool bits = l.range < 0;
  const uint32_t chunk = bits ? 32u * (uint32_t)bit_words_per_lane(r.LB) : (uint32_t)kWarpB;
  auto seg = [&](uint32_t a0, uint32_t a1, uint32_t b0) {
    if (a0 >= a1 || b0 >= r.b1 || (r.tri && a0 + 1 >= r.b1)) return;
    Seg s{};
    s.a_beg = r.A->start[r.La] + a0;
    s.a_end = r.A->start[r.La] + a1;
    s.b_beg = r.B->start[r.LB] + b0;
    s.b_end = r.B->start[r.LB] + r.b1;
    s.aenc_base = r.A->aenc_base[r.La] + a0 * (uint32_t)r.La;
    // (b0 is even: bucket starts, and multiples of 64 and of the strip size)
    s.b_base = bits ? r.B->aenc_base[r.LB] + b0 * (uint32_t)r.LB
                    : (r.B->brec_word_base[r.LB] + (b0 / 2) * (uint32_t)ceil4(r.LB)) / 4;
    s.la = (uint16_t)r.La;
    s.lb = (uint32_t)r.LB;
    s.tri = r.tri ? 1 : 0;
    s.dict = r.dict;
    s.nca = (uint32_t)cdiv(a1 - a0, l.ta);
    s.task0 = l.ntasks;
    l.ntasks += (uint64_t)s.nca * cdiv(r.b1 - b0, chunk);
    l.max_la = std::max(l.max_la, (uint32_t)r.La);
    p.segs.push_back(s);
    ++l.nsegs;
  };
  if (!r.tri) return seg(r.a0, r.a1, r.b0);
  for (uint32_t a = r.a0; a < r.a1; a += l.ta) seg(a, std::min(r.a1, a + l.ta), std::max(r.b0, a));
}

// The DPX launches of a pair list (in order_rects order), one per range of
// longer lengths present, with `ta` A words per task.  Within a launch the
// lengths come one after another, each smallest difference first: the loop
// body of a length is several KB of instructions, and a mix of ten of them
// ran out of the instruction cache.
void plan_dp(Rects rects, uint32_t ta, Plan& p, int only_range = -1, uint32_t bps = 0) {
  std::stable_sort(rects.begin(), rects.end(), [](const Rect& x, const Rect& y) { return x.LB < y.LB; });
  for (int r = 0; r < kDpRanges; ++r) {
    if (only_range >= 0 && r != only_range) continue;
    Launch l;
    l.range = r;
    l.ta = ta;
    l.bps = bps;
    l.seg_first = (uint32_t)p.segs.size();
    for (const Rect& x : rects)
      if (dp_range_of(x.LB) == r) add_rect(p, l, x);
    if (l.ntasks) p.launches.push_back(l);
  }
}

// Estimated SM sub-partition cycles (per warp) of nA words of length a against
// nB words of length b in the lanes of the bit-parallel kernel: a row costs
// ~70 cycles for the lane's words, an A word ~40, each of the lane's words ~12
// to score and file, and each task ~1500 to build its match masks.
uint64_t bit_cost(uint64_t nA, int a, uint64_t nB, int b, uint32_t ta) {
  const uint64_t K = (uint64_t)bit_words_per_lane(b);
  const uint64_t chunks = cdiv(nB, 32 * K), kk = std::min<uint64_t>(K, cdiv(nB, 32));
  return chunks * (nA * ((uint64_t)a * 70 + 40 + 12 * kk) + cdiv(nA, ta) * 1500);
}

// The bit-parallel launch of a pair list.  Rectangles of two lengths take the
// cheaper of the two orientations: short words in the lanes pack more densely.
// Against queries, the first kColdWords words that a query length meets count
// double with the queries in the lanes: while the lists are empty every pair is
// offered, and a warp then offers each of its few A words to hundreds of lists that
// all other warps offer to, where with the queries as A words it offers the best of
// 256 words to one.  256 queries against 20,000 words, all of 8 symbols: 1,770 us
// with the queries in the lanes (cheaper by 1 %), 225 as A words; 4,096: 10.6 ms and
// 0.49.  Once the lists are warm the rows decide: counting double throughout, 4,096
// queries against 600,000 words of lengths 1 .. 25 take 12.2 ms instead of 11.9.
// (Thresholds from 4,096 to 262,144 words measure alike, the least is the best for
// 100,000 words of mixed lengths; factors 1.5, 2 and 3 measure alike.)
constexpr uint64_t kColdWords = 4096, kColdFactor = 2;
void plan_bits(const Rects& rects, int m, int x, uint32_t alphabet, uint32_t ta, Plan& p) {
  Launch l;
  l.range = -1;
  l.m = m;
  l.x = x;
  l.alphabet = alphabet;
  l.ta = ta;
  l.seg_first = (uint32_t)p.segs.size();
  uint32_t sets = 0;
  for (const Rect& r : rects) sets = std::max(sets, std::min(r.dict, r.dict_swapped) + 1);
  std::vector<uint64_t> met((size_t)sets * kBuckets, 0);  // words met so far, by query set and length
  for (Rect r : rects) {
    const uint32_t na = r.a1 - r.a0, nb = r.b1 - r.b0;
    uint64_t cost = bit_cost(na, r.La, nb, r.LB, ta), swapped = bit_cost(nb, r.LB, na, r.La, ta);
    if (r.dict != r.dict_swapped) {
      const bool a_queries = r.dict < r.dict_swapped;  // (rects_queries)
      uint64_t& m = met[(size_t)std::min(r.dict, r.dict_swapped) * kBuckets + (size_t)(a_queries ? r.La : r.LB)];
      if (m < kColdWords) (a_queries ? swapped : cost) *= kColdFactor;
      m += a_queries ? nb : na;
    }
    if (!r.tri && swapped < cost) {
      std::swap(r.A, r.B);
      std::swap(r.La, r.LB);
      std::swap(r.a0, r.b0);
      std::swap(r.a1, r.b1);
      std::swap(r.dict, r.dict_swapped);
    }
    add_rect(p, l, r);
  }
  if (l.ntasks) p.launches.push_back(l);
}

// The chunk of A words per task: 256, halved down to 16 while the plan has
// fewer tasks than these (several per resident block of the bit-parallel
// kernel, several per resident warp of the DPX kernel, on a full GPU).
constexpr uint64_t kBitMinTasks = 12288, kDpMinTasks = 40960;
constexpr uint32_t kMinTA = 16;
template <class Make>
void sized(Plan& p, uint64_t min_tasks, Make make) {
  for (uint32_t ta = kDefaultTA;;) {
    p = Plan{};
    make(ta, p);
    uint64_t n = 0;
    for (const Launch& l : p.launches) n += l.ntasks;
    if (n >= min_tasks || ta <= kMinTA) return;
    do {  // (half the chunk makes at most twice the tasks: sizes that cannot suffice are skipped)
      ta /= 2;
      n *= 2;
    } while (n < min_tasks && ta > kMinTA);
  }
}

// Takes out of a step class's pair list what the DPX kernel scores faster: pairs of
// words of more than 32 symbols, one to a lane in the bit-parallel kernel, for the
// classes with the dearest rows (m >= 4 with x <= m - 2: (4,1), (5,1), (5,2), (5,3)),
// when there are enough of them to pay for another launch.  Top-10 lists and
// histogram of 20,000 words of 33 / 40 symbols: (5,1) 31.1 / 37.6 ms, (5,3) 23.9 / 28.8,
// (4,1) 22.5 / 27.1, the DPX kernel 18.1 / 25.4 whatever the scoring, (5,4) 18.7 / 22.4
// and every other class less; of 3,000 words (4.5M pairs) of 33 symbols (4,1) 0.70, DPX
// 0.64, of 2,000 0.40 and 0.41; 1,024 queries against 4,500 words of 33 symbols (4,1)
// 0.68, DPX 0.67.  (5,1) at 17, 18 and 22 to 25 symbols would gain up to 12 % too.
constexpr uint64_t kLongPairs = (uint64_t)1 << 22;
Rects take_long(Rects& rects, const ShiftedScoring& ss) {
  Rects taken;
  if (ss.bit_m < 4 || ss.bit_x > ss.bit_m - 2) return taken;
  auto is_long = [](const Rect& r) { return bit_words_per_lane(std::min(r.La, r.LB)) == 1; };
  uint64_t pairs = 0;
  for (const Rect& r : rects)
    if (is_long(r)) {
      const uint64_t na = r.a1 - r.a0, nb = r.b1 - r.b0;
      pairs += r.tri ? na * nb / 2 : na * nb;
    }
  if (pairs < kLongPairs) return taken;
  const auto at = std::stable_partition(rects.begin(), rects.end(), [&](const Rect& r) { return !is_long(r); });
  taken.assign(at, rects.end());
  rects.erase(at, rects.end());
  return taken;
}

// Appends a plan's launches and segments (not its counts).
void append_plan(Plan& to, const Plan& p) {
  for (Launch l : p.launches) {
    l.seg_first += (uint32_t)to.segs.size();
    to.launches.push_back(l);
  }
  to.segs.insert(to.segs.end(), p.segs.begin(), p.segs.end());
}

// The launches of a pair list for scoring ss and an alphabet; ta = 0 sizes
// the tasks.
void make_plan(Rects rects, const ShiftedScoring& ss, uint32_t alphabet, uint32_t ta, Plan& p) {
  order_rects(rects);
  p = Plan{};
  count_rects(rects, p.pairs, p.cells);
  const Rects dpx = ss.bit_m ? take_long(rects, ss) : std::move(rects);
  auto add = [&](uint64_t min_tasks, auto make) {
    Plan part;
    if (ta) make(ta, part);
    else sized(part, min_tasks, make);
    append_plan(p, part);
  };
  if (ss.bit_m && !rects.empty())
    add(kBitMinTasks, [&](uint32_t t, Plan& q) { plan_bits(rects, ss.bit_m, ss.bit_x, alphabet, t, q); });
  if (!dpx.empty()) add(kDpMinTasks, [&](uint32_t t, Plan& q) { plan_dp(dpx, t, q); });
}

uint32_t index_bits(uint32_t n) {
  uint32_t b = 1;
  while (b < 32 && ((uint64_t)1 << b) < (uint64_t)n) ++b;
  return b;
}

// Tables of the length-normalised ranking (Section 5 divides each score by
// the longer word's length).  Every value s/m that a pair whose longer word
// has m symbols can reach (s within that length's score bounds and within
// [lo, hi]) is ranked ascending by exact integer cross-multiplication; equal
// fractions share a rank.  Two empty words (m = 0) rank as s/1.
struct NormTables {
  int32_t lo = 0;              // score of row 0 of `rank`
  uint32_t nranks = 0;
  std::vector<uint16_t> rank;  // [(s - lo) * kBuckets + m]: rank of s/m (0 where s is out of reach for m)
  std::vector<int16_t> smin;   // [r * kBuckets + m]: smallest reachable s whose s/m has rank >= r, else above reach
  std::vector<int16_t> frac;   // [2r], [2r + 1]: numerator and denominator of rank r in lowest terms
};

void build_norm_tables(const nw_scoring& sc, int32_t lo, int32_t hi, NormTables& t) {
  int flo[kBuckets], fhi[kBuckets];
  std::vector<std::pair<int32_t, int32_t>> fr;  // reduced (numerator, denominator)
  for (int m = 0; m < kBuckets; ++m) {
    flo[m] = INT32_MAX;
    fhi[m] = INT32_MIN;
    for (int la = 0; la <= m; ++la) {
      int a, b;
      pair_bounds(sc, la, m, a, b);
      flo[m] = std::min(flo[m], a);
      fhi[m] = std::max(fhi[m], b);
    }
    flo[m] = std::max(flo[m], lo);
    fhi[m] = std::min(fhi[m], hi);
    const int32_t den = m > 0 ? m : 1;
    for (int s = flo[m]; s <= fhi[m]; ++s) {
      int32_t g = std::abs(s), h = den;
      while (h) { const int32_t r = g % h; g = h; h = r; }
      fr.push_back({s / g, den / g});
    }
  }
  auto less = [](const std::pair<int32_t, int32_t>& x, const std::pair<int32_t, int32_t>& y) {
    return (int64_t)x.first * y.second < (int64_t)y.first * x.second;
  };
  std::sort(fr.begin(), fr.end(), less);
  fr.erase(std::unique(fr.begin(), fr.end()), fr.end());  // reduced fractions are equal iff their parts are
  t.lo = lo;
  t.nranks = (uint32_t)fr.size();
  t.rank.assign((size_t)(hi - lo + 1) * kBuckets, 0);
  t.frac.resize(2 * fr.size());
  for (size_t r = 0; r < fr.size(); ++r) {
    t.frac[2 * r] = (int16_t)fr[r].first;
    t.frac[2 * r + 1] = (int16_t)fr[r].second;
  }
  for (int m = 0; m < kBuckets; ++m) {
    const int32_t den = m > 0 ? m : 1;
    for (int s = flo[m]; s <= fhi[m]; ++s) {
      const auto it = std::lower_bound(fr.begin(), fr.end(), std::make_pair((int32_t)s, den), less);
      t.rank[(size_t)(s - lo) * kBuckets + m] = (uint16_t)(it - fr.begin());
    }
  }
  // rank grows with s at fixed m, so the smallest s reaching rank r is found
  // by one sweep per length; above reach, the bound no G value attains
  t.smin.assign((size_t)fr.size() * kBuckets, INT16_MAX);
  for (int m = 0; m < kBuckets; ++m) {
    int s = flo[m];
    for (uint32_t r = 0; r < t.nranks; ++r) {
      while (s <= fhi[m] && t.rank[(size_t)(s - lo) * kBuckets + m] < r) ++s;
      if (s > fhi[m]) break;
      t.smin[(size_t)r * kBuckets + m] = (int16_t)s;
    }
  }
}

std::vector<DevBuf*> wordset_bufs(WordSet& w) {
  return {&w.perm, &w.rank, &w.slen, &w.aoff, &w.brec_w, &w.a_enc, &w.b_rec};
}

void free_wordset(nw_ctx* c, WordSet& w) {
  for (DevBuf* b : wordset_bufs(w)) ctx_free(c, *b);
  w = WordSet{};
}

uint64_t wordset_bytes(const WordSet& w) {
  return w.perm.bytes + w.rank.bytes + w.slen.bytes + w.aoff.bytes + w.brec_w.bytes + w.a_enc.bytes +
         w.b_rec.bytes;
}

// Copies (if needed), validates, buckets and encodes a word set.
nw_status ingest(nw_ctx* c, const uint8_t* codes, const uint32_t* offsets, uint32_t n, uint32_t alphabet,
                 uint32_t shift, uint32_t flags, WordSet& ws) {
  const bool dev = flags & NW_DEVICE_PTRS;
  cudaStream_t s = c->stream;
  std::vector<DevBuf> tmp;
  struct Cleanup {
    nw_ctx* c;
    std::vector<DevBuf>& t;
    bool done = false;
    ~Cleanup() {
      for (auto& b : t) done ? ctx_release(c, b) : ctx_free(c, b);
    }
  } cleanup{c, tmp};
  auto talloc = [&](size_t bytes, const char* what, void** out) -> nw_status {
    tmp.emplace_back();
    NW_TRY(ctx_alloc(c, tmp.back(), bytes, what));
    *out = tmp.back().p;
    return NW_OK;
  };

  uint32_t total = 0;
  const uint8_t* d_codes = codes;
  const uint32_t* d_offsets = offsets;
  if (dev) {
    NW_CK(cudaMemcpyAsync(&total, offsets + n, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    NW_CK(cudaStreamSynchronize(s));
  } else {
    if (offsets[0] != 0) return set_err(c, NW_EINVAL, "offsets[0] must be 0");
    for (uint32_t i = 0; i < n; ++i) {
      if (offsets[i + 1] < offsets[i]) return set_err(c, NW_EINVAL, "offsets decrease at word %u", i);
      if (offsets[i + 1] - offsets[i] > (uint32_t)kMaxLen)
        return set_err(c, NW_EINVAL, "word %u has %u codes; at most %d are supported", i, offsets[i + 1] - offsets[i], kMaxLen);
    }
    total = offsets[n];
    void* p;
    NW_TRY(talloc((size_t)total + 16, "input codes", &p));
    if (total) NW_CK(cudaMemcpyAsync(p, codes, total, cudaMemcpyHostToDevice, s));
    d_codes = static_cast<const uint8_t*>(p);
    NW_TRY(talloc(sizeof(uint32_t) * ((size_t)n + 1), "input offsets", &p));
    NW_CK(cudaMemcpyAsync(p, offsets, sizeof(uint32_t) * ((size_t)n + 1), cudaMemcpyHostToDevice, s));
    d_offsets = static_cast<const uint32_t*>(p);
  }

  const uint32_t nblk = (uint32_t)cdiv(n, kIngestBlock);
  void *p_counts, *p_small;
  NW_TRY(talloc(sizeof(uint32_t) * (size_t)nblk * kBuckets, "ingest block counts", &p_counts));
  NW_TRY(talloc(sizeof(uint32_t) * (kBuckets + 4), "ingest counters", &p_small));
  uint32_t* d_counts = static_cast<uint32_t*>(p_counts);
  uint32_t* d_bucket = static_cast<uint32_t*>(p_small);
  uint32_t* d_err = d_bucket + kBuckets;
  NW_CK(cudaMemsetAsync(p_small, 0, sizeof(uint32_t) * (kBuckets + 4), s));
  NW_CK(launch_ingest_count(d_codes, d_offsets, n, alphabet, d_counts, d_err, s));
  NW_CK(launch_ingest_scan(d_counts, nblk, d_bucket, s));
  uint32_t host_small[kBuckets + 1];
  NW_CK(cudaMemcpyAsync(host_small, p_small, sizeof(uint32_t) * (kBuckets + 1), cudaMemcpyDeviceToHost, s));
  NW_CK(cudaStreamSynchronize(s));
  if (host_small[kBuckets])
    return set_err(c, NW_EINVAL,
                   "invalid words: offsets must start at 0 and not decrease, words have at most %d codes and "
                   "every code is < alphabet (%u)", kMaxLen, alphabet);

  ws.n = n;
  std::memcpy(ws.bk.count, host_small, sizeof(uint32_t) * kBuckets);
  fill_buckets(ws.bk);
  ws.min_len = kMaxLen;
  ws.max_len = 0;
  for (int L = 0; L < kBuckets; ++L)
    if (ws.bk.count[L]) { ws.min_len = std::min<uint32_t>(ws.min_len, L); ws.max_len = std::max<uint32_t>(ws.max_len, L); }
  if (n == 0) ws.min_len = 0;
  const uint64_t aw = aenc_words(ws.bk), bw = brec_words(ws.bk);
  if (aw >= (1ull << 32) || bw >= (1ull << 31))
    return set_err(c, NW_EINVAL, "word set too large for 32-bit symbol offsets");

  NW_TRY(ctx_alloc(c, ws.perm, sizeof(uint32_t) * (size_t)n, "word permutation"));
  NW_TRY(ctx_alloc(c, ws.rank, sizeof(uint32_t) * (size_t)n, "word ranks"));
  NW_TRY(ctx_alloc(c, ws.slen, (size_t)n + 16, "word lengths"));
  NW_TRY(ctx_alloc(c, ws.aoff, sizeof(uint32_t) * (size_t)n, "A-side offsets"));
  NW_TRY(ctx_alloc(c, ws.brec_w, sizeof(uint32_t) * (size_t)n, "B-side offsets"));
  NW_TRY(ctx_alloc(c, ws.a_enc, sizeof(uint32_t) * (size_t)(aw + 4), "A-side symbols"));
  NW_TRY(ctx_alloc(c, ws.b_rec, sizeof(uint32_t) * (size_t)(bw + 4), "B-side pair records"));
  NW_CK(cudaMemsetAsync(ws.b_rec.p, 0xff, ws.b_rec.bytes, s));
  if (n) {
    NW_CK(launch_ingest_scatter(d_offsets, n, d_counts, ws.bk, ws.perm.as<uint32_t>(), ws.rank.as<uint32_t>(),
                                ws.slen.as<uint8_t>(), s));
    NW_CK(launch_ingest_encode(d_codes, d_offsets, n, ws.perm.as<uint32_t>(), ws.slen.as<uint8_t>(), ws.bk,
                               shift, ws.a_enc.as<uint32_t>(), ws.aoff.as<uint32_t>(), ws.b_rec.as<uint32_t>(),
                               ws.brec_w.as<uint32_t>(), s));
  }
  NW_CK(cudaStreamSynchronize(s));  // temporaries are released on return
  cleanup.done = true;
  return NW_OK;
}

// ---------------------------------------------------------------------------
// profiling events

struct Timer {
  nw_ctx* c;
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> dp, fin;
  cudaEvent_t first = nullptr, last = nullptr;
  size_t used = 0;
  cudaEvent_t get() {
    if (used == c->events.size()) {
      cudaEvent_t e;
      if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
      c->events.push_back(e);
    }
    return c->events[used++];
  }
  void mark(cudaEvent_t e) {
    if (!e) return;
    cudaEventRecord(e, c->stream);
    if (!first) first = e;
    last = e;
  }
  void begin(bool dp_kind, cudaEvent_t& a) {
    a = c->profiling ? get() : nullptr;
    mark(a);
    (void)dp_kind;
  }
  void end(bool dp_kind, cudaEvent_t a) {
    if (!c->profiling) return;
    cudaEvent_t b = get();
    mark(b);
    if (a && b) (dp_kind ? dp : fin).emplace_back(a, b);
  }
  void collect() {
    if (!c->profiling) return;
    double dms = 0, fms = 0;
    for (auto& pr : dp) { float ms = 0; cudaEventElapsedTime(&ms, pr.first, pr.second); dms += ms; }
    for (auto& pr : fin) { float ms = 0; cudaEventElapsedTime(&ms, pr.first, pr.second); fms += ms; }
    c->prof.dp_ms = dms;
    c->prof.finalize_ms = fms;
    float tot = 0;
    if (first && last) cudaEventElapsedTime(&tot, first, last);
    c->prof.total_ms = tot;
  }
};

// error flag, insert count, task counters: one per DPX range or bit-parallel launch
constexpr size_t kCounterBytes = 64 + sizeof(unsigned long long) * 16;

struct RunOut {
  uint32_t dp_launches = 0;
};

// Launches one alignment launch of a plan on `stream`; `P` brings the terms,
// the epilogue's settings and the counter.
nw_status run_launch(nw_ctx* c, cudaStream_t stream, const Launch& l, const Seg* d_segs, int epi, AlignParams P,
                     Timer& tm, RunOut& ro) {
  const bool bits = l.range < 0;
  const int warps = bits ? kBitWarps : kWarpsPerBlock;
  P.segs = d_segs + l.seg_first;
  P.nsegs = l.nsegs;
  P.TA = l.ta;
  P.ntasks = l.ntasks;
  P.dbg_insert_limit = c->dbg_insert_iters >= 0 ? (uint32_t)c->dbg_insert_iters + 1u : 0u;
  const bool tab = !bits && P.sim_tab != nullptr;
  size_t smem = (epi == kEpiListsLaneHist || epi == kEpiLists ? hist_smem_words(P.hist_mode, P.nbins, warps) : 0) *
                sizeof(uint32_t);
  if (bits) {
    P.sub = std::max<uint32_t>(1, std::min<uint32_t>(kBitSub, l.ta / kBitWarps));
    P.mask_bytes = l.alphabet * kMaskRow;
    P.stage_syms = (P.sub * l.max_la + 2 + 7) & ~7u;
    smem += P.mask_bytes + (size_t)warps * P.stage_syms * sizeof(uint16_t);
  } else {
    P.stage_syms = 32u * std::max<uint32_t>(1, l.max_la);
    smem += (size_t)warps * P.stage_syms * sizeof(uint32_t) + (tab ? kTabBytes : 0);
  }
  const void* fn = bits ? bit_kernel(l.m, l.x, epi) : dp_kernel(l.range, epi, tab);
  if (!fn) return set_err(c, NW_EINVAL, "no alignment kernel for this launch");
  const int block = bits ? kBitBlock : kBlock;
  NW_CK(allow_shared(fn));
  int occ = 0;
  NW_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, block, smem));
  if (occ < 1) occ = 1;
  if (l.bps && occ > (int)l.bps) occ = (int)l.bps;
  const uint64_t grid = std::min<uint64_t>((uint64_t)c->sm_count * occ, bits ? l.ntasks : cdiv(l.ntasks, kWarpsPerBlock));
  void* args[] = {&P};
  cudaEvent_t e0 = nullptr;
  tm.begin(true, e0);
  NW_CK(cudaLaunchKernel(fn, dim3((unsigned)grid), dim3(block), args, smem, stream));
  tm.end(true, e0);
  ++ro.dp_launches;
  return NW_OK;
}

// All launches of a plan, in order; launch i takes counters[i].
nw_status run_plan(nw_ctx* c, cudaStream_t stream, const Plan& plan, const Seg* d_segs, int epi, const AlignParams& base,
                   unsigned long long* counters, Timer& tm, RunOut& ro) {
  for (size_t i = 0; i < plan.launches.size(); ++i) {
    AlignParams P = base;
    P.counter = counters + i;
    NW_TRY(run_launch(c, stream, plan.launches[i], d_segs, epi, P, tm, ro));
  }
  return NW_OK;
}

// Terms of dictionary `d`'s scoring between an A set and a B set.
Terms make_terms(const nw_dict* d, const WordSet& a, const WordSet& b, SideView A, SideView B, int32_t key_lo,
                 uint32_t ib) {
  Terms T{};
  T.a_sym = a.a_enc.as<uint32_t>();
  T.b_sym = b.a_enc.as<uint32_t>();
  T.b_rec = b.b_rec.as<uint4>();
  T.A = A;
  T.B = B;
  T.shift = d->ss.shift;
  T.alphabet = d->alphabet;
  T.coef = (uint32_t)d->ss.bit_coef;
  T.C1 = d->ss.C1;
  T.C2 = d->ss.C2;
  T.match = d->sc.match;
  T.mismatch = d->sc.mismatch;
  T.gap = d->sc.gap;
  T.key_lo = key_lo;
  T.ib = ib;
  T.imask = (uint32_t)(((uint64_t)1 << ib) - 1);
  return T;
}

// The word records for a call that scores m pairs on stream s, or null (the
// kernel then reads the pair records).  Making them takes an allocation, a kernel
// and a wait for it, about 100 us from 65,536 words on, and saves 15 to 40 us a
// million pairs (1,000,003 pairs of 100k words, 40 / 128 codes: 76 / 101 us without,
// 62 / 68 with), so they are made once the dictionary has met kRecordPairs pairs: no
// program pays for them much more than they have saved it.  None are made for pairs
// that another kernel scores, for a call that does not wait for its stream
// (may_wait), and a call that is being captured reads none: the memory may go.
constexpr uint64_t kRecordPairs = (uint64_t)3 << 20;
const uint4* pair_records(nw_dict* d, const PairsParams& P, uint64_t m, bool may_wait, cudaStream_t s) {
  nw_ctx* c = d->ctx;
  if (!pairs_take_bits(P) || d->ws.n == 0) return nullptr;
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &capture) != cudaSuccess || capture != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return nullptr;
  }
  if (d->rec.p) return d->rec.as<uint4>();
  d->pairs_scored += m;
  if (!may_wait || d->pairs_scored < kRecordPairs) return nullptr;
  const std::string err = c->err;
  if (ctx_alloc(c, d->rec, (size_t)d->ws.n * 16, "word records", /*give_up=*/false) != NW_OK) {
    c->err = err;
    return nullptr;
  }
  if (launch_word_records(d->ws.rank.as<uint32_t>(), d->ws.slen.as<uint8_t>(), d->ws.aoff.as<uint32_t>(),
                          d->ws.brec_w.as<uint32_t>(), d->ws.a_enc.as<uint32_t>(), d->ss.shift, d->ws.n, d->rec.as<uint4>(), s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess) {  // other streams may read them next
    cudaGetLastError();
    ctx_free(c, d->rec);
    return nullptr;
  }
  return d->rec.as<uint4>();
}

// the bit-parallel part of a pair list's parameters
void pairs_bits(const nw_dict* d, PairsParams& P) {
  P.bit_m = d->ss.bit_m;
  P.bit_x = d->ss.bit_x;
  P.coef = d->ss.bit_coef;
  P.shift = d->ss.shift;
  P.alphabet = d->alphabet;
  P.min_len = d->ws.min_len;
  P.max_len = d->ws.max_len;
}

int lists_epi(int hist_mode) { return hist_mode == kHistLane ? kEpiListsLaneHist : kEpiLists; }

// The whole pair set of a dictionary, or one shard of it (planned on the spot
// through the context's segment workspace).
nw_status run_dict(nw_dict* d, int epi, const AlignParams& base, unsigned long long* counters, uint32_t shard,
                   uint32_t nshards, Timer& tm, RunOut& ro) {
  nw_ctx* c = d->ctx;
  if (nshards == 1) return run_plan(c, c->stream, d->plan, d->d_segs.as<Seg>(), epi, base, counters, tm, ro);
  Rects rects;
  rects_shard(d->ws.bk, shard, nshards, rects);
  Plan plan;
  make_plan(std::move(rects), d->ss, d->alphabet, 0, plan);
  NW_TRY(ctx_ensure(c, c->ws_segs, sizeof(Seg) * std::max<size_t>(1, plan.segs.size()), "shard segments"));
  if (!plan.segs.empty()) {
    NW_CK(cudaMemcpyAsync(c->ws_segs.p, plan.segs.data(), sizeof(Seg) * plan.segs.size(), cudaMemcpyHostToDevice, c->stream));
    NW_CK(cudaStreamSynchronize(c->stream));  // the host list goes out of scope
  }
  return run_plan(c, c->stream, plan, c->ws_segs.as<Seg>(), epi, base, counters, tm, ro);
}

nw_status check_device_flags(nw_ctx* c, const uint32_t* d_small) {
  uint32_t err = 0;
  NW_CK(cudaMemcpyAsync(&err, d_small, sizeof(uint32_t), cudaMemcpyDeviceToHost, c->stream));
  NW_CK(cudaStreamSynchronize(c->stream));
  if (err & kErrRetry) return set_err(c, NW_ETIMEOUT, "a neighbour-list update exceeded its retry bound");
  if (err & kErrWait) return set_err(c, NW_ETIMEOUT, "a pipeline wait on the device ran out");
  if (err & kErrInput) return set_err(c, NW_EINVAL, "invalid word index in the input (outputs may be partially written)");
  if (err & kErrCapacity) return set_err(c, NW_ERANGE, "a device buffer reached its capacity (outputs are not valid)");
  if (err & kErrHistRange) return set_err(c, NW_ERANGE, "a score fell outside the histogram range");
  return NW_OK;
}

nw_status topk_impl(nw_dict* d, uint32_t shard, uint32_t nshards, uint32_t k, uint32_t* nbr_idx,
                    int16_t* nbr_score, int64_t* hist, int32_t* hist_lo, uint32_t nbins, uint32_t flags) {
  nw_ctx* c = d->ctx;
  const uint32_t n = d->ws.n;
  if (n < 2) return set_err(c, NW_EINVAL, "the dictionary needs at least 2 words (has %u)", n);
  if (k == 0 || k > NW_MAX_K) return set_err(c, NW_EINVAL, "k must be in [1, %d]", NW_MAX_K);
  if (!nbr_idx || !nbr_score) return set_err(c, NW_EINVAL, "null output pointer");
  if (nshards == 0 || shard >= nshards) return set_err(c, NW_EINVAL, "shard %u of %u", shard, nshards);
  const uint32_t need_bins = (uint32_t)(d->score_hi - d->score_lo + 1);
  if (hist && nbins < need_bins)
    return set_err(c, NW_ERANGE, "histogram needs %u bins for scores [%d, %d], got %u", need_bins, d->score_lo,
                   d->score_hi, nbins);
  if (d->score_lo < INT16_MIN + 1 || d->score_hi > INT16_MAX)
    return set_err(c, NW_ERANGE, "scores [%d, %d] do not fit int16", d->score_lo, d->score_hi);
  const uint32_t ib = index_bits(n);
  const int32_t key_lo = d->score_lo - 1;
  const bool norm = flags & NW_RANK_NORMALISED;
  if (norm && nshards != 1)
    return set_err(c, NW_EINVAL, "the normalised ranking is not available for shards (lists merge by raw score)");
  NormTables nt;
  if (norm) {
    build_norm_tables(d->sc, d->score_lo, d->score_hi, nt);
    if (nt.nranks > 65535u || (uint64_t)nt.nranks >= (1ull << (32 - ib)))
      return set_err(c, NW_ERANGE, "%u normalised score values with %u words do not fit 32-bit list keys", nt.nranks,
                     n);
  } else if ((uint64_t)(d->score_hi - key_lo) >= (1ull << (32 - ib))) {
    return set_err(c, NW_ERANGE, "score range %d..%d with %u words does not fit 32-bit list keys", d->score_lo,
                   d->score_hi, n);
  }
  const bool dev = flags & NW_DEVICE_PTRS;
  cudaStream_t s = c->stream;
  NW_TRY(ctx_ensure(c, c->ws_slots, sizeof(uint32_t) * (size_t)n * k, "list slots"));
  NW_TRY(ctx_ensure(c, c->ws_thr, sizeof(uint32_t) * (size_t)n, "list thresholds"));
  NW_TRY(ctx_ensure(c, c->ws_small, kCounterBytes, "task counters"));
  if (hist) NW_TRY(ctx_ensure(c, c->ws_hist, sizeof(unsigned long long) * need_bins, "histogram"));
  uint32_t* out_idx = nbr_idx;
  int16_t* out_score = nbr_score;
  if (!dev) {
    NW_TRY(ctx_ensure(c, c->ws_out_idx, sizeof(uint32_t) * (size_t)n * k, "output indices"));
    NW_TRY(ctx_ensure(c, c->ws_out_score, sizeof(int16_t) * (size_t)n * k, "output scores"));
    out_idx = c->ws_out_idx.as<uint32_t>();
    out_score = c->ws_out_score.as<int16_t>();
  }
  uint32_t* d_err = c->ws_small.as<uint32_t>();
  unsigned long long* d_stats = reinterpret_cast<unsigned long long*>(c->ws_small.as<char>() + 8);
  unsigned long long* d_counters = reinterpret_cast<unsigned long long*>(c->ws_small.as<char>() + 64);

  Timer tm{c};
  cudaEvent_t e_all = nullptr;
  tm.begin(false, e_all);
  NW_CK(cudaMemsetAsync(c->ws_small.p, 0, c->ws_small.bytes, s));
  NW_CK(cudaMemsetAsync(c->ws_slots.p, 0, sizeof(uint32_t) * (size_t)n * k, s));
  NW_CK(cudaMemsetAsync(c->ws_thr.p, 0, sizeof(uint32_t) * (size_t)n, s));
  if (hist) NW_CK(cudaMemsetAsync(c->ws_hist.p, 0, sizeof(unsigned long long) * need_bins, s));

  AlignParams base{};
  base.sim_tab = dict_tab(d);
  base.k = k;
  base.hist_mode = !hist ? kHistNone : hist_mode_for(need_bins);
  base.hist = hist ? c->ws_hist.as<unsigned long long>() : nullptr;
  base.hist_lo = d->score_lo;
  base.nbins = hist ? need_bins : 0;
  base.stats = d_stats;
  base.err = d_err;
  const int16_t* d_frac = nullptr;
  if (norm) {
    // one upload of the three tables, each at a 256-byte aligned offset
    const size_t rank_b = nt.rank.size() * sizeof(uint16_t), smin_b = nt.smin.size() * sizeof(int16_t);
    const size_t o_smin = (rank_b + 255) & ~(size_t)255, o_frac = (o_smin + smin_b + 255) & ~(size_t)255;
    const size_t total = o_frac + nt.frac.size() * sizeof(int16_t);
    NW_TRY(ctx_ensure(c, c->ws_norm, total, "normalised ranking tables"));
    std::vector<char> h(total, 0);
    std::memcpy(h.data(), nt.rank.data(), rank_b);
    std::memcpy(h.data() + o_smin, nt.smin.data(), smin_b);
    std::memcpy(h.data() + o_frac, nt.frac.data(), nt.frac.size() * sizeof(int16_t));
    NW_CK(cudaMemcpyAsync(c->ws_norm.p, h.data(), total, cudaMemcpyHostToDevice, s));
    NW_CK(cudaStreamSynchronize(s));  // the staging vector goes out of scope
    base.norm_rank = c->ws_norm.as<uint16_t>();
    base.norm_smin = reinterpret_cast<const int16_t*>(c->ws_norm.as<char>() + o_smin);
    base.norm_lo = nt.lo;
    d_frac = reinterpret_cast<const int16_t*>(c->ws_norm.as<char>() + o_frac);
  }
  SideView side{d->ws.perm.as<uint32_t>(), c->ws_slots.as<uint32_t>(), c->ws_thr.as<uint32_t>()};
  base.local[0] = make_terms(d, d->ws, d->ws, side, side, key_lo, ib);
  RunOut ro;
  NW_TRY(run_dict(d, lists_epi(base.hist_mode), base, d_counters, shard, nshards, tm, ro));
  cudaEvent_t e_fin = nullptr;
  tm.begin(false, e_fin);
  NW_CK(launch_finalize(c->ws_slots.as<uint32_t>(), n, k, d->ws.perm.as<uint32_t>(), ib, base.local[0].imask, key_lo,
                        out_idx, out_score, s, d_frac, d->ws.slen.as<uint8_t>(), d->ws.rank.as<uint32_t>()));
  tm.end(false, e_fin);
  if (hist && dev) NW_CK(cudaMemcpyAsync(hist, c->ws_hist.p, sizeof(int64_t) * need_bins, cudaMemcpyDeviceToDevice, s));
  if (!dev) {
    NW_CK(cudaMemcpyAsync(nbr_idx, out_idx, sizeof(uint32_t) * (size_t)n * k, cudaMemcpyDeviceToHost, s));
    NW_CK(cudaMemcpyAsync(nbr_score, out_score, sizeof(int16_t) * (size_t)n * k, cudaMemcpyDeviceToHost, s));
    if (hist) NW_CK(cudaMemcpyAsync(hist, c->ws_hist.p, sizeof(int64_t) * need_bins, cudaMemcpyDeviceToHost, s));
  }
  if (hist) {
    if (hist_lo) *hist_lo = d->score_lo;
    if (nbins > need_bins) {
      if (dev) NW_CK(cudaMemsetAsync(hist + need_bins, 0, sizeof(int64_t) * (nbins - need_bins), s));
      else std::memset(hist + need_bins, 0, sizeof(int64_t) * (nbins - need_bins));
    }
  }
  tm.mark(tm.c->profiling ? tm.get() : nullptr);
  if ((flags & NW_ASYNC) && dev) return NW_OK;
  NW_TRY(check_device_flags(c, d_err));
  if (c->profiling) {
    tm.collect();
    unsigned long long ins = 0;
    NW_CK(cudaMemcpy(&ins, d_stats, sizeof ins, cudaMemcpyDeviceToHost));
    c->prof.dp_launches = ro.dp_launches;
    c->prof.launches = ro.dp_launches + 1;
    c->prof.pairs = nshards == 1 ? d->plan.pairs : 0;
    c->prof.cells = nshards == 1 ? d->plan.cells : 0;
    c->prof.list_inserts = ins;
  }
  return NW_OK;
}

}  // namespace

