// nw_batch.cu -- nw_batch_*: many independent dictionaries, each with an
// optional query set, reduced to top-k lists in one CUDA-graph launch.
//
// Every dictionary is loaded as usual (its own word set, scoring and score
// bounds), and its query set is ingested with the dictionary's alphabet and
// code shift.  The pair lists of all dictionaries and query sets are planned
// together, each rectangle tagged with its terms (3d for dictionary d's own
// pairs, 3d + 1 for its queries as A words, 3d + 2 for its queries as B words);
// the kernels (epilogue kEpiOtherLists) read those terms' word sets, lists and
// scoring per task.  Dictionaries whose scoring the bit-parallel kernel takes
// share one launch per step class, on a second stream; the others share one
// DPX launch per range of longer lengths, whose A-chunk size is a tile-shape
// parameter that the autotuner picks by timing candidates on the batch.  The
// whole reduction is captured once into a CUDA graph and replayed by
// nw_batch_run / nw_batch_run_queries.
#include <chrono>
#include <map>
#include <mutex>

#include "nw_host.h"

struct nw_batch {
  nw_ctx* ctx = nullptr;
  cudaStream_t stream = nullptr;  // the batch's own stream (capture needs a non-legacy stream)
  cudaStream_t side = nullptr;    // the bit-parallel launches run here, forked from and joined to `stream`
  cudaEvent_t forked = nullptr, joined = nullptr;
  std::vector<nw_dict*> dicts;
  std::vector<WordSet> qsets;     // each dictionary's query set (n = 0: none)
  std::vector<uint8_t> self;      // 1: the dictionary's own lists are computed
  uint32_t k = 0;
  Rects dp_rects;                      // the DPX launches' pairs, ordered
  uint32_t ta[kDpRanges] = {0};        // their A words per task, by range of longer lengths
  uint32_t bps[kDpRanges] = {0};       // resident blocks per SM at most (0: as many as fit)
  bool has_len[kBuckets] = {false};    // longer lengths with pairs, and of which in DPX launches
  bool dp_len[kBuckets] = {false};
  bool tune_cached = false;
  Plan plan;
  std::vector<size_t> list_off;   // first list of each dictionary's own lists in the combined arrays
  std::vector<size_t> qlist_off;  // first list of each query set in the combined arrays
  std::vector<int32_t> q_key_lo;  // list-key offset of each query set (its lowest score - 1)
  size_t nlists = 0;
  uint32_t query_words = 0;
  uint64_t query_pairs = 0, query_cells = 0;
  DevBuf d_segs, d_terms, d_slots, d_thr, d_small, d_out_idx, d_out_score;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  double tune_ms = 0;
};

namespace {

constexpr uint32_t kTaCandidates[] = {64, 128, 256};

// Terms of dictionary d's own pairs (role 0) and of its query set as A words
// (role 1) or B words (role 2).
uint32_t term_index(size_t d, int role) { return (uint32_t)(3 * d + role); }

AlignParams batch_params(nw_batch* B) {
  AlignParams P{};
  P.k = B->k;
  P.hist_mode = kHistNone;
  P.stats = reinterpret_cast<unsigned long long*>(B->d_small.as<char>() + 8);
  P.err = B->d_small.as<uint32_t>();
  P.terms = B->d_terms.as<Terms>();
  return P;
}

nw_status upload_plan(nw_batch* B, const Plan& plan) {
  nw_ctx* c = B->ctx;
  NW_TRY(ctx_ensure(c, B->d_segs, sizeof(Seg) * std::max<size_t>(1, plan.segs.size()), "batch segments"));
  if (!plan.segs.empty())
    NW_CK(cudaMemcpyAsync(B->d_segs.p, plan.segs.data(), sizeof(Seg) * plan.segs.size(), cudaMemcpyHostToDevice,
                          B->stream));
  return NW_OK;
}

// List resets and the alignment launches of `plan`: the DPX launches on the
// batch's stream, the bit-parallel ones beside them on its side stream.
nw_status issue_lists(nw_batch* B, const Plan& plan) {
  nw_ctx* c = B->ctx;
  cudaStream_t s = B->stream;
  NW_CK(cudaMemsetAsync(B->d_small.p, 0, B->d_small.bytes, s));
  NW_CK(cudaMemsetAsync(B->d_slots.p, 0, sizeof(uint32_t) * B->nlists * B->k, s));
  NW_CK(cudaMemsetAsync(B->d_thr.p, 0, sizeof(uint32_t) * B->nlists, s));
  const bool saved = c->profiling;
  c->profiling = false;
  struct Restore {
    nw_ctx* c;
    bool v;
    ~Restore() { c->profiling = v; }
  } restore{c, saved};
  Timer tm{c};
  RunOut ro;
  NW_CK(cudaEventRecord(B->forked, s));
  NW_CK(cudaStreamWaitEvent(B->side, B->forked, 0));
  nw_status st = NW_OK;
  for (size_t i = 0; i < plan.launches.size() && st == NW_OK; ++i) {
    AlignParams P = batch_params(B);
    P.counter = reinterpret_cast<unsigned long long*>(B->d_small.as<char>() + 64) + i;
    st = run_launch(c, plan.launches[i].range < 0 ? B->side : s, plan.launches[i], B->d_segs.as<Seg>(), kEpiOtherLists,
                    P, tm, ro);
  }
  NW_CK(cudaEventRecord(B->joined, B->side));
  NW_CK(cudaStreamWaitEvent(s, B->joined, 0));
  return st;
}

nw_status issue_finalize(nw_batch* B) {
  nw_ctx* c = B->ctx;
  for (size_t d = 0; d < B->dicts.size(); ++d) {
    const nw_dict* D = B->dicts[d];
    const uint32_t n = D->ws.n;
    const uint32_t ib = index_bits(std::max<uint32_t>(n, 2));
    const uint32_t imask = (uint32_t)(((uint64_t)1 << ib) - 1);
    if (B->self[d] && n) {
      NW_CK(launch_finalize(B->d_slots.as<uint32_t>() + B->list_off[d] * B->k, n, B->k, D->ws.perm.as<uint32_t>(),
                            ib, imask, D->score_lo - 1, B->d_out_idx.as<uint32_t>() + B->list_off[d] * B->k,
                            B->d_out_score.as<int16_t>() + B->list_off[d] * B->k, B->stream));
    }
    const WordSet& Q = B->qsets[d];
    if (Q.n) {  // query lists name dictionary words, as nw_query's do
      NW_CK(launch_finalize(B->d_slots.as<uint32_t>() + B->qlist_off[d] * B->k, Q.n, B->k, Q.perm.as<uint32_t>(),
                            ib, imask, B->q_key_lo[d], B->d_out_idx.as<uint32_t>() + B->qlist_off[d] * B->k,
                            B->d_out_score.as<int16_t>() + B->qlist_off[d] * B->k, B->stream));
    }
  }
  return NW_OK;
}

// The autotuner's choices, kept for the life of the process and keyed by the
// batch's shape (tune_key): a batch of the same shape is not timed again.
struct TunedShape {
  uint32_t ta[kDpRanges];
  uint32_t bps[kDpRanges];
};
std::mutex& tune_mutex() {
  static std::mutex m;
  return m;
}
std::map<uint64_t, TunedShape>& tune_cache() {
  static std::map<uint64_t, TunedShape> m;
  return m;
}

// FNV-1a over the device's SM count, k, and every dictionary's and query
// set's length histogram, scoring and flags: what the launches' work and
// their timing follow.
uint64_t tune_key(const nw_batch* B) {
  uint64_t h = 1469598103934665603ull;
  auto mix = [&h](uint64_t v) {
    for (int i = 0; i < 8; ++i) {
      h ^= (v >> (8 * i)) & 0xffu;
      h *= 1099511628211ull;
    }
  };
  mix((uint64_t)B->ctx->sm_count);
  mix(B->k);
  mix(B->dicts.size());
  for (size_t d = 0; d < B->dicts.size(); ++d) {
    const nw_dict* D = B->dicts[d];
    mix(B->self[d]);
    mix(D->alphabet);
    mix((uint32_t)D->sc.match);
    mix((uint32_t)D->sc.mismatch);
    mix((uint32_t)D->sc.gap);
    mix(D->subst ? 1u : 0u);
    for (int L = 0; L < kBuckets; ++L) mix(D->ws.bk.count[L]);
    for (int L = 0; L < kBuckets; ++L) mix(B->qsets[d].bk.count[L]);
  }
  return h;
}

constexpr uint32_t kBpsCandidates[] = {3, 2};

// Per DPX launch: the fastest A-chunk candidate, then the fastest cap on
// resident blocks per SM at that chunk (whole launches timed on the batch).
nw_status autotune(nw_batch* B) {
  nw_ctx* c = B->ctx;
  const uint64_t key = tune_key(B);
  {
    std::lock_guard<std::mutex> lk(tune_mutex());
    auto it = tune_cache().find(key);
    if (it != tune_cache().end()) {
      std::copy(it->second.ta, it->second.ta + kDpRanges, B->ta);
      std::copy(it->second.bps, it->second.bps + kDpRanges, B->bps);
      B->tune_cached = true;
      B->tune_ms = 0;
      return NW_OK;
    }
  }
  const auto t0 = std::chrono::steady_clock::now();
  cudaEvent_t e0, e1;
  NW_CK(cudaEventCreate(&e0));
  NW_CK(cudaEventCreate(&e1));
  struct EvFree {
    cudaEvent_t a, b;
    ~EvFree() { cudaEventDestroy(a); cudaEventDestroy(b); }
  } evfree{e0, e1};
  constexpr size_t kNta = sizeof(kTaCandidates) / sizeof(kTaCandidates[0]);
  // one timed launch of range r with chunk candidate ci and cap bps; ms < 0 if the range has no pairs
  auto time_launch = [&](int r, size_t ci, uint32_t bps, bool& warm, float& ms) -> nw_status {
    Plan p;
    plan_dp(B->dp_rects, kTaCandidates[ci], p, r, bps);
    ms = -1.f;
    if (p.launches.empty()) return NW_OK;
    NW_TRY(upload_plan(B, p));
    if (!warm) {  // the kernel's first launch pays its set-up; keep it out of the timings
      NW_TRY(issue_lists(B, p));
      warm = true;
    }
    NW_CK(cudaEventRecord(e0, B->stream));
    NW_TRY(issue_lists(B, p));
    NW_CK(cudaEventRecord(e1, B->stream));
    NW_CK(cudaEventSynchronize(e1));
    NW_CK(cudaEventElapsedTime(&ms, e0, e1));
    return NW_OK;
  };
  for (int r = 0; r < kDpRanges; ++r) {
    float best = 0;
    size_t best_ci = kNta;
    bool warm = false;
    for (size_t ci = 0; ci < kNta; ++ci) {
      float ms;
      NW_TRY(time_launch(r, ci, 0, warm, ms));
      if (ms < 0) break;
      if (best_ci == kNta || ms < best) {
        best = ms;
        best_ci = ci;
      }
    }
    if (best_ci == kNta) continue;  // ranges without pairs keep the defaults
    B->ta[r] = kTaCandidates[best_ci];
    for (uint32_t bps : kBpsCandidates) {
      float ms;
      NW_TRY(time_launch(r, best_ci, bps, warm, ms));
      if (ms >= 0 && ms < best) {
        best = ms;
        B->bps[r] = bps;
      }
    }
  }
  B->tune_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
  TunedShape t;
  std::copy(B->ta, B->ta + kDpRanges, t.ta);
  std::copy(B->bps, B->bps + kDpRanges, t.bps);
  std::lock_guard<std::mutex> lk(tune_mutex());
  tune_cache()[key] = t;
  return NW_OK;
}

nw_status check_flags(nw_ctx* c, cudaStream_t stream, const uint32_t* d_err) {
  uint32_t err = 0;
  NW_CK(cudaMemcpyAsync(&err, d_err, sizeof err, cudaMemcpyDeviceToHost, stream));
  NW_CK(cudaStreamSynchronize(stream));
  if (err & kErrRetry) return set_err(c, NW_ETIMEOUT, "a neighbour-list update exceeded its retry bound");
  if (err) return set_err(c, NW_EINVAL, "device-side error flag %u", err);
  return NW_OK;
}

nw_status create_impl(nw_batch* B, const nw_batch_dict* dicts, uint32_t ndicts, uint32_t flags) {
  nw_ctx* c = B->ctx;
  for (uint32_t d = 0; d < ndicts; ++d) {
    nw_dict* D = nullptr;
    const nw_status st = nw_load_dictionary(c, dicts[d].codes, dicts[d].offsets, dicts[d].n, dicts[d].alphabet,
                                            &dicts[d].scoring, flags & NW_DEVICE_PTRS, &D);
    if (st != NW_OK) return st;
    B->dicts.push_back(D);
    B->qsets.emplace_back();
    B->self.push_back(dicts[d].queries_only ? 0 : 1);
    const uint32_t ib = index_bits(std::max<uint32_t>(D->ws.n, 2));
    if (B->self[d] && (D->score_lo < INT16_MIN + 1 || D->score_hi > INT16_MAX ||
                       (uint64_t)(D->score_hi - (D->score_lo - 1)) >= (1ull << (32 - ib))))
      return set_err(c, NW_ERANGE, "dictionary %u: scores [%d, %d] do not fit the list keys", d, D->score_lo,
                     D->score_hi);
    B->list_off.push_back(B->nlists);
    if (B->self[d]) B->nlists += D->ws.n;
    // the query set: ingested with the dictionary's alphabet and code shift;
    // its list keys span the scores of the (query length, dictionary length)
    // pairs present, as in nw_query
    int32_t key_lo = 0;
    if (dicts[d].nq) {
      if (!dicts[d].qoffsets) return set_err(c, NW_EINVAL, "dictionary %u: null query offsets", d);
      NW_TRY(ingest(c, dicts[d].qcodes, dicts[d].qoffsets, dicts[d].nq, D->alphabet, D->ss.shift,
                    flags & NW_DEVICE_PTRS, B->qsets[d]));
      const WordSet& Q = B->qsets[d];
      int lo = INT32_MAX, hi = INT32_MIN;
      for (int La = 0; La < kBuckets; ++La)
        for (int Lb = 0; Lb < kBuckets; ++Lb) {
          if (!Q.bk.count[La] || !D->ws.bk.count[Lb]) continue;
          int l, h;
          pair_bounds(D->sc, La, Lb, l, h);
          lo = std::min(lo, l);
          hi = std::max(hi, h);
        }
      if (D->ws.n == 0) lo = hi = 0;
      if (lo < INT16_MIN + 1 || hi > INT16_MAX || (uint64_t)(hi - (lo - 1)) >= (1ull << (32 - ib)))
        return set_err(c, NW_ERANGE, "query set %u: scores [%d, %d] do not fit the list keys", d, lo, hi);
      key_lo = lo - 1;
      B->query_words += Q.n;
    }
    B->q_key_lo.push_back(key_lo);
    B->qlist_off.push_back(B->nlists);
    B->nlists += B->qsets[d].n;
  }
  const size_t L = std::max<size_t>(1, B->nlists);
  NW_TRY(ctx_alloc(c, B->d_slots, sizeof(uint32_t) * L * B->k, "batch list slots"));
  NW_TRY(ctx_alloc(c, B->d_thr, sizeof(uint32_t) * L, "batch list bounds"));
  NW_TRY(ctx_alloc(c, B->d_out_idx, sizeof(uint32_t) * L * B->k, "batch output indices"));
  NW_TRY(ctx_alloc(c, B->d_out_score, sizeof(int16_t) * L * B->k, "batch output scores"));
  NW_TRY(ctx_alloc(c, B->d_small, kCounterBytes, "batch counters"));
  std::vector<Terms> terms(std::max<size_t>(1, 3 * B->dicts.size()));
  // the pairs: DPX dictionaries together, the others by step class
  struct Group {
    int m, x;
    uint32_t alphabet;
    Rects rects;
  };
  std::vector<Group> groups;
  for (size_t d = 0; d < B->dicts.size(); ++d) {
    const nw_dict* D = B->dicts[d];
    const WordSet& Q = B->qsets[d];
    const uint32_t ib = index_bits(std::max<uint32_t>(D->ws.n, 2));
    const SideView dict_side{D->ws.perm.as<uint32_t>(), B->d_slots.as<uint32_t>() + B->list_off[d] * B->k,
                             B->d_thr.as<uint32_t>() + B->list_off[d]};
    const SideView dict_nolists{D->ws.perm.as<uint32_t>(), nullptr, nullptr};
    const SideView query_side{Q.perm.as<uint32_t>(), B->d_slots.as<uint32_t>() + B->qlist_off[d] * B->k,
                              B->d_thr.as<uint32_t>() + B->qlist_off[d]};
    terms[term_index(d, 0)] = make_terms(D, D->ws, D->ws, dict_side, dict_side, D->score_lo - 1, ib);
    terms[term_index(d, 1)] = make_terms(D, Q, D->ws, query_side, dict_nolists, B->q_key_lo[d], ib);
    terms[term_index(d, 2)] = make_terms(D, D->ws, Q, dict_nolists, query_side, B->q_key_lo[d], ib);
    Rects* rects = &B->dp_rects;  // of the dictionary's pairs, those that are not taken out for the DPX launches
    if (D->ss.bit_m) {
      auto g = std::find_if(groups.begin(), groups.end(),
                            [&](const Group& x) { return x.m == D->ss.bit_m && x.x == D->ss.bit_x; });
      if (g == groups.end()) g = groups.insert(g, Group{D->ss.bit_m, D->ss.bit_x, 0, {}});
      g->alphabet = std::max(g->alphabet, D->alphabet);
      rects = &g->rects;
    }
    Rects own, queries;
    if (B->self[d]) rects_all(D->ws.bk, term_index(d, 0), own);
    if (Q.n) rects_queries(Q.bk, D->ws.bk, term_index(d, 1), queries);
    count_rects(queries, B->query_pairs, B->query_cells);
    for (Rects* list : {&own, &queries}) {
      const Rects dpx = D->ss.bit_m ? take_long(*list, D->ss) : std::move(*list);
      if (D->ss.bit_m)
        for (const Rect& r : *list) {
          rects->push_back(r);
          B->has_len[r.LB] = true;
        }
      for (const Rect& r : dpx) {
        B->dp_rects.push_back(r);
        B->has_len[r.LB] = B->dp_len[r.LB] = true;
      }
    }
  }
  NW_TRY(ctx_alloc(c, B->d_terms, sizeof(Terms) * terms.size(), "batch terms"));
  NW_CK(cudaMemcpyAsync(B->d_terms.p, terms.data(), sizeof(Terms) * terms.size(), cudaMemcpyHostToDevice, B->stream));

  order_rects(B->dp_rects);
  for (uint32_t& t : B->ta) t = kDefaultTA;
  if (flags & NW_BATCH_AUTOTUNE) NW_TRY(autotune(B));
  B->plan = Plan{};
  for (int r = 0; r < kDpRanges; ++r) plan_dp(B->dp_rects, B->ta[r], B->plan, r, B->bps[r]);
  count_rects(B->dp_rects, B->plan.pairs, B->plan.cells);
  for (Group& g : groups) {
    order_rects(g.rects);
    Plan p;
    sized(p, kBitMinTasks, [&](uint32_t ta, Plan& q) { plan_bits(g.rects, g.m, g.x, g.alphabet, ta, q); });
    append_plan(B->plan, p);
    count_rects(g.rects, B->plan.pairs, B->plan.cells);
  }
  NW_TRY(upload_plan(B, B->plan));
  // one uncaptured run sets the kernels' shared-memory attributes
  NW_TRY(issue_lists(B, B->plan));
  NW_TRY(issue_finalize(B));
  NW_TRY(check_flags(c, B->stream, B->d_small.as<uint32_t>()));

  NW_CK(cudaStreamBeginCapture(B->stream, cudaStreamCaptureModeThreadLocal));
  nw_status st = issue_lists(B, B->plan);
  if (st == NW_OK) st = issue_finalize(B);
  cudaGraph_t g = nullptr;
  const cudaError_t ce = cudaStreamEndCapture(B->stream, &g);
  if (st != NW_OK) {
    if (g) cudaGraphDestroy(g);
    return st;
  }
  if (ce != cudaSuccess) return cuda_fail(c, ce, "cudaStreamEndCapture");
  B->graph = g;
  NW_CK(cudaGraphInstantiate(&B->exec, B->graph, 0));
  return NW_OK;
}

void destroy_impl(nw_batch* B) {
  nw_ctx* c = B->ctx;
  if (B->stream) cudaStreamSynchronize(B->stream);
  if (B->exec) cudaGraphExecDestroy(B->exec);
  if (B->graph) cudaGraphDestroy(B->graph);
  for (DevBuf* b : {&B->d_segs, &B->d_terms, &B->d_slots, &B->d_thr, &B->d_small, &B->d_out_idx, &B->d_out_score})
    ctx_free(c, *b);
  for (WordSet& Q : B->qsets) free_wordset(c, Q);
  for (nw_dict* D : B->dicts) nw_dict_free(D);
  if (B->side) {
    cudaStreamSynchronize(B->side);
    cudaStreamDestroy(B->side);
  }
  if (B->forked) cudaEventDestroy(B->forked);
  if (B->joined) cudaEventDestroy(B->joined);
  if (B->stream) cudaStreamDestroy(B->stream);
  delete B;
}

}  // namespace

extern "C" {

nw_status nw_batch_create(nw_ctx* ctx, const nw_batch_dict* dicts, uint32_t ndicts, uint32_t k, uint32_t flags,
                          nw_batch** out) {
  if (!ctx || !out) return NW_EINVAL;
  *out = nullptr;
  if (!dicts && ndicts) return set_err(ctx, NW_EINVAL, "null dictionary array");
  if (k == 0 || k > NW_MAX_K) return set_err(ctx, NW_EINVAL, "k must be in [1, %d]", NW_MAX_K);
  if (flags & NW_RANK_NORMALISED) return set_err(ctx, NW_EINVAL, "batches rank by raw score only");
  if (cudaSetDevice(ctx->device) != cudaSuccess) return cuda_fail(ctx, cudaGetLastError(), "cudaSetDevice");
  nw_batch* B = new nw_batch();
  B->ctx = ctx;
  B->k = k;
  nw_status st = NW_OK;
  if (cudaStreamCreateWithFlags(&B->stream, cudaStreamNonBlocking) != cudaSuccess ||
      cudaStreamCreateWithFlags(&B->side, cudaStreamNonBlocking) != cudaSuccess ||
      cudaEventCreateWithFlags(&B->forked, cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&B->joined, cudaEventDisableTiming) != cudaSuccess)
    st = cuda_fail(ctx, cudaGetLastError(), "cudaStreamCreateWithFlags");
  if (st == NW_OK) st = create_impl(B, dicts, ndicts, flags);
  if (st != NW_OK) {
    const std::string msg = ctx->err;
    destroy_impl(B);
    ctx->err = msg;
    return st;
  }
  *out = B;
  return NW_OK;
}

nw_status nw_batch_run_queries(nw_batch* B, uint32_t* const* nbr_idx, int16_t* const* nbr_score,
                               uint32_t* const* qnbr_idx, int16_t* const* qnbr_score, uint32_t flags) {
  if (!B) return NW_EINVAL;
  nw_ctx* c = B->ctx;
  NW_ENTER(c);
  if (flags & NW_RANK_NORMALISED) return set_err(c, NW_EINVAL, "batches rank by raw score only");
  const bool want_q = qnbr_idx || qnbr_score;
  if (want_q && (!qnbr_idx || !qnbr_score)) return set_err(c, NW_EINVAL, "null query output arrays");
  // every buffer the copies need, checked before the graph runs
  for (size_t d = 0; d < B->dicts.size(); ++d) {
    if (B->self[d] && B->dicts[d]->ws.n &&
        (!nbr_idx || !nbr_score || !nbr_idx[d] || !nbr_score[d]))
      return set_err(c, NW_EINVAL, "null output for dictionary %zu", d);
    if (want_q && B->qsets[d].n && (!qnbr_idx[d] || !qnbr_score[d]))
      return set_err(c, NW_EINVAL, "null query output for dictionary %zu", d);
  }
  const bool dev = flags & NW_DEVICE_PTRS;
  const cudaMemcpyKind kind = dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
  NW_CK(cudaGraphLaunch(B->exec, B->stream));
  auto copy_out = [&](uint32_t* idx, int16_t* score, size_t first, size_t lists) -> nw_status {
    const size_t cnt = lists * B->k;
    NW_CK(cudaMemcpyAsync(idx, B->d_out_idx.as<uint32_t>() + first * B->k, sizeof(uint32_t) * cnt, kind, B->stream));
    NW_CK(cudaMemcpyAsync(score, B->d_out_score.as<int16_t>() + first * B->k, sizeof(int16_t) * cnt, kind,
                          B->stream));
    return NW_OK;
  };
  for (size_t d = 0; d < B->dicts.size(); ++d) {
    if (B->self[d] && B->dicts[d]->ws.n) NW_TRY(copy_out(nbr_idx[d], nbr_score[d], B->list_off[d], B->dicts[d]->ws.n));
    if (want_q && B->qsets[d].n) NW_TRY(copy_out(qnbr_idx[d], qnbr_score[d], B->qlist_off[d], B->qsets[d].n));
  }
  if ((flags & NW_ASYNC) && dev) return NW_OK;
  return check_flags(c, B->stream, B->d_small.as<uint32_t>());
}

nw_status nw_batch_run(nw_batch* B, uint32_t* const* nbr_idx, int16_t* const* nbr_score, uint32_t flags) {
  return nw_batch_run_queries(B, nbr_idx, nbr_score, nullptr, nullptr, flags);
}

nw_status nw_batch_info_get(const nw_batch* B, nw_batch_info* out) {
  if (!B || !out) return NW_EINVAL;
  nw_batch_info i{};
  i.ndicts = (uint32_t)B->dicts.size();
  i.launches = (uint32_t)B->plan.launches.size();
  i.pairs = B->plan.pairs;
  i.cells = B->plan.cells;
  i.tune_ms = B->tune_ms;
  // lengths met in bit-parallel launches alone: the size their chunks start from
  for (int L = 0; L < kBuckets; ++L) {
    i.words_per_task[L] = B->dp_len[L] ? B->ta[dp_range_of(L)] : (B->has_len[L] ? kDefaultTA : 0);
    i.blocks_per_sm[L] = B->dp_len[L] ? B->bps[dp_range_of(L)] : 0;
  }
  i.tune_cached = B->tune_cached ? 1u : 0u;
  i.query_words = B->query_words;
  i.query_pairs = B->query_pairs;
  i.query_cells = B->query_cells;
  *out = i;
  return NW_OK;
}

void nw_batch_free(nw_batch* B) {
  if (!B) return;
  cudaSetDevice(B->ctx->device);
  destroy_impl(B);
}

}  // extern "C"
