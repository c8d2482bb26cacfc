// Fused verify pass: tree mask -> attention -> LM-head statistics -> acceptance scan on one
// stream (one verification round of Algorithm 1 for one verifier).
#include <mutex>
#include <optional>
#include <stdlib.h>

#include "attn_common.cuh"

namespace trispec {
// Second streams (with their events) of the fused passes. A set belongs to one stream of the caller's, so that callers on
// different streams never wait for each other's work, and a set that is part of a capture is used by that capture only.
// Per device at most 16, made on first use and kept until the process exits; a set whose work is done is handed on to
// another stream. A pass that finds none free runs in stream order: the same results without the overlap.
struct SideStream {
  cudaStream_t stream = nullptr;
  cudaEvent_t fork = nullptr, done = nullptr, inputs = nullptr;
  bool made = false;
  const void* owner = nullptr;       // the caller's stream
  unsigned long long used = 0;       // when it was taken last
  int users = 0;                     // calls that hold it
  std::mutex enqueue;                // callers that share the owner record and wait on its events one after the other
};
constexpr int kSideStreams = 16;
struct SidePool {
  std::mutex mu;
  unsigned long long clock = 0;
  SideStream set[kSideStreams];
};

static bool side_make(SideStream* s) {
  if (cudaStreamCreateWithFlags(&s->stream, cudaStreamNonBlocking) != cudaSuccess) return false;
  cudaEvent_t* const ev[3] = {&s->fork, &s->done, &s->inputs};
  for (int i = 0; i < 3; ++i) {
    if (cudaEventCreateWithFlags(ev[i], cudaEventDisableTiming) == cudaSuccess) continue;
    while (i-- > 0) cudaEventDestroy(*ev[i]);
    cudaStreamDestroy(s->stream);
    return false;
  }
  s->made = true;
  return true;
}

// The set for a pass on `st` while this object lives; operator-> of one without a set may not be used.
class SideLease {
 public:
  explicit SideLease(cudaStream_t st) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return;
    take(pools()[dev], st);
    if (s_) s_->enqueue.lock();
  }
  ~SideLease() {
    if (!s_) return;
    s_->enqueue.unlock();
    std::lock_guard<std::mutex> lock(pool_->mu);
    --s_->users;
  }
  SideLease(const SideLease&) = delete;
  SideLease& operator=(const SideLease&) = delete;
  explicit operator bool() const { return s_ != nullptr; }
  SideStream* operator->() const { return s_; }

 private:
  static SidePool* pools() {
    static SidePool per_dev[64];
    return per_dev;
  }
  // the id of the capture `st` is part of, 0 if it is in none; false where that cannot be told or the capture is broken
  static bool capture_of(cudaStream_t st, unsigned long long* id) {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    *id = 0;
    if (cudaStreamGetCaptureInfo(st, &status, id) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    if (status == cudaStreamCaptureStatusNone) *id = 0;
    return status != cudaStreamCaptureStatusInvalidated;
  }
  // a set that belongs to nobody yet, or the one of those whose work is done that was taken the longest ago
  static SideStream* fresh(SidePool& pool) {
    SideStream* got = nullptr;
    unsigned long long theirs = 0;
    for (SideStream& s : pool.set) {
      if (!s.made) {
        if (side_make(&s)) return &s;
        cudaGetLastError();
        return nullptr;
      }
      if (s.users > 0 || (got && got->used < s.used) || !capture_of(s.stream, &theirs) || theirs != 0) continue;
      if (cudaStreamQuery(s.stream) == cudaSuccess) got = &s;
      else cudaGetLastError();
    }
    return got;
  }
  void take(SidePool& pool, cudaStream_t st) {
    unsigned long long capture = 0, theirs = 0;
    static thread_local char per_thread;       // (one handle stands for every thread's default stream)
    const void* const id = st == cudaStreamPerThread ? static_cast<const void*>(&per_thread) : st;
    if (!capture_of(st, &capture)) return;
    std::lock_guard<std::mutex> lock(pool.mu);
    SideStream* got = nullptr;
    for (SideStream& s : pool.set)
      if (s.made && s.owner == id) {
        // (a set that an earlier capture of the owner's has not given back yet stays with it)
        if (!capture_of(s.stream, &theirs) || (theirs != 0 && theirs != capture)) return;
        got = &s;
        break;
      }
    if (!got) {
      // making a stream, and asking one for its state, must not disturb a capture of this or another thread's
      cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
      cudaThreadExchangeStreamCaptureMode(&mode);
      got = fresh(pool);
      cudaThreadExchangeStreamCaptureMode(&mode);
      if (!got) return;
    }
    got->owner = id;
    got->used = ++pool.clock;
    ++got->users;
    pool_ = &pool;
    s_ = got;
  }
  SidePool* pool_ = nullptr;
  SideStream* s_ = nullptr;
};
}  // namespace trispec

namespace trispec {
// How a pass arranges its attention and its LM head (they do not depend on each other).
enum PassForm { PASS_ATTENTION_FIRST = 0, PASS_LM_FIRST = 1, PASS_SIDE_BY_SIDE = 2 };
struct PassPlan {
  PassForm form;
  bool beside;        // the attention runs beside the LM head, which leaves it `attn_ctas` SMs
  int attn_ctas;
  bool in_turn;       // that attention takes the splits of its plan one after the other, in few CTAs: in the LM head's launch (in
                      // trispec_verify_host on the second stream, as the attention's own plan always is)
  bool pair;          // two CTAs per item, in the LM head's launch
};

// The memory that one of the two streams of a pass reads and writes.
class Footprint {
 public:
  void reads(const void* p, size_t bytes) { add(p, bytes, false); }
  void writes(const void* p, size_t bytes) { add(p, bytes, true); }
  bool clashes(const Footprint& o) const {
    for (int i = 0; i < n_; ++i)
      for (int j = 0; j < o.n_; ++j) {
        const Span &a = span_[i], &b = o.span_[j];
        if ((a.written || b.written) && a.at < b.at + b.bytes && b.at < a.at + a.bytes) return true;
      }
    return false;
  }

 private:
  struct Span { uintptr_t at; size_t bytes; bool written; };
  void add(const void* p, size_t bytes, bool written) {
    if (p && bytes > 0 && n_ < kMax) span_[n_++] = {reinterpret_cast<uintptr_t>(p), bytes, written};
  }
  static constexpr int kMax = 48;     // 16 arrays on one side, 37 on the other
  Span span_[kMax];
  int n_ = 0;
};

static void tree_footprint(Footprint* f, const trispec_tree_args* tree) {
  const size_t n = static_cast<size_t>(tree->B) * tree->T;
  f->reads(tree->parent, n * 4);
  f->writes(tree->mask, n * 8);
  f->writes(tree->depth, n * 4);
}
static void attn_footprint(Footprint* f, const trispec_attn_args* attn) {
  const size_t B = attn->B, T = attn->T, Hq = attn->Hq, Hkv = attn->Hkv, D = attn->D;
  const bool paged = attn->kv_layout == TRISPEC_KV_PAGED;
  const size_t kv = (paged ? static_cast<size_t>(attn->num_blocks) * attn->block_size : B * attn->Lmax) * Hkv * D * 2;
  f->reads(attn->q, B * T * Hq * D * 2);
  f->reads(attn->k_tree, B * T * Hkv * D * 2);
  f->reads(attn->v_tree, B * T * Hkv * D * 2);
  f->reads(attn->k_cache, kv);
  f->reads(attn->v_cache, kv);
  if (paged) f->reads(attn->block_table, B * attn->max_blocks_per_seq * 4);
  f->reads(attn->ctx_len, B * 4);
  if (attn->seq_index) f->reads(attn->seq_index, static_cast<size_t>(attn->B_active) * 4);
  f->reads(attn->n_nodes, B * 4);
  f->writes(attn->o, B * T * Hq * D * 2);
  f->writes(attn->lse, B * T * Hq * 4);
  f->writes(attn->workspace, trispec_verify_attn_workspace(attn));
}

// Whether the tree step and the attention share more than the mask: then the one comes after the other, also where a launch of
// both would compute the masks on the way.
static bool tree_shares_memory(const trispec_tree_args* tree, const trispec_attn_args* attn) {
  Footprint masks, attention;
  tree_footprint(&masks, tree);
  attn_footprint(&attention, attn);
  return masks.clashes(attention);
}

// Whether the steps that would run beside each other share memory that one of them writes (a workspace used by both, an
// escalation list written over the index list that the attention reads): in stream order that is no conflict.
static bool pass_shares_memory(const trispec_tree_args* tree, const trispec_attn_args* attn, const trispec_lmhead_args* lm,
                               const trispec_scan_args* scan) {
  Footprint beside, main;
  if (tree) tree_footprint(&beside, tree);
  attn_footprint(&beside, attn);
  beside.reads(attn->mask, static_cast<size_t>(attn->B) * attn->T * 8);
  {
    const size_t n = static_cast<size_t>(lm->B) * lm->T;
    main.reads(lm->h, n * lm->d * 2);
    main.reads(lm->W, static_cast<size_t>(lm->V) * lm->d * 2);
    main.reads(lm->parent, n * 4);
    main.reads(lm->tok, n * 4);
    if (lm->seq_index) main.reads(lm->seq_index, static_cast<size_t>(lm->B_active) * 4);
    const trispec_stats& o = lm->out;
    const void* const out[11] = {o.max, o.lse, o.top1_val, o.top2_val, o.p_top1, o.p_top2, o.top1_idx, o.top2_idx,
                                 o.draft_logit, o.p_draft, o.entropy};
    for (const void* p : out) main.writes(p, n * 4);
    const size_t need = trispec_lmhead_stats_workspace(lm);
    main.writes(lm->workspace, need < lm->workspace_bytes ? need : lm->workspace_bytes);
  }
  if (scan) {
    const size_t B = scan->B, n = B * scan->T;
    const trispec_stats& in = scan->in;
    const void* const by_node[9] = {scan->parent, scan->tok, scan->q_draft, scan->u_accept, in.top1_idx, in.p_top1,
                                    in.p_top2, in.entropy, in.p_draft};
    for (const void* p : by_node) main.reads(p, n * 4);
    main.reads(scan->active, B);
    main.reads(scan->start_node, B * 4);
    const void* const by_sequence[5] = {scan->accept_len, scan->bonus_tok, scan->last_node, scan->near_thr, scan->esc_index};
    for (const void* p : by_sequence) main.writes(p, B * 4);
    main.writes(scan->path, n * 4);
    main.writes(scan->escalate, B);
    main.writes(scan->n_escalated, 4);
    main.writes(scan->compact_scratch, (B + 65535) / 65536 * 4);
  }
  return beside.clashes(main) || (scan && scan->esc_index && attn->seq_index == scan->esc_index);
}

// `one_launch`: the attention in turn and the LM head share a launch (everything is on the device already).
static PassPlan pass_plan(const trispec_tree_args* tree, const trispec_attn_args* attn, const trispec_lmhead_args* lm,
                          const trispec_scan_args* scan, bool one_launch = true) {
  PassPlan pl = {PASS_ATTENTION_FIRST, false, attn ? attn_planned_ctas(attn) : 0, false, false};
  const int lm_seqs = lm->seq_index ? lm->B_active : lm->B;
  if (!attn || pl.attn_ctas <= 0 || !lm_runs_small_rows(lm)) return pl;      // the pair kernel takes every SM
  const int sms = device_sm_count();
  const bool in_order = pass_shares_memory(tree, attn, lm, scan);
  // TRISPEC_PASS_FORM = attention_first | lm_first | side_by_side overrides the rules below for so few
  // rows (a tuning and testing aid, read at every call; lm_first is then one after the other, and side by
  // side, with the attention's own plan, still needs at most SMs / 2 CTAs)
  if (const char* e = getenv("TRISPEC_PASS_FORM")) {
    if (e[0] == 'a') return pl;
    if (e[0] == 'l') { pl.form = PASS_LM_FIRST; return pl; }
    if (e[0] == 's' && pl.attn_ctas * 2 <= sms && !in_order) { pl.form = PASS_SIDE_BY_SIDE; pl.beside = true; return pl; }
  }
  // With so few rows the LM head is a pure stream of W that does not need every SM to saturate HBM, and the attention
  // a chain of tiles that does not need bandwidth: the attention runs beside the LM head in as FEW CTAs as it can,
  // one or two per (sequence, KV head, M tile), each taking the splits of the attention's own plan in turn (attn_split.cuh: the
  // same bits), where they end well before the LM head (W streams at 6 TB/s) and are at most a quarter of the chip. One
  // sequence of 61 nodes, 4096 context tokens, 151936 x 2048 weights: 8 pairs of CTAs, 65 tiles each, beside 132 CTAs of the LM
  // head, 117 us a pass (8 single CTAs beside 140 of it, 126 us).
  const double lm_us = static_cast<double>(lm->V) * lm->d * 2.0 / 6.0e6;
  const int compact_ctas = in_order ? 0 : attn_compact_ctas(attn, 0.8 * lm_us, sms / 4, one_launch ? &pl.pair : nullptr);
  if (lm_seqs == 1) {
    // Behind the attention the LM head would stall as a programmatic dependent, so for one sequence it goes first
    // whatever the form. The attention's own plan runs side by side where it can be given one SM per CTA for less
    // than about 40 us of the LM head's time, which then takes SMs / (SMs - CTAs) times as long. (Where only its form
    // in few CTAs does, the pass still is called LM head first.)
    const double own_lm_us = lm_us * 6.0 / 5.0;
    const bool own_fits = pl.attn_ctas * 2 <= sms && !in_order && own_lm_us * pl.attn_ctas <= 40.0 * (sms - pl.attn_ctas);
    pl.form = own_fits ? PASS_SIDE_BY_SIDE : PASS_LM_FIRST;
    pl.beside = compact_ctas > 0 || own_fits;
  } else if (compact_ctas > 0) {
    pl.form = PASS_SIDE_BY_SIDE;
    pl.beside = true;
  }
  if (compact_ctas > 0) {
    pl.attn_ctas = compact_ctas;
    pl.in_turn = true;
  }
  return pl;
}

// Argument errors of any step are found before anything is launched.
static int pass_check(const trispec_tree_args* tree, const trispec_attn_args* attn, const trispec_lmhead_args* lm,
                      const trispec_scan_args* scan, const PassPlan& plan) {
  int rc = tree_mask_check(tree);
  if (rc == TRISPEC_OK && attn) rc = attn_check(attn);
  if (rc == TRISPEC_OK) {
    lm_reserve_sms_once(plan.beside ? plan.attn_ctas : 0);
    rc = lmhead_check(lm);
    lm_reserve_sms_once(0);
  }
  return rc == TRISPEC_OK ? scan_check(scan) : rc;
}
}  // namespace trispec

extern "C" const char* trispec_verify_plan(const trispec_attn_args* attn, const trispec_lmhead_args* lm,
                                           const trispec_scan_args* scan) {
  if (!lm) return "none";
  switch (trispec::pass_plan(nullptr, attn, lm, scan).form) {
    case trispec::PASS_LM_FIRST: return "lm_first";
    case trispec::PASS_SIDE_BY_SIDE: return "side_by_side";
    default: return "attention_first";
  }
}

extern "C" int trispec_verify_beside(const trispec_attn_args* attn, const trispec_lmhead_args* lm, const trispec_scan_args* scan) {
  if (!lm) return 0;
  const trispec::PassPlan plan = trispec::pass_plan(nullptr, attn, lm, scan);
  return plan.beside ? plan.attn_ctas : 0;
}

extern "C" int trispec_verify(const trispec_tree_args* tree, const trispec_attn_args* attn,
                              const trispec_lmhead_args* lm, const trispec_scan_args* scan, void* stream) {
  trispec::EntryScope entry_scope;   // the first kernel launched below is an ordinary launch
  if (!tree || !lm || !scan) return TRISPEC_ERR_INVALID_ARG;
  // The attention and the LM head do not depend on each other, so their order is free. A kernel launched as
  // a programmatic dependent gets its launch latency and prologue hidden, but its loads make almost no
  // progress while the kernel before it still runs (measured: the stages of the single-sequence LM head
  // arrive within a microsecond of the attention's end, whenever it started). For one active sequence the
  // LM head is a pure stream of W and loses more behind an attention than the hidden latency is worth (one
  // sequence of 4096 context tokens: 166 us against 156 us the other way round), so there the LM head goes
  // first, or the two run side by side (pass_plan above).
  const trispec::PassPlan plan = trispec::pass_plan(tree, attn, lm, scan);
  const bool lm_first = plan.form == trispec::PASS_LM_FIRST;
  int rc = trispec::pass_check(tree, attn, lm, scan, plan);
  if (rc != TRISPEC_OK) return rc;
  // Few rows and an attention in turn that fits beside the LM head (pass_plan): masks, attention and LM head in one launch, the
  // scan behind its merge. (On a second stream, forked and joined by events, until now: one short chain 36.4 -> 31.0 us a pass,
  // host 29 -> 18 us a call.)
  if (plan.in_turn) {
    trispec::AttnBeside beside;
    rc = trispec::attn_beside(attn, trispec::tree_shares_memory(tree, attn) ? nullptr : tree, plan.pair, &beside);
    if (rc == TRISPEC_OK && !beside.masks) rc = trispec_build_tree_mask(tree, stream);
    if (rc == TRISPEC_OK) rc = trispec::lmhead_stats_beside(lm, beside, stream);
    return rc == TRISPEC_OK ? trispec_accept_scan(scan, stream) : rc;
  }
  // The attention's own plan beside the LM head: mask and attention go to a second stream behind an event recorded on `stream` at the
  // start of the call; the LM head, whose grid is one persistent CTA per SM, leaves them one SM per attention
  // CTA and starts at once, the scan follows it, and `stream` then waits for the second stream: everything
  // the call enqueues is complete before anything enqueued on `stream` after it.
  if (plan.beside) {
    using namespace trispec;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    SideLease side(st);
    if (side) {
      TRISPEC_CUDA_OK(cudaEventRecord(side->fork, st));
      TRISPEC_CUDA_OK(cudaStreamWaitEvent(side->stream, side->fork, 0));
      rc = trispec_build_tree_mask(tree, side->stream);      // ordinary launch: first kernel of the call
      if (rc == TRISPEC_OK) {
        rc = trispec_verify_attn(attn, side->stream);        // dependent of the mask kernel
      }
      TRISPEC_CUDA_OK(cudaEventRecord(side->done, side->stream));
      if (rc == TRISPEC_OK) {
        entry_scope_next_launch_ordinary();                  // first kernel on `stream`
        lm_reserve_sms_once(plan.attn_ctas);
        rc = trispec_lmhead_stats(lm, stream);
        lm_reserve_sms_once(0);
      }
      if (rc == TRISPEC_OK) rc = trispec_accept_scan(scan, stream);   // dependent of the LM head's last kernel
      // joined after an error too: what has been launched ends before whatever `stream` gets next
      TRISPEC_CUDA_OK(cudaStreamWaitEvent(st, side->done, 0));
      return rc;
    }
  }
  rc = trispec_build_tree_mask(tree, stream);
  if (rc != TRISPEC_OK) return rc;
  if (attn && !lm_first) {
    rc = trispec_verify_attn(attn, stream);
    if (rc != TRISPEC_OK) return rc;
  }
  // (a pass that would have left SMs free, but found no second stream, keeps the LM head's plan: the same bits)
  trispec::lm_reserve_sms_once(plan.beside ? plan.attn_ctas : 0);
  rc = trispec_lmhead_stats(lm, stream);
  if (rc != TRISPEC_OK) return rc;
  if (lm_first) {
    rc = trispec_verify_attn(attn, stream);
    if (rc != TRISPEC_OK) return rc;
  }
  return trispec_accept_scan(scan, stream);
}

// The host-buffer form of the pass. The LM head needs only h (and the tree), the attention
// needs q and the tree keys/values: the latter are copied on a side stream while the LM-head
// GEMM, the longest step, already runs, and the attention follows the GEMM. The caller's
// stream sees one ordered unit of work: everything enqueued here completes before anything
// the caller enqueues on `stream` afterwards.
extern "C" int trispec_verify_host(const trispec_host_io* io, const trispec_tree_args* tree,
                                   const trispec_attn_args* attn, const trispec_lmhead_args* lm,
                                   const trispec_scan_args* scan, void* stream) {
  trispec::EntryScope entry_scope;   // the first kernel launched below is an ordinary launch
  using namespace trispec;
  if (!io || !tree || !lm || !scan) return TRISPEC_ERR_INVALID_ARG;
  // the copies below land in the buffers the structs name: they must describe one and the same pass
  if (tree->parent != lm->parent || tree->parent != scan->parent || lm->tok != scan->tok)
    return TRISPEC_ERR_INVALID_ARG;
  const PassPlan plan = pass_plan(tree, attn, lm, scan, false);
  int rc = pass_check(tree, attn, lm, scan, plan);
  if (rc != TRISPEC_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t BT = static_cast<size_t>(tree->B) * tree->T;
  // A copy list is issued with neighbours merged: requests whose source AND destination follow
  // each other in memory become one transfer (each transfer costs a few microseconds of set-up
  // whatever its size, and a pass moves eleven arrays). Callers get this by carving the arrays
  // out of one host and one device buffer in the order used here.
  struct CopyReq { void* dst; const void* src; size_t bytes; };
  auto copy_list = [](CopyReq* r, int n, cudaMemcpyKind kind, cudaStream_t s) -> cudaError_t {
    int i = 0;
    while (i < n) {
      if (!r[i].dst || !r[i].src || r[i].bytes == 0) { ++i; continue; }
      size_t bytes = r[i].bytes;
      int j = i + 1;
      while (j < n && r[j].dst && r[j].src &&
             static_cast<const char*>(r[j].dst) == static_cast<const char*>(r[i].dst) + bytes &&
             static_cast<const char*>(r[j].src) == static_cast<const char*>(r[i].src) + bytes) {
        bytes += r[j].bytes;
        ++j;
      }
      cudaError_t e = cudaMemcpyAsync(r[i].dst, r[i].src, bytes, kind, s);
      if (e != cudaSuccess) return e;
      i = j;
    }
    return cudaSuccess;
  };
  // the attention's inputs are copied on a second stream (in stream order where there is none free); it may not overwrite
  // q / k_tree / v_tree before earlier work on `stream` (a previous pass reading them) is done
  std::optional<SideLease> side;
  if (attn) side.emplace(st);
  const bool forked = side && *side;
  if (forked) TRISPEC_CUDA_OK(cudaEventRecord((*side)->fork, st));
  // what the LM head needs goes first through the copy engine
  {
    CopyReq in[3] = {{const_cast<int32_t*>(tree->parent), io->parent, BT * 4},
                     {const_cast<int32_t*>(lm->tok), io->tok, BT * 4},
                     {const_cast<void*>(lm->h), io->h, BT * static_cast<size_t>(lm->d) * 2}};
    TRISPEC_CUDA_OK(copy_list(in, 3, cudaMemcpyHostToDevice, st));
  }
  const bool side_by_side = plan.beside && forked;
  if (side_by_side) TRISPEC_CUDA_OK(cudaEventRecord((*side)->inputs, st));
  if (attn) {
    if (forked) TRISPEC_CUDA_OK(cudaStreamWaitEvent((*side)->stream, (*side)->fork, 0));
    CopyReq in[3] = {{const_cast<void*>(attn->q), io->q, BT * static_cast<size_t>(attn->Hq) * attn->D * 2},
                     {const_cast<void*>(attn->k_tree), io->k_tree, BT * static_cast<size_t>(attn->Hkv) * attn->D * 2},
                     {const_cast<void*>(attn->v_tree), io->v_tree, BT * static_cast<size_t>(attn->Hkv) * attn->D * 2}};
    TRISPEC_CUDA_OK(copy_list(in, 3, cudaMemcpyHostToDevice, forked ? (*side)->stream : st));
    if (forked && !side_by_side) TRISPEC_CUDA_OK(cudaEventRecord((*side)->done, (*side)->stream));
  }
  if (side_by_side) {
    // few rows (as in trispec_verify): mask and attention follow their inputs on
    // the second stream, the LM head and the scan run on `stream`, which then waits for the second stream
    TRISPEC_CUDA_OK(cudaStreamWaitEvent((*side)->stream, (*side)->inputs, 0));   // the tree's parents have arrived
    rc = trispec_build_tree_mask(tree, (*side)->stream);
    if (rc == TRISPEC_OK) {
      attn_in_turn_once(plan.in_turn);
      rc = trispec_verify_attn(attn, (*side)->stream);
      attn_in_turn_once(false);
    }
    TRISPEC_CUDA_OK(cudaEventRecord((*side)->done, (*side)->stream));
    if (rc == TRISPEC_OK) {
      entry_scope_next_launch_ordinary();                            // first kernel on `stream`
      lm_reserve_sms_once(plan.attn_ctas);
      rc = trispec_lmhead_stats(lm, stream);
      lm_reserve_sms_once(0);
    }
    if (rc == TRISPEC_OK) rc = trispec_accept_scan(scan, stream);
    TRISPEC_CUDA_OK(cudaStreamWaitEvent(st, (*side)->done, 0));
    if (rc != TRISPEC_OK) return rc;
  } else {
    rc = trispec_build_tree_mask(tree, stream);
    if (rc != TRISPEC_OK) return rc;
    lm_reserve_sms_once(plan.beside ? plan.attn_ctas : 0);   // (as in trispec_verify)
    rc = trispec_lmhead_stats(lm, stream);
    if (rc != TRISPEC_OK) return rc;
    if (attn) {
      if (forked) TRISPEC_CUDA_OK(cudaStreamWaitEvent(st, (*side)->done, 0));
      rc = trispec_verify_attn(attn, stream);
      if (rc != TRISPEC_OK) return rc;
    }
    rc = trispec_accept_scan(scan, stream);
    if (rc != TRISPEC_OK) return rc;
  }
  const size_t B = static_cast<size_t>(scan->B);
  CopyReq out[5] = {{io->accept_len, scan->accept_len, B * 4},
                    {io->bonus_tok, scan->bonus_tok, B * 4},
                    {io->last_node, scan->last_node, B * 4},
                    {io->path, scan->path, B * static_cast<size_t>(scan->T) * 4},
                    {io->escalate, scan->escalate, B}};
  TRISPEC_CUDA_OK(copy_list(out, 5, cudaMemcpyDeviceToHost, st));
  return TRISPEC_OK;
}
