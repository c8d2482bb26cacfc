// Verification attention, host side of the split-KV forms (kernel body: attn_split.cuh) and the merge of more than eight splits.
#include <stdlib.h>

#include "attn_split.cuh"

namespace trispec {

template <int kMerge, int NP>
__global__ void __launch_bounds__(AT_THREADS, kMerge == MERGE_IN_TURN ? 1 : 2)
verify_attn_split_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                         const __grid_constant__ CUtensorMap tm_kt, const __grid_constant__ CUtensorMap tm_vt,
                         const AttnParams p) {
  pdl_launch_dependents();
  attn_split_cta<kMerge, NP>(tm_k, tm_v, tm_kt, tm_vt, p, blockIdx.x);
}


// ---------------------------------------------------------------------------------------
// Merge of the KV splits: one warp per output row (sequence, node, query head).
// ---------------------------------------------------------------------------------------
struct AttnMergeParams {
  int B, T, Hq, Hkv, G, NPT, n_mt, n_splits, n_seq, Lcap;
  const int32_t *ctx_len, *seq_index, *n_nodes;
  const float *part_o, *part_ml;
  uint16_t* o;   // bf16 [B][T][Hq][128]
  float* lse;    // [B][Hq][T] or null
};

__global__ void __launch_bounds__(256)
verify_attn_merge_kernel(const AttnMergeParams p) {
  pdl_launch_dependents();
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const long long w = static_cast<long long>(blockIdx.x) * 8 + (threadIdx.x >> 5);
  const long long total = static_cast<long long>(p.n_seq) * p.T * p.Hq;
  if (w >= total) return;
  const int hq = static_cast<int>(w % p.Hq);
  const int node = static_cast<int>((w / p.Hq) % p.T);
  const int a = static_cast<int>(w / (static_cast<long long>(p.Hq) * p.T));
  const int b = attn_sequence(p.seq_index, a, p.B);
  if (b < 0) return;
  if (p.n_nodes && node >= __ldg(p.n_nodes + b)) return;   // not a node of this (pruned) tree
  const int g = hq / p.G, j = hq % p.G;
  const int mtile = node / p.NPT;
  const int row = (node % p.NPT) * p.G + j;
  const int L = max(0, min(__ldg(p.ctx_len + b), p.Lcap));   // clamped as in the split kernel
  const int n_ctx_tiles = (L + AT_BN - 1) / AT_BN;
  const int tiles_per_split = max(1, (n_ctx_tiles + p.n_splits - 1) / p.n_splits);
  const int n_valid = max(0, (n_ctx_tiles + tiles_per_split - 1) / tiles_per_split - 1) + 1;
  const size_t item0 = ((static_cast<size_t>(a) * p.Hkv + g) * p.n_mt + mtile) * p.n_splits;
  // Bound by the latency of the partials in L2: four splits' loads go out together, then they are folded (before, a pass
  // for the maximum and one for the sums, each load behind the last).
  float M = -INFINITY, Lsum = 0.f;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int s0 = 0; s0 < n_valid; s0 += 4) {
    float2 ml[4];
    float4 v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      ml[k] = make_float2(-INFINITY, 0.f);
      v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (s0 + k < n_valid) {
        const size_t item = item0 + static_cast<size_t>(s0 + k);
        ml[k] = __ldg(reinterpret_cast<const float2*>(p.part_ml + (item * AT_BM + row) * 2));
        v[k] = __ldg(reinterpret_cast<const float4*>(p.part_o + (item * AT_BM + row) * AT_D) + lane);
      }
    }
    float Mn = M;
#pragma unroll
    for (int k = 0; k < 4; ++k) Mn = fmaxf(Mn, ml[k].x);
    const float keep = (M == -INFINITY) ? 0.f : ex2f(M - Mn);
    Lsum *= keep;
    acc.x *= keep; acc.y *= keep; acc.z *= keep; acc.w *= keep;
    M = Mn;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float wgt = (ml[k].x == -INFINITY) ? 0.f : ex2f(ml[k].x - M);
      Lsum = fmaf(ml[k].y, wgt, Lsum);
      acc.x = fmaf(v[k].x, wgt, acc.x); acc.y = fmaf(v[k].y, wgt, acc.y);
      acc.z = fmaf(v[k].z, wgt, acc.z); acc.w = fmaf(v[k].w, wgt, acc.w);
    }
  }
  const float inv = 1.f / Lsum;
  uint2 out;
  out.x = pack_bf16(acc.x * inv, acc.y * inv);
  out.y = pack_bf16(acc.z * inv, acc.w * inv);
  uint16_t* orow = p.o + ((static_cast<size_t>(b) * p.T + node) * p.Hq + hq) * AT_D;
  *reinterpret_cast<uint2*>(orow + lane * 4) = out;
  if (p.lse && lane == 0) p.lse[(static_cast<size_t>(b) * p.Hq + hq) * p.T + node] = (M + log2f(Lsum)) * kLn2;
}

struct AttnPlan {
  int n_seq, G, NPT, n_mt, tiles_max, n_splits;
  bool cluster;      // splits merged inside a thread-block cluster (no workspace)
  bool pieces;       // persistent CTAs over balanced pieces of the work (attn_pieces.cu)
  int n_cta;         // CTAs of the persistent launch
  size_t items;
};

// TRISPEC_ATTN_PLAN = "pieces" or "splits" overrides the planner's choice between the persistent kernel
// and the split kernels where both apply (a tuning and testing aid; read at every call).
static int attn_plan_override() {
  const char* e = getenv("TRISPEC_ATTN_PLAN");
  if (!e) return 0;
  if (e[0] == 'p') return 1;
  if (e[0] == 's') return 2;
  return 0;
}

static thread_local bool tl_attn_in_turn = false;
void attn_in_turn_once(bool on) { tl_attn_in_turn = on; }

static int attn_plan(const trispec_attn_args* a, AttnPlan* pl) {
  if (!a || a->B <= 0 || a->T <= 0 || a->Hq <= 0 || a->Hkv <= 0) return TRISPEC_ERR_INVALID_ARG;
  if (a->D != AT_D || a->T > 64 || a->Hq % a->Hkv != 0) return TRISPEC_ERR_UNSUPPORTED;
  const int G = a->Hq / a->Hkv;
  if (!(G == 1 || G == 2 || G == 4 || G == 8 || G == 16)) return TRISPEC_ERR_UNSUPPORTED;
  int Lmax;
  if (a->kv_layout == TRISPEC_KV_CONTIGUOUS) {
    if (a->Lmax < 0) return TRISPEC_ERR_INVALID_ARG;
    Lmax = a->Lmax;
  } else if (a->kv_layout == TRISPEC_KV_PAGED) {
    if (a->block_size != AT_BN) return TRISPEC_ERR_UNSUPPORTED;
    if (a->max_blocks_per_seq <= 0 || a->num_blocks <= 0) return TRISPEC_ERR_INVALID_ARG;
    Lmax = a->max_blocks_per_seq * AT_BN;
  } else {
    return TRISPEC_ERR_INVALID_ARG;
  }
  pl->n_seq = a->seq_index ? a->B_active : a->B;
  if (pl->n_seq <= 0 || pl->n_seq > a->B) return TRISPEC_ERR_INVALID_ARG;
  pl->G = G;
  pl->NPT = (AT_BM / G < 64) ? AT_BM / G : 64;
  pl->n_mt = (a->T + pl->NPT - 1) / pl->NPT;
  pl->tiles_max = (Lmax + AT_BN - 1) / AT_BN;
  const long long fixed = static_cast<long long>(pl->n_seq) * a->Hkv * pl->n_mt;
  // Number of KV splits (1..8 form a cluster; 16, 32, ... go through the workspace). Measured on the
  // five workloads: more than about 1.25 waves of CTAs with at least 32 tiles each run best (the fixed
  // costs of a CTA - pipeline fill, Q load, merge - hide behind other CTAs); when tiles are too few
  // for that, one wave filled as far as possible; very few (sequence, head) pairs are cut further.
  const long long slots = static_cast<long long>(device_sm_count()) * 2;   // two CTAs per SM (split kernels)
  const int tiles = pl->tiles_max;
  int best_s = 0;
  for (int sp = 1; sp <= 8 && !best_s; ++sp)
    if (fixed * sp * 4 >= slots * 5 && tiles / sp >= 32) best_s = sp;
  if (!best_s) {
    best_s = 1;
    for (int sp = 2; sp <= 8; ++sp)
      if (fixed * sp <= slots && tiles / sp >= 4) best_s = sp;
    if (best_s == 8 && fixed * 8 * 2 <= slots)
      for (int sp = 16; sp <= 1024 && fixed * sp <= slots && tiles / sp >= 8; sp *= 2) best_s = sp;
  }
  pl->n_splits = best_s;
  pl->cluster = pl->n_splits <= 8;
  // Clusters do not reach every CTA slot (measured: 142 of the 148 SMs take clusters of 3 or 4, 284 slots), and
  // a grid a little larger than that runs as two waves. When plain CTAs would fill the chip in ONE wave
  // (at least 92 % of all slots, long enough tile loops), that wave plus the small merge kernel is faster than
  // the clustered choice: target_escalated (96 items x 3 splits = 288 CTAs) 148 -> 118 us.
  {
    const long long cluster_slots = slots * 96 / 100;
    const int sp_full = fixed > 0 ? static_cast<int>(slots / fixed) : 0;
    if (pl->cluster && fixed * best_s > cluster_slots && sp_full >= 2 && fixed * sp_full * 100 >= slots * 92 &&
        tiles / sp_full >= 16) {
      pl->n_splits = sp_full;
      pl->cluster = false;
    }
  }
  pl->items = static_cast<size_t>(fixed) * pl->n_splits;
  if (pl->items > 0x7fffffffull) return TRISPEC_ERR_UNSUPPORTED;
  // The persistent kernel: every CTA slot of the chip gets the same number of tile steps whatever the
  // shape. It pays where the split plan cannot fill the slots evenly: fewer CTAs than slots, a last
  // wave that is mostly empty, or clusters that cannot be placed everywhere.
  pl->pieces = false;
  pl->n_cta = 0;
  if (pl->n_seq <= AT_PIECES_MAX_SEQ) {
    // groups of n_mt neighbouring CTAs (one per M tile) share a range of the (sequence, head, tile) steps
    const long long steps_max = static_cast<long long>(pl->n_seq) * a->Hkv * (tiles + 1);   // upper bound of the work
    long long n_grp = steps_max / 4;                                  // at least four steps per CTA on average
    if (n_grp > slots / pl->n_mt) n_grp = slots / pl->n_mt;
    if (n_grp < 1) n_grp = 1;
    pl->n_cta = static_cast<int>(n_grp) * pl->n_mt;
    const long long ctas = static_cast<long long>(pl->items);
    const long long waves = (ctas + slots - 1) / slots;
    const bool uneven = ctas * 100 < waves * slots * 93;              // the split plan leaves 7 % of the slots idle or more
    // The partials' trip through the workspace and the merge launch cost 15-20 us whatever the size:
    // worth it from a few hundred tile steps per CTA on (long_paged: 555 steps, 1.09 -> 0.98 ms; at 110
    // steps, llama_tree, the split plan is still ahead, 165 against 180 us).
    const int ov = attn_plan_override();
    pl->pieces = ov == 1 || (ov == 0 && uneven && steps_max >= 256 * n_grp);
  }
  return TRISPEC_OK;
}

int attn_compact_ctas(const trispec_attn_args* a, double budget_us, int max_ctas, bool* pair) {
  AttnPlan pl;
  if (pair) *pair = false;
  if (attn_plan(a, &pl) != TRISPEC_OK || pl.pieces || !pl.cluster) return 0;
  const size_t ctas = pl.items / pl.n_splits;
  if (ctas > static_cast<size_t>(max_ctas)) return 0;
  // Two CTAs per item where that is at most an eighth of the chip (half of `max_ctas`): beside the stream of W an item of 65
  // tiles takes 120 us in one CTA and 60 in two, and the LM head's stream does not miss 8 more SMs (one sequence of 61
  // nodes at 4096 tokens beside 151936 x 2048 weights: 131 -> 117 us a pass; 64 query heads at 8192 tokens, 64 CTAs: 258 -> 317).
  const bool two = pair && pl.n_splits >= 2 && 4 * ctas <= static_cast<size_t>(max_ctas);
  if (two) *pair = true;
  const int launched = static_cast<int>(two ? 2 * ctas : ctas);
  // A CTA alone on its SM, launch included (measured: 18.5 us with 9 tiles in 2 splits, 28.7 with 17 in 4, 80.0 with 65 in 8,
  // 137.4 with 125 in 8). The context's capacity stands for its length, which only the device knows.
  const double us = 8.5 + 0.96 * (pl.tiles_max + 1) + 1.3 * (pl.n_splits - 1);
  if (us <= budget_us) return launched;
  const int own = (pl.n_splits + 1) / 2;         // splits of a pair's longer half
  const double half = static_cast<double>(own) * ((pl.tiles_max + pl.n_splits - 1) / pl.n_splits);
  if (two && 8.5 + 0.96 * (half + 1) + 1.3 * own <= budget_us) return launched;
  if (pair) *pair = false;
  return 0;
}

int attn_planned_ctas(const trispec_attn_args* a) {
  AttnPlan pl;
  if (attn_plan(a, &pl) != TRISPEC_OK) return 0;
  return pl.pieces ? pl.n_cta : static_cast<int>(pl.items);
}

}  // namespace trispec

extern "C" size_t trispec_verify_attn_workspace(const trispec_attn_args* a) {
  using namespace trispec;
  AttnPlan pl;
  if (attn_plan(a, &pl) != TRISPEC_OK) return 0;
  if (pl.pieces) return attn_pieces_workspace(pl.n_cta);
  if (pl.cluster) return 0;
  return pl.items * AT_BM * (AT_D + 2) * sizeof(float);
}

extern "C" const char* trispec_verify_attn_plan(const trispec_attn_args* a) {
  using namespace trispec;
  AttnPlan pl;
  if (attn_plan(a, &pl) != TRISPEC_OK) return "none";
  return pl.pieces ? "pieces" : (pl.cluster ? "cluster" : "splits");
}

namespace trispec {
static int attn_checked_plan(const trispec_attn_args* a, AttnPlan* plan) {
  const int rc = attn_plan(a, plan);
  if (rc != TRISPEC_OK) return rc;
  const AttnPlan& pl = *plan;
  if (!a->q || !a->k_tree || !a->v_tree || !a->ctx_len || !a->mask || !a->o) return TRISPEC_ERR_INVALID_ARG;
  if ((pl.pieces || !pl.cluster) && !a->workspace) return TRISPEC_ERR_INVALID_ARG;
  if (pl.tiles_max > 0 && (!a->k_cache || !a->v_cache)) return TRISPEC_ERR_INVALID_ARG;
  if (a->kv_layout == TRISPEC_KV_PAGED && !a->block_table) return TRISPEC_ERR_INVALID_ARG;
  if (!aligned16(a->q) || !aligned16(a->k_tree) || !aligned16(a->v_tree) || !aligned16(a->k_cache) ||
      !aligned16(a->v_cache) || !aligned16(a->o) || (reinterpret_cast<uintptr_t>(a->workspace) & 255u))
    return TRISPEC_ERR_INVALID_ARG;
  if (!(a->scale > 0.f) || !isfinite(a->scale)) return TRISPEC_ERR_INVALID_ARG;
  if (a->workspace_bytes < trispec_verify_attn_workspace(a)) return TRISPEC_ERR_WORKSPACE;
  return TRISPEC_OK;
}
int attn_check(const trispec_attn_args* a) {
  AttnPlan pl;
  return attn_checked_plan(a, &pl);
}
}  // namespace trispec

namespace trispec {
static bool attn_maps(const trispec_attn_args* a, const AttnPlan& pl, CUtensorMap& tm_k, CUtensorMap& tm_v, CUtensorMap& tm_kt,
                      CUtensorMap& tm_vt) {
  const uint64_t D = AT_D, Hkv = a->Hkv, T = a->T, B = a->B;
  {
    const uint64_t dims[4] = {D, Hkv, T, B};
    const uint64_t str[3] = {D * 2, Hkv * D * 2, T * Hkv * D * 2};
    const uint32_t box[4] = {64, 1, 64, 1};
    if (!cached_tmap_bf16(&tm_kt, a->k_tree, 4, dims, str, box)) return false;
    if (!cached_tmap_bf16(&tm_vt, a->v_tree, 4, dims, str, box)) return false;
  }
  if (pl.tiles_max > 0) {
    uint64_t dims[4], str[3];
    if (a->kv_layout == TRISPEC_KV_CONTIGUOUS) {
      dims[0] = D; dims[1] = Hkv; dims[2] = a->Lmax; dims[3] = B;
      str[0] = D * 2; str[1] = Hkv * D * 2; str[2] = static_cast<uint64_t>(a->Lmax) * Hkv * D * 2;
    } else {
      dims[0] = D; dims[1] = Hkv; dims[2] = AT_BN; dims[3] = a->num_blocks;
      str[0] = D * 2; str[1] = Hkv * D * 2; str[2] = static_cast<uint64_t>(AT_BN) * Hkv * D * 2;
    }
    const uint32_t box[4] = {64, 1, 64, 1};
    if (!cached_tmap_bf16(&tm_k, a->k_cache, 4, dims, str, box)) return false;
    if (!cached_tmap_bf16(&tm_v, a->v_cache, 4, dims, str, box)) return false;
  } else {
    tm_k = tm_kt;   // never dereferenced: every sequence has zero context tiles
    tm_v = tm_vt;
  }
  return true;
}
static AttnParams attn_params(const trispec_attn_args* a, const AttnPlan& pl) {
  AttnParams p;
  p.B = a->B; p.T = a->T; p.Hq = a->Hq; p.Hkv = a->Hkv; p.G = pl.G; p.NPT = pl.NPT; p.n_mt = pl.n_mt;
  p.n_splits = pl.n_splits;
  p.paged = (a->kv_layout == TRISPEC_KV_PAGED); p.max_blocks_per_seq = a->max_blocks_per_seq;
  p.num_blocks = a->num_blocks;
  p.Lcap = p.paged ? a->max_blocks_per_seq * AT_BN : a->Lmax;
  p.scale_log2 = a->scale * kLog2e;
  p.q = static_cast<const uint16_t*>(a->q);
  p.block_table = a->block_table; p.ctx_len = a->ctx_len; p.seq_index = a->seq_index; p.mask = a->mask;
  p.n_nodes = a->n_nodes;
  p.part_o = static_cast<float*>(a->workspace);
  p.part_ml = p.part_o + pl.items * AT_BM * AT_D;
  p.o = static_cast<uint16_t*>(a->o);
  p.lse = a->lse;
  p.dev_status = a->dev_status;
  p.n_seq = pl.n_seq;
  p.parent = nullptr;
  p.n_cta = pl.n_cta;
  return p;
}

int attn_beside(const trispec_attn_args* a, const trispec_tree_args* tree, bool pair, AttnBeside* out) {
  AttnPlan pl;
  const int rc = attn_checked_plan(a, &pl);
  if (rc != TRISPEC_OK) return rc;
  if (pl.pieces || !pl.cluster || (pair && pl.n_splits < 2)) return TRISPEC_ERR_UNSUPPORTED;
  if (!attn_maps(a, pl, out->k, out->v, out->kt, out->vt)) return TRISPEC_ERR_CUDA;
  out->p = attn_params(a, pl);
  out->pair = pair;
  // the masks of a decode batch: by the same launch, where the attention reads what the tree step writes
  out->masks = tree && tree->mask == a->mask && tree->B == a->B && tree->T == a->T && tree->B < 2048;
  if (out->masks) {
    out->tree = *tree;
    out->p.parent = tree->parent;
  }
  out->ctas = static_cast<int>(pl.items / pl.n_splits) * (pair ? 2 : 1);
  return TRISPEC_OK;
}
}  // namespace trispec

extern "C" int trispec_verify_attn(const trispec_attn_args* a, void* stream) {
  trispec::EntryScope entry_scope;   // the first kernel launched below is an ordinary launch
  using namespace trispec;
  AttnPlan pl;
  int rc = attn_checked_plan(a, &pl);
  if (rc != TRISPEC_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);

  CUtensorMap tm_k, tm_v, tm_kt, tm_vt;
  if (!attn_maps(a, pl, tm_k, tm_v, tm_kt, tm_vt)) return TRISPEC_ERR_CUDA;
  // Two P buffers for CTAs with few tiles (their time is the S -> softmax -> P V chain, tile after
  // tile, and never reaches the HBM-bound steady state); one P buffer and the deeper V ring for long
  // tile loops. Measured: proxy_tree (16 tiles per CTA) 45.1 -> 43.2 us with two; long_paged
  // (128-512) 1005 -> 1023 us, target_escalated (64) 150 -> 154 us, llama_tree (129) unchanged.
  const bool two_p = pl.pieces ? (static_cast<long long>(pl.n_seq) * a->Hkv * pl.n_mt * (pl.tiles_max + 1) / pl.n_cta <= 32)
                               : (pl.tiles_max / pl.n_splits <= 32);
  const bool in_turn = tl_attn_in_turn && pl.cluster && !pl.pieces && pl.n_splits > 1;
  typedef void (*AttnKernel)(CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, AttnParams);
  static const AttnKernel table[5] = {verify_attn_split_kernel<MERGE_WORKSPACE, 1>, verify_attn_split_kernel<MERGE_WORKSPACE, 2>,
                                      verify_attn_split_kernel<MERGE_CLUSTER, 1>, verify_attn_split_kernel<MERGE_CLUSTER, 2>,
                                      verify_attn_split_kernel<MERGE_IN_TURN, 1>};
  const int which = in_turn ? 4 : (pl.cluster ? 2 : 0) + (two_p ? 1 : 0);
  const AttnKernel kernel = table[which];
  const int smem_bytes = in_turn ? AT_TURN_SMEM_BYTES : AT_SMEM_BYTES;
  static bool smem_set[5][64] = {};
  rc = ensure_smem_limit(reinterpret_cast<const void*>(kernel), smem_bytes, smem_set[which]);
  if (rc != TRISPEC_OK) return rc;
  const AttnParams p = attn_params(a, pl);
  if (pl.pieces) {
    const CUtensorMap maps[4] = {tm_k, tm_v, tm_kt, tm_vt};
    return attn_launch_pieces(p, maps, two_p, a->workspace, st);
  }
  if (in_turn) {
    TRISPEC_CUDA_OK(launch_dependent(kernel, static_cast<unsigned>(pl.items / pl.n_splits), AT_THREADS, smem_bytes, st, 1, tm_k, tm_v,
                                     tm_kt, tm_vt, p));
    count_launch();
    return TRISPEC_OK;
  }
  if (pl.cluster) {
    TRISPEC_CUDA_OK(launch_dependent(kernel, static_cast<unsigned>(pl.items), AT_THREADS,
                                     AT_SMEM_BYTES, st, static_cast<unsigned>(pl.n_splits), tm_k, tm_v, tm_kt, tm_vt,
                                     p));
    count_launch();
    return TRISPEC_OK;
  }
  TRISPEC_CUDA_OK(launch_dependent(kernel, static_cast<unsigned>(pl.items), AT_THREADS,
                                   AT_SMEM_BYTES, st, 1, tm_k, tm_v, tm_kt, tm_vt, p));
  count_launch();

  AttnMergeParams m;
  m.B = a->B; m.T = a->T; m.Hq = a->Hq; m.Hkv = a->Hkv; m.G = pl.G; m.NPT = pl.NPT; m.n_mt = pl.n_mt;
  m.n_splits = pl.n_splits; m.n_seq = pl.n_seq; m.Lcap = p.Lcap;
  m.ctx_len = a->ctx_len; m.seq_index = a->seq_index; m.n_nodes = a->n_nodes;
  m.part_o = p.part_o; m.part_ml = p.part_ml;
  m.o = static_cast<uint16_t*>(a->o); m.lse = a->lse;
  const long long rows = static_cast<long long>(pl.n_seq) * a->T * a->Hq;
  TRISPEC_CUDA_OK(launch_dependent(verify_attn_merge_kernel, static_cast<unsigned>((rows + 7) / 8), 256, 0, st, 1, m));
  count_launch();
  return TRISPEC_OK;
}
