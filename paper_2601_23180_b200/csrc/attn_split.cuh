// Verification attention (the attention of the parallel verification pass, Eq. 2 / Eq. 5):
// every draft-tree node attends to the whole committed context plus the tree keys its mask
// row allows. Split-KV: one CTA handles (sequence, KV head, M tile, KV split) and produces an
// unnormalised partial (O, m, l). With up to 8 splits the CTAs of one (sequence, KV head,
// M tile) form a thread-block cluster: each leaves its partial in its own shared memory and
// the cluster merges them through distributed shared memory, every CTA normalising and
// writing a slice of the rows - no scratch traffic and no second launch. With more splits
// (few sequences, long contexts) partials go to a caller-provided workspace and a second
// kernel merges them.
//
// GQA packing: the G = Hq / Hkv query heads that share a KV head are stacked on the M axis,
// row = node_local * G + head_in_group, so one K/V tile serves all of them. An M tile holds
// NPT = min(128 / G, 64) nodes.
//
// Per 64-key tile:  S = Q K^T  (tcgen05.mma M=128, N=64, K=128; Q is the A operand and lives
//                   in tensor memory for the whole kernel, K is the K-major B operand)
//                   online softmax in registers, one TMEM lane (row) per thread, exp2 domain,
//                   lazy rescaling of O (only when the running max grows by more than 2^8)
//                   P (bf16) -> shared memory, O += P V (V is the MN-major B operand)
// The kernel is bound by shared-memory bandwidth before anything else (TMA writes, operand
// reads of the MMAs, P), which is why Q is kept out of shared memory: per tile the MMAs read
// K, P and V only.
// Warps 0-3: softmax. Warp 4: one thread streams K and V by TMA (no multicast) through two
// independent rings (a K slot is free once S has read it, a V slot after O += P V); it
// initialises the ring barriers itself and starts loading before the CTA-wide set-up barrier.
// Warp 5: one thread issues the MMAs, polling for whichever of S(i+1) / P V(i) can go.
// A softmax thread computes and packs the exponentials of tile i before it waits for the P
// buffer to be free, so that only the 16-byte stores of P sit behind that wait.
// Two CTAs fit on one SM (~112 KB shared memory, 256 TMEM columns each). The 112 KB are either
// K ring 3 + V ring 3 + one P buffer (long tile loops: bytes in flight) or K ring 3 + V ring 2 +
// two P buffers (short loops: tile i waits for P V of tile i - 2 only).
// A sequence may carry fewer than T tree nodes (a pruned tree): rows past its count are not
// computed and M tiles past it do nothing.
// In-turn form: one CTA takes all the splits of a (sequence, KV head, M tile) of the cluster form one after the other and
// merges them itself, with the same arithmetic in the same order: the same bits from an eighth of the CTAs. The fused
// pass runs it beside an LM head that streams W and can spare few SMs, see there. The CTA is alone on its SM: partials
// (bf16, as the cluster form exchanges them) 0-3 lie in the other half of tensor memory, 4-6 in the other half of shared
// memory, and partial 7, if there is one the last, in the K ring. It is bound by the latency of its copies, which the stream
// of W beside it raises: one P buffer and a V ring of three (beside 151936 x 2048 weights, 65 tiles: 121 us a pass; with
// two P buffers and a V ring of two 139).
// In turn in a pair: a cluster of two, the first CTA takes the first half of the splits, all partials in shared memory, each CTA
// merges half of the rows (65 tiles beside that stream 120 -> 60 us).
#pragma once

#include "attn_common.cuh"
#include "tree_mask.cuh"

namespace trispec {

// NP = number of P buffers. With one, the softmax of tile i waits for O += P V of tile i - 1 before
// it may overwrite P; with two (and a V ring of two slots instead of three, same shared memory) it
// waits for tile i - 2, which has long completed: the variant for short tile loops, which are bound
// by the S -> softmax -> P V chain of a CTA rather than by the bytes in flight.
enum AttnMerge { MERGE_WORKSPACE = 0, MERGE_CLUSTER = 1, MERGE_IN_TURN = 2, MERGE_IN_TURN_PAIR = 3 };
__device__ __forceinline__ void attn_sync() { asm volatile("bar.sync 3, %0;" ::"n"(AT_THREADS) : "memory"); }

// One output row from the partials of its splits (bf16 O / l, m, l; weight zero: none), 16 bytes of it per lane: the merge of
// a cluster and of a pair, in the order of the splits.
__device__ __forceinline__ void attn_merge_row(const AttnParams& p, const uint4 (&v)[8], const float2 (&ml)[8], int b, int node,
                                               int hq, int chunk) {
  float M = -INFINITY;
#pragma unroll
  for (int s = 0; s < 8; ++s) M = fmaxf(M, ml[s].x);
  float Lsum = 0.f;
  float acc[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) acc[j] = 0.f;
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const float wgt = (ml[s].x != -INFINITY) ? ex2f(ml[s].x - M) * ml[s].y : 0.f;
    Lsum += wgt;
    const uint32_t w[4] = {v[s].x, v[s].y, v[s].z, v[s].w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      acc[2 * j] = fmaf(__uint_as_float(w[j] << 16), wgt, acc[2 * j]);
      acc[2 * j + 1] = fmaf(__uint_as_float(w[j] & 0xffff0000u), wgt, acc[2 * j + 1]);
    }
  }
  const float inv = 1.f / Lsum;
  uint4 out;
  out.x = pack_bf16(acc[0] * inv, acc[1] * inv);
  out.y = pack_bf16(acc[2] * inv, acc[3] * inv);
  out.z = pack_bf16(acc[4] * inv, acc[5] * inv);
  out.w = pack_bf16(acc[6] * inv, acc[7] * inv);
  uint16_t* orow = p.o + ((static_cast<size_t>(b) * p.T + node) * p.Hq + hq) * AT_D;
  *reinterpret_cast<uint4*>(orow + chunk * 8) = out;
  if (p.lse && chunk == 0)
    p.lse[(static_cast<size_t>(b) * p.Hq + hq) * p.T + node] = (M + log2f(Lsum)) * kLn2;
}

// The seventh warp of a CTA in turn that computes the mask of its tree: into shared memory, for the softmax threads.
template <bool kPair>
__device__ __forceinline__ void attn_mask_warp(const AttnParams& p, int block) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + (((smem_u32(smem_raw) + 1023u) & ~1023u) - smem_u32(smem_raw));
  const int lane = threadIdx.x & 31, idx = kPair ? block >> 1 : block;
  const int mtile = idx % p.n_mt, b = attn_sequence(p.seq_index, idx / (p.n_mt * p.Hkv), p.B);
  const int nn = b < 0 ? 0 : (p.n_nodes ? max(0, min(p.T, __ldg(p.n_nodes + b))) : p.T);
  if (mtile * p.NPT >= nn) return;               // (the CTA does nothing)
  const int32_t* parent = p.parent + static_cast<long long>(b) * p.T;
  const WarpMask m = tree_mask_climb(lane < p.T ? __ldg(parent + lane) : -1, lane + 32 < p.T ? __ldg(parent + lane + 32) : -1, p.T, lane);
  uint64_t* out = reinterpret_cast<uint64_t*>(smem + AT_TURN_MASK_OFF);
  out[lane] = m.bits0;
  out[lane + 32] = m.bits1;
  const int n_rows = min(p.NPT, nn - mtile * p.NPT) * p.G;
  asm volatile("bar.arrive 4, %0;" ::"r"(32 * ((n_rows + 31) >> 5) + 32) : "memory");
}

// CTA `block` of the launch, its first AT_THREADS threads (a kernel that hosts it may have more)
template <int kMerge, int NP>
__device__ __forceinline__ void attn_split_cta(const CUtensorMap& tm_k, const CUtensorMap& tm_v, const CUtensorMap& tm_kt,
                                               const CUtensorMap& tm_vt, const AttnParams& p, int block) {
  constexpr bool kCluster = kMerge == MERGE_CLUSTER, kPair = kMerge == MERGE_IN_TURN_PAIR, kInTurn = kPair || kMerge == MERGE_IN_TURN;
  // ---- which work item: the split index varies fastest, so that in cluster mode the CTAs of
  // one cluster are the splits of one (sequence, KV head, M tile) and cluster rank == split
  int idx = block;
  const int rank = kPair ? idx & 1 : 0;
  if (kPair) idx >>= 1;
  const int split = kInTurn ? 0 : idx % p.n_splits;
  if (!kInTurn) idx /= p.n_splits;
  const int mtile = idx % p.n_mt; idx /= p.n_mt;
  const int g = idx % p.Hkv;
  const int a = idx / p.Hkv;
  // a sequence that does not exist has no nodes: its CTAs do nothing
  const int listed = attn_sequence(p.seq_index, a, p.B), b = max(listed, 0);
  if (listed < 0 && threadIdx.x == 0 && p.dev_status) atomicExch(p.dev_status, TRISPEC_ERR_BAD_INDEX);
  // a length outside [0, capacity] (a stale or corrupt entry) is clamped and flagged: the block
  // table row and the cache are never read past their ends
  int L = listed < 0 ? 0 : __ldg(p.ctx_len + b);
  if (L < 0 || L > p.Lcap) {
    if (threadIdx.x == 0 && p.dev_status) atomicExch(p.dev_status, TRISPEC_ERR_BAD_LENGTH);
    L = max(0, min(L, p.Lcap));
  }
  // a pruned tree has fewer nodes: rows past them are not computed, M tiles past them do nothing
  const int nn = listed < 0 ? 0 : (p.n_nodes ? max(0, min(p.T, __ldg(p.n_nodes + b))) : p.T);
  const int n_ctx_tiles = (L + AT_BN - 1) / AT_BN;
  // every sequence spreads its own context tiles evenly over the splits, so that the CTAs that
  // merge with each other finish together whatever the sequence's length
  const int tiles_per_split = max(1, (n_ctx_tiles + p.n_splits - 1) / p.n_splits);
  const int last_split = max(0, (n_ctx_tiles + tiles_per_split - 1) / tiles_per_split - 1);
  const int own = (p.n_splits + 1) >> 1;        // a pair: the first CTA takes the first `own` splits
  const int t_cut = kPair ? min(n_ctx_tiles, own * tiles_per_split) : 0;
  const int t_begin = kPair ? (rank ? t_cut : 0) : split * tiles_per_split;
  const int t_end = kPair ? (rank ? n_ctx_tiles : t_cut) : (kInTurn ? n_ctx_tiles : min(n_ctx_tiles, t_begin + tiles_per_split));
  const bool has_tree = kPair ? ((last_split >= own) == (rank != 0)) : (kInTurn || (split == last_split));
  const int n_tiles = (t_end - t_begin) + (has_tree ? 1 : 0);   // >= 1 unless this split is empty

  extern __shared__ uint8_t smem_raw[];
  const uint32_t base_u32 = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base_u32 - smem_u32(smem_raw));
  // first and last tile of a split (the tree tile ends the last one)
  auto opens_split = [&](int i) { return i == 0 || (kInTurn && t_begin + i < n_ctx_tiles && i % tiles_per_split == 0); };
  auto ends_split = [&](int i) {
    return i == n_tiles - 1 || (kInTurn && t_begin + i + 1 < n_ctx_tiles && (i + 1) % tiles_per_split == 0);
  };
  const uint32_t smem_slack = kInTurn ? AT_TURN_SMEM_BYTES - AT_TURN_SMEM_USED - 64 * 8 : AT_SMEM_BYTES - AT_SMEM_USED;
  const bool misaligned = base_u32 - smem_u32(smem_raw) > smem_slack;
  if (misaligned && threadIdx.x == 0 && p.dev_status) atomicExch(p.dev_status, TRISPEC_ERR_SMEM_ALIGN);
  // a split past the end of this sequence's context has nothing to do; in cluster mode it
  // still takes part in the merge (with weight zero), so it may not leave early
  const bool idle_cta = (split > last_split) || misaligned || (mtile * p.NPT >= nn);
  if (!kCluster && idle_cta) {                 // the merge kernel skips it too
    pdl_wait();                                // (no grid ends before the one ahead of it)
    return;
  }

  constexpr int NV = (NP == 2) ? 2 : 3;         // V ring slots: K ring + V ring + P buffers = 112 KB either way
  uint8_t* sK = smem;                           // [AT_STAGES] K tiles
  uint8_t* sV = sK + AT_STAGES * AT_TILE_BYTES; // [NV] V tiles
  uint8_t* sP = sV + NV * AT_TILE_BYTES;        // [NP] P tiles
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + AT_STAGES * AT_KV_STAGE_BYTES + AT_P_BYTES);
  uint64_t* k_full = bars;                      // [3]  K tile landed
  uint64_t* k_empty = bars + AT_STAGES;         // [3]  S = Q K^T has consumed it
  uint64_t* v_full = bars + 2 * AT_STAGES;      // [NV] V tile landed
  uint64_t* v_empty = bars + 3 * AT_STAGES;     // [NV] O += P V has consumed it
  uint64_t* s_bar = bars + 4 * AT_STAGES;       // S ready in TMEM
  uint64_t* s_free = s_bar + 1;                 // S read into registers by the 128 softmax threads
  uint64_t* q_bar = s_bar + 2;                  // Q stored to TMEM by the 128 softmax threads
  uint64_t* o_bar = s_bar + 3;                  // [NP] O += P V of a tile using P buffer b complete (buffer free)
  uint64_t* p_bar = s_bar + 5;                  // [NP] P buffer b written by the 128 softmax threads
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(s_bar + 7);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Softmax warps that hold at least one row of the M tile (a chain of 9 nodes with 4 query heads per KV head fills 36
  // rows, two warps). The others take no part in the tile loop: their rows of P and O are whatever memory holds, never
  // read, and the exponential unit, which the two CTAs of an SM share, is left to the rows that exist.
  const int n_rows = min(p.NPT, nn - mtile * p.NPT) * p.G;         // > 0 unless idle_cta
  const int sm_threads = 32 * ((n_rows + 31) >> 5);
  uint8_t* sPartO = smem;                                               // reuses the K/V ring at the end
  float2* sPartML = reinterpret_cast<float2*>(smem + AT_PART_ML_OFF);
  uint8_t* sTurn = smem + AT_SMEM_USED_ALIGNED;                         // in turn: partials 4-6, then (m, l) of all
  float2* sTurnML = reinterpret_cast<float2*>(sTurn + AT_TURN_SMEM_PARTS * AT_TURN_PART_BYTES);   // [8][128]
  uint32_t tmem_base = 0;

  if (!idle_cta) {   // uniform for the whole CTA
  if (warp == 4) {
    // the loader owns the ring barriers: it signals the set-up barrier without waiting on it
    // and starts streaming while the other warps are still allocating TMEM and storing Q
    if (lane == 0) {
      for (int i = 0; i < AT_STAGES; ++i) { mbar_init(k_full + i, 1); mbar_init(k_empty + i, 1); }
      for (int i = 0; i < NV; ++i) { mbar_init(v_full + i, 1); mbar_init(v_empty + i, 1); }
      fence_mbar_init();
    }
    __syncwarp();
    asm volatile("bar.arrive 1, 192;" ::: "memory");
  } else {
    if (threadIdx.x == 0) {
      mbar_init(s_bar, 1); mbar_init(s_free, sm_threads); mbar_init(q_bar, sm_threads);
      for (int i = 0; i < NP; ++i) { mbar_init(o_bar + i, 1); mbar_init(p_bar + i, sm_threads); }
      fence_mbar_init();
    }
    if (warp == 5) {
      tmem_alloc(tmem_slot, kInTurn ? 2 * AT_TMEM_COLS : AT_TMEM_COLS);
      tmem_relinquish();
    }
    tc_fence_before();
    asm volatile("bar.sync 1, 192;" ::: "memory");
    tc_fence_after();
    tmem_base = *tmem_slot;
  }

  if (warp == 4) {
    // ------------------------------------------------------------------ TMA loader
    if (lane == 0) {
      prefetch_tmap(&tm_k); prefetch_tmap(&tm_kt); prefetch_tmap(&tm_v); prefetch_tmap(&tm_vt);
      const int32_t* table = p.block_table + static_cast<long long>(b) * p.max_blocks_per_seq;
      auto block_id = [&](int t) -> int {      // fetched two tiles before it is used
        if (!p.paged || t >= t_end) return 0;
        int v = __ldg(table + t);
        if (v < 0 || v >= p.num_blocks) {
          if (p.dev_status) atomicExch(p.dev_status, TRISPEC_ERR_BAD_BLOCK);   // clamped, flagged
          v = 0;
        }
        return v;
      };
      auto load_tile = [&](int i, bool is_v, int blk) {
        const bool tree = has_tree && (i == n_tiles - 1);
        const int stage = is_v ? i % NV : i % AT_STAGES;
        uint64_t* full = (is_v ? v_full : k_full) + stage;
        uint8_t* dst = (is_v ? sV : sK) + stage * AT_TILE_BYTES;
        mbar_expect_tx(full, 2 * AT_BOX_BYTES);
        if (tree) {
          const CUtensorMap* tm = is_v ? &tm_vt : &tm_kt;
          tma_load_4d(dst, tm, full, 0, g, 0, b);
          tma_load_4d(dst + AT_BOX_BYTES, tm, full, 64, g, 0, b);
        } else {
          const CUtensorMap* tm = is_v ? &tm_v : &tm_k;
          const int c2 = p.paged ? 0 : (t_begin + i) * AT_BN;
          const int c3 = p.paged ? blk : b;
          tma_load_4d(dst, tm, full, 0, g, c2, c3);
          tma_load_4d(dst + AT_BOX_BYTES, tm, full, 64, g, c2, c3);
        }
      };
      int kblk0 = block_id(t_begin), kblk1 = block_id(t_begin + 1);
      int vblk0 = kblk0, vblk1 = kblk1;
      int next_k = 0, next_v = 0;
      uint32_t idle = 0;
      while (next_v < n_tiles) {
        bool progressed = false;
        if (next_k < n_tiles && mbar_test(k_empty + next_k % AT_STAGES, ((next_k / AT_STAGES) & 1u) ^ 1u)) {
          load_tile(next_k, false, kblk0);
          kblk0 = kblk1;
          kblk1 = block_id(t_begin + next_k + 2);
          ++next_k;
          progressed = true;
        }
        if (mbar_test(v_empty + next_v % NV, ((next_v / NV) & 1u) ^ 1u)) {
          load_tile(next_v, true, vblk0);
          vblk0 = vblk1;
          vblk1 = block_id(t_begin + next_v + 2);
          ++next_v;
          progressed = true;
        }
        if (progressed) {
          idle = 0;
        } else {
          __nanosleep(32);                    // leave the issue slots to the softmax warps
          if (++idle > kWaitPolls) {          // bounded: give up, flag, and let the kernel end
            if (p.dev_status) atomicExch(p.dev_status, 5);
            break;
          }
        }
      }
    }
  } else if (warp == 5) {
    // ------------------------------------------------------------------ MMA issuer
    // S(i) may be issued once the softmax threads have read S(i-1) out of TMEM and K(i) has
    // landed; P V(i) once P(i) is in shared memory and V(i) has landed.
    if (lane == 0) {
      const uint32_t idesc_s = idesc_bf16(AT_BM, AT_BN, false, false);
      const uint32_t idesc_o = idesc_bf16(AT_BM, AT_D, false, true);
      const uint32_t sK_u = base_u32, sV_u = sK_u + AT_STAGES * AT_TILE_BYTES, sP_u = sV_u + NV * AT_TILE_BYTES;
      mbar_wait(q_bar, 0, p.dev_status);
      tc_fence_after();
      int next_s = 0, next_pv = 0;
      uint32_t idle = 0;
      while (next_pv < n_tiles) {
        bool progressed = false;
        if (next_s < n_tiles && (next_s == 0 || mbar_test(s_free, (next_s - 1) & 1u)) &&
            mbar_test(k_full + next_s % AT_STAGES, (next_s / AT_STAGES) & 1u)) {
          const int stage = next_s % AT_STAGES;
          tc_fence_after();
          const uint32_t sk = sK_u + stage * AT_TILE_BYTES;
#pragma unroll
          for (int kk = 0; kk < AT_D / 16; ++kk) {
            const uint64_t bd = smem_desc_sw128(sk + (kk >> 2) * AT_BOX_BYTES + (kk & 3) * 32, 1024, 16);
            tc_mma_ts(tmem_base + AT_TM_S, tmem_base + AT_TM_Q + kk * 8, bd, idesc_s, kk != 0);
          }
          tc_commit(s_bar);
          tc_commit(k_empty + stage);
          ++next_s;
          progressed = true;
        }
        if (next_pv < next_s && mbar_test(p_bar + next_pv % NP, (next_pv / NP) & 1u) &&
            mbar_test(v_full + next_pv % NV, (next_pv / NV) & 1u)) {
          const int stage = next_pv % NV;
          tc_fence_after();
          const uint32_t sv = sV_u + stage * AT_TILE_BYTES;
          const uint32_t sp = sP_u + (next_pv % NP) * AT_P_BYTES;
          const bool add = !opens_split(next_pv);
#pragma unroll
          for (int kk = 0; kk < AT_BN / 16; ++kk) {
            const uint64_t ad = smem_desc_sw128(sp + kk * 32, 1024, 16);
            // V: MN-major, 64-dim blocks 8 KB apart (LBO), 8-key groups 1 KB apart (SBO)
            const uint64_t bd = smem_desc_sw128(sv + kk * 2048, 1024, AT_BOX_BYTES);
            tc_mma_ss(tmem_base + AT_TM_O, ad, bd, idesc_o, add || kk != 0);
          }
          tc_commit(v_empty + stage);
          tc_commit(o_bar + next_pv % NP);
          ++next_pv;
          progressed = true;
        }
        if (progressed) {
          idle = 0;
        } else {
          // (no sleep here: the sooner an MMA is issued, the sooner its K or V slot is free again)
          if (++idle > kWaitPolls) {          // bounded: give up, flag, and let the kernel end
            if (p.dev_status) atomicExch(p.dev_status, 5);
            break;
          }
        }
      }
    }
  } else if (static_cast<int>(threadIdx.x) < sm_threads) {
    // ------------------------------------------------------------------ softmax (warps 0-3)
    const int row = warp * 32 + lane;
    const int node = mtile * p.NPT + row / p.G;
    const bool row_valid = (row < p.NPT * p.G) && (node < nn);
    const uint32_t lane_base = static_cast<uint32_t>(warp * 32) << 16;
    // Q row -> TMEM (A operand of S = Q K^T): lane = row, column c = dims (2c, 2c + 1)
    {
      const int hq = g * p.G + row % p.G;
      const uint4* src = reinterpret_cast<const uint4*>(
          p.q + ((static_cast<long long>(b) * p.T + (row_valid ? node : 0)) * p.Hq + hq) * AT_D);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        uint32_t r[32];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          uint4 v = make_uint4(0, 0, 0, 0);
          if (row_valid) v = __ldg(src + c * 8 + j);
          r[4 * j] = v.x; r[4 * j + 1] = v.y; r[4 * j + 2] = v.z; r[4 * j + 3] = v.w;
        }
        tmem_st32(tmem_base + lane_base + AT_TM_Q + c * 32, r);
      }
      tc_wait_st();
      tc_fence_before();
      mbar_arrive(q_bar);
    }
    float m_ref = -INFINITY, l = 0.f;
    int turn = 0;                                // in turn: the split at hand

    for (int i = 0; i < n_tiles; ++i) {
      const bool tree = has_tree && (i == n_tiles - 1);
      const bool opens = opens_split(i);
      mbar_wait(s_bar, i & 1u, p.dev_status);
      tc_fence_after();
      uint32_t sr[64];
      {
        uint32_t r0[32], r1[32];
        tmem_ld32(tmem_base + lane_base + AT_TM_S, r0);
        tmem_ld32(tmem_base + lane_base + AT_TM_S + 32, r1);
        tc_wait_ld();
#pragma unroll
        for (int j = 0; j < 32; ++j) { sr[j] = r0[j]; sr[32 + j] = r1[j]; }
      }
      tc_fence_before();
      mbar_arrive(s_free);                       // S(i + 1) may overwrite the buffer now
      // which keys of this tile does this row see
      uint64_t vis;
      int nvalid = AT_BN;
      if (tree) {
        // the mask comes from the kernel before this one on the stream: first dependent read
        if (kInTurn && p.parent) {
          asm volatile("bar.sync 4, %0;" ::"r"(sm_threads + 32) : "memory");   // the host kernel's mask warp has arrived
          vis = row_valid ? reinterpret_cast<const uint64_t*>(smem + AT_TURN_MASK_OFF)[node] : 0ull;
        } else {
          pdl_wait();
          vis = row_valid ? __ldg(p.mask + static_cast<long long>(b) * p.T + node) : 0ull;
        }
      } else {
        nvalid = min(AT_BN, L - (t_begin + i) * AT_BN);
        vis = (nvalid >= 64) ? ~0ull : ((1ull << nvalid) - 1ull);
      }
      // running maximum on the raw scores (the scale is positive, so it commutes with max);
      // four chains for instruction-level parallelism
      float tm[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
      if (!tree && nvalid >= AT_BN) {
#pragma unroll
        for (int j = 0; j < 64; j += 8) {
          tm[0] = fmax3(tm[0], __uint_as_float(sr[j]), __uint_as_float(sr[j + 1]));
          tm[1] = fmax3(tm[1], __uint_as_float(sr[j + 2]), __uint_as_float(sr[j + 3]));
          tm[2] = fmax3(tm[2], __uint_as_float(sr[j + 4]), __uint_as_float(sr[j + 5]));
          tm[3] = fmax3(tm[3], __uint_as_float(sr[j + 6]), __uint_as_float(sr[j + 7]));
        }
      } else {
#pragma unroll
        for (int j = 0; j < 64; ++j) {
          const float v = ((vis >> j) & 1ull) ? __uint_as_float(sr[j]) : -INFINITY;
          sr[j] = __float_as_uint(v);
          tm[j & 3] = fmaxf(tm[j & 3], v);
        }
      }
      const float tmax = fmaxf(fmaxf(tm[0], tm[1]), fmaxf(tm[2], tm[3])) * p.scale_log2;
      // new reference maximum (lazy: only when the running one is exceeded by more than the
      // threshold); the rescaling of O it implies is applied further down, after P V of the
      // previous tile, so that the exponentials below do not wait for that MMA
      bool need = false;
      float f = 1.f;
      if (opens) {
        m_ref = tmax;
        l = 0.f;
      } else {
        need = tmax > m_ref + kRescaleThreshold;
        if (need) { f = (m_ref == -INFINITY) ? 0.f : ex2f(m_ref - tmax); m_ref = tmax; l *= f; }
      }
      const float nmu = (m_ref == -INFINITY) ? 0.f : -m_ref;
      float2 ls[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
      const float2 sc2 = make_float2(p.scale_log2, p.scale_log2), nmu2 = make_float2(nmu, nmu);
      uint4 pk[8];
#pragma unroll
      for (int cch = 0; cch < 8; ++cch) {
        float e[8];
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
          // exp2(s * scale - m) on two scores at a time
          const float2 t = ffma2(make_float2(__uint_as_float(sr[cch * 8 + j]), __uint_as_float(sr[cch * 8 + j + 1])),
                                 sc2, nmu2);
          e[j] = ex2f(t.x);
          e[j + 1] = ex2f(t.y);
          ls[(j >> 1) & 1] = fadd2(ls[(j >> 1) & 1], make_float2(e[j], e[j + 1]));
        }
        pk[cch].x = pack_bf16(e[0], e[1]); pk[cch].y = pack_bf16(e[2], e[3]);
        pk[cch].z = pack_bf16(e[4], e[5]); pk[cch].w = pack_bf16(e[6], e[7]);
      }
      if (i >= NP) {
        // the P buffer is free once O += P V of the tile that used it last is complete
        mbar_wait(o_bar + i % NP, ((i / NP) - 1) & 1u, p.dev_status);
        tc_fence_after();
      }
      if (!opens) {
        if (__any_sync(0xffffffffu, need)) {
          if (NP > 1) {   // O is stable only after the previous tile's P V
            mbar_wait(o_bar + (i - 1) % NP, ((i - 1) / NP) & 1u, p.dev_status);
            tc_fence_after();
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            uint32_t o[32];
            tmem_ld32(tmem_base + lane_base + AT_TM_O + c * 32, o);
            tc_wait_ld();
#pragma unroll
            for (int j = 0; j < 32; ++j) o[j] = __float_as_uint(__uint_as_float(o[j]) * f);
            tmem_st32(tmem_base + lane_base + AT_TM_O + c * 32, o);
          }
          tc_wait_st();
        }
      }
      uint8_t* prow = sP + (i % NP) * AT_P_BYTES + row * 128;
#pragma unroll
      for (int cch = 0; cch < 8; ++cch) *reinterpret_cast<uint4*>(prow + ((cch ^ (row & 7)) << 4)) = pk[cch];
      l += (ls[0].x + ls[0].y) + (ls[1].x + ls[1].y);
      // keys past the end of the context, and tree nodes past the end of a pruned tree, have
      // probability 0 but their V rows may hold anything (0 * NaN = NaN): zero them
      const int vrows = tree ? ((nn < p.T) ? nn : AT_BN) : nvalid;
      if (vrows < AT_BN) {
        mbar_wait(v_full + i % NV, (i / NV) & 1u, p.dev_status);
        uint8_t* sv = sV + (i % NV) * AT_TILE_BYTES;
        for (int e = threadIdx.x; e < (AT_BN - vrows) * 16; e += sm_threads) {
          const int r = vrows + (e >> 4), c16 = e & 15;
          *reinterpret_cast<uint4*>(sv + (c16 >> 3) * AT_BOX_BYTES + r * 128 + ((c16 & 7) << 4)) = make_uint4(0, 0, 0, 0);
        }
      }
      fence_async_smem();
      tc_fence_before();
      mbar_arrive(p_bar + i % NP);
      if (kInTurn && p.n_splits > 1 && ends_split(i)) {
        // This split's partial, normalised and rounded as the cluster form does it. The next split's first P V, which
        // overwrites O, comes after its P, and that after these reads.
        mbar_wait(o_bar + i % NP, (i / NP) & 1u, p.dev_status);
        tc_fence_after();
        const float invl = (l > 0.f) ? 1.f / l : 0.f;
        constexpr int kInTmem = kPair ? 0 : AT_TURN_TMEM_PARTS;
        uint8_t* part = (turn == kInTmem + AT_TURN_SMEM_PARTS ? smem : sTurn + (turn - kInTmem) * AT_TURN_PART_BYTES) + row * (AT_D * 2);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint32_t o0[32], o1[32], pk2[32];
          tmem_ld32(tmem_base + lane_base + AT_TM_O + c * 64, o0);
          tmem_ld32(tmem_base + lane_base + AT_TM_O + c * 64 + 32, o1);
          tc_wait_ld();
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            pk2[j] = pack_bf16(__uint_as_float(o0[2 * j]) * invl, __uint_as_float(o0[2 * j + 1]) * invl);
            pk2[16 + j] = pack_bf16(__uint_as_float(o1[2 * j]) * invl, __uint_as_float(o1[2 * j + 1]) * invl);
          }
          if (turn < kInTmem) {
            tmem_st32(tmem_base + lane_base + AT_TMEM_COLS + turn * 64 + c * 32, pk2);
          } else {
#pragma unroll
            for (int j = 0; j < 8; ++j)
              *reinterpret_cast<uint4*>(part + (((c * 8 + j) ^ (row & 7)) << 4)) =
                  make_uint4(pk2[4 * j], pk2[4 * j + 1], pk2[4 * j + 2], pk2[4 * j + 3]);
          }
        }
        if (turn < kInTmem) tc_wait_st();
        sTurnML[turn * AT_BM + row] = make_float2(m_ref, l);
        tc_fence_before();
        ++turn;
      }
    }
    if (kPair && p.parent && !has_tree) asm volatile("bar.sync 4, %0;" ::"r"(sm_threads + 32) : "memory");
    // ---------------------------------------------------------------- epilogue
    if (!kPair || n_tiles > 0)                   // the last P V, hence all of them
      mbar_wait(o_bar + (n_tiles - 1) % NP, ((n_tiles - 1) / NP) & 1u, p.dev_status);
    tc_fence_after();
    if (kPair) {
      for (int s = turn; s < own; ++s) sTurnML[s * AT_BM + row] = make_float2(-INFINITY, 0.f);   // splits without a tile
    } else if (kInTurn && p.n_splits > 1) {
      // merge of this row's partials: the arithmetic of the cluster merge below, in its order
      pdl_wait();                                // before the first global write
      const int hq = g * p.G + row % p.G;
      float wgt[8];
      float M = -INFINITY, Lsum = 0.f;
#pragma unroll
      for (int s = 0; s < 8; ++s)
        if (s < turn) M = fmaxf(M, sTurnML[s * AT_BM + row].x);
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        const float2 ml = s < turn ? sTurnML[s * AT_BM + row] : make_float2(-INFINITY, 0.f);
        wgt[s] = (ml.x != -INFINITY) ? ex2f(ml.x - M) * ml.y : 0.f;
        Lsum += wgt[s];
      }
      const float inv = 1.f / Lsum;
      uint16_t* orow = p.o + ((static_cast<size_t>(b) * p.T + (row_valid ? node : 0)) * p.Hq + hq) * AT_D;
#pragma unroll
      for (int c = 0; c < 8; ++c) {              // 16 dims at a time
        float acc[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) acc[j] = 0.f;
#pragma unroll
        for (int s = 0; s < 8; ++s) {
          if (s >= turn) break;                  // (an empty split adds nothing)
          uint32_t w[8];
          if (s < AT_TURN_TMEM_PARTS) {
            tmem_ld8(tmem_base + lane_base + AT_TMEM_COLS + s * 64 + c * 8, w);
            tc_wait_ld();
          } else {
            const uint8_t* part = (s == 7 ? smem : sTurn + (s - AT_TURN_TMEM_PARTS) * AT_TURN_PART_BYTES) + row * (AT_D * 2);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              const uint4 v = *reinterpret_cast<const uint4*>(part + (((c * 2 + j) ^ (row & 7)) << 4));
              w[4 * j] = v.x; w[4 * j + 1] = v.y; w[4 * j + 2] = v.z; w[4 * j + 3] = v.w;
            }
          }
          const bool used = sTurnML[s * AT_BM + row].x != -INFINITY;   // a fully masked row's partial counts as 0
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint32_t x = used ? w[j] : 0u;
            acc[2 * j] = fmaf(__uint_as_float(x << 16), wgt[s], acc[2 * j]);
            acc[2 * j + 1] = fmaf(__uint_as_float(x & 0xffff0000u), wgt[s], acc[2 * j + 1]);
          }
        }
        if (row_valid) {
#pragma unroll
          for (int j = 0; j < 16; j += 8) {
            uint4 out;
            out.x = pack_bf16(acc[j] * inv, acc[j + 1] * inv);
            out.y = pack_bf16(acc[j + 2] * inv, acc[j + 3] * inv);
            out.z = pack_bf16(acc[j + 4] * inv, acc[j + 5] * inv);
            out.w = pack_bf16(acc[j + 6] * inv, acc[j + 7] * inv);
            *reinterpret_cast<uint4*>(orow + c * 16 + j) = out;
          }
        }
      }
      if (row_valid && p.lse) p.lse[(static_cast<size_t>(b) * p.Hq + hq) * p.T + node] = (M + log2f(Lsum)) * kLn2;
    } else if (kInTurn || (kCluster && p.n_splits == 1)) {
      // a single split is the whole result: normalise and store it straight from tensor memory
      pdl_wait();                                // before the first global write
      const float invl = (l > 0.f) ? 1.f / l : 0.f;
      const int hq = g * p.G + row % p.G;
      uint16_t* orow = p.o + ((static_cast<size_t>(b) * p.T + (row_valid ? node : 0)) * p.Hq + hq) * AT_D;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint32_t o[32];
        tmem_ld32(tmem_base + lane_base + AT_TM_O + c * 32, o);
        tc_wait_ld();
        if (row_valid) {
#pragma unroll
          for (int j = 0; j < 32; j += 8) {
            uint4 pk;
            pk.x = pack_bf16(__uint_as_float(o[j]) * invl, __uint_as_float(o[j + 1]) * invl);
            pk.y = pack_bf16(__uint_as_float(o[j + 2]) * invl, __uint_as_float(o[j + 3]) * invl);
            pk.z = pack_bf16(__uint_as_float(o[j + 4]) * invl, __uint_as_float(o[j + 5]) * invl);
            pk.w = pack_bf16(__uint_as_float(o[j + 6]) * invl, __uint_as_float(o[j + 7]) * invl);
            *reinterpret_cast<uint4*>(orow + c * 32 + j) = pk;
          }
        }
      }
      if (row_valid && p.lse) p.lse[(static_cast<size_t>(b) * p.Hq + hq) * p.T + node] = (m_ref + log2f(l)) * kLn2;
    } else if (kCluster) {
      // partial (O / l as bf16, m, l) -> this CTA's shared memory (the K/V ring is idle: every
      // tile has been consumed by its MMAs). The exchange between the CTAs of a cluster goes
      // over the SM-to-SM network, whose bandwidth is a small fraction of shared memory's, so the
      // partial travels normalised and in the output precision; m and l stay fp32. Rows are
      // padded by 16 bytes so that the 16-byte stores of a warp spread over the banks.
      uint8_t* po = sPartO + row * AT_PART_PITCH;
      const float invl = (l > 0.f) ? 1.f / l : 0.f;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint32_t o[32];
        tmem_ld32(tmem_base + lane_base + AT_TM_O + c * 32, o);
        tc_wait_ld();
#pragma unroll
        for (int j = 0; j < 32; j += 8) {
          uint4 pk;
          pk.x = pack_bf16(__uint_as_float(o[j]) * invl, __uint_as_float(o[j + 1]) * invl);
          pk.y = pack_bf16(__uint_as_float(o[j + 2]) * invl, __uint_as_float(o[j + 3]) * invl);
          pk.z = pack_bf16(__uint_as_float(o[j + 4]) * invl, __uint_as_float(o[j + 5]) * invl);
          pk.w = pack_bf16(__uint_as_float(o[j + 6]) * invl, __uint_as_float(o[j + 7]) * invl);
          *reinterpret_cast<uint4*>(po + (c * 32 + j) * 2) = pk;
        }
      }
      sPartML[row] = make_float2(m_ref, l);
    } else {
      pdl_wait();                                // before the first global write
      const size_t item = static_cast<size_t>(block);
      float* po = p.part_o + (item * AT_BM + row) * AT_D;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint32_t o[32];
        tmem_ld32(tmem_base + lane_base + AT_TM_O + c * 32, o);
        tc_wait_ld();
        if (row_valid) {
#pragma unroll
          for (int j = 0; j < 32; j += 4)
            *reinterpret_cast<float4*>(po + c * 32 + j) =
                make_float4(__uint_as_float(o[j]), __uint_as_float(o[j + 1]), __uint_as_float(o[j + 2]),
                            __uint_as_float(o[j + 3]));
        }
      }
      if (row_valid) {
        float2 ml = make_float2(m_ref, l);
        *reinterpret_cast<float2*>(p.part_ml + (item * AT_BM + row) * 2) = ml;
      }
    }
  }
  tc_fence_before();
  attn_sync();
  if (warp == 5) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kInTurn ? 2 * AT_TMEM_COLS : AT_TMEM_COLS);
  }
  }   // !idle_cta

  if (kPair) {
    // ---------------------------------------------------------------- merge of a pair
    // Both CTAs hold their splits' partials in shared memory; each normalises half of the rows that exist, in the order of
    // the splits, as the cluster merge below does it.
    pdl_wait();                                  // before the first global write
    cluster_sync_all();
    const int share = (((n_rows + 1) >> 1) + 1) & ~1;           // rows of the first CTA, an even number
    const int row_end = rank ? n_rows : min(n_rows, share);
    const uint32_t ml_u = smem_u32(sTurnML), turn_u = smem_u32(sTurn), ring_u = smem_u32(smem);
    const int half = lane >> 4, chunk = lane & 15;
    for (int row = (rank ? share : 0) + 2 * warp + half; row < row_end; row += 2 * (AT_THREADS / 32)) {
      uint4 v[8];
      float2 ml[8];
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        v[s] = make_uint4(0u, 0u, 0u, 0u);
        ml[s] = make_float2(-INFINITY, 0.f);
        if (s < p.n_splits) ml[s] = ld_cluster_f2(cluster_map(ml_u + ((s < own ? s : s - own) * AT_BM + row) * 8, s < own ? 0 : 1));
      }
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        const int local = s < own ? s : s - own;
        if (ml[s].x != -INFINITY)                 // an empty split's partial was never written
          v[s] = ld_cluster_u4(cluster_map((local == AT_TURN_SMEM_PARTS ? ring_u : turn_u + local * AT_TURN_PART_BYTES) +
                                           row * (AT_D * 2) + ((chunk ^ (row & 7)) << 4), s < own ? 0 : 1));
      }
      attn_merge_row(p, v, ml, b, mtile * p.NPT + row / p.G, g * p.G + row % p.G, chunk);
    }
    cluster_sync_all();   // nobody leaves while its shared memory may still be read
  }

  if (kCluster && p.n_splits > 1) {
    // ---------------------------------------------------------------- cluster merge
    // Every CTA of the cluster holds one partial in its shared memory (idle CTAs: weight zero).
    // CTA `split` normalises rows [split * rpc, (split + 1) * rpc) of the 128.
    if (idle_cta) {
      for (int r = threadIdx.x; r < AT_BM; r += AT_THREADS) sPartML[r] = make_float2(-INFINITY, 0.f);
    }
    pdl_wait();                                  // before the first global write (o, lse)
    cluster_sync_all();
    // Requests over the SM-to-SM network are expensive per instruction, whatever their size,
    // so they are few and wide: one gather of the (m, l) pairs of all splits for this CTA's
    // rows, then per pair of rows one 16-byte-per-lane load from every split.
    // rows this CTA normalises: an even share of the 128 (the last CTA may get fewer)
    const int rpc = (((AT_BM + p.n_splits - 1) / p.n_splits) + 1) & ~1;
    const uint32_t po_u = smem_u32(sPartO), pml_u = smem_u32(sPartML);
    float2* sML2 = reinterpret_cast<float2*>(smem + AT_PART_ML2_OFF);   // [n_splits][rpc]
    for (int t = threadIdx.x; t < p.n_splits * rpc; t += AT_THREADS) {
      const int s_src = t / rpc, row = split * rpc + t % rpc;
      if (row < AT_BM) sML2[t] = ld_cluster_f2(cluster_map(pml_u + row * 8, s_src));
    }
    attn_sync();
    constexpr int kWarps = AT_THREADS / 32;
    const int half = lane >> 4, chunk = lane & 15;
    for (int pr = warp; pr < rpc / 2; pr += kWarps) {
      const int rl = 2 * pr + half;               // row within this CTA's slice
      const int row = split * rpc + rl;
      const int node = mtile * p.NPT + row / p.G;
      const bool ok = (row < AT_BM) && (row < p.NPT * p.G) && (node < nn);
      uint4 v[8];
      float2 ml[8];
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        v[s] = make_uint4(0u, 0u, 0u, 0u);
        ml[s] = make_float2(-INFINITY, 0.f);
        if (s < p.n_splits) {
          ml[s] = sML2[s * rpc + rl];
          if (ok && ml[s].x != -INFINITY)         // an empty partial's rows hold arbitrary bits
            v[s] = ld_cluster_u4(cluster_map(po_u + row * AT_PART_PITCH + chunk * 16, s));
        }
      }
      if (!ok) continue;
      attn_merge_row(p, v, ml, b, node, g * p.G + row % p.G, chunk);
    }
    cluster_sync_all();   // nobody leaves while its shared memory may still be read
  }
}

}  // namespace trispec
