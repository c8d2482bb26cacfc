// LM head fused with per-row softmax statistics (distributions p_i of Eq. 5 reduced to what
// the margin rule of Eq. 8 and the acceptance test of Eq. 6 need). The [rows x V] logits
// never reach global memory: each CTA streams a slice of the vocabulary through
// tcgen05.mma (bf16 x bf16 -> fp32 in tensor memory) and its epilogue keeps, per row, a
// running (max, sum of exponentials, top-1, top-2) in registers across all of its vocabulary
// tiles (and the sum the entropy needs, when the caller asks for the entropy). A small second
// kernel merges the per-slice partials and computes the drafted-token probabilities.
//
// GEMM kernel layout (two CTAs on two SMs work as a pair on one 256 x 256 tile)
//   M tile  = up to 256 rows, up to 128 per CTA of the pair. The rows of the active sequences are packed, row = a * T + node,
//             so that a chain of 9 nodes costs 9 rows: 64 chains of 9 nodes (128256 x 4096 weights) are 3 M tiles,
//             where a slot of 64 rows per sequence made them 16 (2571 -> 600 us). Past the last row: zero fill.
//   N tile  = 256 vocabulary entries, plus one narrower tile (a multiple of 32) for the rest of
//             the CTA pair's vocabulary range; each CTA loads one half of a tile
//   K block = 64 bf16 = one 128-byte swizzle row; 4 MMAs of K = 16 per block
//   Per k-block a CTA stages its own half of the M tile's rows of H (up to 128, 16 KB) and half
//   of the W tile (16 KB): 32 KB for 128 x 256 x 64 multiply-adds per SM, against 48 KB when
//   every SM works alone. The pipeline is bound by how fast W tiles reach shared memory, so this is what
//   lifts the tensor-core duty cycle.
//   warps 0-3: epilogue (one TMEM lane = one row per thread), warp 4: TMA producer,
//   warp 5: TMEM owner; in the leader CTA (cluster rank 0) one of its threads issues the
//   MMAs of the pair. Accumulators are double-buffered in TMEM (2 x 256 columns per CTA)
//   so that the epilogue of tile i overlaps the MMAs of tile i + 1.
//   Pair c works on M tile (c % n_mt) and vocabulary range (c / n_mt): pairs that share a
//   vocabulary range are neighbours and stream the same W tiles at the same time, so W is
//   read from HBM once and re-hit in L2.
//   Barriers: `full` lives in the leader and counts the bytes of both CTAs' loads; `empty`
//   and `tmem_full` exist in both CTAs and are signalled by the leader's commits;
//   `tmem_empty` lives in the leader and collects the epilogue warps of both CTAs.
#include <math.h>

#include <mutex>

#include "attn_split.cuh"

namespace trispec {

constexpr int LM_BM = 128;                      // rows per CTA
constexpr int LM_BN = 256;
constexpr int LM_BK = 64;
constexpr int LM_STAGES = 6;
constexpr int LM_A_BYTES = LM_BM * LM_BK * 2;         // 16 KB
constexpr int LM_B_BYTES = (LM_BN / 2) * LM_BK * 2;   // 16 KB: this CTA's half of the W tile
constexpr int LM_BOX_BYTES = 64 * LM_BK * 2;    // one TMA box: 64 rows x 64 k
constexpr int LM_STAGE_BYTES = LM_A_BYTES + LM_B_BYTES;
constexpr int LM_THREADS = 192;
constexpr int LM_SMEM_BYTES = LM_STAGES * LM_STAGE_BYTES + 1024 /*alignment slack*/ + 256 /*barriers*/;

struct __align__(16) LmPartial {
  float m, s, v1, v2;  // raw (unscaled) running max, sum of 2^((z-m)c), top-1 / top-2 raw logits
  int i1, i2;
  float t;             // sum of 2^((z-m)c) * z over the range (for the entropy: H = lse - E_p[z])
  int pad;
};

struct LmParams {
  int T, d, V;
  int n_seq;      // active sequences
  int n_mt;       // M tiles
  int tile_rows;  // packed rows per M tile, a multiple of 16 up to 256 (4 sequence slots: 256)
  int slots;      // rows are not packed: an M tile is 4 slots of 64 node rows, read through seq_index
  int wait_rows;  // the packed rows are written by the kernel before this one
  int n_ranges;   // vocabulary ranges of the main part: pair c < n_mt * n_ranges works on M tile c % n_mt, range c / n_mt
  int n_tail;     // pairs beyond those: each sweeps ALL M tiles over its slice of the vocabulary's tail
  int main_units; // 32-column units [0, main_units) belong to the main part, the rest to the tail
  float c;        // logit_scale * log2(e)
  const int32_t* seq_index;
  int part_rows;       // rows of a vocabulary range's partials: n_mt * tile_rows
  LmPartial* partial;  // [n_ranges + n_tail][part_rows]
  int32_t* dev_status;
};

// Vocabulary range r of n_ranges, cut into tiles of 256 columns plus one narrower tile for the
// rest; all boundaries are multiples of 32 columns so that each CTA of a pair takes a half that
// is a multiple of 16. (A tile of 224 columns costs as much as one of 256 - its k-loop is as long
// and the MMA time does not shrink in proportion - so the rest is not spread over the tiles.)
struct TileIter {
  int u0, units, n_tiles;
  // part r of n_parts of the 32-column units [first, first + count)
  __device__ TileIter(int first, int count, int n_parts, int r) {
    // Every part gets count / n_parts units. What is left over goes to the first parts in chunks that
    // cost as few extra tiles as possible: a tile costs a whole k-loop whatever its width, so a chunk
    // first fills up a part's last, partial tile (no extra tile), and where the parts consist of whole
    // tiles it is a whole tile (few parts run one tile longer, instead of many).
    const int base = count / n_parts, rem = count - base * n_parts;
    const int chunk = 8 - (base & 7);               // 1..8
    u0 = first + r * base + min(rem, r * chunk);
    units = base + min(chunk, max(0, rem - r * chunk));
    n_tiles = (units + 7) >> 3;
  }
  __device__ void tile(int t, int& n0, int& nw) const {
    n0 = (u0 + 8 * t) << 5;
    nw = min(8, units - 8 * t) << 5;
  }
};

// What a CTA pair works on. A main pair computes one M tile over one vocabulary range (one sweep). When
// the M tiles do not divide the pairs of the chip, the pairs left over take the tail of the vocabulary:
// each of them takes all M tiles over its own slice of that tail, one W tile after the other and on each of them one M tile
// after the other, so that W comes from HBM once (M tile by M tile the slices, 84 MB with 16 M tiles, did not stay in L2
// beside the main stream: 2.05 GB of DRAM reads for 0.64, an eighth of the energy of a launch that runs at the power limit;
// 3904 rows, 151936 x 2048 weights: 1862 -> 1780 us). The main ranges shrink accordingly, so that every
// pair of the chip runs about the same number of tiles.
struct PairWork {
  int n_sweeps, mt0, part;      // M tiles mt0 .. mt0 + n_sweeps - 1; `part` = row block of the partial array
  TileIter tiles;
  __device__ PairWork(const LmParams& p, int pair)
      : n_sweeps(1), mt0(0), part(0), tiles(0, 0, 1, 0) {
    const int V32 = (p.V + 31) >> 5;
    const int n_main = p.n_mt * p.n_ranges;
    if (pair < n_main) {
      mt0 = pair % p.n_mt;
      part = pair / p.n_mt;
      tiles = TileIter(0, p.main_units, p.n_ranges, part);
    } else {
      n_sweeps = p.n_mt;
      part = p.n_ranges + (pair - n_main);
      tiles = TileIter(p.main_units, V32 - p.main_units, p.n_tail, pair - n_main);
    }
  }
};

// Next logit of a scan in ascending vocabulary order (an equal one never displaces): selects, no branches, because the
// lanes of a warp rarely agree.
__device__ __forceinline__ void lm_scan2(float v, int i, float& v1, int& i1, float& v2, int& i2) {
  const bool first = v > v1, second = v > v2;
  v2 = first ? v1 : (second ? v : v2);
  i2 = first ? i1 : (second ? i : i2);
  v1 = first ? v : v1;
  i1 = first ? i : i1;
}

// Order-preserving key of (logit, vocabulary entry): larger logit first, lower entry on ties; 0 = no entry. Merging two
// top-two lists is then three 64-bit minima and maxima.
__device__ __forceinline__ unsigned long long lm_key(float z, int v) {
  const uint32_t b = __float_as_uint(z + 0.f);           // -0 ties with +0
  const uint32_t u = (b & 0x80000000u) ? ~b : (b | 0x80000000u);
  return v < 0 ? 0ull : (static_cast<unsigned long long>(u) << 32) | (0xffffffffu - static_cast<uint32_t>(v));
}
__device__ __forceinline__ float lm_key_value(unsigned long long k) {
  const uint32_t u = static_cast<uint32_t>(k >> 32);
  return k == 0ull ? -INFINITY : __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}
__device__ __forceinline__ int lm_key_entry(unsigned long long k) {
  return k == 0ull ? -1 : static_cast<int>(0xffffffffu - static_cast<uint32_t>(k));
}
struct LmTop2 { unsigned long long a, b; };              // a >= b
__device__ __forceinline__ void lm_merge(LmTop2& t, unsigned long long a, unsigned long long b) {
  const unsigned long long lo = a < t.a ? a : t.a;
  t.a = a < t.a ? t.a : a;
  t.b = b < t.b ? t.b : b;
  t.b = lo < t.b ? t.b : lo;
}

struct LmRowStats { float m, s, t, v1, v2; int i1, i2; };    // of a row (or a column) over the entries a lane has seen

// 32 logits of a row, vocabulary entries v0 + j, of which the first nv exist. All lanes of the warp, a row each.
template <bool kEntropy>
__device__ __forceinline__ void lm_fold32(uint32_t (&r)[32], int v0, int nv, float c, LmRowStats& st) {
  if (nv < 32) {                                  // ragged end of the vocabulary: columns past V count as -inf
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (j >= nv) r[j] = __float_as_uint(-INFINITY);
  }
  // maxima of groups of eight: three-input max and, below, packed fp32 pairs halve the instruction count
  float gm[4];
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    const float* z = reinterpret_cast<const float*>(r + 8 * g);
    gm[g] = fmaxf(fmax3(fmax3(z[0], z[1], z[2]), z[3], z[4]), fmax3(z[5], z[6], z[7]));
  }
  const float cmax = fmaxf(fmax3(gm[0], gm[1], gm[2]), gm[3]);
  if (cmax > st.m) {
    const float f = ex2f((st.m - cmax) * c);
    st.s *= f;
    if (kEntropy) st.t *= f;
    st.m = cmax;
  }
  const float nmc = -st.m * c;
  const float2 c2 = make_float2(c, c), nmc2 = make_float2(nmc, nmc);
  float2 acc2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  float2 acz2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
  for (int j = 0; j < 32; j += 2) {
    float2 z = make_float2(__uint_as_float(r[j]), __uint_as_float(r[j + 1]));
    const float2 x = ffma2(z, c2, nmc2);
    const float2 e = make_float2(ex2f(x.x), ex2f(x.y));
    acc2[(j >> 1) & 1] = fadd2(acc2[(j >> 1) & 1], e);
    if (kEntropy) {
      if (nv < 32) {                              // masked columns hold -inf with e = 0: keep 0 * inf out of the sum
        if (j >= nv) z.x = 0.f;
        if (j + 1 >= nv) z.y = 0.f;
      }
      acz2[(j >> 1) & 1] = ffma2(e, z, acz2[(j >> 1) & 1]);
    }
  }
  st.s += (acc2[0].x + acc2[0].y) + (acc2[1].x + acc2[1].y);
  if (kEntropy) st.t += (acz2[0].x + acz2[0].y) + (acz2[1].x + acz2[1].y);
  // The top two change once every few hundred entries of a row, but among a warp's 32 rows about once per 32 columns: eight
  // entries at a time, without branches between them (a branch per entry took 1000 of the 1500 clocks of 32 columns). Where no
  // row of the warp gets a new one, one test is enough (2880 rows, 151936 x 1024 weights, 651 -> 640 us).
  if (__any_sync(0xffffffffu, cmax > st.v2)) {
#pragma unroll
    for (int g = 0; g < 4; ++g)
      if (gm[g] > st.v2) {
#pragma unroll
        for (int j = 8 * g; j < 8 * g + 8; ++j) lm_scan2(__uint_as_float(r[j]), v0 + j, st.v1, st.i1, st.v2, st.i2);
      }
  }
}

template <bool kEntropy>
__global__ void __launch_bounds__(LM_THREADS, 1)
lmhead_gemm_kernel(const __grid_constant__ CUtensorMap tmap_h, const __grid_constant__ CUtensorMap tmap_w,
                   const LmParams p) {
  pdl_launch_dependents();
  extern __shared__ uint8_t smem_raw[];
  // the dynamic window starts at the same offset in both CTAs of the pair, so the aligned
  // layouts coincide, as the paired MMA requires
  const uint32_t base_u32 = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base_u32 - smem_u32(smem_raw));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + LM_STAGES * LM_STAGE_BYTES);
  uint64_t* full_bar = bars;                      // [LM_STAGES]  (used in the leader)
  uint64_t* empty_bar = bars + LM_STAGES;         // [LM_STAGES]
  uint64_t* tmem_full = bars + 2 * LM_STAGES;     // [2]
  uint64_t* tmem_empty = bars + 2 * LM_STAGES + 2;  // [2]        (used in the leader)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * LM_STAGES + 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();        // 0 = leader
  const int pair = blockIdx.x >> 1;
  const PairWork work(p, pair);
  const TileIter& tiles = work.tiles;
  const int n_kb = p.d / LM_BK;

  if (threadIdx.x == 0) {
    for (int i = 0; i < LM_STAGES; ++i) { mbar_init(full_bar + i, 1); mbar_init(empty_bar + i, 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(tmem_full + i, 1); mbar_init(tmem_empty + i, 8); }
    fence_mbar_init();
  }
  // Operand rows that no copy writes are zero: nobody reads what comes of them, but multiplying stale data costs power,
  // and with it clock (16 sequences of 49 nodes, 104 of 128 rows fetched: 1010 us a pass against 985).
  {
    const int words = (LM_BM - (p.tile_rows >> 1)) * 8;          // 16-byte words per stage
    for (int i = threadIdx.x; i < LM_STAGES * words; i += LM_THREADS)
      *reinterpret_cast<uint4*>(smem + (i / words) * LM_STAGE_BYTES + (p.tile_rows >> 1) * 128 + (i % words) * 16) = make_uint4(0, 0, 0, 0);
    fence_async_smem();
  }
  if (warp == 5) {
    tmem_alloc_pair(tmem_slot, 512);
    tmem_relinquish_pair();
  }
  if (warp == 4 && lane == 0) { prefetch_tmap(&tmap_h); prefetch_tmap(&tmap_w); }
  tc_fence_before();
  cluster_sync_all();                             // both CTAs' barriers and TMEM are ready
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 4) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      if (p.wait_rows) pdl_wait();
      // the rows are spread evenly over the M tiles, and only those that a tile has are fetched
      const int half_rows = p.tile_rows >> 1;
      for (int t = 0; t < tiles.n_tiles; ++t) {
      int n0, nw;
      tiles.tile(t, n0, nw);
      for (int sweep = 0; sweep < work.n_sweeps; ++sweep) {
      const int row0 = (work.mt0 + sweep) * p.tile_rows + static_cast<int>(rank) * half_rows;
      int s0 = 0, s1 = 0;
      if (p.slots) {
        // sequence slots of this CTA; a slot past the last active sequence re-reads the M tile's
        // first sequence (its rows are computed and never looked at), which keeps the byte count
        // of a stage the same in both CTAs
        const int a_first = 4 * (work.mt0 + sweep);
        int a0 = a_first + 2 * static_cast<int>(rank), a1 = a0 + 1;
        if (a0 >= p.n_seq) a0 = a_first;
        if (a1 >= p.n_seq) a1 = a_first;
        s0 = __ldg(p.seq_index + a0);
        s1 = __ldg(p.seq_index + a1);
      }
        const int nh = nw >> 1;                   // rows of W this CTA stages
        const int nbox = (nh + 63) >> 6;
        const int w0 = n0 + static_cast<int>(rank) * nh;
        const uint32_t tx_pair = 2u * static_cast<uint32_t>(half_rows + 64 * nbox) * (LM_BK * 2);
        for (int kb = 0; kb < n_kb; ++kb) {
          mbar_wait(empty_bar + stage, phase ^ 1u, p.dev_status);
          uint8_t* sa = smem + stage * LM_STAGE_BYTES;
          uint8_t* sb = sa + LM_A_BYTES;
          if (rank == 0) mbar_expect_tx(full_bar + stage, tx_pair);
          const uint32_t fb = cluster_map(smem_u32(full_bar + stage), 0);
          if (p.slots) {
            tma_load_3d_pair(sa, &tmap_h, fb, kb * LM_BK, 0, s0);
            tma_load_3d_pair(sa + LM_BOX_BYTES, &tmap_h, fb, kb * LM_BK, 0, s1);
          } else {
            tma_load_2d_pair(sa, &tmap_h, fb, kb * LM_BK, row0);
          }
          for (int j = 0; j < nbox; ++j)
            tma_load_2d_pair(sb + j * LM_BOX_BYTES, &tmap_w, fb, kb * LM_BK, w0 + 64 * j);
          if (++stage == LM_STAGES) { stage = 0; phase ^= 1u; }
        }
      }   // sweeps
      }
    }
  } else if (warp == 5) {
    // ------------------------------------------------------------------ MMA issuer (leader CTA)
    if (lane == 0 && rank == 0) {
      int stage = 0;
      uint32_t phase = 0;
      const int n_all = work.n_sweeps * tiles.n_tiles;      // the accumulator buffers alternate over all sweeps
      for (int tt = 0; tt < n_all; ++tt) {
        const int t = tt / work.n_sweeps;
        int n0, nw;
        tiles.tile(t, n0, nw);
        const int buf = tt & 1;
        mbar_wait(tmem_empty + buf, ((tt >> 1) & 1u) ^ 1u, p.dev_status);
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(buf * LM_BN);
        const uint32_t idesc = idesc_bf16(2 * LM_BM, nw, false, false);
        for (int kb = 0; kb < n_kb; ++kb) {
          mbar_wait(full_bar + stage, phase, p.dev_status);
          tc_fence_after();
          const uint32_t sa = base_u32 + stage * LM_STAGE_BYTES;
          const uint64_t adesc = smem_desc_sw128(sa, 1024, 16);
          const uint64_t bdesc = smem_desc_sw128(sa + LM_A_BYTES, 1024, 16);
#pragma unroll
          for (int k = 0; k < LM_BK / 16; ++k) {
            // advancing 16 elements (32 bytes) along K inside the swizzle row: +2 in the
            // 16-byte-granular start address field
            tc_mma_ss_pair(d_tmem, adesc + 2u * k, bdesc + 2u * k, idesc, (kb | k) != 0);
          }
          tc_commit_pair(empty_bar + stage, 3);   // the stage is free again in both CTAs
          if (++stage == LM_STAGES) { stage = 0; phase ^= 1u; }
        }
        tc_commit_pair(tmem_full + buf, 3);       // both CTAs' accumulators are complete
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 0-3)
    const int row = warp * 32 + lane;  // TMEM lane == row of this CTA's half of the M tile
    const bool no_rows = warp * 32 >= (p.tile_rows >> 1);
    const float c = p.c;
    const uint32_t tmem_empty_leader = cluster_map(smem_u32(tmem_empty), 0);
    LmRowStats st = {-INFINITY, 0.f, 0.f, -INFINITY, -INFINITY, -1, -1};
    for (int t = 0, tt = 0; t < tiles.n_tiles; ++t)
    for (int sweep = 0; sweep < work.n_sweeps; ++sweep, ++tt) {
      int n0, nw;
      tiles.tile(t, n0, nw);
      const int buf = tt & 1;
      // several M tiles: this row's statistics over the tiles so far wait in its place of the partials
      LmPartial* const place = p.partial + static_cast<size_t>(work.part) * p.part_rows +
                               ((work.mt0 + sweep) * 2 + rank) * (p.tile_rows >> 1) + row;
      const bool mine = row < (p.tile_rows >> 1);
      if (work.n_sweeps > 1) {
        st = {-INFINITY, 0.f, 0.f, -INFINITY, -INFINITY, -1, -1};
        if (t > 0 && mine) {
          const LmPartial q = *place;
          st = {q.m, q.s, q.t, q.v1, q.v2, q.i1, q.i2};
        }
      }
      mbar_wait(tmem_full + buf, (tt >> 1) & 1u, p.dev_status);
      tc_fence_after();
      const int ncols = no_rows ? 0 : min(nw, p.V - n0);  // valid columns of this tile
      const uint32_t taddr = tmem_base + (static_cast<uint32_t>(warp * 32) << 16) + static_cast<uint32_t>(buf * LM_BN);
      // (The next 32 columns on their way to registers while the warp folds the ones at hand: 0.3 to 1 % slower, 488 rows, 151936
      // x 2048 weights, 230 -> 232 us; the MMAs hide the wait for them.)
      for (int c0 = 0; c0 < ncols; c0 += 32) {
        uint32_t r[32];
        tmem_ld32(taddr + c0, r);
        tc_wait_ld(r);
        lm_fold32<kEntropy>(r, n0 + c0, ncols - c0, c, st);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(tmem_empty_leader + static_cast<uint32_t>(buf) * 8u);
      if (work.n_sweeps > 1 || t == tiles.n_tiles - 1) {
        if (tt == 0 || work.n_sweeps == 1) pdl_wait();   // the previous pass's partials may be read until earlier kernels are done
        LmPartial out;
        out.m = st.m; out.s = st.s; out.v1 = st.v1; out.v2 = st.v2; out.i1 = st.i1; out.i2 = st.i2; out.t = st.t; out.pad = 0;
        if (mine) *place = out;
      }
    }
  }

  pdl_wait();
  // nobody leaves, and tensor memory stays allocated, until both CTAs are done: the leader's
  // MMAs write the peer's tensor memory and its commits arrive on the peer's barriers
  tc_fence_before();
  cluster_sync_all();
  if (warp == 5) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, 512);
  }
}

// Packs the activation rows of the active sequences (an index list) without gaps: one warp per row. Beside the stream
// of W it is small: 3 sequences of 61 rows of 5120 are 1.9 MB.
__global__ void __launch_bounds__(256)
lmhead_pack_rows_kernel(const uint4* __restrict__ h, const int32_t* __restrict__ seq_index, uint4* __restrict__ out, int B, int T,
                        int vecs /* 16-byte words per row */, long long n_rows) {
  pdl_launch_dependents();
  const int lane = threadIdx.x & 31;
  const long long r = static_cast<long long>(blockIdx.x) * 8 + (threadIdx.x >> 5);
  const bool active = r < n_rows;
  const int a = active ? static_cast<int>(r / T) : 0;
  const int seq = __ldg(seq_index + a);
  const bool there = static_cast<unsigned>(seq) < static_cast<unsigned>(B);   // (finalize skips a sequence that is not)
  const uint4* src = h + (static_cast<long long>(there ? seq : 0) * T + (active ? r % T : 0)) * vecs;
  pdl_wait();
  if (!active) return;
  uint4* dst = out + r * vecs;
#pragma unroll 4
  for (int i = lane; i < vecs; i += 32) dst[i] = __ldg(src + i);
}

// ---------------------------------------------------------------------------------------
// Merge of the per-range partials + drafted-token logits.
// ---------------------------------------------------------------------------------------
struct LmFinalizeParams {
  int B, T, d, V, n_ranges;
  int stride;       // partial rows per vocabulary range
  int pitch;        // partial rows per active sequence (T: packed rows)
  float scale, c;
  const int32_t* seq_index;
  const LmPartial* partial;
  const uint16_t *h, *W;
  const int32_t *parent, *tok;
  int32_t* dev_status;
  trispec_stats out;
};

constexpr int LM_FIN_THREADS = 256;   // 8 warps = 8 rows per block

__device__ __forceinline__ float bf16_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }

// what a sum relative to maximum m is worth relative to M >= m
__device__ __forceinline__ float lm_weight(float m, float M, float c) { return (m == -INFINITY) ? 0.f : ex2f((m - M) * c); }

// One warp per (active sequence, node): merges the row's partial statistics and, for a child
// node, computes the logit of its drafted token in its parent's row (a d-long dot product).
// The dot product needs only the kernel's inputs, so it runs before the wait for the GEMM and
// overlaps that kernel's tail; after the wait every lane loads its share of the partials of
// the node's row and of the parent's row in one go and the warp folds them by shuffles.
// Bound by latency. (Going over the partials once before the wait, to have code and pages at hand, gave nothing beside the pair
// kernel: 150 rows, 50257 x 1024 weights, 34.8 us either way.) kCg: loads that bypass L1, where the blocks come to wait on the SMs
// of an attention in the same launch (one chain of 9 nodes 34.1 -> 33.4 us a pass); elsewhere they cost 1 to 4 us (LM head alone,
// 32000 x 1024 weights, 18 rows 21.3 -> 23.9 us, 61 rows 25.1 -> 28.7; 9 rows, 32000 x 2048, 31.6 -> 32.6).
template <bool kCg>
__global__ void __launch_bounds__(LM_FIN_THREADS)
lmhead_finalize_kernel(const LmFinalizeParams p, int n_seq) {
  pdl_launch_dependents();
  const int lane = threadIdx.x & 31;
  const long long w = static_cast<long long>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int T = p.T;
  bool active = w < static_cast<long long>(n_seq) * T;
  const int a = active ? static_cast<int>(w / T) : 0, node = active ? static_cast<int>(w % T) : 0;
  int seq = p.seq_index ? __ldg(p.seq_index + a) : a;
  if (static_cast<unsigned>(seq) >= static_cast<unsigned>(p.B)) {   // no such sequence: its rows are computed and dropped
    if (active && lane == 0 && p.dev_status) atomicExch(p.dev_status, TRISPEC_ERR_BAD_INDEX);
    active = false;
    seq = 0;
  }
  const long long row0 = static_cast<long long>(seq) * T;

  // ---- drafted-token logit z[parent(node)][tok[node]]: inputs only
  bool has_draft = false;
  int par = 0;
  float dot = 0.f;
  if (active && node >= 1) {
    par = __ldg(p.parent + row0 + node);
    const int tk = __ldg(p.tok + row0 + node);
    has_draft = par >= 0 && par < node && tk >= 0 && tk < p.V;
    if (has_draft) {
      const uint4* hv = reinterpret_cast<const uint4*>(p.h + (row0 + par) * p.d);
      const uint4* wv = reinterpret_cast<const uint4*>(p.W + static_cast<long long>(tk) * p.d);
      float acc[2] = {0.f, 0.f};
#pragma unroll 4
      for (int i = lane; i < p.d / 8; i += 32) {
        const uint4 x = __ldg(hv + i), y = __ldg(wv + i);
        acc[0] = fmaf(bf16_lo(x.x), bf16_lo(y.x), acc[0]); acc[1] = fmaf(bf16_hi(x.x), bf16_hi(y.x), acc[1]);
        acc[0] = fmaf(bf16_lo(x.y), bf16_lo(y.y), acc[0]); acc[1] = fmaf(bf16_hi(x.y), bf16_hi(y.y), acc[1]);
        acc[0] = fmaf(bf16_lo(x.z), bf16_lo(y.z), acc[0]); acc[1] = fmaf(bf16_hi(x.z), bf16_hi(y.z), acc[1]);
        acc[0] = fmaf(bf16_lo(x.w), bf16_lo(y.w), acc[0]); acc[1] = fmaf(bf16_hi(x.w), bf16_hi(y.w), acc[1]);
      }
      dot = acc[0] + acc[1];
      for (int o2 = 16; o2 > 0; o2 >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o2);
    }
  }
  if (!has_draft) par = node;                    // a valid row to load; the result is not used

  pdl_wait();                                    // the partials come from the GEMM kernel
  if (!active) return;

  // ---- merge of the per-range partials: own row (all statistics) and parent row (max, sum)
  const size_t stride = static_cast<size_t>(p.stride);
  const LmPartial* own = p.partial + static_cast<size_t>(a) * p.pitch + node;
  const LmPartial* parp = p.partial + static_cast<size_t>(a) * p.pitch + par;
  // Up to 148 ranges are five per lane: loaded at once, folded relative to the row's maximum, so that the chains
  // across the lanes are one maximum, the sums, and the top two as 64-bit keys, side by side.
  float m_own = -INFINITY, s_own = 0.f, t_own = 0.f, m_par = -INFINITY, s_par = 0.f;
  LmTop2 top = {0ull, 0ull};
  constexpr int kPer = 5;
  for (int r0 = 0; r0 < p.n_ranges; r0 += 32 * kPer) {
    float4 qa[kPer], qb[kPer];
    float2 qp[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int r = r0 + lane + 32 * u;
      qa[u] = make_float4(-INFINITY, 0.f, -INFINITY, -INFINITY);
      qb[u] = make_float4(__int_as_float(-1), __int_as_float(-1), 0.f, 0.f);
      qp[u] = make_float2(-INFINITY, 0.f);
      if (r < p.n_ranges) {
        const float4* q4 = reinterpret_cast<const float4*>(own + r * stride);
        const float2* qp2 = reinterpret_cast<const float2*>(parp + r * stride);
        qa[u] = kCg ? __ldcg(q4) : q4[0];        // m, s, v1, v2
        qb[u] = kCg ? __ldcg(q4 + 1) : q4[1];    // i1, i2, t, pad
        qp[u] = kCg ? __ldcg(qp2) : *qp2;        // m, s of the parent's row
      }
    }
    float mo = m_own, mp = m_par;
#pragma unroll
    for (int u = 0; u < kPer; ++u) { mo = fmaxf(mo, qa[u].x); mp = fmaxf(mp, qp[u].x); }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      mo = fmaxf(mo, __shfl_xor_sync(0xffffffffu, mo, o));
      mp = fmaxf(mp, __shfl_xor_sync(0xffffffffu, mp, o));
    }
    const float fo = lm_weight(m_own, mo, p.c), fp = lm_weight(m_par, mp, p.c);
    s_own *= fo; t_own *= fo; s_par *= fp;
    m_own = mo; m_par = mp;
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const float w = lm_weight(qa[u].x, mo, p.c);
      s_own = fmaf(qa[u].y, w, s_own);
      t_own = fmaf(qb[u].z, w, t_own);
      s_par = fmaf(qp[u].y, lm_weight(qp[u].x, mp, p.c), s_par);
      lm_merge(top, lm_key(qa[u].z, __float_as_int(qb[u].x)), lm_key(qa[u].w, __float_as_int(qb[u].y)));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s_own += __shfl_xor_sync(0xffffffffu, s_own, o);
    t_own += __shfl_xor_sync(0xffffffffu, t_own, o);
    s_par += __shfl_xor_sync(0xffffffffu, s_par, o);
    const unsigned long long a = __shfl_xor_sync(0xffffffffu, top.a, o), b = __shfl_xor_sync(0xffffffffu, top.b, o);
    lm_merge(top, a, b);
  }
  const float v1 = lm_key_value(top.a), v2 = lm_key_value(top.b);
  const int i1 = lm_key_entry(top.a), i2 = lm_key_entry(top.b);
  if (lane == 0) {
    const float lse = m_own * p.scale + logf(s_own);
    const long long o = row0 + node;
    p.out.max[o] = m_own * p.scale;
    p.out.lse[o] = lse;
    p.out.top1_val[o] = v1 * p.scale;
    p.out.top2_val[o] = v2 * p.scale;
    p.out.top1_idx[o] = i1;
    p.out.top2_idx[o] = i2;
    p.out.p_top1[o] = expf(v1 * p.scale - lse);
    p.out.p_top2[o] = expf(v2 * p.scale - lse);
    // entropy in nats: H = lse - E_p[z], E_p[z] = scale * sum(e * z_raw) / sum(e); never below 0
    if (p.out.entropy) p.out.entropy[o] = fmaxf(lse - p.scale * (t_own / s_own), 0.f);
    float dl = __int_as_float(0x7fc00000), pd = dl;
    if (has_draft) {
      dl = dot * p.scale;
      pd = expf(dl - (m_par * p.scale + logf(s_par)));
    }
    p.out.draft_logit[o] = dl;
    p.out.p_draft[o] = pd;
  }
}

// ---------------------------------------------------------------------------------------
// At most 64 columns, and at most 128 over a long W (batch-1 decoding, the paper's own setting; two trees; a batch of
// chains): operands swapped. With so few rows the GEMM is bound by streaming W, and the pair kernel above spends half of its ring
// on H tiles. Here W is the M-side operand, the rows are the N side (16-128 columns), and one CTA per SM takes one
// vocabulary range. A tile is up to 2 x 128 vocabulary entries, two MMAs that share the k-block of H: a stage is
// 32 KB of W and 2-16 KB of H, so that up to 160 KB of W are in flight per SM and H, which every SM reads, adds 25 %
// (64 rows) to what L2 delivers (with 128 entries per tile it was 50 %, in the pair kernel it is 100 %).
// A range is cut into tiles of equal height, so that none ends in a tile that is nearly empty and W is streamed once.
// TMEM lane = vocabulary entry, column = row. Epilogue: warps 0-3 take the first 128 entries of a tile, warps
// 4-7 the others. A warp passes 32 entries x 16 columns through 2 KB of shared memory, after which a lane holds 16
// entries of one column and folds them into the running statistics it keeps for that column (the MMAs leave
// shared memory idle most of the time here; the butterflies over (value, index) tuples that did this before
// took 5 us for the last tile, which nothing overlaps).
// ---------------------------------------------------------------------------------------
constexpr int LW_BM = 128, LW_SUBS = 2, LW_BK = 64, LW_MAX_STAGES = 6, LW_EPI_WARPS = 8;
constexpr int LW_THREADS = 32 * (LW_EPI_WARPS + 2);
constexpr int LW_A_BYTES = LW_SUBS * LW_BM * LW_BK * 2;  // 32 KB of W per stage
// partial rows per vocabulary range
constexpr int lw_rows(long long n_rows) { return n_rows <= 64 ? 64 : static_cast<int>((n_rows + 15) / 16 * 16); }
constexpr int LW_XPOSE_BYTES = 2048;                     // 32 entries x 16 columns per epilogue warp
constexpr int LW_SMEM_BYTES = 227 * 1024;
constexpr int LW_RING_BYTES = LW_SMEM_BYTES - 1024 /*alignment slack*/ - LW_EPI_WARPS * LW_XPOSE_BYTES - 256 /*barriers*/;

struct LmRowsParams {
  LmParams base;
  int n_rows, N;    // columns that are rows, and the same rounded up to 16
  int slot_rows;    // > 0: not packed rows but slots of this many (a multiple of 8) per sequence of the index list
  int wait_rows;    // the rows are written by the kernel before this one
  int n_tiles;      // tiles per vocabulary range
  int box_rows;     // W rows per copy: the height of half a tile
  int stages, stage_bytes;
};

typedef LmRowStats LmColStats;                              // of one column
struct LmColMerge { LmTop2 top; float m, s, t, pad; };     // the same on its way to the other warps

// 16 logits of one column, vocabulary entries v0 + j, of which those below v_end exist.
template <bool kEntropy>
__device__ __forceinline__ void lm_fold16(float (&z)[16], int v0, int v_end, float c, LmColStats& st) {
  if (v0 + 16 > v_end) {                          // ragged end: entries that do not exist count as -inf
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (v0 + j >= v_end) z[j] = -INFINITY;
  }
  float gm[2];
#pragma unroll
  for (int g = 0; g < 2; ++g)
    gm[g] = fmaxf(fmax3(fmax3(z[8 * g], z[8 * g + 1], z[8 * g + 2]), z[8 * g + 3], z[8 * g + 4]),
                  fmax3(z[8 * g + 5], z[8 * g + 6], z[8 * g + 7]));
  const float cmax = fmaxf(gm[0], gm[1]);
  if (cmax > st.m) {
    const float f = ex2f((st.m - cmax) * c);
    st.s *= f;
    if (kEntropy) st.t *= f;
    st.m = cmax;
  }
  const float nmc = (st.m == -INFINITY) ? 0.f : -st.m * c;
  const float2 c2 = make_float2(c, c), nmc2 = make_float2(nmc, nmc);
  float2 acc = make_float2(0.f, 0.f), acz = make_float2(0.f, 0.f);
#pragma unroll
  for (int j = 0; j < 16; j += 2) {
    const float2 x = ffma2(make_float2(z[j], z[j + 1]), c2, nmc2);
    const float2 e = make_float2(ex2f(x.x), ex2f(x.y));
    acc = fadd2(acc, e);
    if (kEntropy)                                 // keep 0 * inf out of the sum
      acz = ffma2(e, make_float2(z[j] == -INFINITY ? 0.f : z[j], z[j + 1] == -INFINITY ? 0.f : z[j + 1]), acz);
  }
  st.s += acc.x + acc.y;
  if (kEntropy) st.t += acz.x + acz.y;
#pragma unroll
  for (int g = 0; g < 2; ++g)
    if (gm[g] > st.v2) {
#pragma unroll
      for (int j = 8 * g; j < 8 * g + 8; ++j) lm_scan2(z[j], v0 + j, st.v1, st.i1, st.v2, st.i2);
    }
}

// 32 entries x 16 columns of an accumulator (r: on their way): lane (entry) x columns -> 16 entries of one column per lane,
// ascending, through the warp's 2 KB at xb; `more`: the next 16 columns are sent for. The upper lanes read their entries in the order j ^ 1: entries of other parity lie in the other 16 banks.
__device__ __forceinline__ void lm_block16(uint32_t (&r)[16], uint32_t next, bool more, float* xb, int lane, float (&z)[16]) {
  const int col = lane & 15, upper = lane >> 4, flip = upper;
  tc_wait_ld(r);
  __syncwarp();                           // the block before this one has been read
#pragma unroll
  for (int j = 0; j < 4; ++j)             // word (entry e, column c): 16 e + 4 (c / 4 ^ (e / 2) % 4) + c % 4
    *reinterpret_cast<uint4*>(xb + lane * 16 + ((j ^ ((lane >> 1) & 3)) << 2)) =
        make_uint4(r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
  if (more) tmem_ld16(next, r);
  __syncwarp();
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int e = 16 * upper + (j ^ flip);
    z[j] = xb[e * 16 + (((col >> 2) ^ ((j >> 1) & 3)) << 2) + (col & 3)];
  }
#pragma unroll
  for (int j = 0; j < 16; j += 2) {       // back to ascending entries
    const float a = z[j], b = z[j + 1];
    z[j] = flip ? b : a;
    z[j + 1] = flip ? a : b;
  }
}

// The lanes l and l + 16 covered different entries of a column.
template <bool kEntropy>
__device__ __forceinline__ LmColMerge lm_merge_halves(const LmColStats& q, float c) {
  LmColMerge o;
  o.top.a = lm_key(q.v1, q.i1); o.top.b = lm_key(q.v2, q.i2); o.pad = 0.f;
  const float om = __shfl_xor_sync(0xffffffffu, q.m, 16), os = __shfl_xor_sync(0xffffffffu, q.s, 16);
  const float ot = kEntropy ? __shfl_xor_sync(0xffffffffu, q.t, 16) : 0.f;
  const unsigned long long oa = __shfl_xor_sync(0xffffffffu, o.top.a, 16), ob = __shfl_xor_sync(0xffffffffu, o.top.b, 16);
  lm_merge(o.top, oa, ob);
  o.m = fmaxf(q.m, om);
  const float f = lm_weight(q.m, o.m, c), g = lm_weight(om, o.m, c);
  o.s = fmaf(q.s, f, os * g);
  o.t = kEntropy ? fmaf(q.t, f, ot * g) : 0.f;
  return o;
}

// A column's eight shares, relative to their common maximum: no chain from share to share.
template <bool kEntropy>
__device__ __forceinline__ LmPartial lm_merge_shares(const LmColMerge (&q)[8], float c) {
  LmTop2 top = {0ull, 0ull};
  LmPartial out;
  out.m = -INFINITY; out.s = 0.f; out.t = 0.f; out.pad = 0;
#pragma unroll
  for (int s = 0; s < 8; ++s) out.m = fmaxf(out.m, q[s].m);
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const float f = lm_weight(q[s].m, out.m, c);
    out.s = fmaf(q[s].s, f, out.s);
    if (kEntropy) out.t = fmaf(q[s].t, f, out.t);
    lm_merge(top, q[s].top.a, q[s].top.b);
  }
  out.v1 = lm_key_value(top.a); out.v2 = lm_key_value(top.b);
  out.i1 = lm_key_entry(top.a); out.i2 = lm_key_entry(top.b);
  return out;
}

// kRows = 64 or 128: columns that the tensor memory and the statistics are laid out for
template <bool kEntropy, int kRows>
__device__ __forceinline__ void lm_rows_cta(const CUtensorMap& tmap_w, const CUtensorMap& tmap_h, const LmRowsParams& sp, int range) {
  const LmParams& p = sp.base;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base_u32 = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base_u32 - smem_u32(smem_raw));
  uint8_t* xpose = smem + sp.stages * sp.stage_bytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(xpose + LW_EPI_WARPS * LW_XPOSE_BYTES);
  uint64_t* full_bar = bars;
  uint64_t* empty_bar = bars + LW_MAX_STAGES;
  uint64_t* tmem_full = bars + 2 * LW_MAX_STAGES;
  uint64_t* tmem_empty = bars + 2 * LW_MAX_STAGES + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * LW_MAX_STAGES + 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int V16 = (p.V + 15) >> 4;
  const int v_begin = static_cast<int>((static_cast<long long>(V16) * range) / p.n_ranges) << 4;
  const int v_stop = min(static_cast<int>((static_cast<long long>(V16) * (range + 1)) / p.n_ranges) << 4, p.V);
  const int n_tiles = sp.n_tiles;
  const int n_kb = p.d / LW_BK;
  // 8-entry units of the range, spread evenly over 2 n_tiles halves
  const int units = (v_stop - v_begin + 7) >> 3;
  auto half_begin = [&](int i) { return min(v_begin + 8 * ((units * i) / (LW_SUBS * n_tiles)), v_stop); };

  if (threadIdx.x == 0) {
    for (int i = 0; i < sp.stages; ++i) { mbar_init(full_bar + i, 1); mbar_init(empty_bar + i, 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(tmem_full + i, 1); mbar_init(tmem_empty + i, LW_EPI_WARPS); }
    fence_mbar_init();
  }
  if (warp == LW_EPI_WARPS + 1) {
    tmem_alloc(tmem_slot, 4 * kRows);             // two buffers of two accumulators of kRows columns
    tmem_relinquish();
  }
  if (warp == LW_EPI_WARPS && lane == 0) { prefetch_tmap(&tmap_h); prefetch_tmap(&tmap_w); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == LW_EPI_WARPS) {
    if (lane == 0) {   // ---------------------------------------------------------- TMA producer
      int stage = 0;
      uint32_t phase = 0;
      const int n_slots = sp.slot_rows > 0 ? p.n_seq : 1;      // one box per slot; packed rows are one box
      const int slot_bytes = sp.slot_rows * (LW_BK * 2);
      if (sp.wait_rows) pdl_wait();
      const uint32_t tx = static_cast<uint32_t>(LW_SUBS * sp.box_rows + (sp.slot_rows > 0 ? sp.n_rows : sp.N)) * (LW_BK * 2);
      for (int t = 0; t < n_tiles; ++t) {
        const int w0 = half_begin(LW_SUBS * t), w1 = half_begin(LW_SUBS * t + 1);
        for (int kb = 0; kb < n_kb; ++kb) {
          mbar_wait(empty_bar + stage, phase ^ 1u, p.dev_status);
          uint8_t* sa = smem + stage * sp.stage_bytes;
          mbar_expect_tx(full_bar + stage, tx);     // a box always delivers its full size (rows past V: zero fill)
          tma_load_2d(sa, &tmap_w, full_bar + stage, kb * LW_BK, w0);
          tma_load_2d(sa + LW_A_BYTES / 2, &tmap_w, full_bar + stage, kb * LW_BK, w1);
          for (int a = 0; a < n_slots; ++a)       // rows past the last: zero fill
            tma_load_3d(sa + LW_A_BYTES + a * slot_bytes, &tmap_h, full_bar + stage, kb * LW_BK, 0,
                        p.seq_index ? __ldg(p.seq_index + a) : 0);
          if (++stage == sp.stages) { stage = 0; phase ^= 1u; }
        }
      }
      // The kernels after this one may start when its last copies are on their way. Earlier their blocks keep an attention on
      // a second stream off the SMs left to it (a pass of one sequence behind other work: 197 us, now 133), and their
      // first loads, behind the stream of W, take longer than it saves (LM head alone, 9 rows: 34.2 -> 32.8 us).
      pdl_launch_dependents();
    }
  } else if (warp == LW_EPI_WARPS + 1) {
    if (lane == 0) {   // ---------------------------------------------------------- MMA issuer
      int stage = 0;
      uint32_t phase = 0;
      const uint32_t idesc = idesc_bf16(LW_BM, sp.N, false, false);
      for (int t = 0; t < n_tiles; ++t) {
        const int buf = t & 1;
        mbar_wait(tmem_empty + buf, ((t >> 1) & 1u) ^ 1u, p.dev_status);
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(buf * (2 * kRows));
        for (int kb = 0; kb < n_kb; ++kb) {
          mbar_wait(full_bar + stage, phase, p.dev_status);
          tc_fence_after();
          const uint32_t sa = base_u32 + stage * sp.stage_bytes;
          const uint64_t bdesc = smem_desc_sw128(sa + LW_A_BYTES, 1024, 16);
#pragma unroll
          for (int u = 0; u < LW_SUBS; ++u) {
            const uint64_t adesc = smem_desc_sw128(sa + u * (LW_A_BYTES / 2), 1024, 16);
#pragma unroll
            for (int k = 0; k < LW_BK / 16; ++k)
              tc_mma_ss(d_tmem + static_cast<uint32_t>(kRows) * u, adesc + 2u * k, bdesc + 2u * k, idesc, (kb | k) != 0);
          }
          tc_commit(empty_bar + stage);
          if (++stage == sp.stages) { stage = 0; phase ^= 1u; }
        }
        tc_commit(tmem_full + buf);
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 0-7)
    const int quad = warp & 3, half = warp >> 2;
    const int col = lane & 15, upper = lane >> 4;           // column within 16, entries 0-15 or 16-31 of the warp's 32
    float* xb = reinterpret_cast<float*>(xpose + warp * LW_XPOSE_BYTES);
    LmColStats run[kRows / 16];                 // columns 16 h + col, this lane's share of the entries
#pragma unroll
    for (int h = 0; h < kRows / 16; ++h) {
      run[h].m = -INFINITY; run[h].s = 0.f; run[h].t = 0.f;
      run[h].v1 = -INFINITY; run[h].v2 = -INFINITY; run[h].i1 = -1; run[h].i2 = -1;
    }
    const float c = p.c;
    for (int t = 0; t < n_tiles; ++t) {
      const int buf = t & 1;
      mbar_wait(tmem_full + buf, (t >> 1) & 1u, p.dev_status);
      tc_fence_after();
      const int v_warp = half_begin(LW_SUBS * t + half) + quad * 32;            // first entry of this warp
      const int v_end = half_begin(LW_SUBS * t + half + 1);
      const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + static_cast<uint32_t>(buf * (2 * kRows) + half * kRows);
      if (v_warp < v_end) {
        uint32_t r[16];
        tmem_ld16(taddr, r);
#pragma unroll
        for (int h = 0; h < kRows / 16; ++h) {
          if (16 * h >= sp.N) break;
          float z[16];
          lm_block16(r, taddr + 16 * (h + 1), 16 * (h + 1) < sp.N, xb, lane, z);
          if (v_warp + 16 * upper < v_end) lm_fold16<kEntropy>(z, v_warp + 16 * upper, v_end, c, run[h]);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tmem_empty + buf);
    }
    // The lanes l and l + 16 and the eight warps covered different vocabulary entries: merge through the ring's
    // memory (every copy has landed and every MMA has read it: the last accumulator is complete).
    LmColMerge* red = reinterpret_cast<LmColMerge*>(smem);          // [8 warps][kRows columns]
#pragma unroll
    for (int h = 0; h < kRows / 16; ++h) {
      if (16 * h >= sp.N) break;
      const LmColMerge o = lm_merge_halves<kEntropy>(run[h], c);
      if (upper == 0) red[warp * kRows + 16 * h + col] = o;
    }
    asm volatile("bar.sync 2, 256;" ::: "memory");   // the eight epilogue warps
    if (warp < kRows / 32) {
      const int column = warp * 32 + lane;
      pdl_wait();   // the partials of the previous pass may still be read until earlier kernels are done
      if (column < sp.n_rows) {
        LmColMerge q[LW_EPI_WARPS];
#pragma unroll
        for (int w2 = 0; w2 < LW_EPI_WARPS; ++w2) q[w2] = red[w2 * kRows + column];
        p.partial[static_cast<size_t>(range) * p.part_rows + column] = lm_merge_shares<kEntropy>(q, c);
      }
    }
  }
  pdl_wait();
  tc_fence_before();
  __syncthreads();
  if (warp == LW_EPI_WARPS + 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 4 * kRows);
  }
}

template <bool kEntropy, int kRows>
__global__ void __launch_bounds__(LW_THREADS, 1)
lmhead_rows_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_h,
                   const LmRowsParams sp) {
  lm_rows_cta<kEntropy, kRows>(tmap_w, tmap_h, sp, blockIdx.x);
}

// The attention beside the LM head in one launch: the first CTAs take its items, the others a vocabulary range each. Neither
// waits for the other. Before, the attention was a launch of its own on a second stream, forked and joined by events.
template <bool kEntropy, int kRows, bool kPair>
__global__ void __launch_bounds__(LW_THREADS, 1)
lmhead_rows_beside_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_h, const LmRowsParams sp,
                          const __grid_constant__ AttnBeside at) {
  const int block = blockIdx.x;
  if (block < at.ctas) {
    pdl_launch_dependents();
    const int spare = static_cast<int>(threadIdx.x >> 5) - AT_THREADS / 32;
    if (spare == 0 && at.masks) attn_mask_warp<kPair>(at.p, block);
    if (spare == 1 && at.masks) {                      // what the tree step returns, of all sequences
      const int lane = threadIdx.x & 31, T = at.tree.T;
      for (int b = block; b < at.tree.B; b += at.ctas) {
        const int32_t* parent = at.tree.parent + static_cast<long long>(b) * T;
        const WarpMask m = tree_mask_climb(lane < T ? __ldg(parent + lane) : -1, lane + 32 < T ? __ldg(parent + lane + 32) : -1, T, lane);
        pdl_wait();                                    // before the first global write
        tree_mask_store(m, b, T, lane, at.tree.mask, at.tree.depth, at.tree.dev_status);
      }
    }
    if (spare < 0)
      attn_split_cta<kPair ? MERGE_IN_TURN_PAIR : MERGE_IN_TURN, 1>(at.k, at.v, at.kt, at.vt, at.p, block);
  } else if (block - at.ctas < sp.base.n_ranges) {     // (clusters of two: the grid may hold one CTA more)
    lm_rows_cta<kEntropy, kRows>(tmap_w, tmap_h, sp, block - at.ctas);
  }
}

// ---------------------------------------------------------------------------------------
// More rows than the small-row kernel takes, in tiles that leave a quarter of the pair kernel's M lanes or more empty: operands
// swapped in a CTA pair. W is the M side (256 vocabulary entries per tile, 128 per CTA), the rows are the N side, exactly as
// many columns as there are (to 16): no MMA cycle goes to padding (312 rows run as 2 x 160 columns instead of 2 x 256 lanes).
// What bounds both kernels beside the power limit is how fast L2 delivers operands (about 53 of 64 bytes per clock and SM);
// the statistics cross the lanes through shared memory as in the small-row kernel, twice the work per logit of the pair
// kernel's, hidden behind the MMAs of 32 k-blocks and more. Both CTAs' statistics meet through distributed shared memory, so
// that a range still is one row block of the partials. Up to 8 stages of 16 KB of W and up to 12 KB of H per CTA.
// ---------------------------------------------------------------------------------------
constexpr int LC_EPI_WARPS = 8, LC_THREADS = 32 * (LC_EPI_WARPS + 2), LC_MAX_STAGES = 8, LC_MAX_COLS = 256;
constexpr int LC_MIN_V = 96 << 10;                                // vocabulary from which it is taken
constexpr int LC_A_BYTES = 128 * LM_BK * 2;                        // 16 KB: this CTA's half of the W tile
constexpr int LC_RING_BYTES = LW_SMEM_BYTES - 1024 - LC_EPI_WARPS * LW_XPOSE_BYTES - 256;

struct LmColsParams {
  LmParams base;    // tile_rows: columns of a tile, a multiple of 16
  int n_rows;
  int stages, stage_bytes;
};

template <bool kEntropy>
__global__ void __launch_bounds__(LC_THREADS, 1)
lmhead_cols_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_h, const LmColsParams sp) {
  pdl_launch_dependents();
  const LmParams& p = sp.base;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base_u32 = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base_u32 - smem_u32(smem_raw));
  uint8_t* xpose = smem + sp.stages * sp.stage_bytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(xpose + LC_EPI_WARPS * LW_XPOSE_BYTES);
  uint64_t* full_bar = bars;                          // (used in the leader)
  uint64_t* empty_bar = bars + LC_MAX_STAGES;
  uint64_t* tmem_full = bars + 2 * LC_MAX_STAGES;
  uint64_t* tmem_empty = bars + 2 * LC_MAX_STAGES + 2;   // (used in the leader)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * LC_MAX_STAGES + 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();            // 0 = leader
  const PairWork work(p, blockIdx.x >> 1);
  const TileIter& tiles = work.tiles;
  const int n_kb = p.d / LM_BK;
  const int cols = p.tile_rows, half_cols = cols >> 1;

  if (threadIdx.x == 0) {
    for (int i = 0; i < sp.stages; ++i) { mbar_init(full_bar + i, 1); mbar_init(empty_bar + i, 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(tmem_full + i, 1); mbar_init(tmem_empty + i, 2 * LC_EPI_WARPS); }
    fence_mbar_init();
  }
  if (warp == LC_EPI_WARPS + 1) {
    tmem_alloc_pair(tmem_slot, 512);
    tmem_relinquish_pair();
  }
  if (warp == LC_EPI_WARPS && lane == 0) { prefetch_tmap(&tmap_h); prefetch_tmap(&tmap_w); }
  tc_fence_before();
  cluster_sync_all();                                 // both CTAs' barriers and TMEM are ready
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  LmColMerge* red = reinterpret_cast<LmColMerge*>(smem);           // [4 warps][columns], in the ring's memory at the end

  if (warp == LC_EPI_WARPS) {
    if (lane == 0) {   // ---------------------------------------------------------- TMA producer
      int stage = 0;
      uint32_t phase = 0;
      if (p.wait_rows) pdl_wait();
      const int row0 = work.mt0 * cols + static_cast<int>(rank) * half_cols;
      for (int t = 0; t < tiles.n_tiles; ++t) {
        int n0, nw;
        tiles.tile(t, n0, nw);
        const int nh = nw >> 1, nbox = (nh + 63) >> 6;
        const int w0 = n0 + static_cast<int>(rank) * nh;
        const uint32_t tx_pair = 2u * static_cast<uint32_t>(half_cols + 64 * nbox) * (LM_BK * 2);
        for (int kb = 0; kb < n_kb; ++kb) {
          mbar_wait(empty_bar + stage, phase ^ 1u, p.dev_status);
          uint8_t* sa = smem + stage * sp.stage_bytes;
          if (rank == 0) mbar_expect_tx(full_bar + stage, tx_pair);
          const uint32_t fb = cluster_map(smem_u32(full_bar + stage), 0);
          for (int j = 0; j < nbox; ++j) tma_load_2d_pair(sa + j * LM_BOX_BYTES, &tmap_w, fb, kb * LM_BK, w0 + 64 * j);
          tma_load_2d_pair(sa + LC_A_BYTES, &tmap_h, fb, kb * LM_BK, row0);
          if (++stage == sp.stages) { stage = 0; phase ^= 1u; }
        }
      }
    }
  } else if (warp == LC_EPI_WARPS + 1) {
    if (lane == 0 && rank == 0) {   // --------------------------------------------- MMA issuer (leader CTA)
      int stage = 0;
      uint32_t phase = 0;
      const uint32_t idesc = idesc_bf16(256, cols, false, false);
      for (int t = 0; t < tiles.n_tiles; ++t) {
        const int buf = t & 1;
        mbar_wait(tmem_empty + buf, ((t >> 1) & 1u) ^ 1u, p.dev_status);
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(buf * LC_MAX_COLS);
        for (int kb = 0; kb < n_kb; ++kb) {
          mbar_wait(full_bar + stage, phase, p.dev_status);
          tc_fence_after();
          const uint32_t sa = base_u32 + stage * sp.stage_bytes;
          const uint64_t adesc = smem_desc_sw128(sa, 1024, 16), bdesc = smem_desc_sw128(sa + LC_A_BYTES, 1024, 16);
#pragma unroll
          for (int k = 0; k < LM_BK / 16; ++k) tc_mma_ss_pair(d_tmem, adesc + 2u * k, bdesc + 2u * k, idesc, (kb | k) != 0);
          tc_commit_pair(empty_bar + stage, 3);
          if (++stage == sp.stages) { stage = 0; phase ^= 1u; }
        }
        tc_commit_pair(tmem_full + buf, 3);
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 0-7)
    const int quad = warp & 3, side = warp >> 2;              // lanes of tensor memory; every other block of 16 columns
    const int col = lane & 15, upper = lane >> 4;
    float* xb = reinterpret_cast<float*>(xpose + warp * LW_XPOSE_BYTES);
    const float c = p.c;
    const uint32_t tmem_empty_leader = cluster_map(smem_u32(tmem_empty), 0);
    LmColStats run[LC_MAX_COLS / 32];                         // columns 32 h + 16 side + col
#pragma unroll
    for (int h = 0; h < LC_MAX_COLS / 32; ++h) {
      run[h].m = -INFINITY; run[h].s = 0.f; run[h].t = 0.f;
      run[h].v1 = -INFINITY; run[h].v2 = -INFINITY; run[h].i1 = -1; run[h].i2 = -1;
    }
    for (int t = 0; t < tiles.n_tiles; ++t) {
      int n0, nw;
      tiles.tile(t, n0, nw);
      const int buf = t & 1;
      mbar_wait(tmem_full + buf, (t >> 1) & 1u, p.dev_status);
      tc_fence_after();
      const int v_first = n0 + static_cast<int>(rank) * (nw >> 1), v_end = min(v_first + (nw >> 1), p.V), v_warp = v_first + quad * 32;
      const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + static_cast<uint32_t>(buf * LC_MAX_COLS + 16 * side);
      if (v_warp < v_end && 16 * side < cols) {
        uint32_t r[16];
        tmem_ld16(taddr, r);
#pragma unroll
        for (int h = 0; h < LC_MAX_COLS / 32; ++h) {
          if (32 * h + 16 * side >= cols) break;
          float z[16];
          lm_block16(r, taddr + 32 * (h + 1), 32 * (h + 1) + 16 * side < cols, xb, lane, z);
          if (v_warp + 16 * upper < v_end) lm_fold16<kEntropy>(z, v_warp + 16 * upper, v_end, c, run[h]);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(tmem_empty_leader + static_cast<uint32_t>(buf) * 8u);
    }
#pragma unroll
    for (int h = 0; h < LC_MAX_COLS / 32; ++h) {
      if (32 * h + 16 * side >= cols) break;
      const LmColMerge o = lm_merge_halves<kEntropy>(run[h], c);
      if (upper == 0) red[quad * LC_MAX_COLS + 32 * h + 16 * side + col] = o;
    }
  }
  tc_fence_before();
  cluster_sync_all();    // both CTAs' statistics are in shared memory; the leader's MMAs and commits on the peer are over
  if (warp == LC_EPI_WARPS + 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, 512);
  }
  pdl_wait();            // the partials of the previous pass may still be read until earlier kernels are done
  // a column's eight shares, four of them the peer's; each CTA merges half of the columns
  for (int column = static_cast<int>(rank) * half_cols + threadIdx.x; column < (static_cast<int>(rank) + 1) * half_cols; column += LC_THREADS) {
    const int row = work.mt0 * cols + column;
    if (row >= sp.n_rows) break;
    LmColMerge q[8];
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const uint32_t at = cluster_map(smem_u32(red + (s & 3) * LC_MAX_COLS + column), s >> 2);
      const uint4 a = ld_cluster_u4(at), b = ld_cluster_u4(at + 16);
      q[s].top.a = (static_cast<unsigned long long>(a.y) << 32) | a.x;
      q[s].top.b = (static_cast<unsigned long long>(a.w) << 32) | a.z;
      q[s].m = __uint_as_float(b.x); q[s].s = __uint_as_float(b.y); q[s].t = __uint_as_float(b.z);
    }
    p.partial[static_cast<size_t>(work.part) * p.part_rows + row] = lm_merge_shares<kEntropy>(q, p.c);
  }
  cluster_sync_all();    // nobody leaves while its shared memory may still be read
}

static thread_local int tl_lm_reserved_sms = 0;
void lm_reserve_sms_once(int n) { tl_lm_reserved_sms = n > 0 ? n : 0; }

struct LmPlan {
  int n_seq;
  bool few_rows;   // at most 128 rows: lmhead_rows_kernel, one CTA and one vocabulary range per SM
  bool pack;       // the rows of an index list are gathered into the workspace first
  bool slots;      // (no workspace to gather into) four slots of 64 node rows per M tile
  bool cols;       // lmhead_cols_kernel: the rows of an M tile are the columns
  int slot_rows;   // few_rows and an index list of several: columns per sequence, read without gathering; 0 = packed
  int n_mt;        // M tiles of 256 rows
  int n_ranges;    // vocabulary ranges of the main part (few_rows: one per CTA, at most this many)
  int tile_rows;   // rows per M tile (the rows are spread evenly over the tiles)
  int part_rows;   // partial rows per vocabulary range
  int n_tail;      // pairs that sweep all M tiles over a slice of the vocabulary's tail
  int main_units;  // 32-column units of the main part
  size_t required;   // workspace the call cannot do without
  size_t pack_bytes; // and what it needs on top of it to pack listed rows
  size_t partial_bytes() const {
    return static_cast<size_t>(n_ranges + n_tail) * part_rows * sizeof(LmPartial);
  }
};

// W is streamed from HBM for long enough (about twice L2) that what happens before and after it matters less
static bool lm_long_stream(const trispec_lmhead_args* a) { return static_cast<long long>(a->V) * a->d * 2 >= (256ll << 20); }

static bool lm_takes_few_rows(const trispec_lmhead_args* a, long long columns) {
  return columns <= (lm_long_stream(a) ? LM_FEW_ROWS : 64);
}

static int lm_ranges_within(size_t max_ws, int part_rows, int ranges) {
  const size_t fit = max_ws / (static_cast<size_t>(part_rows) * sizeof(LmPartial));
  return fit >= static_cast<size_t>(ranges) ? ranges : (fit > 0 ? static_cast<int>(fit) : 1);
}
// Plans the launch for rows that are packed, or that sit in slots of 64 per sequence. `max_ws` bounds the partial
// array: tail pairs, which cost a block of partial rows for every M tile each, are given up until it fits, and packed rows
// are cut into fewer ranges.
static void lm_plan_rows(const trispec_lmhead_args* a, int n_seq, bool slots, size_t max_ws, LmPlan* pl) {
  const long long rows = static_cast<long long>(n_seq) * a->T;
  pl->n_seq = n_seq;
  pl->slots = slots;
  pl->pack = false;
  pl->pack_bytes = 0;
  pl->n_tail = 0;
  pl->main_units = (a->V + 31) / 32;
  // From 65 rows on the small-row kernel's last tile, which nothing overlaps, costs more than the pair kernel's (7 us
  // at 128 columns): it pays once the stream of W is long (112 rows, 225 MB of W 86 -> 95 us a pass; 72 rows, 622 MB
  // 142 -> 123 us).
  pl->few_rows = lm_takes_few_rows(a, rows) && !slots;
  pl->slot_rows = 0;
  pl->cols = false;
  if (pl->few_rows) {
    pl->n_mt = 1;
    pl->tile_rows = 0;
    pl->part_rows = lw_rows(rows);
    const int V16 = (a->V + 15) / 16;
    int sms = device_sm_count() - tl_lm_reserved_sms;
    if (sms < 1) sms = 1;
    pl->n_ranges = sms < V16 ? sms : V16;
    return;
  }
  pl->n_mt = slots ? (n_seq + 3) / 4 : static_cast<int>((rows + 2 * LM_BM - 1) / (2 * LM_BM));
  pl->tile_rows = slots ? 2 * LM_BM : static_cast<int>(((rows + pl->n_mt - 1) / pl->n_mt + 15) / 16 * 16);
  pl->part_rows = pl->n_mt * pl->tile_rows;
  const int pairs = device_sm_count() / 2;       // one CTA pair per two SMs
  int r = pairs / pl->n_mt;
  if (r < 1) r = 1;
  const int V32 = (a->V + 31) / 32;
  if (r > V32) r = V32;
  if (!slots) r = lm_ranges_within(max_ws, pl->part_rows, r);
  pl->n_ranges = r;
  // Pairs that the M tiles leave over (74 = 16 x 4 + 10 for 16 M tiles) take the tail of the vocabulary,
  // every one of them for all M tiles in turn. Balance in whole tiles (a tile costs a k-loop whatever its
  // width): a main pair runs ceil(main_units / r / 8) tiles, a tail pair n_mt x ceil(slice / 8).
  int tail = pairs - pl->n_mt * r;
  if (pl->n_mt < 2 || tail < 1 || pl->n_mt * r > pairs) tail = 0;
  while (tail > 0 && static_cast<size_t>(r + tail) * pl->part_rows * sizeof(LmPartial) > max_ws) --tail;
  // Rows as columns where the M tiles would be a quarter padding or more, over rows long enough to hide the heavier statistics and
  // a vocabulary of five tiles and more per pair and M tile, behind which the last tile's do not count. Such a call costs less energy, not
  // fewer clocks. LM head alone, pair kernel and this one, in loops at the power limit: 183 rows of 5120 x 151936 weights 386 and
  // 362 us, 312 of 4096 x 128256 426 and 394, 576 of 4096 x 128256 619 and 580, 150 of 2048 x 151936 144 and 135; one call now and
  // then: 314 and 303, 352 and 333, 501 and 513, 124 and 127. Shorter vocabularies, loops and single calls: 183 of 5120 x 32000 91 and 97,
  // 77 and 87; 576 of 4096 x 33000 173 and 177, 144 and 154; 150 of 2048 x 65600 73 and 75, 63 and 70; 150 of 3072 x 100000 153
  // and 148, 124 and 127. Without padding or over short rows it loses: 488 of 2048 262 and 278, 150 of 1024 31 and 42.
  pl->cols = !slots && pl->tile_rows <= 192 && a->d >= 2048 && a->V >= LC_MIN_V;
  if (pl->cols) tail = 0;
  if (tail > 0) {
    int best_slice = 0, best_cost = (V32 / r + 7) / 8 + 1;    // without a tail: the longest main range
    {
      const int base = V32 / r, rem = V32 - base * r;
      best_cost = (base + (rem ? ((8 - (base & 7)) < rem ? (8 - (base & 7)) : rem) : 0) + 7) / 8;
    }
    const int ideal = static_cast<int>((static_cast<long long>(V32) * tail) / (static_cast<long long>(pl->n_mt) * r + tail) / tail);
    for (int slice = (ideal / 8 > 1 ? ideal / 8 - 1 : 1) * 8; slice <= (ideal / 8 + 2) * 8; slice += 8) {
      const int main_u = V32 - slice * tail;
      if (main_u < r) break;
      const int base = main_u / r, rem = main_u - base * r;
      const int chunk = 8 - (base & 7);
      const int longest = base + (rem ? (chunk < rem ? chunk : rem) : 0);
      const int main_tiles = (longest + 7) / 8, tail_tiles = pl->n_mt * (slice / 8);
      const int cost = main_tiles > tail_tiles ? main_tiles : tail_tiles;
      if (cost < best_cost) { best_cost = cost; best_slice = slice; }
    }
    if (best_slice > 0) {
      pl->n_tail = tail;
      pl->main_units = V32 - best_slice * tail;
    }
  }
}

// Rows of all sequences of the batch lie back to back already. Rows of an index list are gathered into the
// workspace first (a few MB at most beside the hundreds of MB of W) where the caller's workspace has room for
// them; without (a workspace that was sized for a call without a list, or the entry point that has none) they
// are read in slots of 64 per sequence. Every call needs the slots' workspace at least, so that how much a
// call asks for does not depend on how it reads its rows.
static int lm_plan(const trispec_lmhead_args* a, LmPlan* pl, size_t room, size_t max_ws = ~static_cast<size_t>(0)) {
  if (!a || a->B <= 0 || a->T <= 0 || a->d <= 0 || a->V <= 0) return TRISPEC_ERR_INVALID_ARG;
  if (a->T > 64 || (a->d % LM_BK) != 0 || a->V < 2) return TRISPEC_ERR_UNSUPPORTED;
  const int n_seq = a->seq_index ? a->B_active : a->B;
  if (n_seq <= 0 || n_seq > a->B) return TRISPEC_ERR_INVALID_ARG;
  if (n_seq == 1) {
    lm_plan_rows(a, n_seq, false, max_ws, pl);
    pl->required = pl->partial_bytes();
    return TRISPEC_OK;
  }
  // the slots' workspace is what a call of several sequences asks for, however it reads its rows (a packed plan that would
  // take more, one M tile of more than 248 rows from 9 to 12 sequences, has 72 ranges instead of 74)
  LmPlan slots;
  lm_plan_rows(a, n_seq, true, max_ws, &slots);
  const size_t required = slots.partial_bytes();
  lm_plan_rows(a, n_seq, false, required, pl);
  pl->required = slots.required = required;
  if (pl->few_rows) pl->n_ranges = lm_ranges_within(required, pl->part_rows, pl->n_ranges);
  if (!a->seq_index) return TRISPEC_OK;
  // A few listed sequences whose rows, rounded up to 8 each, still are columns of the small-row kernel: one copy per
  // sequence and stage instead of a gather, whose launch would come before the stream of W can start (3 of 5 sequences
  // of 23 nodes, 50257 x 2048 weights: 93.5 us with the gather, 87.5 us in slots of 64 in the pair kernel).
  const int slot_rows = (a->T + 7) / 8 * 8;
  if (pl->few_rows && n_seq <= 8 && lm_takes_few_rows(a, static_cast<long long>(n_seq) * slot_rows)) {
    pl->slot_rows = slot_rows;
    pl->part_rows = lw_rows(static_cast<long long>(n_seq) * slot_rows);
    pl->n_ranges = lm_ranges_within(required, pl->part_rows, pl->n_ranges);
    return TRISPEC_OK;
  }
  const size_t pack_bytes = static_cast<size_t>(n_seq) * a->T * a->d * 2;
  // The gather is a launch before the stream of W: not for a short stream that it does not make any shorter.
  const bool worth = pl->few_rows || lm_long_stream(a) || pl->n_mt < slots.n_mt;
  if (worth && room >= pl->required && room - pl->required >= pack_bytes) {
    pl->pack = true;
    pl->pack_bytes = pack_bytes;
  } else {
    *pl = slots;
  }
  return TRISPEC_OK;
}

}  // namespace trispec

extern "C" size_t trispec_lmhead_stats_workspace(const trispec_lmhead_args* a) {
  using namespace trispec;
  LmPlan pl;
  if (lm_plan(a, &pl, ~static_cast<size_t>(0)) != TRISPEC_OK) return 0;
  return pl.required + pl.pack_bytes;
}

namespace trispec {
bool lm_runs_small_rows(const trispec_lmhead_args* a) {
  LmPlan pl;
  return lm_plan(a, &pl, a->workspace_bytes) == TRISPEC_OK && pl.few_rows;
}
static int lm_check_planned(const trispec_lmhead_args* a, const LmPlan& pl) {
  if (!a->h || !a->W || !a->parent || !a->tok || !a->workspace) return TRISPEC_ERR_INVALID_ARG;
  if (!aligned16(a->h) || !aligned16(a->W) || (reinterpret_cast<uintptr_t>(a->workspace) & 255u))
    return TRISPEC_ERR_INVALID_ARG;
  if (!(a->logit_scale > 0.f) || !isfinite(a->logit_scale)) return TRISPEC_ERR_INVALID_ARG;
  const trispec_stats& o = a->out;
  if (!o.max || !o.lse || !o.top1_val || !o.top2_val || !o.p_top1 || !o.p_top2 || !o.top1_idx || !o.top2_idx ||
      !o.draft_logit || !o.p_draft)
    return TRISPEC_ERR_INVALID_ARG;
  if (a->workspace_bytes < pl.required) return TRISPEC_ERR_WORKSPACE;
  return TRISPEC_OK;
}
int lmhead_check(const trispec_lmhead_args* a) {
  LmPlan pl;
  const int rc = lm_plan(a, &pl, a ? a->workspace_bytes : 0);
  return rc != TRISPEC_OK ? rc : lm_check_planned(a, pl);
}
static int lmhead_stats_planned(const trispec_lmhead_args* a, const LmPlan& pl, void* stream, const AttnBeside* beside = nullptr);

int lmhead_stats_beside(const trispec_lmhead_args* a, const AttnBeside& beside, void* stream) {
  LmPlan pl;
  lm_reserve_sms_once(beside.ctas);
  const int rc = lm_plan(a, &pl, a->workspace_bytes);
  tl_lm_reserved_sms = 0;
  if (rc != TRISPEC_OK) return rc;
  return pl.few_rows ? lmhead_stats_planned(a, pl, stream, &beside) : TRISPEC_ERR_UNSUPPORTED;
}
}

extern "C" int trispec_lmhead_stats(const trispec_lmhead_args* a, void* stream) {
  trispec::EntryScope entry_scope;   // the first kernel launched below is an ordinary launch
  using namespace trispec;
  LmPlan pl;
  const int rc = lm_plan(a, &pl, a ? a->workspace_bytes : 0);
  tl_lm_reserved_sms = 0;            // a reservation holds for one call
  if (rc != TRISPEC_OK) return rc;
  return lmhead_stats_planned(a, pl, stream);
}

static int trispec::lmhead_stats_planned(const trispec_lmhead_args* a, const LmPlan& pl, void* stream, const AttnBeside* beside) {
  int n_ranges = pl.n_ranges;
  if (pl.few_rows) {
    // few units per range: as many ranges as keep the longest one as short, all of the same length where that comes
    // out even (a small vocabulary's statistics then do not depend on how many SMs the launch was given)
    const int V16 = (a->V + 15) / 16, per = (V16 + n_ranges - 1) / n_ranges;
    if (per <= 8) n_ranges = (V16 + per - 1) / per;
  }
  const int n_seq = pl.n_seq;
  const long long n_rows = static_cast<long long>(n_seq) * a->T;
  int rc = lm_check_planned(a, pl);
  if (rc != TRISPEC_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);

  // the entropy sum costs two more instructions per logit: only computed when it is asked for
  const bool want_entropy = a->out.entropy != nullptr;
  LmFinalizeParams f;
  f.B = a->B; f.T = a->T; f.d = a->d; f.V = a->V; f.n_ranges = n_ranges + pl.n_tail;
  f.scale = a->logit_scale; f.c = a->logit_scale * kLog2e;
  f.seq_index = a->seq_index;
  f.partial = static_cast<LmPartial*>(a->workspace);
  f.h = static_cast<const uint16_t*>(a->h);
  f.W = static_cast<const uint16_t*>(a->W);
  f.parent = a->parent; f.tok = a->tok; f.dev_status = a->dev_status;
  f.out = a->out;
  f.pitch = pl.slots ? 64 : (pl.slot_rows > 0 ? pl.slot_rows : a->T);

  LmParams p;
  p.T = a->T; p.d = a->d; p.V = a->V;
  p.n_seq = n_seq; p.n_mt = pl.n_mt; p.n_ranges = n_ranges;
  p.n_tail = pl.n_tail; p.main_units = pl.main_units;
  p.slots = pl.slots ? 1 : 0;
  p.tile_rows = pl.tile_rows;
  p.part_rows = pl.part_rows;
  p.wait_rows = pl.pack ? 1 : 0;
  p.c = f.c;
  p.seq_index = a->seq_index;
  p.partial = static_cast<LmPartial*>(a->workspace);
  p.dev_status = a->dev_status;

  const void* rows_base = a->h;
  if (pl.pack) {
    uint4* packed = reinterpret_cast<uint4*>(static_cast<char*>(a->workspace) + pl.required);
    rows_base = packed;
    TRISPEC_CUDA_OK(launch_dependent(lmhead_pack_rows_kernel, static_cast<unsigned>((n_rows + 7) / 8), 256, 0, st, 1,
                                     static_cast<const uint4*>(a->h), a->seq_index, packed, a->B, a->T, a->d / 8, n_rows));
    count_launch();
  }
  if (pl.few_rows) {
    LmRowsParams sp;
    sp.base = p;
    if (pl.pack) sp.base.seq_index = nullptr;
    sp.slot_rows = pl.slot_rows;
    sp.n_rows = pl.slot_rows > 0 ? n_seq * pl.slot_rows : static_cast<int>(n_rows);
    sp.wait_rows = p.wait_rows;
    sp.N = ((sp.n_rows + 15) / 16) * 16;
    sp.stage_bytes = LW_A_BYTES + sp.N * LW_BK * 2;
    sp.stages = LW_RING_BYTES / sp.stage_bytes;
    if (sp.stages > LW_MAX_STAGES) sp.stages = LW_MAX_STAGES;
    // tiles of equal height: as few as the longest range (in 8-entry units; the lengths differ by two) allows
    {
      const int V16 = (a->V + 15) / 16;
      const int u_max = 2 * ((V16 + n_ranges - 1) / n_ranges);
      sp.n_tiles = (u_max + LW_SUBS * LW_BM / 8 - 1) / (LW_SUBS * LW_BM / 8);
      sp.box_rows = 8 * ((u_max + LW_SUBS * sp.n_tiles - 1) / (LW_SUBS * sp.n_tiles));
    }
    CUtensorMap tm_wr, tm_hn;
    {
      const uint64_t dims[2] = {static_cast<uint64_t>(a->d), static_cast<uint64_t>(a->V)};
      const uint64_t strides[1] = {static_cast<uint64_t>(a->d) * 2};
      const uint32_t box[2] = {LW_BK, static_cast<uint32_t>(sp.box_rows)};
      if (!cached_tmap_bf16(&tm_wr, a->W, 2, dims, strides, box)) return TRISPEC_ERR_CUDA;
    }
    {
      // listed sequences: their nodes, one box each; otherwise all rows, back to back
      const bool listed = sp.base.seq_index != nullptr;
      const uint64_t n = listed ? static_cast<uint64_t>(a->T) : static_cast<uint64_t>(n_rows);
      const uint64_t dims[3] = {static_cast<uint64_t>(a->d), n, listed ? static_cast<uint64_t>(a->B) : 1};
      const uint64_t strides[2] = {static_cast<uint64_t>(a->d) * 2, static_cast<uint64_t>(a->d) * 2 * n};
      const uint32_t box[3] = {LW_BK, static_cast<uint32_t>(pl.slot_rows > 0 ? pl.slot_rows : sp.N), 1};
      if (!cached_tmap_bf16(&tm_hn, rows_base, 3, dims, strides, box)) return TRISPEC_ERR_CUDA;
    }
    typedef void (*RowsKernel)(CUtensorMap, CUtensorMap, LmRowsParams);
    static const RowsKernel table[2][2] = {{lmhead_rows_kernel<false, 64>, lmhead_rows_kernel<false, 128>},
                                           {lmhead_rows_kernel<true, 64>, lmhead_rows_kernel<true, 128>}};
    const int wide = sp.n_rows > 64 ? 1 : 0, which = (want_entropy ? 2 : 0) + wide;
    if (beside) {
      typedef void (*BesideKernel)(CUtensorMap, CUtensorMap, LmRowsParams, AttnBeside);
      static const BesideKernel beside_table[2][4] = {
          {lmhead_rows_beside_kernel<false, 64, false>, lmhead_rows_beside_kernel<false, 128, false>,
           lmhead_rows_beside_kernel<true, 64, false>, lmhead_rows_beside_kernel<true, 128, false>},
          {lmhead_rows_beside_kernel<false, 64, true>, lmhead_rows_beside_kernel<false, 128, true>,
           lmhead_rows_beside_kernel<true, 64, true>, lmhead_rows_beside_kernel<true, 128, true>}};
      const BesideKernel kernel = beside_table[beside->pair ? 1 : 0][which];
      static bool smem_set_beside[2][4][64] = {};
      rc = ensure_smem_limit(reinterpret_cast<const void*>(kernel), LW_SMEM_BYTES, smem_set_beside[beside->pair ? 1 : 0][which]);
      if (rc != TRISPEC_OK) return rc;
      const unsigned cluster = beside->pair ? 2u : 1u, ctas = static_cast<unsigned>(beside->ctas + n_ranges);
      TRISPEC_CUDA_OK(launch_dependent(kernel, (ctas + cluster - 1) / cluster * cluster, LW_THREADS, static_cast<size_t>(LW_SMEM_BYTES), st,
                                       cluster, tm_wr, tm_hn, sp, *beside));
    } else {
      const RowsKernel kernel = table[want_entropy ? 1 : 0][wide];
      static bool smem_set_rows[4][64] = {};
      rc = ensure_smem_limit(reinterpret_cast<const void*>(kernel), LW_SMEM_BYTES, smem_set_rows[which]);
      if (rc != TRISPEC_OK) return rc;
      TRISPEC_CUDA_OK(launch_dependent(kernel, static_cast<unsigned>(n_ranges), LW_THREADS,
                                       static_cast<size_t>(LW_SMEM_BYTES), st, 1, tm_wr, tm_hn, sp));
    }
    count_launch();
    f.stride = pl.part_rows;
    // One row per block: as many SMs as rows fetch the merge's operands (LM head alone, 151936 x 2048 weights, 9 rows 102.1 -> 101.0
    // us, 61 rows 105.2 -> 104.2; 61 rows, 32000 x 1024, 27.0 -> 26.5). More rows than 64 are eight per block (122 rows 138.8 -> 136.8).
    const unsigned per_block = sp.n_rows > 64 ? LM_FIN_THREADS / 32 : 1;
    TRISPEC_CUDA_OK(launch_dependent(beside ? lmhead_finalize_kernel<true> : lmhead_finalize_kernel<false>,
                                     (static_cast<unsigned>(n_rows) + per_block - 1) / per_block, 32 * per_block, 0, st, 1, f, n_seq));
    count_launch();
    return TRISPEC_OK;
  }
  CUtensorMap tm_h, tm_w;
  if (pl.slots) {
    const uint64_t dims[3] = {static_cast<uint64_t>(a->d), static_cast<uint64_t>(a->T), static_cast<uint64_t>(a->B)};
    const uint64_t strides[2] = {static_cast<uint64_t>(a->d) * 2, static_cast<uint64_t>(a->d) * 2 * a->T};
    const uint32_t box[3] = {LM_BK, 64, 1};
    if (!cached_tmap_bf16(&tm_h, a->h, 3, dims, strides, box)) return TRISPEC_ERR_CUDA;
  } else {
    const uint64_t dims[2] = {static_cast<uint64_t>(a->d), static_cast<uint64_t>(n_rows)};
    const uint64_t strides[1] = {static_cast<uint64_t>(a->d) * 2};
    const uint32_t box[2] = {LM_BK, static_cast<uint32_t>(p.tile_rows / 2)};
    if (!cached_tmap_bf16(&tm_h, rows_base, 2, dims, strides, box)) return TRISPEC_ERR_CUDA;
  }
  {
    const uint64_t dims[2] = {static_cast<uint64_t>(a->d), static_cast<uint64_t>(a->V)};
    const uint64_t strides[1] = {static_cast<uint64_t>(a->d) * 2};
    const uint32_t box[2] = {LM_BK, 64};
    if (!cached_tmap_bf16(&tm_w, a->W, 2, dims, strides, box)) return TRISPEC_ERR_CUDA;
  }
  if (pl.cols) {
    LmColsParams sp;
    sp.base = p;
    sp.n_rows = static_cast<int>(n_rows);
    sp.stage_bytes = LC_A_BYTES + p.tile_rows / 2 * (LM_BK * 2);
    sp.stages = LC_RING_BYTES / sp.stage_bytes < LC_MAX_STAGES ? LC_RING_BYTES / sp.stage_bytes : LC_MAX_STAGES;
    typedef void (*ColsKernel)(CUtensorMap, CUtensorMap, LmColsParams);
    const ColsKernel kernel = want_entropy ? lmhead_cols_kernel<true> : lmhead_cols_kernel<false>;
    static bool smem_set_cols[2][64] = {};
    rc = ensure_smem_limit(reinterpret_cast<const void*>(kernel), LW_SMEM_BYTES, smem_set_cols[want_entropy ? 1 : 0]);
    if (rc != TRISPEC_OK) return rc;
    TRISPEC_CUDA_OK(launch_dependent(kernel, static_cast<unsigned>(2 * p.n_mt * n_ranges), LC_THREADS, static_cast<size_t>(LW_SMEM_BYTES),
                                     st, 2, tm_w, tm_h, sp));
    count_launch();
    f.stride = pl.part_rows;
    TRISPEC_CUDA_OK(launch_dependent(lmhead_finalize_kernel<false>, static_cast<unsigned>((n_rows + 7) / 8), LM_FIN_THREADS, 0, st, 1, f, n_seq));
    count_launch();
    return TRISPEC_OK;
  }
  static bool smem_set[2][64] = {};
  typedef void (*GemmKernel)(CUtensorMap, CUtensorMap, LmParams);
  const GemmKernel kernel = want_entropy ? lmhead_gemm_kernel<true> : lmhead_gemm_kernel<false>;
  rc = ensure_smem_limit(reinterpret_cast<const void*>(kernel), LM_SMEM_BYTES, smem_set[want_entropy ? 1 : 0]);
  if (rc != TRISPEC_OK) return rc;
  TRISPEC_CUDA_OK(launch_dependent(kernel, static_cast<unsigned>(2 * (p.n_mt * n_ranges + pl.n_tail)), LM_THREADS,
                                   LM_SMEM_BYTES, st, 2, tm_h, tm_w, p));
  count_launch();
  f.stride = pl.part_rows;
  TRISPEC_CUDA_OK(launch_dependent(lmhead_finalize_kernel<false>, static_cast<unsigned>((n_rows + 7) / 8),
                                   LM_FIN_THREADS, 0, st, 1, f, n_seq));
  count_launch();
  return TRISPEC_OK;
}

// ---------------------------------------------------------------------------------------
// No-allocation variant: the partial statistics live in an array that is part of the library
// image instead of a caller-provided workspace.
// ---------------------------------------------------------------------------------------
namespace trispec {
// Scratch shared by every call on a device. In host code this name is only a handle for the
// runtime's symbol table, not an address a kernel could use: the device address is looked up
// once per device with cudaGetSymbolAddress and that pointer is what the kernels receive.
static __device__ __align__(256) unsigned char g_lm_noalloc_scratch[TRISPEC_NOALLOC_SCRATCH_BYTES];

// Device address of the scratch array on the current device; looked up on the first call per
// device (with that device current) and remembered.
static int lm_noalloc_scratch(void** out) {
  static void* addr[64] = {};
  static std::mutex mu;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return TRISPEC_ERR_CUDA;
  if (dev < 0 || dev >= 64) return TRISPEC_ERR_UNSUPPORTED;
  std::lock_guard<std::mutex> lock(mu);
  if (!addr[dev]) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_lm_noalloc_scratch) != cudaSuccess || !ptr) return TRISPEC_ERR_CUDA;
    addr[dev] = ptr;
  }
  *out = addr[dev];
  return TRISPEC_OK;
}
}  // namespace trispec

extern "C" int trispec_lmhead_stats_noalloc(const trispec_lmhead_args* a, void* stream) {
  trispec::EntryScope entry_scope;   // the first kernel launched below is an ordinary launch
  using namespace trispec;
  // planned so that the partial array fits the built-in scratch (fewer tail pairs where they would not)
  LmPlan pl;
  int rc = lm_plan(a, &pl, 0, TRISPEC_NOALLOC_SCRATCH_BYTES);
  if (rc != TRISPEC_OK) return rc;
  if (pl.required > TRISPEC_NOALLOC_SCRATCH_BYTES) return TRISPEC_ERR_TOO_LARGE;
  void* scratch = nullptr;
  rc = lm_noalloc_scratch(&scratch);
  if (rc != TRISPEC_OK) return rc;
  trispec_lmhead_args b = *a;     // same call, with the built-in array as its workspace
  b.workspace = scratch;
  b.workspace_bytes = TRISPEC_NOALLOC_SCRATCH_BYTES;
  return lmhead_stats_planned(&b, pl, stream);
}
