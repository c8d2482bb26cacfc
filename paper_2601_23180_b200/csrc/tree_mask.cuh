// The ancestor mask of one sequence's tree, computed by a warp: lane l has the parents of the nodes l and l + 32, all nodes climb
// to the root together, one shuffle per level.
#pragma once
#include "host_common.h"

namespace trispec {

struct WarpMask {
  uint64_t bits0, bits1;   // of the nodes lane and lane + 32
  bool bad;                // not a tree (the same in every lane)
};

__device__ __forceinline__ WarpMask tree_mask_climb(int par0, int par1, int T, int lane) {
  const bool has0 = lane < T, has1 = lane + 32 < T;
  WarpMask m;
  // parent[i] must satisfy -1 <= parent[i] < i (and parent[0] == -1); anything else marks the
  // node, and every node whose walk meets it, as malformed: mask 0, depth -1
  int q0 = par0, q1 = par1;
  if (has0 && !(q0 >= -1 && q0 < lane && (lane != 0 || q0 == -1))) q0 = -2;
  if (has1 && !(q1 >= -1 && q1 < lane + 32)) q1 = -2;
  // not a tree (a parent out of range, or a second root): reported through the status word
  const bool bad = (has0 && (q0 == -2 || (lane != 0 && q0 == -1))) || (has1 && q1 < 0);
  m.bad = __any_sync(0xffffffffu, bad) != 0;
  // both parents of a lane in one register (a byte each, biased by 2), so that a walk needs
  // one shuffle per level
  const int packed = (q0 + 2) | ((q1 + 2) << 8);
  m.bits0 = m.bits1 = 0;
  int p0 = has0 ? lane : -1, p1 = has1 ? lane + 32 : -1;   // node each walk currently stands on
  // the walks strictly descend, so T levels are enough; stop as soon as every walk has ended
  for (int it = 0; it < T; ++it) {
    if (!__any_sync(0xffffffffu, (p0 & p1) >= 0)) break;   // some walk is still on a node
    const int g0 = __shfl_sync(0xffffffffu, packed, p0 & 31);
    const int g1 = __shfl_sync(0xffffffffu, packed, p1 & 31);
    if (p0 >= 0) { m.bits0 |= (1ull << p0); p0 = ((g0 >> ((p0 >> 5) << 3)) & 0xff) - 2; }
    if (p1 >= 0) { m.bits1 |= (1ull << p1); p1 = ((g1 >> ((p1 >> 5) << 3)) & 0xff) - 2; }
  }
  // a walk ends at -1 (above the root) or at -2 (malformed parent on the way)
  if (p0 != -1) m.bits0 = 0;
  if (p1 != -1) m.bits1 = 0;
  return m;
}

// Masks and depths of sequence b, a word of the status set where its parents are no tree.
__device__ __forceinline__ void tree_mask_store(const WarpMask& m, long long b, int T, int lane, uint64_t* mask, int32_t* depth,
                                                int32_t* status) {
  const long long base = b * T;
  if (m.bad && lane == 0 && status) atomicExch(status, TRISPEC_ERR_BAD_TREE);
  if (lane < T) { mask[base + lane] = m.bits0; if (depth) depth[base + lane] = __popcll(m.bits0) - 1; }
  if (lane + 32 < T) { mask[base + lane + 32] = m.bits1; if (depth) depth[base + lane + 32] = __popcll(m.bits1) - 1; }
}

}  // namespace trispec
