// How the clock warps of a ragged launch (ragged.cu) share the warp-groups:
// the host's cuts and the pieces that a clock warp reads off them.  Plain C++,
// so that the cuts can be checked without a GPU.
//
// A warp-group needs as many blocks of 128 clocks as its longest lane.  The
// even share is all blocks over all clock warps.  A warp-group above it cannot
// be split over more warps (its clocks follow one another) and decides how
// long the call takes, so it gets a clock warp to itself; what is left is
// shared evenly again by the clock warps that are left, until no warp-group is
// above the share.  Those go on one line of blocks, which is cut into equal
// segments of that share, a segment per clock warp.  So
//   * a warp-group spans two segments at most: the head piece at the end of
//     one and the tail piece at the start of the next;
//   * a segment runs its head first and its tail last, and head and tail of a
//     warp-group together are at most a segment, so the tail comes to its
//     hand-off when the head is done, or before it by less than a block per
//     segment (the last segment may be that much shorter).
// (Cutting at the longest warp-group instead, whatever the others are, made
// the tail of a short last segment wait for nearly all of it: 42 s where one
// stream of 2^27 bits lay among 2^20 of 2^13.)
#pragma once

#include <algorithm>
#include <cstdint>
#include <numeric>

#ifdef __CUDACC__
#define MICKEY_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define MICKEY_HOST_DEVICE inline
#endif

namespace mickey {

// The warp-groups by position: order[0 .. alone-1] have a clock warp each (slot
// p takes position p), order[alone .. W-1] lie on the line, slot alone + j
// taking its blocks [j L, j L + L).
struct RaggedLine {
  const uint64_t *blocks;   // W + 1 prefix sums of the blocks of order[0], order[1], ...
  const uint64_t *order;    // W warp-groups
  uint32_t W, alone;
  uint64_t L;
};

// Fill order (W) and blocks (W + 1) for warp-groups of c[w] blocks on `slots`
// clock warps.
inline RaggedLine ragged_cuts(const uint64_t *c, uint32_t W, uint64_t slots, uint64_t *order,
                              uint64_t *blocks) {
  std::iota(order, order + W, uint64_t(0));
  uint64_t rest = 0, longest = 0;
  for (uint32_t w = 0; w < W; ++w) {
    rest += c[w];
    longest = std::max(longest, c[w]);
  }
  auto share = [&](uint64_t warps) { return std::max<uint64_t>((rest + warps - 1) / warps, 1); };
  uint32_t alone = W <= slots ? W : 0;
  uint64_t L = share(slots);
  if (!alone && longest > L) {
    std::stable_sort(order, order + W, [c](uint64_t x, uint64_t y) { return c[x] > c[y]; });
    while (c[order[alone]] > L) {            // ends with a clock warp left: its share is the rest
      rest -= c[order[alone]];
      L = share(slots - ++alone);
    }
    std::sort(order + alone, order + W);     // the line in the streams' order
  }
  blocks[0] = 0;
  for (uint32_t p = 0; p < W; ++p) blocks[p + 1] = blocks[p] + c[order[p]];
  return RaggedLine{blocks, order, W, alone, L};
}

// The position on the line that holds block x: the last p with blocks[p] <= x
// (x below blocks[W]).
MICKEY_HOST_DEVICE uint32_t ragged_find(const RaggedLine &q, uint64_t x) {
  uint32_t lo = q.alone, hi = q.W;
  while (hi - lo > 1) {
    const uint32_t mid = lo + (hi - lo) / 2;
    if (q.blocks[mid] <= x) lo = mid;
    else hi = mid;
  }
  return lo;
}

// Piece k of a slot: blocks [ba, bb) of the warp-group at position p.  Returns
// false past the last piece.  The order is head, whole warp-groups (empty ones
// among them), tail; tails_first turns it round.
MICKEY_HOST_DEVICE bool ragged_piece(const RaggedLine &q, bool tails_first, uint32_t slot,
                                     uint32_t k, uint32_t &p, uint64_t &ba, uint64_t &bb) {
  if (slot < q.alone) {
    p = slot;
    ba = 0;
    bb = q.blocks[slot + 1] - q.blocks[slot];
    return k == 0;
  }
  const uint64_t total = q.blocks[q.W];
  const uint64_t a = q.blocks[q.alone] + uint64_t(slot - q.alone) * q.L;
  const uint64_t b = a + q.L < total ? a + q.L : total;
  if (a >= b) return false;
  const uint32_t pf = ragged_find(q, a), pl = ragged_find(q, b - 1);
  const bool tail = a > q.blocks[pf];
  const bool head = b < q.blocks[pl + 1] && (pl != pf || !tail);
  const uint32_t lo = pf + (tail ? 1 : 0), hi = b < q.blocks[pl + 1] ? pl : pl + 1;   // whole
  const uint32_t whole = hi > lo ? hi - lo : 0, n = whole + (head ? 1 : 0) + (tail ? 1 : 0);
  if (k >= n) return false;
  if (tails_first) k = n - 1 - k;
  p = head && k == 0 ? pl : k < whole + (head ? 1 : 0) ? lo + k - (head ? 1 : 0) : pf;
  ba = p == pf && tail ? a - q.blocks[p] : 0;
  bb = (b < q.blocks[p + 1] ? b : q.blocks[p + 1]) - q.blocks[p];
  return true;
}

}  // namespace mickey
