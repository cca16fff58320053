// Where the level blocks of the IC(0) substitutions lie in the ring of a CTA's shared memory (host
// arithmetic only, so that it can be checked without a GPU; team.cuh: ic_levels_team uses it).
//
// A producer writes the blocks in order; block l may be written once `need` levels have been consumed.
// The consumers announce l levels consumed at the barrier before level l, and that barrier waits for
// block l. So a block may need at most all levels but the one right before it: with two neighbours in
// each other's place, producer and consumers would wait for one another.
#pragma once
#include <algorithm>
#include <vector>

namespace mpcg {

// A block's place in the blob, its size, its place in the ring (all in 16-byte units), and `need`.
struct IcBlock {
  int from, size, at, need;
};

// Fills in `at` and `need` for a ring of `cap` units and `inflight` blocks in flight at most: blocks in
// order from the ring's start, one that would cross the end back at the start. False when a block does
// not fit the ring or would take its left neighbour's place.
inline bool ic_ring_places(std::vector<IcBlock>& blocks, int cap, int inflight) {
  int at = 0;
  for (int l = 0; l < (int)blocks.size(); ++l) {
    IcBlock& b = blocks[l];
    if (b.size > cap) return false;
    if (at + b.size > cap) at = 0;
    b.at = at;
    at += b.size;
    int need = std::max(0, l - inflight + 1);
    for (int j = l - 1; j >= need; --j)
      if (blocks[j].at < b.at + b.size && b.at < blocks[j].at + blocks[j].size) need = j + 1;
    if (l > 0 && need >= l) return false;
    b.need = need;
  }
  return true;
}

}  // namespace mpcg
