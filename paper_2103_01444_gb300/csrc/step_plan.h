// How a run of steps is split into launches of four, two and one steps.  Host
// only, without CUDA headers.
#pragma once
#include <cstdint>
#include <vector>

namespace pemlbm {

struct StepPlan {
  int64_t quads, pairs, singles;   // launched in this order
  int64_t launches() const { return quads + pairs + singles; }
  int steps(int64_t launch) const { return launch < quads ? 4 : launch < quads + pairs ? 2 : 1; }
};

// The plan of n steps: fours where the lattice takes them (quad, which
// includes pair), pairs, then single steps.  A run ends with a single step
// unless it goes on (open): that leaves the state before its last step in the
// other buffer, where the read-outs of that step look for it.
// keep: every launch swaps the two buffers, and an even number of steps is to
// end in the buffer it began in, as single steps do.  A four is then taken as
// two pairs, or a pair as two single steps.
inline StepPlan plan_steps(bool quad, bool pair, int64_t n, bool open, bool keep) {
  StepPlan p{0, 0, open || n == 0 ? 0 : 1};
  int64_t left = n - p.singles;
  if (quad) p.quads = left / 4;
  left -= 4 * p.quads;
  if (pair) p.pairs = left / 2;
  p.singles += left - 2 * p.pairs;
  if (keep && ((p.quads + p.pairs) & 1)) {
    if (p.quads > 0) {
      p.quads -= 1;
      p.pairs += 2;
    } else {
      p.pairs -= 1;
      p.singles += 2;
    }
  }
  return p;
}

// Which of the two graphs that a batch keeps was captured for given buffers
// (one per case).  A run of an even number of steps leaves each case where it
// was or in its other buffer, the same at every call of that count, so calls
// alternate between two sets of buffers at most.
struct GraphSlots {
  std::vector<int> bufs[2];   // empty: no graph in that slot
  int newest = 1;
  // the slot of the graph for these buffers, -1 for none
  int find(const std::vector<int> &b) const {
    for (int k = 0; k < 2; ++k)
      if (!bufs[k].empty() && bufs[k] == b) return k;
    return -1;
  }
  // the slot that a new graph for these buffers takes: the older one
  int take(const std::vector<int> &b) {
    newest ^= 1;
    bufs[newest] = b;
    return newest;
  }
  void clear(int slot) { bufs[slot].clear(); }
};

}  // namespace pemlbm
