// How a run of steps is split into launches of four, two and one steps.  Host
// only, without CUDA headers.
#pragma once
#include <cstdint>

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

}  // namespace pemlbm
