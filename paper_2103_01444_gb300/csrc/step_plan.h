// How a run of steps is split into launches of four, two and one steps.  Host
// only, without CUDA headers.
#pragma once
#include <cstdint>
#include <vector>

namespace pemlbm {

// The four-step kernel's blocks finish kQuadCols x kQuadRows cells.
constexpr int kQuadCols = 26, kQuadRows = 10;
// Two states above this do not stay in the L2 cache (129 MB) from pass to pass.
constexpr double kStatesInL2 = 96e6;

// How many steps a launch takes in a run of steps of a lattice that may take
// several (can_pair): 4 (k_step4), 2 (k_step2) or 1.  us a step one by one, in
// pairs and in fours, replayed from a graph:
//   - fours up to three of their blocks per SM.  FP32 cathodes: 200 x 40 (32
//     blocks) 3.1, 3.5, 2.0; 640 x 160 (400) 4.7, 5.8, 4.1; 720 x 180 (504)
//     5.2, 6.4, 5.1; 1024 x 256 (1040) 7.6, 9.8, 8.5.  BF16: 640 x 160 4.4,
//     6.3, 4.2; 720 x 180 4.6, 6.8, 5.2.  Grains FP32 and BF16, 640 x 160: 4.9,
//     6.5, 4.5 and 5.2, 6.2, 4.7; closed cavities 320 x 320: 4.3, 5.7, 4.3 and
//     4.0, 5.8, 4.5.
//   - pairs where a pass over the two states is one over HBM: FP32 1300 x 320
//     (80 MB) 10.9, 12.5; 1500 x 375 (108 MB) 17.2, 15.9; 4096 x 1024 121, 83;
//     BF16 1750 x 440 (74 MB) 14.6, 17.1; 2400 x 600 (138 MB) 30.3, 29.6; 4096 x
//     1024 78, 70.  Not on narrow lattices, whose strips are mostly ends and
//     unused columns (400 MB: FP32 128 columns 63, 67; 180 columns 69, 63;
//     BF16 512 columns 41, 46; 1024 columns 41, 39), nor in 16 bits with a thick
//     catalyst, whose repeated reaction costs more than the bytes saved (4096 x
//     500, 250 rows of it: 43, 45; FP32 62, 54).
//   - one by one between them.
inline int steps_at_once(int nx, int ny, int nxp, int ny_cl, int esize) {
  const int64_t blocks = (int64_t)((nx + kQuadCols - 1) / kQuadCols) * ((ny + kQuadRows - 1) / kQuadRows);
  if (blocks <= 3 * 152) return 4;
  if (48.0 * nxp * ny * esize <= kStatesInL2) return 1;
  if (esize == 4) return nx >= 180 ? 2 : 1;
  return nx >= 1024 && 4 * ny_cl <= ny ? 2 : 1;
}

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
