// The coupled step kernel (one cell per thread, pull scheme) and its
// launcher, templated on the population storage type S.  Kept apart from
// the read-out, batch and adjoint kernels so that its sources can be
// identified on their own.
#pragma once
#include <type_traits>

#include "lbm_core.cuh"
#include "lbm_launch.h"

namespace pemlbm {

// Own-state and pulled records of a listed cell (see RecPtrs): the values
// the reverse of its reaction and of its boundary links needs.  `cell`
// holds the post-stream values before the surface reaction.
template <typename S, typename R, int CG>
__device__ __forceinline__ void write_listed_records(const Pops<S, CG> &src, const KArgsT<R> &a,
                                                     const RecPtrs<R> &rp, uint8_t m, long long c,
                                                     int x, int y, const Cell<R> &cell) {
  const bool cat = a.mode == 1 && (m & REG_MASK) == REG_CATALYST;
  if (!(m & M_EDGE) && !cat) return;
  const long long sl = rp.slot[c];
  R th = 0, cv = 0, jx = 0, jy = 0;
  if ((a.mode == 0 && (m & M_YLO)) || cat) th = own_sum<S, R, CG>(src, 0, x, y) + a.theta0;
  if (cat) cv = own_sum<S, R, CG>(src, 1, x, y) + R(a.Cref[1]);
  if (has_vcol(a, x)) {
    R d[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) d[k] = R(src.at(k, x, y));
    jx = d[1] - d[3] + d[5] - d[6] - d[7] + d[8];
    jy = d[2] - d[4] + d[5] + d[6] - d[7] - d[8];
  }
  stq(rp.own + 4 * sl, th, cv, jx, jy);
  if (m & M_EDGE) {
    R *p = rp.pulled + 24 * sl;
#pragma unroll
    for (int i = 0; i < 9; ++i) p[i] = cell.f[i];
#pragma unroll
    for (int s = 0; s < 3; ++s)
#pragma unroll
      for (int i = 0; i < 5; ++i) p[9 + 5 * s + i] = cell.g[s][i];
  }
}

// ------------------------------------------------------------- step (K1)
// The update of cell (x, y) once its interior pulls are in `cell`: boundary
// links, reaction, collisions, store.  c is its index in the lattice, m its
// node bits; the 24 new values go to cell k of dst, a buffer whose planes
// hold P cells (I = unsigned: the lattice's planes, addressed by one uniform
// base per plane and a 32-bit byte offset).  jout, when not NULL, is where
// reacting cells leave the O2 they consume in this step, [row][nx]; write_j
// says whether this cell's caller owns it.  seed: the step counter of
// stochastic rounding.
// Shared by the single-domain step, the batched steps and the two-step
// kernel.  X: closed ends, fixed wall values and buoyancy compiled in (see
// pull_flow_edge).  REC: the step also writes its reverse records
// (RecPtrs) for the discrete adjoint.
template <typename S, int CG, bool SR, bool X, bool REC, typename I>
__device__ __forceinline__ void finish_cell(const Pops<S, CG> &src, S *__restrict__ dst, I k, I P,
                                            const uint8_t *__restrict__ mask,
                                            const uint16_t *__restrict__ mid,
                                            const MatCoef<typename Real<S>::type> *__restrict__ pal,
                                            const KArgsT<typename Real<S>::type> &a, long long c,
                                            int x, int y, uint8_t m,
                                            const MatCoef<typename Real<S>::type> &mc,
                                            Cell<typename Real<S>::type> &cell,
                                            typename Real<S>::type *__restrict__ jout,
                                            bool write_j, unsigned seed,
                                            const RecPtrs<typename Real<S>::type> &rp) {
  using R = typename Real<S>::type;
  // solid cells run the same arithmetic on their (unused) values and only
  // skip the stores, so no branch stands between the mask and the loads
  const bool live = (m & REG_MASK) != REG_SOLID;
  auto edges = [&] {
    // next to grains but away from the lattice's edges: bounce-back only
    if ((m & M_EDGE) == M_NEAR_SOLID)
      bounce_solid<S, R, CG>(src, x, y, ld_mask(mask, a.plane + c, a, 23), cell);
    else fix_edges<S, R, CG, X>(src, a, mask, mid, pal, mc, x, y, m, cell);
  };
  R S_vol = 0;
  auto reaction = [&] {
    if (a.mode == 0 && (m & M_YLO)) {
      const R J = surface_reaction<S, R, CG>(src, a, mc, x, cell);
      if (jout && write_j && live) jout[(long long)y * a.nx + x] = J;
    }
    if (a.mode == 1 && (m & REG_MASK) == REG_CATALYST) {
      S_vol = volume_sink<S, R, CG>(src, a, x, y);
      if (jout && write_j) jout[(long long)y * a.nx + x] = -S_vol;
    }
  };
  if constexpr (REC) {
    if (m & M_EDGE) edges();
    if (live) write_listed_records<S, R, CG>(src, a, rp, m, c, x, y, cell);
    reaction();
  } else if ((m & M_EDGE) || (m & REG_MASK) == REG_CATALYST) {
    // one branch for everything an interior cell of a layer without reaction
    // skips (a surface reaction is on the bottom edge)
    if (m & M_EDGE) edges();
    reaction();
  }
  const Macro<R> u = macros<R, X>(a, mc, cell);
  if constexpr (REC) {
    if (live) {
      R *r = rp.cell + 8 * c;
      stq(r, u.vx, u.vy, u.C[0], u.C[1]);
      stq(r + 4, u.C[2], cell.g[1][1] - cell.g[1][3], cell.g[1][2] - cell.g[1][4], R(0));
    }
  }
  R o[9];
  collide_flow<R, X>(a, mc, u, cell.f, o);
  // 16-bit storage with stochastic rounding: a random stream per cell and
  // step (hash of the cell and the device step counter), twelve 32-bit
  // xorshift draws; population q (0-8 flow, 9 + 5 s + i scalar s) takes half
  // q & 1 of draw q >> 1.  Each draw's two halves thus round populations of
  // one lattice (the pair f_8, T_0 aside): giving both halves of a draw to
  // f_i and T_i of the same link correlated the rounding of u and of T, and
  // the mean of their product then biased the advected heat (at 50 k steps
  // on the 8192 x 2048 grain cathode the BF16 current was off by 271%
  // against 2% with this assignment).
  unsigned rnd[12] = {};
  if constexpr (SR) {
    unsigned rs = hash32((unsigned)c * 0x9e3779b9u ^ hash32(seed + 0x632be5abu)) | 1u;
#pragma unroll
    for (int j = 0; j < 12; ++j) rnd[j] = xorshift32(rs);
  }
  auto r16 = [&](int q) { return (q & 1) ? rnd[q >> 1] >> 16 : rnd[q >> 1] & 0xffffu; };
  // (the bounds-checked build skips a store outside the 24 planes)
  auto st_ok = [&](long long i, int width) {
    const long long n = 24 * (long long)(std::is_same<I, unsigned>::value ? a.plane : P);
    return in_bounds(i, n, 24) && in_bounds(i + width - 1, n, 24);
  };
  // where population q (a group's first, or a diagonal link) of cell k goes
  auto at = [&](int q) {
    if constexpr (std::is_same<I, unsigned>::value) {
      const int n = q < 5 ? 4 : 1;
      return reinterpret_cast<S *>(reinterpret_cast<char *>(dst) +
                                   (q < 5 ? 4 * q : 15 + q) * a.plane * (long long)sizeof(S) +
                                   k * (unsigned)(n * sizeof(S)));
    } else {
      return dst + (I)pop_index(q, k, P);
    }
  };
  if (live) {   // the diagonal flow links
    if constexpr (SR) {
#pragma unroll
      for (int i = 5; i < 9; ++i)
        if (st_ok(pop_index(i, k, std::is_same<I, unsigned>::value ? a.plane : (long long)P), 1)) st_sr(at(i), o[i], r16(i));
    } else {
#pragma unroll
      for (int i = 5; i < 9; ++i)
        if (st_ok(pop_index(i, k, std::is_same<I, unsigned>::value ? a.plane : (long long)P), 1)) st_r(at(i), o[i]);
    }
  }
  const R srcv[3] = {-S_vol * R(a.hpo) * mc.inv_sigma, S_vol, R(-2) * S_vol};
  R g[3][5];
#pragma unroll
  for (int s = 0; s < 3; ++s)
    collide_scalar<R>(a, mc, s, u.ux, u.uy, u.C[s], cell.g[s], srcv[s], g[s], S_vol != R(0));
  if (live) {   // links 0-4 of the flow and the three scalars, one group each
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      if (!st_ok(pop_index(i, k, std::is_same<I, unsigned>::value ? a.plane : (long long)P), 4)) continue;
      if constexpr (SR) {
        stq_sr(at(i), o[i], g[0][i], g[1][i], g[2][i], r16(i), r16(9 + i),
               r16(14 + i), r16(19 + i));
      } else {
        stq(at(i), o[i], g[0][i], g[1][i], g[2][i]);
      }
    }
  }
}

// One coupled update of cell (x, y) of a global buffer: src -> dst.
template <typename S, int CG = kLdg, bool SR = false, bool X = false, bool REC = false>
__device__ __forceinline__ void cell_update(const S *__restrict__ src_p, S *__restrict__ dst,
                                            const uint8_t *__restrict__ mask,
                                            const uint16_t *__restrict__ mid,
                                            const MatCoef<typename Real<S>::type> *__restrict__ pal,
                                            const KArgsT<typename Real<S>::type> &a, int x, int y,
                                            typename Real<S>::type *__restrict__ jout = nullptr,
                                            const RecPtrs<typename Real<S>::type> &rp = {}) {
  using R = typename Real<S>::type;
  const long long c = (long long)y * a.nxp + x;
  const Pops<S, CG> src{src_p, a.plane, a.nxp};
  const uint8_t m = ld_mask(mask, c, a, 20);
  Cell<R> cell;
  load_interior<S, R, CG>(src, a, x, y, cell);
  const MatCoef<R> mc = pal[ld_mid(mid, c, a, 21)];
  unsigned seed = 0;
  if constexpr (SR) seed = __ldg(a.seed_ctr) + a.seed_off;
  finish_cell<S, CG, SR, X, REC, long long>(src, dst, c, a.plane, mask, mid, pal, a, c, x, y, m, mc,
                                            cell, jout, true, seed, rp);
}

// The cell of a thread in blocks of BX x BY cells.  FP64: the first blocks
// walk up the two end columns and the others cover the columns between.  An
// FP64 instruction costs the same with one active lane as with 32, and the
// boundary links of the ends (inlet parabola, the outlet's virtual column)
// are almost as many as a cell's own: in row blocks every row paid for them
// twice, now each 32 rows do.  (509 x 127: 44.4 -> 40 us a step, 1024 x
// 256: 140 -> 136; 250 x 64, bound by a warp's latency, 16.2 both ways.)
template <typename S, int BX, int BY>
__device__ __forceinline__ bool cell_of_thread(int nx, int ny, int &x, int &y) {
  if constexpr (sizeof(S) == 8) {
    constexpr int T = BX * BY;
    const int per_end = (ny + T - 1) / T;
    int b = blockIdx.x;
    if (b < 2 * per_end) {
      x = b < per_end ? 0 : nx - 1;
      y = (b < per_end ? b : b - per_end) * T + threadIdx.x;
      return y < ny;
    }
    b -= 2 * per_end;
    const int across = (nx - 2 + BX - 1) / BX;
    x = 1 + b % across * BX + threadIdx.x % BX;
    y = b / across * BY + threadIdx.x / BX;
    return x < nx - 1 && y < ny;
  } else {
    x = blockIdx.x * BX + threadIdx.x % BX;
    y = blockIdx.y * BY + threadIdx.x / BX;
    return x < nx && y < ny;
  }
}
inline dim3 ends_first_grid(int nx, int ny, StepShape sh) {
  const int T = sh.bx * sh.by;
  return dim3(2 * ((ny + T - 1) / T) + (nx - 2 + sh.bx - 1) / sh.bx * ((ny + sh.by - 1) / sh.by));
}

// SR: 16-bit stores with stochastic rounding (a separate instantiation, so
// the round-to-nearest kernel carries none of its code); X as cell_update.
template <typename S, int BX, int BY, int MINB, bool SR = false, bool X = false>
__global__ void __launch_bounds__(BX * BY, MINB)
k_step(const S *__restrict__ src_p, S *__restrict__ dst, const uint8_t *__restrict__ mask,
       const uint16_t *__restrict__ mid, const MatCoef<typename Real<S>::type> *__restrict__ pal,
       KArgsT<typename Real<S>::type> a, typename Real<S>::type *__restrict__ jout) {
  int x, y;
  if (!cell_of_thread<S, BX, BY>(a.nx, a.ny, x, y)) return;
  cell_update<S, kLdg, SR, X>(src_p, dst, mask, mid, pal, a, x, y, jout);
}

// -------------------------------------------------------- two steps (K1b)
// Two coupled steps in one pass over memory: src -> (row ring) -> dst.  A
// warp owns a strip of kStripCols columns and walks up the rows [ya, yb): a
// round takes the first step of one row, of kRingCols columns (one more on
// either side), into the ring, and the second step of the row below from
// the ring to dst.  The two steps of a cell are exactly two single steps.
//
// A single step of this lattice is bound by HBM (FP32, 0.95 of the measured
// copy rate at 4096 x 1024) or by latency and issue (16 bits); a pair moves
// the same bytes for two steps and is bound by issue and by what is left of
// the memory latency (FP32: 64% of issue slots, 2.0 of 5.5 warp cycles per
// issue wait for loads, 848 MB of DRAM a pass at 5.1 TB/s; BF16: 78% of issue
// slots).  One warp alone owns its ring, so no block barrier
// ties warps in different phases together (with blocks of 128 x 2 cells and
// __syncthreads: 184 us a step).  The next row's pulls are copied into the
// stage while both steps of this round run, and a column's material stays in
// registers.  Per step, two at a time against single steps: 4096 x 1024 FP32 83
// against 121 us, BF16 70 against 78; 1000 x 1000 cavity, FP32, 26 against 32
// (steps_at_once: where they pay).
template <typename S, bool X>
__device__ __forceinline__ void two_steps(const S *__restrict__ src_p, S *__restrict__ dst,
                                          const uint8_t *__restrict__ mask,
                                          const uint16_t *__restrict__ mid,
                                          const MatCoef<typename Real<S>::type> *__restrict__ pal,
                                          const KArgsT<typename Real<S>::type> &a, int strip,
                                          int ya, int yb, typename Real<S>::type *__restrict__ jout,
                                          long long jstep, S *__restrict__ ring,
                                          unsigned char *__restrict__ stage) {
  using R = typename Real<S>::type;
  const int lane = threadIdx.x & 31;
  const int x0 = strip * kStripCols - 1, x = x0 + lane;
  const bool in_x = x >= 0 && x < a.nx;
  const bool own_x = in_x && lane >= 1 && lane <= kStripCols;
  const Pops<S, kLdg> src{src_p, a.plane, a.nxp};
  const Pops<S, kRing> between{ring, x0};
  R *const jout2 = jout ? jout + jstep : nullptr;
  const int y_top = yb < a.ny ? yb : a.ny - 1;   // the last row the second step pulls from
  // this lane's cell in ring row y1 (row y1 - 1 follows two ring rows on,
  // row y1 - 2 one), and its node bits and palette index in the rows y1 - 1
  // and y1
  int hi = between.row(ya - 1) + lane;
  unsigned m_lo = REG_SOLID, m_hi = REG_SOLID, e_lo = 0, e_hi = 0;
  unsigned c1 = (unsigned)(ya - 1) * (unsigned)a.nxp + (unsigned)x;   // cell (x, y1)
  // the lines of a coming row that this lane prefetches into the L2 cache:
  // five 128-byte lines of each group plane, one of each diagonal, palette
  // indices and node bits
  const long long pf_cell = (long long)(ya - 1 + a.pair_ahead) * a.nxp + (x0 > 0 ? x0 : 0);
  const char *pf;
  int pf_row;
  if (lane < 25) {
    pf = (const char *)(src_p + 4 * ((lane / 5) * a.plane + pf_cell)) + 128 * (lane % 5);
    pf_row = a.nxp * 4 * (int)sizeof(S);
  } else if (lane < 29) {
    pf = (const char *)(src_p + (lane - 5) * a.plane + pf_cell);
    pf_row = a.nxp * (int)sizeof(S);
  } else if (lane == 29) {
    pf = (const char *)(mid + pf_cell);
    pf_row = 2 * a.nxp;
  } else {
    pf = (const char *)(mask + pf_cell);
    pf_row = a.nxp;
  }
  const int pf_top = a.pair_ahead ? y_top - a.pair_ahead : -2;   // last row y1 that prefetches
  S diag[4] = {};
  int asked = 0;   // rows asked for and not taken (only the bounds-checked build looks at it)
  if (in_x) {
    const unsigned c = ya > 0 ? c1 : c1 + a.nxp;   // the first row taken
    request_interior(src, a, c, lane, stage, diag);
    asked = 1;
    m_hi = ld_mask(mask, c, a, 20);
    e_hi = ld_mid(mid, c, a, 21);
  }
  // the material of a column changes rarely from row to row: its
  // coefficients stay in registers until the palette index differs
  MatCoef<R> mc{};
  unsigned e_mc = ~0u;
  auto material = [&](unsigned e) {
    if (e != e_mc) {
      mc = pal[e];
      e_mc = e;
    }
  };
  for (int y1 = ya - 1; y1 <= yb; ++y1, c1 += a.nxp) {
    unsigned m_next = REG_SOLID, e_next = 0;
    if (y1 <= pf_top) asm volatile("prefetch.global.L2 [%0];" ::"l"(pf));
    pf += pf_row;
    const bool first = in_x && y1 >= 0 && y1 <= y_top;
    if (first) {   // first step of row y1
      Cell<R> cell;
      in_bounds(asked - 1, 1, 7);   // the row to take was asked for, once
      asked -= 1;
      take_interior<S, R>(lane, stage, diag, cell);
      material(e_hi);
      // the next row is on its way during both steps; none is asked for past
      // the last, so that every copy into the stage has been waited for when
      // the warp leaves its shared memory to another block
      if (y1 < y_top) {
        const unsigned c2 = c1 + a.nxp;
        request_interior(src, a, c2, lane, stage, diag);
        asked += 1;
        m_next = ld_mask(mask, c2, a, 20);
        e_next = ld_mid(mid, c2, a, 21);
      }
      finish_cell<S, kLdg, false, X, false, int>(
          src, ring, hi, kRingCells, mask, mid, pal, a, c1, x, y1, (uint8_t)m_hi, mc, cell, jout,
          own_x && y1 >= ya && y1 < yb, 0u, RecPtrs<R>{});
    }
    __syncwarp();
    const int y = y1 - 1;
    if (own_x && y >= ya) {   // second step of row y (y < yb)
      const unsigned c = c1 - a.nxp;
      const int lo = hi >= 2 * kRingCols ? hi - 2 * kRingCols : hi + kRingCols;
      const int c0 = hi >= kRingCols ? hi - kRingCols : hi + 2 * kRingCols;
      Cell<R> cell;
      load_shared(between, lo, c0, hi, cell);
      material(e_lo);
      finish_cell<S, kRing, false, X, false, unsigned>(
          between, dst, c, 0u, mask, mid, pal, a, c, x, y, (uint8_t)m_lo, mc, cell, jout2, true,
          0u, RecPtrs<R>{});
    }
    __syncwarp();   // the next first step overwrites ring row y1 - 2
    hi = hi >= 2 * kRingCols ? hi - 2 * kRingCols : hi + kRingCols;
    if (first) {
      m_lo = m_hi;
      e_lo = e_hi;
      m_hi = m_next;
      e_hi = e_next;
    }
  }
  in_bounds(asked, 1, 7);   // no copy may still be on its way
}

// Unit u of a lattice's strips x row chunks, one per warp.
template <typename S, bool X>
__device__ __forceinline__ void two_steps_unit(const S *src_p, S *dst, const uint8_t *mask,
                                               const uint16_t *mid,
                                               const MatCoef<typename Real<S>::type> *pal,
                                               const KArgsT<typename Real<S>::type> &a, int u,
                                               typename Real<S>::type *jout, long long jstep) {
  extern __shared__ __align__(16) unsigned char pair_smem[];
  const int w = threadIdx.x >> 5, strips = (a.nx + kStripCols - 1) / kStripCols;
  S *ring = reinterpret_cast<S *>(pair_smem) + w * (24 * kRingCells);
  unsigned char *stage = pair_smem + kPairWarps * (24 * kRingCells * (int)sizeof(S)) + w * Stage<S>::kBytes;
  // chunks of equal weight: a catalyst row counts two rows
  const int chunks = (a.ny + a.ny_cl + a.pair_rows - 1) / a.pair_rows;
  if (u >= strips * chunks) return;   // (whole warps leave)
  // the slow units first: the end columns, then the bottom chunk upwards
  int strip, chunk;
  if (strips > 2) {
    const int ends = 2 * chunks, v = u - ends, inner = strips - 2;
    chunk = u < ends ? u >> 1 : v / inner;
    strip = u < ends ? (u & 1) * (strips - 1) : 1 + (v - chunk * inner);
  } else {
    chunk = u / strips;
    strip = u - chunk * strips;
  }
  auto row_at = [&](int w) { return w < 2 * a.ny_cl ? (w + 1) >> 1 : min(w - a.ny_cl, a.ny); };
  const int ya = row_at(chunk * a.pair_rows), yb = row_at((chunk + 1) * a.pair_rows);
  if (ya >= yb) return;
  two_steps<S, X>(src_p, dst, mask, mid, pal, a, strip, ya, yb, jout, jstep, ring, stage);
}

template <typename S, bool X>
__global__ void __launch_bounds__(32 * kPairWarps, pair_blocks_per_sm(sizeof(S)))
k_step2(const S *__restrict__ src_p, S *__restrict__ dst, const uint8_t *__restrict__ mask,
        const uint16_t *__restrict__ mid, const MatCoef<typename Real<S>::type> *__restrict__ pal,
        KArgsT<typename Real<S>::type> a, typename Real<S>::type *__restrict__ jout,
        long long jstep) {
  two_steps_unit<S, X>(src_p, dst, mask, mid, pal, a, blockIdx.x * kPairWarps + (threadIdx.x >> 5),
                           jout, jstep);
}

// ------------------------------------------------------- four steps (K1c)
// Four steps of a small lattice: each warp takes one row of 32 columns through
// four steps in shared memory, and every step gives up a column and a row on
// each side, so a block finishes kQuadCols x kQuadRows cells (62% of its
// work).  Small lattices are bound by the latency of a cell's dependent
// instructions (about 1.6 us) and of a launch; here four steps pay for one
// launch, one load from the L2 cache and four times that latency, where
// k_step2's warps walk four rows in turn for two steps.  200 x 40, FP32: 2.0
// us a step against 3.5 in pairs and 3.1 one by one (steps_at_once: where the
// repeated work outweighs it).
template <typename S, bool X>
__global__ void __launch_bounds__(32 * kTileWarps, 1)
k_step4(const S *__restrict__ src_p, S *__restrict__ dst, const uint8_t *__restrict__ mask,
        const uint16_t *__restrict__ mid, const MatCoef<typename Real<S>::type> *__restrict__ pal,
        KArgsT<typename Real<S>::type> a, typename Real<S>::type *__restrict__ jout,
        long long jstep) {
  using R = typename Real<S>::type;
  extern __shared__ __align__(16) unsigned char quad_smem[];
  S *const buf = reinterpret_cast<S *>(quad_smem);   // two tiles
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int x_lo = blockIdx.x * kQuadCols - 3, y_lo = blockIdx.y * kQuadRows - 3;
  const int x = x_lo + lane, y = y_lo + w, k = w * 32 + lane;
  const bool in = x >= 0 && x < a.nx && y >= 0 && y < a.ny;
  const bool own = in && lane >= 3 && lane < 3 + kQuadCols && w >= 3 && w < 3 + kQuadRows;
  const unsigned c = (unsigned)y * (unsigned)a.nxp + (unsigned)x;
  uint8_t m = REG_SOLID;
  MatCoef<R> mc{};
  Cell<R> cell;
  if (in) {
    const Pops<S, kLdg> src{src_p, a.plane, a.nxp};
    m = ld_mask(mask, c, a, 20);
    load_interior<S, R, kLdg>(src, a, x, y, cell);
    mc = pal[ld_mid(mid, c, a, 21)];
    finish_cell<S, kLdg, false, X, false, int>(src, buf, k, kTileCells, mask, mid, pal, a, c, x, y, m, mc,
                                               cell, jout, own, 0u, RecPtrs<R>{});
  }
  for (int t = 1; t < 3; ++t) {
    __syncthreads();
    const Pops<S, kTile> tile{buf + (t == 1 ? 0 : 24 * kTileCells), x_lo, y_lo};
    if (in && lane >= t && lane < 32 - t && w >= t && w < kTileWarps - t) {
      load_shared(tile, k - 32, k, k + 32, cell);
      finish_cell<S, kTile, false, X, false, int>(
          tile, buf + (t == 1 ? 24 * kTileCells : 0), k, kTileCells, mask, mid, pal, a, c, x, y, m, mc, cell,
          jout ? jout + t * jstep : nullptr, own, 0u, RecPtrs<R>{});
    }
  }
  __syncthreads();
  if (own) {
    const Pops<S, kTile> tile{buf, x_lo, y_lo};
    load_shared(tile, k - 32, k, k + 32, cell);
    finish_cell<S, kTile, false, X, false, unsigned>(tile, dst, c, 0u, mask, mid, pal, a, c, x, y, m, mc, cell,
                                                     jout ? jout + 3 * jstep : nullptr, true, 0u,
                                                     RecPtrs<R>{});
  }
}

// The step with its reverse records (plain cathode set-ups, round-to-
// nearest storage: what the adjoint covers).
template <typename S, int BX, int BY, int MINB>
__global__ void __launch_bounds__(BX * BY, MINB)
k_step_rec(const S *__restrict__ src_p, S *__restrict__ dst, const uint8_t *__restrict__ mask,
           const uint16_t *__restrict__ mid, const MatCoef<typename Real<S>::type> *__restrict__ pal,
           KArgsT<typename Real<S>::type> a, RecPtrs<typename Real<S>::type> rp) {
  const int x = blockIdx.x * BX + (threadIdx.x % BX);
  const int y = blockIdx.y * BY + (threadIdx.x / BX);
  if (x >= a.nx || y >= a.ny) return;
  cell_update<S, kLdg, false, false, true>(src_p, dst, mask, mid, pal, a, x, y, nullptr, rp);
}

// ------------------------------------------------------ launcher
template <typename S, int V>
void launch_step_v(const void *src, void *dst, const DevGeom &g, const KArgs &a, void *jout, cudaStream_t st) {
  constexpr StepShape sh = step_shape(sizeof(S), V);
  dim3 grid((a.nx + sh.bx - 1) / sh.bx, (a.ny + sh.by - 1) / sh.by);
  if (sizeof(S) == 8) grid = ends_first_grid(a.nx, a.ny, sh);
  using R = typename Real<S>::type;
  if (needs_extended(a)) {
    // two shapes of the extended step: 128 x 2 at 80 registers (variants
    // 0-2) and 64 x 2 at 64 registers (the rest); the tuner picks one (FP64:
    // 64 x 1 and 256 x 1)
    constexpr StepShape sx = step_shape(sizeof(S), V <= 2 ? 1 : 7);
    dim3 gx((a.nx + sx.bx - 1) / sx.bx, (a.ny + sx.by - 1) / sx.by);
    if (sizeof(S) == 8) gx = ends_first_grid(a.nx, a.ny, sx);
    k_step<S, sx.bx, sx.by, sx.minb, false, true><<<gx, sx.bx * sx.by, 0, st>>>(
        (const S *)src, (S *)dst, g.mask, g.mid, (const MatCoef<R> *)g.pal, narrow_args<R>(a), (R *)jout);
    return;
  }
  if constexpr (sizeof(S) == 2) {
    if (a.stochastic) {
      k_step<S, sh.bx, sh.by, sh.minb, true><<<grid, sh.bx * sh.by, 0, st>>>(
          (const S *)src, (S *)dst, g.mask, g.mid, (const MatCoef<R> *)g.pal, narrow_args<R>(a), (R *)jout);
      return;
    }
  }
  k_step<S, sh.bx, sh.by, sh.minb><<<grid, sh.bx * sh.by, 0, st>>>(
      (const S *)src, (S *)dst, g.mask, g.mid, (const MatCoef<R> *)g.pal, narrow_args<R>(a), (R *)jout);
}

// (FP64: see kStepShapes64)
template <typename S> constexpr StepShape kRecShape = sizeof(S) == 8 ? StepShape{32, 1, 1} : StepShape{64, 2, 6};
template <typename S>
void launch_step_rec(const void *src, void *dst, const DevGeom &g, const KArgs &a,
                     const RecBufs &r, cudaStream_t st) {
  using R = typename Real<S>::type;
  constexpr StepShape sh = kRecShape<S>;
  dim3 grid((a.nx + sh.bx - 1) / sh.bx, (a.ny + sh.by - 1) / sh.by);
  const RecPtrs<R> rp{(R *)r.cell, (R *)r.own, (R *)r.pulled, r.slot};
  k_step_rec<S, sh.bx, sh.by, sh.minb><<<grid, sh.bx * sh.by, 0, st>>>(
      (const S *)src, (S *)dst, g.mask, g.mid, (const MatCoef<R> *)g.pal, narrow_args<R>(a), rp);
}

template <typename S>
void launch_step(const void *src, void *dst, const DevGeom &g, const KArgs &a, int variant,
                 void *jout, cudaStream_t st) {
  switch (variant) {
    case 1: launch_step_v<S, 1>(src, dst, g, a, jout, st); break;
    case 2: launch_step_v<S, 2>(src, dst, g, a, jout, st); break;
    case 3: launch_step_v<S, 3>(src, dst, g, a, jout, st); break;
    case 4: launch_step_v<S, 4>(src, dst, g, a, jout, st); break;
    case 5: launch_step_v<S, 5>(src, dst, g, a, jout, st); break;
    case 6: launch_step_v<S, 6>(src, dst, g, a, jout, st); break;
    case 7: launch_step_v<S, 7>(src, dst, g, a, jout, st); break;
    default: launch_step_v<S, 0>(src, dst, g, a, jout, st); break;
  }
}

// Two steps, one warp per strip and row chunk.
template <typename S>
void launch_step2(const void *src, void *dst, const DevGeom &g, const KArgs &a, void *jout,
                  long long jstep, cudaStream_t st) {
  if constexpr (sizeof(S) < 8) {
    using R = typename Real<S>::type;
    auto kern = needs_extended(a) ? k_step2<S, true> : k_step2<S, false>;
    kern<<<pair_blocks(a.nx, a.ny, a.ny_cl, a.pair_rows), 32 * kPairWarps, pair_smem_bytes(sizeof(S)), st>>>(
        (const S *)src, (S *)dst, g.mask, g.mid, (const MatCoef<R> *)g.pal, narrow_args<R>(a), (R *)jout,
        jstep);
  }
}
template <typename S>
void launch_step4(const void *src, void *dst, const DevGeom &g, const KArgs &a, void *jout,
                  long long jstep, cudaStream_t st) {
  if constexpr (sizeof(S) < 8) {
    using R = typename Real<S>::type;
    const dim3 grid((a.nx + kQuadCols - 1) / kQuadCols, (a.ny + kQuadRows - 1) / kQuadRows);
    auto kern = needs_extended(a) ? k_step4<S, true> : k_step4<S, false>;
    kern<<<grid, 32 * kTileWarps, quad_smem_bytes(sizeof(S)), st>>>(
        (const S *)src, (S *)dst, g.mask, g.mid, (const MatCoef<R> *)g.pal, narrow_args<R>(a), (R *)jout,
        jstep);
  }
}

}  // namespace pemlbm
