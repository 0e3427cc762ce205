// Internal definitions of the batched Newton-Raphson solver (Alg. 2) shared
// by its host analysis (dpf_nr_symbolic.cpp) and its CUDA part (dpf_nr.cu).
//
// The Newton system J_f dx = -f of Alg. 2 is written per bus as 2x2 blocks:
// block row i holds the (P_i, Q_i) equations, block column j the (theta_j,
// |V|_j) unknowns.  Equations and unknowns that Alg. 2 leaves out (P and Q at
// the slack, Q at pv buses; theta at the slack, |V| at pv and slack buses)
// become identity rows and columns with a zero right-hand side, so that every
// case of a batch has the same block pattern: that of Y_bus.  The blocks are
// factorised as A = L U with unit block-lower L and block-upper U, pivoting
// only inside the 2x2 diagonal blocks (inverted), in a fill-reducing order
// found on the host.
#pragma once

#include <stdint.h>

#include <vector>

#include "dpf_internal.h"

namespace dpf {

enum { NR_U = 0, NR_DIAG = 1, NR_L = 2 };

struct NrSymbolic {
  int n = 0;                       // block rows (buses)
  std::vector<int32_t> order;      // order[r] = internal bus at elimination step r
  std::vector<int32_t> rank;       // rank[i] = elimination step of internal bus i
  // filled block pattern of L + U in elimination order, CSR by rows with
  // sorted columns: row r = its L columns (< r), r itself, its U columns (> r)
  std::vector<int32_t> row_ptr, col, diag;  // diag[r]: position of (r, r)
  std::vector<int32_t> ymap;       // Y_bus CSR entry (internal order) of a position, -1 for fill
  std::vector<int32_t> level;      // elimination-tree height of every row (leaves 0)
  int n_levels = 0;
  // factorisation schedule: positions grouped by the level of their pivot
  // p = min(row, col), 8 ints per target:
  //   {pos, pair_begin, pair_end, kind, dpos, dpair_begin, dpair_end, r}
  // kind NR_U: a U position; NR_DIAG: the diagonal of row r (its inverse
  // is stored; the forward substitution of row r, over its L positions from
  // dpos = row_ptr[r] up to the diagonal, follows); NR_L: an L
  // position, which also needs the pivot's diagonal block: position dpos
  // with its own update range
  std::vector<int32_t> lvl_ptr;    // [n_levels + 1] into targets
  std::vector<int32_t> targets;    // 8 ints per target
  std::vector<int32_t> pairs;      // 2 ints per pair: L(i,k) position, U(k,j) position
  // triangular solves: rows grouped by level, 4 ints per row:
  // {r, first U position of row r, end of row r, 0}
  std::vector<int32_t> rlvl_ptr;   // [n_levels + 1]
  std::vector<int32_t> rows;       // [4 n]
};

// Minimum-degree order of Y_bus's graph, the filled pattern it produces, the
// elimination tree's levels and the update lists.  Host only; fails with
// DPF_E_UNSUPPORTED when the update lists would exceed `max_pairs`.
int nr_symbolic(const dpf_ybus* y, int64_t max_pairs, NrSymbolic* s);

// Most cases the shared-memory form of the factor takes (per_sm: its CTAs an SM
// holds).  Its time grows by waves of CTAs, each about one case's latency; the
// global form's hardly grows until it fills the GPU, the sooner the smaller the
// grid's factor.  Whole N-1 solve in us, shared-memory / global, by cases:
//   FP32   30 buses (10 an SM)  1,216 482 / 548    2,432 634 / 599
//          64 (9)      1,216 538 / 702    2,432 738 / 751
//          118 (5)     1,216 753 / 793    1,824 962 / 871    2,432 1172 / 938
//          200 (4)     1,216 1187 / 1386  1,824 1566 / 1508
//          256 (4)     1,824 1675 / 1850  2,432 2051 / 2072
//          300 (2)     912 1227 / 1281    1,216 1514 / 1341  1,824 2133 / 1604
//          450 (2)     912 2118 / 2110    1,216 2711 / 2327
//          600 (2)     1,216 2570 / 2642  1,520 3130 / 2981
//          800 (2)     1,520 5182 / 6275  1,824 6036 / 6663
//          2,000 (1)   300 2300 / 4300    850 6200 / 7500    2,379 17100 / 12800
//   FP64   one wave of a few CTAs keeps its pipe busy: 30 buses, 1 case 1.2 / 1.4
//          ms; 118, 500 1.0 / 1.3; 300, 300 2.3 / 3.7; 1,000, 120 2.9 / 5.0; but
//          30, 1,500 (10 CTAs an SM) 2.1 / 1.7 and 118, 3,000 3.5 / 2.7
inline int nr_smem_cases(int n, bool fp64, int sms, int per_sm) {
  if (fp64) return sms * (per_sm < 4 ? per_sm : 4);
  if (per_sm >= 9) return sms * per_sm * 27 / 20;
  const int waves = per_sm >= 3 ? (n < 240 ? 2 : 3) : per_sm == 1 ? 6 : n < 500 ? 3 : n < 750 ? 4 : 5;
  return sms * per_sm * waves;
}

}  // namespace dpf
