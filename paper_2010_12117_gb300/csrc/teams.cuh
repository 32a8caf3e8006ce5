// Per-order launch tables of the condensation and fused kernels.
#pragma once

#include "../../include/polydet.h"

// The condensation kernel of order n (condense_kernel): lanes per matrix (T),
// columns its fast pass takes at a time (step_at: 2 pairs, 3 triples, 4 two
// nested pairs), the CTAs per SM it is compiled for (its __launch_bounds__
// minimum, which sets the registers per thread), threads per CTA, and where
// the pivots are folded into (numerator, denominator): by every lane as they
// come (lane_pivots) or by one thread per matrix at the end.
//
// What bounds the kernel is the integer multiply pipe and how many warps fill
// it: 12 to 20 warps per SM, each with its whole matrix in registers.  Chosen
// per order by timing every candidate on three primes of 140001 random
// matrices (and on 5329 nodes, a single wave), in microseconds, the previous
// table's choice (pairs or triples, pivots folded by every lane) first:
//   n = 8 41.4 -> 35.0   9 45.3 -> 43.2  10 57.4 -> 53.3  11 65.6  12 90.2 -> 82.0
//   13 123 -> 102   14 139 -> 123   15 164 -> 145   16 204 -> 170   17 230 -> 220
//   18 287 -> 244   19 327 -> 297   20 390 -> 338   21 450 -> 414   22 507 -> 474
//   23 573 -> 531   24 643 -> 570   25 991 -> 667   26 1062 -> 804  27 1171 -> 858
//   28 1223 -> 962  29 1407 -> 1312 30 1513 -> 1399 31 1684 -> 1436 32 1777 -> 1592
// Quads (five products and one reduction for four columns) win from order 14
// on, where the trailing matrix is large enough to pay for their panel.  Four
// lanes beat eight up to order 28: the panel is computed once per lane, and
// the registers that spill (up to 700 bytes at order 28) cost less; from 29
// on they cost more (order 29: 1454 with four lanes).  Folding the pivots at
// the end saves 5 to 9 % where a lane has registers to spare (triples, orders
// 15 and 22 to 25) and costs as much in spills where it has not (order 16:
// 204 instead of 171).
struct CondCfg {
  int team, step, ctas, threads;
  bool lane_pivots;
};
constexpr CondCfg kCond[POLYDET_MAX_N + 1] = {
    {1, 2, 1, 128, false},                                                                       // (none)
    {1, 2, 1, 128, false}, {1, 2, 1, 128, false}, {1, 2, 1, 128, false}, {1, 2, 3, 128, false},  // 1 - 4
    {1, 2, 2, 128, false}, {1, 2, 4, 128, false}, {1, 2, 4, 128, false}, {1, 3, 5, 128, false},  // 5 - 8
    {1, 3, 5, 128, false}, {1, 4, 5, 128, false}, {1, 3, 4, 128, false}, {1, 3, 4, 128, false},  // 9 - 12
    {1, 3, 3, 128, true},  {2, 4, 4, 128, true},  {2, 4, 4, 128, false}, {2, 4, 2, 256, true},   // 13 - 16
    {2, 4, 3, 128, false}, {2, 4, 3, 128, true},  {4, 4, 4, 128, false}, {4, 4, 4, 128, true},   // 17 - 20
    {4, 4, 4, 128, true},  {4, 4, 2, 256, false}, {4, 4, 4, 128, false}, {4, 4, 2, 192, false},  // 21 - 24
    {4, 4, 2, 192, false}, {4, 4, 3, 128, true},  {4, 4, 3, 128, true},  {4, 4, 2, 192, false},  // 25 - 28
    {8, 4, 3, 128, true},  {8, 4, 2, 192, true},  {8, 4, 3, 128, false}, {8, 4, 2, 192, true}};  // 29 - 32

// Launches of at most kCondFew matrices, about one wave, take as long as one
// matrix does, or as the wave's last CTA: for some orders more lanes, fewer
// columns at a time or smaller CTAs than large launches like.  In
// microseconds, the large launches' choice / this one: 100 matrices, order 16
// 10.4 / 8.9, 30 17.5 / 15.5, 8 to 10 4.1 / 3.9, 4.7 / 4.5, 5.4 / 5.1; 16 k
// matrices, order 25 43.1 / 41.0, 27 48.1 / 47.5, 28 57.2 / 51.5 (four lanes
// take nearly twice as long as eight with one matrix per warp).
constexpr int64_t kCondFew = 128 * 152;
constexpr CondCfg cond_few(int n) {
  return n == 8 || n == 10   ? CondCfg{1, 3, 4, 128, true}
         : n == 9            ? CondCfg{1, 2, 4, 128, true}
         : n == 13           ? CondCfg{2, 3, 4, 128, true}
         : n == 16           ? CondCfg{2, 2, 4, 128, true}
         : n >= 25 && n <= 28 ? CondCfg{8, 4, 4, 128, true}
         : n == 30           ? CondCfg{8, 2, 3, 128, true}
                             : kCond[n];
}

// Launches that hold a prime above PD_FOLD3_MAX, which pairs and quads can only
// redo one step at a time.  Orders whose triples come near the quads (or win in
// small launches) take triples, which any prime passes; 25 to 28, whose large
// launches have four lanes, redo with eight.  The others stay with their
// pairs or quads and redo.  30000 matrices and three such primes, microseconds, redone
// quads / this choice: order 10 28.2 / 13.5, 15 86 / 37, 17 144 / 56, 18 189 /
// 73, 19 180 / 77, 21 254 / 104, 23 439 / 128, 26 707 / 527, 28 1182 / 672.
constexpr CondCfg cond_wide(int n) {
  return n == 10              ? CondCfg{1, 3, 4, 128, true}
         : n == 15 || n == 17 ? CondCfg{2, 3, 4, 128, true}
         : n == 18 || n == 19 ? CondCfg{2, 3, 3, 128, true}
         : n == 21            ? CondCfg{4, 3, 2, 256, true}
         : n == 23            ? CondCfg{4, 3, 4, 128, true}
         : n >= 25 && n <= 28 ? CondCfg{8, 4, 4, 128, true}
                              : kCond[n];
}

constexpr bool cond_same(CondCfg a, CondCfg b) {
  return a.team == b.team && a.step == b.step && a.ctas == b.ctas && a.threads == b.threads &&
         a.lane_pivots == b.lane_pivots;
}

// The kernel of a launch of `matrices` matrices of order n, `wide` where it
// holds a prime above PD_FOLD3_MAX: 0 kCond, 1 cond_few, 2 cond_wide.
constexpr bool cond_has_wide(int n) { return !cond_same(cond_wide(n), kCond[n]); }
constexpr int cond_pick(int n, int64_t matrices, bool wide) {
  return wide && cond_has_wide(n) ? 2 : !cond_same(cond_few(n), kCond[n]) && matrices <= kCondFew ? 1 : 0;
}
constexpr CondCfg cond_cfg(int n, int pick) { return pick == 2 ? cond_wide(n) : pick == 1 ? cond_few(n) : kCond[n]; }

// A range of primes that straddles PD_FOLD3_MAX is launched in two parts where
// the lower part is long enough for its kernel's lead (5 % at order 21) to pay
// for the second launch's last wave (about half a wave): a dozen waves.
constexpr int64_t kCondSplit = 1 << 18;

// The fused kernels (fused.cuh): lanes per matrix and columns per step.  One
// lane while the whole matrix fits in registers (n <= 12), then 2, 4 and 8:
// fewer lanes would need entry slices that do not fit in shared memory.
constexpr int kTeam[POLYDET_MAX_N + 1] = {1, 1, 1, 1, 1, 1, 1, 1, 1, 1, 1, 1, 1, 2, 2, 2, 2,
                                          2, 2, 2, 4, 4, 4, 4, 4, 8, 8, 8, 8, 8, 8, 8, 8};
constexpr int kFusedStep[POLYDET_MAX_N + 1] = {2, 2, 2, 2, 2, 2, 2, 2, 3, 2, 3, 3, 3, 3, 2, 3, 2,
                                               3, 3, 3, 2, 3, 2, 3, 2, 2, 2, 2, 2, 2, 2, 2, 2};
