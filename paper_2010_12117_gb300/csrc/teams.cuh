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
//   28 1223 -> 962  29 1407 -> 1312 30 1524 -> 1417 31 1684 -> 1436 32 1777 -> 1592
// Quads (five products and one reduction for four columns) win at order 10 and
// from 14 on, where the trailing matrix is large enough to pay for their panel.  Four
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
    {8, 4, 3, 128, true},  {8, 4, 3, 128, true},  {8, 4, 3, 128, false}, {8, 4, 2, 192, true}};  // 29 - 32

// Launches of one or a few waves take as long as one matrix does, or as the
// wave's last CTA: more lanes, fewer columns at a time, more registers per
// thread or smaller CTAs than large launches like.  Up to how many matrices is a
// matter of each order (a wave is ctas x threads / team x 152 matrices); both
// sides were timed from 30 to 140000 matrices.  Microseconds, kCond / this
// choice, at 100 matrices, just below the limit and at the next size above it
// that was timed:
//   n = 8  4.1 / 4.0, 7.9 / 7.8, 9.2 / 9.5    9  4.7 / 4.6, 5.8 / 5.8, 7.7 / 7.8
//   10  5.5 / 5.1, 13.2 / 13.2, 19.4 / 19.4   13  7.6 / 5.9, 8.2 / 7.6, 10.3 / 10.5
//   16  10.6 / 7.8, 32.1 / 28.7, 40.1 / 42.4  23  13.5 / 11.2, 22.6 / 20.6, 28.0 / 31.5
//   25  18.0 / 10.8, 18.4 / 18.0 (26.9 / 23.0 with four CTAs at 9700), 27.9 / 32.1
//   26  16.8 / 11.2, 22.8 / 19.9, 22.9 / 30.1  27  18.8 / 12.0, 23.4 / 20.6, 23.5 / 31.6
//   28  23.4 / 12.6, 24.1 / 22.6 (34.1 / 29.4 with four CTAs at 9700), 36.0 / 41.8
//   31  16.2 / 15.9, 73.7 / 68.8, 98.7 / 96.1 (119 / 121 at 30000)
//   32  20.7 / 17.6, 243 / 239, 355 / 356
// Order 19's kernel has waves of 19456 matrices and a slow full one (17.1 us at
// 19300); two lanes pass the sizes next to it in 15.8.
struct CondSmall {
  int64_t from, upto;  // matrices
  CondCfg cfg;
};
constexpr int kCondSmall = 2;  // choices per order
constexpr CondSmall cond_small(int n, int i) {
  const CondSmall none = {0, -1, kCond[n]};
  if (i == 1) return n == 25 || n == 28 ? CondSmall{7297, 9728, {8, 4, 4, 128, true}} : none;
  return n == 8               ? CondSmall{0, 65536, {1, 3, 4, 128, true}}
         : n == 9             ? CondSmall{0, 32768, {1, 2, 4, 128, true}}
         : n == 10            ? CondSmall{0, 131072, {1, 3, 4, 128, true}}
         : n == 13            ? CondSmall{0, 19456, {2, 3, 4, 128, true}}
         : n == 16            ? CondSmall{0, 65536, {2, 4, 3, 128, true}}
         : n == 19            ? CondSmall{14593, 19456, {2, 4, 3, 128, true}}
         : n == 23            ? CondSmall{0, 14592, {4, 4, 3, 128, true}}
         : n >= 25 && n <= 28 ? CondSmall{0, 7296, {8, 4, 3, 128, true}}
         : n == 31            ? CondSmall{0, 21888, {8, 4, 3, 128, true}}
         : n == 32            ? CondSmall{0, 65536, {8, 4, 3, 128, true}}
                              : none;
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
// holds a prime above PD_FOLD3_MAX: 0 kCond, 1 + i cond_small(n, i), then
// cond_wide.  Triples come before the small launches' choices, eight lanes after.
constexpr int kPickWide = 1 + kCondSmall;
constexpr bool cond_has_wide(int n) { return !cond_same(cond_wide(n), kCond[n]); }
constexpr int cond_pick(int n, int64_t matrices, bool wide) {
  if (wide && cond_has_wide(n) && cond_wide(n).step == 3) return kPickWide;
  for (int i = 0; i < kCondSmall; ++i) {
    if (wide && kCond[n].step == 3 && cond_small(n, i).cfg.step != 3) continue;  // nor redo what triples pass
    if (matrices >= cond_small(n, i).from && matrices <= cond_small(n, i).upto) return 1 + i;
  }
  return wide && cond_has_wide(n) ? kPickWide : 0;
}
constexpr CondCfg cond_cfg(int n, int pick) {
  return pick == kPickWide ? cond_wide(n) : pick ? cond_small(n, pick - 1).cfg : kCond[n];
}
// The first choice with the same kernel as `pick` (kernels are compiled once).
constexpr int cond_canonical(int n, int pick) {
  for (int i = 0; i < pick; ++i)
    if (cond_same(cond_cfg(n, i), cond_cfg(n, pick))) return i;
  return pick;
}

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
