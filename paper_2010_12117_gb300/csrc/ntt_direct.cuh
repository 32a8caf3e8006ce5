// The arguments of one batched 1-D pass (ntt.cu) and the register-direct
// forward kernel for short inputs (Lin <= 8), kept in a header of their own
// so that launch shapes can be timed apart from the library.
#pragma once

#include "common.cuh"

struct TxArgs {
  const void *in;
  uint32_t *out;
  int64_t in_prime_stride, in_item_stride;
  int64_t out_prime_stride, out_item_stride;
  int64_t A, B;
  int Lin, Lout, N, logN;
  int Ct, logCt;
  int in_is_i32;
  int inverse;
  int prime_lo;
  const ModP *mod;
  const uint32_t *tw;
  const uint2 *tws;  // forward passes: (w^j, floor(w^j 2^32 / p)), same offsets as tw
  int tw_len, tw_off;
  const uint32_t *ninv;
  int nvars, var;
  uint32_t *status;
  // interleaved output (partial evaluation, A == 1): element (r, b) of entry
  // e goes to ((r * (B / il_L) + b / il_L) * il_n2 + e) * il_Lp + b % il_L
  int il_L, il_Lp;
  int64_t il_n2;
  // output row stride (words between rows r and r + 1 of a column); 0: B
  int64_t out_row;
  // node order of the output rows (forward passes): row k holds the value at
  // w^node_exp(k, N, olp); 0 or 1: natural order
  int olp;
  // register-direct kernel only: 0 = one grid row per item (blockIdx.y);
  // otherwise the number of items, and the grid's x axis runs over
  // (item, column, coset group) triples, so that short rows still fill whole
  // CTAs; each column's cosets are cut into flat_groups consecutive groups
  int flat_items, flat_groups;
  // forward passes: only output rows [row_lo, row_hi) are stored, as rows
  // 0 .. row_hi - row_lo of the output (row_hi = 0: all Lout rows).  The
  // register-direct kernel takes a window only in coset order, with row_lo
  // a multiple of the coset size
  int row_lo, row_hi;
  // items from zero_item_plus1 - 1 on read nothing and write zeros (the zero
  // entry of an entry map, one item past the evaluated ones); 0: none
  int zero_item_plus1;
};

// Output rows one column of a pass stores.
PD_HD int out_rows(const TxArgs &a) { return a.row_hi ? a.row_hi - a.row_lo : a.Lout; }

// Forward pass for short inputs (Lin <= 8).  The N outputs
// y_i = sum_{e<Lin} c_e w^(i e) are produced coset by coset: for
// i = j + (N/LP) t (LP = Lin rounded up to a power of two),
// y = DFT_LP(c_e w^(j e))[t] with the LP-th root psi = w^(N/LP): Lin - 1
// twiddle products and a register DFT of size LP per LP outputs, in which
// the LP - Lin inputs that are zero are folded away at compile time.  A
// thread owns CPT columns, 32 apart, so that a warp's columns are consecutive
// and every store of a row is coalesced, and loads each coset's twiddles once
// for all of them.
// With one column per thread the grid may instead run over (item, column,
// coset group) triples (TxArgs::flat_items): short rows then fill whole CTAs,
// and a pass with few columns in all spreads each column's cosets over
// several threads.
//
// The pass writes far more than it reads, and its bound is the write
// bandwidth (6.0 TB/s on rows that start on 32-byte sectors) as long as the
// instructions per word stay few and few sectors are written in parts:
//  - a warp's columns are consecutive and its CPT stores of a row follow one
//    another, because rows of an odd number of words split a sector at both
//    ends of every 128-byte store: with a thread's columns a CTA apart the
//    other part came from another warp, and a trivariate x_1 pass of 583 MB
//    (rows of 1369 words) took 127 us, now 104 us; the same with the part
//    arriving even later (146 us) is what a leaner loop alone gave;
//  - a twiddle product is Shoup's: with w' = floor(w 2^32 / p) at hand,
//    x w - umulhi(x, w') p lies in [0, 2p) for any x < 2^32, two low products
//    and a high one where a Montgomery product needs a wide, a low and a high
//    one; the operand may be an unreduced difference (23 -> 18 instructions
//    per word; aligned rows 5.3 -> 6.0 TB/s);
//  - the twiddle circle (pairs w, w') is staged in shared memory;
//  - stores go to a base pointer that is the same for the whole CTA plus a
//    running offset per output row, 32-bit wherever the output of a CTA's
//    prime (flat grid) or item fits in 4 GB (Off = uint32_t, launch_pass);
//  - the cosets whose rows are all stored take no predicate but that of a
//    thread's second to fourth column.
// Plans keep D_v <= n d_v, so with at most 8 inputs (d_v <= 7) and n <= 32 a
// circle has N <= 256 points; launch_pass sends anything longer to the
// shared-memory pass kernel.
constexpr int kDirectThreads = 256;  // at most
constexpr int kDirectTwSmem = 256;

// x w mod p in [0, p), tw = (w, floor(w 2^32 / p)), any x < 2^32.
PD_D uint32_t smul(uint32_t x, uint2 tw, uint32_t p) {
  const uint32_t r = x * tw.x - __umulhi(x, tw.y) * p;
  return min(r, r - p);
}

// x + y and x - y mod p where ZX / ZY say that x / y is known to be zero.
template <bool ZX, bool ZY>
PD_D uint32_t add_z(uint32_t x, uint32_t y, uint32_t p) {
  if (ZY) return x;
  if (ZX) return y;
  return addm(x, y, p);
}
template <bool ZX, bool ZY>
PD_D uint32_t sub_z(uint32_t x, uint32_t y, uint32_t p) {
  if (ZY) return x;
  if (ZX) return y ? p - y : 0u;
  return subm(x, y, p);
}

// DFT_4 of (x0, x1, x2, x3), xe known zero where Ze; r4 = primitive 4th root
// (Montgomery form).  y_t = sum_e x_e r4^(t e).
template <bool Z0, bool Z1, bool Z2, bool Z3>
PD_D void dft4(const uint32_t (&x)[4], uint32_t (&y)[4], uint32_t r4, uint32_t p, uint32_t pinv) {
  const uint32_t a0 = add_z<Z0, Z2>(x[0], x[2], p), a1 = sub_z<Z0, Z2>(x[0], x[2], p);
  constexpr bool ZA = Z0 && Z2, ZB = Z1 && Z3;
  const uint32_t b0 = add_z<Z1, Z3>(x[1], x[3], p);
  const uint32_t b1 = ZB ? 0u : mmul(r4, sub_z<Z1, Z3>(x[1], x[3], p), p, pinv);
  y[0] = add_z<ZA, ZB>(a0, b0, p);
  y[2] = sub_z<ZA, ZB>(a0, b0, p);
  y[1] = add_z<ZA, ZB>(a1, b1, p);
  y[3] = sub_z<ZA, ZB>(a1, b1, p);
}

// The same with a Shoup pair for the root; the product takes the difference
// x1 - x3 + p unreduced.
template <bool Z0, bool Z1, bool Z2, bool Z3>
PD_D void dft4s(const uint32_t (&x)[4], uint32_t (&y)[4], uint2 r4, uint32_t p) {
  const uint32_t a0 = add_z<Z0, Z2>(x[0], x[2], p), a1 = sub_z<Z0, Z2>(x[0], x[2], p);
  constexpr bool ZA = Z0 && Z2, ZB = Z1 && Z3;
  const uint32_t b0 = add_z<Z1, Z3>(x[1], x[3], p);
  const uint32_t b1 = ZB ? 0u : smul(Z3 ? x[1] : x[1] + p - x[3], r4, p);
  y[0] = add_z<ZA, ZB>(a0, b0, p);
  y[2] = sub_z<ZA, ZB>(a0, b0, p);
  y[1] = add_z<ZA, ZB>(a1, b1, p);
  y[3] = sub_z<ZA, ZB>(a1, b1, p);
}

template <int LIN>
struct DirectLP {
  static constexpr int value = LIN <= 1 ? 1 : LIN <= 2 ? 2 : LIN <= 4 ? 4 : 8;
};

// The roots of the register DFT: psi^1, psi^2, psi^3 of order 8 (psi^2 alone
// of order 4).
struct DirectRoots {
  uint2 psi1, psi2, psi3;
};

// The outputs y[t] of a coset with twiddles w[e] = w^(j e) for one column.
template <int LIN>
PD_D void direct_coset(const uint32_t (&c)[LIN], const uint2 (&w)[LIN], uint32_t (&y)[DirectLP<LIN>::value],
                       const DirectRoots &rt, uint32_t p) {
  constexpr int LP = DirectLP<LIN>::value;
  uint32_t z[LP];
  z[0] = c[0];
#pragma unroll
  for (int e = 1; e < LP; ++e) z[e] = (e < LIN) ? smul(c[e % LIN], w[e % LIN], p) : 0u;
  if constexpr (LP == 1) {
    y[0] = z[0];
  } else if constexpr (LP == 2) {
    y[0] = addm(z[0], z[1], p);
    y[1] = subm(z[0], z[1], p);
  } else if constexpr (LP == 4) {
    dft4s<false, false, (LIN <= 2), (LIN <= 3)>(z, y, rt.psi2, p);
  } else {
    // even and odd halves, then y_t = E_t + psi^t O_t, y_{t+4} = E_t - psi^t O_t
    const uint32_t xe[4] = {z[0], z[2], z[4], z[6]}, xo[4] = {z[1], z[3], z[5], z[7]};
    uint32_t E[4], O[4];
    dft4s<false, false, (LIN <= 4), (LIN <= 6)>(xe, E, rt.psi2, p);
    dft4s<false, (LIN <= 3), (LIN <= 5), (LIN <= 7)>(xo, O, rt.psi2, p);
    O[1] = smul(O[1], rt.psi1, p);
    O[2] = smul(O[2], rt.psi2, p);
    O[3] = smul(O[3], rt.psi3, p);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      y[t] = addm(E[t], O[t], p);
      y[t + 4] = subm(E[t], O[t], p);
    }
  }
}

// Off: the type of byte offsets into the output (see above).  FLAT (CPT == 1):
// the grid's x axis runs over the columns of all items (TxArgs::flat_items).
template <int LIN, int CPT, class Off, bool FLAT>
__global__ void __launch_bounds__(kDirectThreads) coltx_direct_kernel(TxArgs a) {
  constexpr int LP = DirectLP<LIN>::value;
  __shared__ uint2 s_tw[kDirectTwSmem];
  const int q = a.prime_lo + blockIdx.z;
  const uint2 *tw = a.tws + (size_t)q * a.tw_len + a.tw_off;
  // every twiddle index used is below N (j < N / LP and e < LP), and
  // N <= kDirectTwSmem (launch_pass); staged before any thread leaves
  for (int i = threadIdx.x; i < a.N; i += blockDim.x) s_tw[i] = __ldg(tw + i);
  __syncthreads();
  const uint32_t p = a.mod[q].p;
  const int64_t ncols = a.A * a.B;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int grp = 0;
  int64_t item = blockIdx.y;
  // the first column, the others 32 apart
  int64_t first = (int64_t)blockIdx.x * blockDim.x * CPT + warp * (32 * CPT) + lane;
  // the CTA's output: its prime's, or its item's
  char *base = reinterpret_cast<char *>(a.out + (int64_t)blockIdx.z * a.out_prime_stride);
  if (FLAT) {  // items * ncols * groups < 2^31 (launch_pass)
    const int pair = (int)first / a.flat_groups;
    grp = (int)first - pair * a.flat_groups;
    item = pair / (int)ncols;
    first = pair - item * ncols;
    if (item >= a.flat_items) return;
  } else {
    if (first >= ncols) return;
    if (!a.il_L) base += 4 * item * a.out_item_stride;
  }
  const int64_t in_base = (int64_t)blockIdx.z * a.in_prime_stride + item * a.in_item_stride;
  const bool zero_item = a.zero_item_plus1 && item >= a.zero_item_plus1 - 1;
  // bytes between output rows
  const Off ostride = (Off)(4 * (a.il_L ? (a.B / a.il_L) * a.il_n2 * a.il_Lp  // row r -> row index r * (B / L)
                                        : a.out_row ? a.out_row : a.B));
  uint32_t c[CPT][LIN];
  Off op[CPT];  // output row 0 of each column
  int nc = 0;   // columns that exist
#pragma unroll
  for (int k = 0; k < CPT; ++k) {
    const bool ok = first + 32 * k < ncols;
    nc += ok;
    const int64_t col = ok ? first + 32 * k : first;
    const int64_t aa = (a.A == 1) ? 0 : col / a.B, bb = col - aa * a.B;
#pragma unroll
    for (int e = 0; e < LIN; ++e) {
      const int64_t idx = in_base + (aa * LIN + e) * a.B + bb;
      c[k][e] = zero_item ? 0u
                          : (a.in_is_i32 ? reduce_i32(((const int32_t *)a.in)[idx], p)
                                         : ((const uint32_t *)a.in)[idx]);
    }
    if (a.il_L)
      op[k] = (Off)(4 * (((bb / a.il_L) * a.il_n2 + item) * a.il_Lp + bb % a.il_L));
    else
      op[k] = (Off)(4 * ((FLAT ? item * a.out_item_stride : 0) +
                         aa * out_rows(a) * (int64_t)(a.out_row ? a.out_row : a.B) + bb));
  }
  const bool coset_rows = a.olp > 1;
  const int N = a.N, J = N / LP;
  const int rhi = a.row_hi ? a.row_hi : a.Lout;
  const int jbeg = coset_rows ? a.row_lo / LP : 0;
  const int jend = coset_rows ? (rhi + LP - 1) / LP : J;
  // Natural order (olp <= 1): coset j holds rows j + J t, stored while
  // j < lim[t].  Coset order (olp == LP): coset j holds rows j LP + t, so
  // only the cosets of the stored rows are computed: those of
  // [row_lo, row_hi) (row_lo a multiple of LP), whose first one lands in
  // output row 0.
  const Off tstep = (Off)(coset_rows ? 1 : J) * ostride;   // a coset's row t to row t + 1
  const Off jstep = (Off)(coset_rows ? LP : 1) * ostride;  // next coset's first row
  int jlo = jbeg, jhi = jend;  // this thread's cosets
  if (FLAT && a.flat_groups > 1) {
    const int nj = jend - jbeg;
    const int per = (nj + a.flat_groups - 1) / a.flat_groups;
    jlo = jbeg + min(nj, grp * per);
    jhi = jbeg + min(nj, (jlo - jbeg) + per);
#pragma unroll
    for (int k = 0; k < CPT; ++k) op[k] += (Off)(jlo - jbeg) * jstep;
  }
  DirectRoots rt = {};
  if (LP >= 4) rt.psi2 = s_tw[N >> 2];  // w^(N/4), a primitive 4th root
  if (LP == 8) {
    rt.psi1 = s_tw[N >> 3];
    rt.psi3 = s_tw[3 * (N >> 3)];
  }
  auto twiddles = [&](int j, uint2 (&w)[LIN]) {
#pragma unroll
    for (int e = 1; e < LIN; ++e) w[e] = s_tw[j * e];
  };
  // the full cosets: column k sits 32 k words after column 0 in every row (with
  // more than one, launch_pass sees to one block of columns in the plain
  // layout); only the stores of a row's missing last columns are predicated
  int j = jlo;
  {
    const int jfull = min(jhi, coset_rows ? rhi / LP : a.Lout - J * (LP - 1));
    Off ro[LP];
#pragma unroll
    for (int t = 0; t < LP; ++t) ro[t] = op[0] + (Off)t * tstep;
    for (; j < jfull; ++j) {
      uint2 w[LIN];
      twiddles(j, w);
      uint32_t y[CPT][LP];
#pragma unroll
      for (int k = 0; k < CPT; ++k) direct_coset<LIN>(c[k], w, y[k], rt, p);
#pragma unroll
      for (int t = 0; t < LP; ++t)
#pragma unroll
        for (int k = 0; k < CPT; ++k)
          if (k == 0 || k < nc) reinterpret_cast<uint32_t *>(base + ro[t])[32 * k] = y[k][t];
#pragma unroll
      for (int t = 0; t < LP; ++t) ro[t] += jstep;
    }
#pragma unroll
    for (int k = 0; k < CPT; ++k) op[k] += (Off)(j - jlo) * jstep;
  }
  for (; j < jhi; ++j) {  // ragged cosets: a predicate per store
    uint2 w[LIN];
    twiddles(j, w);
#pragma unroll
    for (int k = 0; k < CPT; ++k) {
      if (k >= nc) break;
      uint32_t y[LP];
      direct_coset<LIN>(c[k], w, y, rt, p);
#pragma unroll
      for (int t = 0; t < LP; ++t) {
        const bool st = coset_rows ? j * LP + t < rhi : j + J * t < a.Lout;
        if (st) *reinterpret_cast<uint32_t *>(base + op[k] + (Off)t * tstep) = y[t];
      }
      op[k] += jstep;
    }
  }
}
