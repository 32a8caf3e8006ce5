// Evaluation (Sec. 3.1, Algorithm 2) and interpolation (Sec. 3.3) as passes of
// one batched 1-D NTT kernel, one pass per variable.
//
// A pass views every batch item (one matrix entry, or one prime's determinant
// values) as a tensor [A][L][B] and transforms the middle axis: column (a, b)
// of Lin input values becomes Lout output values of the N-point NTT (zero
// padded when Lin < N, truncated when Lout < N).  Evaluating x_k first and
// x_1 last grows the tensor from [L_1..L_k] to [N_1..N_k] = G while every
// pass reads and writes whole 128-byte rows; this replaces the paper's
// transposition kernel and rotation of d (Algorithm 2).
//
// A CTA owns Ct columns: it stages their Lin x Ct tile in shared memory in
// bit-reversed row order, runs the log2(N) radix-2 stages there (decimation
// in time; the output is in natural order) and writes Lout x Ct back.  Data
// are plain residues; twiddles are stored in Montgomery form so one REDC per
// butterfly gives a plain product.
#include <stdio.h>

#include <type_traits>

#include "common.cuh"
#include "ntt_direct.cuh"

__global__ void __launch_bounds__(256) coltx_kernel(TxArgs a) {
  extern __shared__ uint32_t sm[];
  const int q = a.prime_lo + blockIdx.z;
  const ModP md = a.mod[q];
  const int Ct = a.Ct, S = a.Ct + 1;  // padded row stride
  const int N = a.N;
  const int64_t ncols = a.A * a.B;
  const int64_t col0 = (int64_t)blockIdx.x * Ct;
  const int64_t in_base = (int64_t)blockIdx.z * a.in_prime_stride + (int64_t)blockIdx.y * a.in_item_stride;
  const int64_t out_base = (int64_t)blockIdx.z * a.out_prime_stride + (int64_t)blockIdx.y * a.out_item_stride;
  const bool rowmajor = (a.B == 1);  // columns are contiguous rows of the item
  const int tot = Ct * N;

  for (int f = threadIdx.x; f < tot; f += blockDim.x) {
    int r, c;
    if (rowmajor) {
      c = f >> a.logN;
      r = f & (N - 1);
    } else {
      r = f >> a.logCt;
      c = f & (Ct - 1);
    }
    const int64_t col = col0 + c;
    uint32_t v = 0;
    const bool zero_item = a.zero_item_plus1 && (int)blockIdx.y >= a.zero_item_plus1 - 1;
    if (r < a.Lin && col < ncols && !zero_item) {
      const int64_t aa = col / a.B, bb = col - aa * a.B;
      const int64_t idx = in_base + (aa * a.Lin + r) * a.B + bb;
      v = a.in_is_i32 ? reduce_i32(((const int32_t *)a.in)[idx], md.p) : ((const uint32_t *)a.in)[idx];
    }
    const int rr = a.logN ? (int)(__brev((unsigned)r) >> (32 - a.logN)) : 0;
    sm[rr * S + c] = v;
  }
  __syncthreads();

  const uint32_t *tw = a.tw + (size_t)q * a.tw_len + a.tw_off;
  for (int s = 0; s < a.logN; ++s) {
    const int h = 1 << s;
    const int step = N >> (s + 1);
    for (int j = threadIdx.x; j < (N >> 1) * Ct; j += blockDim.x) {
      const int c = j & (Ct - 1);
      const int bj = j >> a.logCt;
      const int pos = bj & (h - 1);
      const int i0 = ((bj >> s) << (s + 1)) + pos;
      const int i1 = i0 + h;
      const uint32_t w = __ldg(tw + pos * step);
      const uint32_t u = sm[i0 * S + c];
      const uint32_t t = mmul(w, sm[i1 * S + c], md.p, md.pinv);
      sm[i0 * S + c] = addm(u, t, md.p);
      sm[i1 * S + c] = subm(u, t, md.p);
    }
    __syncthreads();
  }

  const uint32_t scale = a.inverse ? a.ninv[q * a.nvars + a.var] : 0u;
  bool bad = false;
  for (int f = threadIdx.x; f < tot; f += blockDim.x) {
    int r, c;
    if (rowmajor) {
      c = f >> a.logN;
      r = f & (N - 1);
    } else {
      r = f >> a.logCt;
      c = f & (Ct - 1);
    }
    const int64_t col = col0 + c;
    if (col >= ncols) continue;
    uint32_t v = sm[r * S + c];
    // natural output index r -> its row in the node order (r = j + (N/L) t
    // is node j L + t)
    const int L = a.olp > 1 ? a.olp : 1;
    const int J = N / L;
    const int rk = (r % J) * L + r / J;
    const int rlo = a.row_lo, rhi = a.row_hi ? a.row_hi : a.Lout;
    if (rk >= rlo && rk < rhi) {
      if (a.inverse) v = mmul(scale, v, md.p, md.pinv);
      const int64_t aa = col / a.B, bb = col - aa * a.B;
      if (a.il_L) {
        const int64_t row = (int64_t)rk * (a.B / a.il_L) + bb / a.il_L;
        a.out[(int64_t)blockIdx.z * a.out_prime_stride + (row * a.il_n2 + blockIdx.y) * a.il_Lp +
              bb % a.il_L] = v;
      } else {
        const int64_t orow = a.out_row ? a.out_row : a.B;
        a.out[out_base + (aa * (rhi - rlo) + rk - rlo) * orow + bb] = v;
      }
    } else if (a.inverse && rk >= a.Lout && v != 0u) {
      bad = true;
    }
  }
  if (bad) atomicOr(a.status, POLYDET_STATUS_BOUND);
}

static int ilog2(int64_t x) {
  int l = 0;
  while (((int64_t)1 << l) < x) ++l;
  return l;
}

// How a pass is split over threads: columns per thread, threads per CTA, a
// flattened grid (TxArgs::flat_items), and the CTAs an SM may hold (0: any).
struct DirectShape {
  int cpt, threads;
  bool flat;
  int ctas;
};

// The dynamic shared memory that keeps a CTA's SM to `ctas` of them.
static size_t direct_reserve_bytes(int ctas) {
  if (ctas <= 0) return 0;
  int per_sm = 0, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  // static twiddles and the 1 KB the system keeps per CTA count as well
  return (size_t)std::max(0, per_sm / (ctas + 1) + 256 - (int)(kDirectTwSmem * sizeof(uint2)) - 1024);
}

template <int CPT, class Off, bool FLAT>
static int launch_direct_as(const TxArgs &a, dim3 grid, const DirectShape &s, cudaStream_t st) {
  const size_t reserve = direct_reserve_bytes(s.ctas);
  auto launch = [&](auto lin) {
    auto kern = coltx_direct_kernel<decltype(lin)::value, CPT, Off, FLAT>;
    if (reserve) {
      static PdPerDevice attr;
      const int rc = pd_once_per_device(attr, [&] {
        PD_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 120 * 1024));
        return POLYDET_OK;
      });
      if (rc) return rc;
    }
    kern<<<grid, s.threads, reserve, st>>>(a);
    PD_CUDA(cudaGetLastError());
    return POLYDET_OK;
  };
  switch (a.Lin) {
    case 1: return launch(std::integral_constant<int, 1>());
    case 2: return launch(std::integral_constant<int, 2>());
    case 3: return launch(std::integral_constant<int, 3>());
    case 4: return launch(std::integral_constant<int, 4>());
    case 5: return launch(std::integral_constant<int, 5>());
    case 6: return launch(std::integral_constant<int, 6>());
    case 7: return launch(std::integral_constant<int, 7>());
    default: return launch(std::integral_constant<int, 8>());
  }
}

template <int CPT>
static int launch_direct(const TxArgs &a, int64_t ncols, int items, int nprimes, const DirectShape &s,
                         cudaStream_t st) {
  const int64_t per = (int64_t)s.threads * CPT;
  dim3 grid((unsigned)((ncols + per - 1) / per), (unsigned)items, (unsigned)nprimes);
  if (a.flat_items)
    grid = dim3((unsigned)((ncols * items * a.flat_groups + s.threads - 1) / s.threads), 1u, (unsigned)nprimes);
  // 32-bit byte offsets where all the output a CTA's base pointer covers lies
  // within 4 GB of it (rows the kernel steps over past the last one included)
  const int64_t rows = (int64_t)a.N + 8;
  int64_t span;
  if (a.il_L)
    span = (rows * (a.B / a.il_L) + 1) * a.il_n2 * a.il_Lp;
  else
    span = (a.flat_items ? (int64_t)items * a.out_item_stride : 0) +
           a.A * rows * (a.out_row ? a.out_row : a.B) + per;
  const bool near = span < ((int64_t)1 << 30);
  if constexpr (CPT == 1) {
    if (a.flat_items)
      return near ? launch_direct_as<CPT, uint32_t, true>(a, grid, s, st)
                  : launch_direct_as<CPT, int64_t, true>(a, grid, s, st);
  }
  return near ? launch_direct_as<CPT, uint32_t, false>(a, grid, s, st)
              : launch_direct_as<CPT, int64_t, false>(a, grid, s, st);
}

// Columns per thread: a warp's are consecutive, so that with more of them
// fewer of the sectors that rows off the 32-byte grid split are shared between
// warps, and they share each coset's twiddles; fewer leave fewer idle lanes at
// the end of a row of B columns and need fewer registers.  The times below are
// of x_1 passes of 24 x 24 matrices, relative to the Montgomery kernel before
// unless two are compared.
//
// On the sector grid nothing is shared: one column over a flattened grid (no
// idle lanes) up to 127 columns, two from 128 on: one / two / four columns, 8
// words in: 72 columns .90 / 1.26 / 2.8, 104 .88 / .95 / 2.1, 128 .85 / .81 /
// 1.8, 168 .86 / .87 / 1.6, 1024 .94 / .87 / .87, 8192 .98 / .93 / .94, 36864
// .97 / .90 / .91.  Long rows of at most four words take four, which the whole
// circle hardly tells from two (4 words, 36864 columns .96 and .97) but one
// word and slabs do: one word, 16384 columns 257 us against 278; a 15 x 15
// matrix of 1.1e8 nodes streamed in slabs, 4 words, 86.0 ms in all against 87.5.
//
// Off the grid a split sector costs a read as well where it leaves L2 before
// its other part arrives, so it matters once the output is larger than L2
// (kSplitBytes), and then
//  - the columns of a row want to be few warps': four per thread from 384 on
//    (545 columns, 8 words .96 / 1.05 / .95, 5 words 1.06 / 1.04 / .97), two
//    from 129 on;
//  - a row's warps want to be one CTA's: 97 to 127 columns two per thread on 64
//    threads (97 columns, 4 words .75 of the flattened grid's time, 5 words
//    .77), 49 to 63 one on 64 (4 words .82, 6 words .86), 73 to 95 one on 128,
//    eight CTAs per SM (85 columns, 4 words .96 of 256 threads without that
//    limit, 1.09 of 128 without it; 6 words .92 and .93);
//  - the others, whose last warp would be nearly empty, stay flattened, with
//    few CTAs at work, so that the other part of a sector is written soon: 65
//    columns, per SM three CTAs of 128 threads with 8 words .78 of the time
//    without a limit, 6 words .83; four with 5 words .88, five with 4 words
//    .84, four of 256 with 3 words .88.  With outputs that stay in L2 the
//    limit costs (65 columns, 8 primes: 6 words .91, 4 words 1.05, 4 primes 1.22
//    and 1.10).  Eight words take it up to 1023 columns (129 columns .86 against
//    1.02 with two columns, 257 .92 and .99, 385 .91 and .98), six and seven up
//    to 144 (129 columns, 7 words .87 and 1.00; 193 1.00 and .95).
//
// Blocks of columns (A > 1), interleaved output, and passes too small to fill
// the chip take one column over a flattened grid.
static DirectShape direct_shape(const TxArgs &a, int items, int nprimes) {
  constexpr int64_t kSplitBytes = 128000000;
  const bool flat_ok = a.A * a.B * items < ((int64_t)1 << 31) - kDirectThreads;
  const DirectShape flat = {1, kDirectThreads, flat_ok, 0};
  if (a.A != 1 || a.il_L || a.B < 8) return flat;
  const int64_t row = a.out_row ? a.out_row : a.B;
  const bool many = a.B * items * nprimes >= 152 * 4096;
  const DirectShape one = {1, kDirectThreads, false, 0}, two = {2, kDirectThreads, false, 0},
                    four = {4, kDirectThreads, false, 0};
  if (row % 8 == 0) {
    if (!many || a.B < 64 || (a.B < 128 && a.Lin > 1)) return flat;
    return a.B < 128 ? one : a.Lin <= 4 && a.B >= 8192 ? four : two;
  }
  if (4 * row * out_rows(a) * items * nprimes < kSplitBytes) {
    if (!many || a.B < 64 || (a.B < 128 && a.Lin > 1)) return flat;
    return a.B < 128 ? one : a.B >= 512 ? four : two;
  }
  const DirectShape capped = a.Lin <= 2   ? DirectShape{1, 128, true, 0}
                             : a.Lin == 3 ? DirectShape{1, 256, true, 4}
                                          : DirectShape{1, 128, true, a.Lin == 4 ? 5 : a.Lin == 5 ? 4 : 3};
  if (flat_ok && a.B < (a.Lin == 8 ? 1024 : a.Lin >= 6 && a.B > 128 ? 145 : 0)) return capped;
  if (a.B >= 384) return four;
  if (a.B > 128) return two;
  if (a.B > 96 && a.Lin < 7) return {2, 64, false, 0};
  if (a.Lin <= 2 && flat_ok) return capped;
  if (a.B >= 48 && a.B <= 64) return {1, 64, false, 0};
  if ((a.B >= (a.Lin <= 5 ? 72 : 80) && a.B <= 96) || !flat_ok) return {1, 128, false, 8};
  return capped;
}

static int launch_pass(TxArgs a, int items, int nprimes, cudaStream_t st) {
  int64_t ncols = a.A * a.B;
  // short forward transforms over many columns: the register-direct kernel
  const int lp_in = a.Lin <= 1 ? 1 : a.Lin <= 2 ? 2 : a.Lin <= 4 ? 4 : 8;
  // rows of fewer than 8 columns (a job's first pass: B = 1) only with the
  // flattened grid below, and not into the interleaved partial layout
  const bool rows_ok = a.B >= 8 || (!a.il_L && ncols * items < ((int64_t)1 << 31) - 256);
  const bool window_ok = a.row_hi == 0 || (a.olp > 1 && a.olp == lp_in && a.row_lo % lp_in == 0);
  if (!a.inverse && a.Lin <= 8 && a.N <= kDirectTwSmem && rows_ok && window_ok &&
      (a.olp <= 1 || a.olp == lp_in)) {
    const DirectShape shape = direct_shape(a, items, nprimes);
    // short rows: one grid axis over (item, column) pairs, so that rows
    // shorter than a CTA, or a row's last CTA, leave no threads idle
    a.flat_items = shape.flat ? items : 0;
    // few columns in all (a job's first pass): cut each column's cosets into
    // groups until the grid holds about 152 x 1024 threads
    a.flat_groups = 1;
    if (a.flat_items) {
      const int J = a.N / lp_in;
      const int rhi = a.row_hi ? a.row_hi : a.Lout;
      const int Jc = (a.olp > 1) ? (rhi + lp_in - 1) / lp_in - a.row_lo / lp_in : J;
      const int64_t base = ncols * items * nprimes;
      int64_t g = (152 * 1024 + base - 1) / base;
      g = std::min<int64_t>(g, Jc);
      while (g > 1 && ncols * items * g >= ((int64_t)1 << 31) - 256) --g;
      a.flat_groups = (int)std::max<int64_t>(1, g);
    }
    switch (shape.cpt) {
      case 4: return launch_direct<4>(a, ncols, items, nprimes, shape, st);
      case 2: return launch_direct<2>(a, ncols, items, nprimes, shape, st);
      default: return launch_direct<1>(a, ncols, items, nprimes, shape, st);
    }
  }
  // Ct: columns per CTA, a power of two with N * (Ct + 1) words <= 64 KB.
  int ct = 32;
  while (ct > 1 && (int64_t)a.N * (ct + 1) > 16384) ct >>= 1;
  while (ct > 1 && ct / 2 >= ncols) ct >>= 1;
  a.Ct = ct;
  a.logCt = ilog2(ct);
  size_t smem = (size_t)a.N * (ct + 1) * sizeof(uint32_t);
  static PdPerDevice attr;
  int rc = pd_once_per_device(attr, [] {
    PD_CUDA(cudaFuncSetAttribute(coltx_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    return POLYDET_OK;
  });
  if (rc) return rc;
  dim3 grid((unsigned)((ncols + ct - 1) / ct), (unsigned)items, (unsigned)nprimes);
  coltx_kernel<<<grid, 256, smem, st>>>(a);
  PD_CUDA(cudaGetLastError());
  return POLYDET_OK;
}

static int check_range(const polydet_plan_s *pl, int lo, int hi) {
  return (pl && lo >= 0 && hi <= pl->P && lo < hi) ? POLYDET_OK : POLYDET_EINVAL;
}

extern "C" int polydet_eval(polydet_plan_t pl, const int32_t *coeffs, int lo, int hi,
                            uint32_t *evals, uint32_t *ws, void *stream) {
  if (check_range(pl, lo, hi) || !coeffs || !evals) return POLYDET_EINVAL;
  if (pl->eval_ws_words && !ws) return POLYDET_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  const int k = pl->nvars, np = hi - lo;
  const int64_t n2 = (int64_t)pl->n * pl->n;
  const uint64_t slot = n2 ? pl->eval_ws_words / (uint64_t)n2 : 0;
  // with an entry map only the distinct entries are evaluated, and the zero
  // entry's slot is cleared
  const int64_t items = pl->nitems, nent = pl->nent;
  const void *cur_in = coeffs;
  int64_t cur_item = pl->E, cur_prime = 0;
  int cur_i32 = 1;
  for (int v = k - 1; v >= 0; --v) {
    TxArgs a = {};
    a.A = 1;
    for (int u = 0; u < v; ++u) a.A *= pl->d[u] + 1;
    a.B = 1;
    for (int u = v + 1; u < k; ++u) a.B *= pl->M[u];
    a.Lin = pl->d[v] + 1;
    a.N = pl->N[v];
    a.logN = pl->logN[v];
    a.Lout = pl->M[v];  // the first M_v nodes (in the plan's order) of the N_v-point transform
    a.olp = pl->LPo[v];
    a.in = cur_in;
    a.in_item_stride = cur_item;
    a.in_prime_stride = cur_prime;
    a.in_is_i32 = cur_i32;
    if (v % 2 == 0) {  // even passes land in the output array (slot G per entry)
      a.out = evals;
      a.out_item_stride = pl->G;
      a.out_prime_stride = nent * pl->G;
    } else {
      a.out = ws;
      a.out_item_stride = (int64_t)slot;
      a.out_prime_stride = items * a.out_item_stride;
    }
    a.inverse = 0;
    a.prime_lo = lo;
    a.mod = pl->d_mod;
    a.tw = pl->d_tw_fwd;
    a.tws = pl->d_tw_shoup;
    a.tw_len = pl->tw_len;
    a.tw_off = pl->tw_off[v];
    a.ninv = pl->d_ninv;
    a.nvars = k;
    a.var = v;
    a.status = pl->d_status;
    // the last pass also writes the zero entry's slot (entry map): one more
    // item that reads nothing; earlier passes skip a map without entries
    int launch_items = (int)items;
    if (v == 0 && nent > items) {
      a.zero_item_plus1 = (int)items + 1;
      launch_items = (int)nent;
    }
    if (launch_items > 0) {
      int rc = launch_pass(a, launch_items, np, st);
      if (rc) return rc;
    }
    cur_in = a.out;
    cur_item = a.out_item_stride;
    cur_prime = a.out_prime_stride;
    cur_i32 = 0;
  }
  return POLYDET_OK;
}

// Node-grid interpolation of one variable (Sec. 3.3 on the node grid): every
// column (a, b) of the tensor [A][m][B] holds the values at the m nodes (in
// coset order: node k = j L + t is w^j psi^t, psi = w^(N/L)) of a polynomial
// P of degree < m in that variable; its coefficients replace them.  With
// P(x) = sum_{r<L} x^r Q_r(x^L) and x^L = z_j = w^(L j) on coset j:
//  1. per whole coset j < Jf: an inverse DFT of size L of its L values, times
//     L^-1 w^(-j r), gives Q_r(z_j) for every r;
//  2. the s = m - Jf L nodes of the last coset fix the top coefficient
//     lambda_r of Q_r for r < s (Q_r = I_r + lambda_r Pi, I_r the interpolant
//     through z_0..z_{Jf-1}, Pi = prod_j (z - z_j)): E_r = I_r(z_Jf) is one
//     dot product of the Q_r(z_j), and lambda = B y - (B X) E with the nodes'
//     values y and the plan's s x s and s x L matrices;
//  3. per r: the coefficients of Q_r are dot products of (Q_r(z_j), lambda_r)
//     with the inverse Vandermonde matrix of size Jf, extended by the
//     coefficients of Pi (Jf (Jf + 1) L products per column instead of m^2).
// A CTA stages Ct columns.  Step 3 is nearly all of the work; a thread
// computes kCiU coefficients of two columns there, so that the table words
// (one 16-byte load, the same for the whole warp) and the values each serve
// several products: 3 loads per 8 products.  One dot product per thread (two
// loads per product) was bound by the load pipe at a quarter of the integer
// pipe's rate: 73^3 nodes and 18 primes took 369 us, now 172 us.
struct CiArgs {
  const uint32_t *in;
  uint32_t *out;
  int64_t in_prime_stride, out_prime_stride;
  int64_t A, B;
  int m, Jf, s, Ct, logCt;
  int rows;  // B == 1: columns are contiguous rows of m words, staged through shared memory
  int prime_lo;
  const ModP *mod;
  const uint32_t *tab;  // this variable's tables for prime 0 (layout: CiTab)
  int tab_len;          // words per prime
};

// A table word from shared memory (TAB) or global memory.
template <bool TAB>
PD_D uint32_t ci_ld(const uint32_t *x) {
  if constexpr (TAB)
    return *x;
  else
    return __ldg(x);
}

// sum_{j<len} x[j] y[j s] / R mod p (x a table, y in shared memory with stride
// s): four products per REDC (redc4: 4 p^2 < p 2^32 for any p < 2^31; fewer in
// the last one).
template <bool TAB>
PD_D uint32_t dot_strided(const uint32_t *x, const uint32_t *y, int s, int len, uint32_t p, uint32_t pinv) {
  uint32_t acc = 0u;
  int j = 0;
  for (; j + 3 < len; j += 4)
    acc = addm(acc,
               redc4((uint64_t)ci_ld<TAB>(x + j) * y[j * s] + (uint64_t)ci_ld<TAB>(x + j + 1) * y[(j + 1) * s] +
                         (uint64_t)ci_ld<TAB>(x + j + 2) * y[(j + 2) * s] +
                         (uint64_t)ci_ld<TAB>(x + j + 3) * y[(j + 3) * s],
                     p, pinv),
               p);
  uint64_t t = 0u;
  for (; j < len; ++j) t += (uint64_t)ci_ld<TAB>(x + j) * y[j * s];
  return addm(acc, redc4(t, p, pinv), p);
}

// X_r = sum_t x_t rho^(t r) for L in {1, 2, 4, 8}; rk[k] = rho^k (Montgomery).
template <int L>
PD_D void small_dft(uint32_t (&x)[L], const uint32_t *rk, uint32_t p, uint32_t pinv) {
  if constexpr (L == 2) {
    const uint32_t a = x[0], b = x[1];
    x[0] = addm(a, b, p);
    x[1] = subm(a, b, p);
  } else if constexpr (L == 4) {
    uint32_t y[4], xx[4] = {x[0], x[1], x[2], x[3]};
    dft4<false, false, false, false>(xx, y, __ldg(rk + 1), p, pinv);
#pragma unroll
    for (int r = 0; r < 4; ++r) x[r] = y[r];
  } else if constexpr (L == 8) {
    uint32_t xe[4] = {x[0], x[2], x[4], x[6]}, xo[4] = {x[1], x[3], x[5], x[7]}, E[4], O[4];
    const uint32_t r2 = __ldg(rk + 2);
    dft4<false, false, false, false>(xe, E, r2, p, pinv);
    dft4<false, false, false, false>(xo, O, r2, p, pinv);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const uint32_t o = r ? mmul(__ldg(rk + r), O[r], p, pinv) : O[r];
      x[r] = addm(E[r], o, p);
      x[r + 4] = subm(E[r], o, p);
    }
  }
}

constexpr int kCiU = 4;  // coefficients per thread and column (one 16-byte table load)

// U: coefficients per thread, kCiU, or 1 where a pass is too small to fill the
// chip and its time is one thread's chain of products.
// TAB (U == 1): the tables staged in shared memory, one trip to L2 for all of
// them instead of one per four products of that chain; chains of more than two
// such steps, tables of at most 16 KB (longer ones pass through 1024 threads
// that cover the trips for each other).  One prime, microseconds, tables in
// global memory and 256 threads / now: 24 x 24 univariate, degree 7 (169
// nodes) 5.9 / 5.1; 32 x 32, degree 3 6.0 / 4.6; 19 x 19, degree 200 (3801
// nodes) 380 / 193; 8 x 8, degrees 5 and 200 150 / 48; but 3 x 3, degree 1
// (chains of one step) 2.3 / 2.6 staged.
constexpr int kCiSmallThreads = 1024, kCiTabWords = 4096;
template <int L, int U, bool TAB>
__global__ void __launch_bounds__(U == 1 ? kCiSmallThreads : 256) cinterp_kernel(CiArgs a) {
  extern __shared__ __align__(16) uint32_t sm[];
  const int q = a.prime_lo + blockIdx.z;
  const ModP md = a.mod[q];
  const uint32_t p = md.p, pinv = md.pinv;
  const int m = a.m, Jf = a.Jf, s = a.s, Ct = a.Ct, logCt = a.logCt;
  const int JJ = Jf + (s > 0);  // length of the dot products
  const int64_t ncols = a.A * a.B;
  const int64_t col0 = (int64_t)blockIdx.x * Ct;
  const uint32_t *in = a.in + (int64_t)blockIdx.z * a.in_prime_stride;
  uint32_t *out = a.out + (int64_t)blockIdx.z * a.out_prime_stride;
  const CiTab T(m, L);
  const uint32_t *gtab = a.tab + (size_t)q * a.tab_len, *tab = TAB ? sm : gtab;
  uint32_t *Qv = sm + (TAB ? T.words : 0);           // [L][JJ][Ct] Q_r(z_j), then lambda_r
  uint32_t *Es = Qv + (size_t)L * JJ * Ct;           // [L][Ct] E_r (s > 0)
  uint32_t *Y = Es + (s > 0 ? (size_t)L * Ct : 0);   // [Ct][mp] node values, then coefficients (rows)
  const int mp = m | 1;                              // odd: lanes of different columns in different banks
  const int tid = threadIdx.x, bd = blockDim.x;
  const int ncol = (int)min((int64_t)Ct, ncols - col0);
  // word of row 0 of column c of the tile (row e: + e B)
  auto word0 = [&](int c) -> int64_t {
    const int64_t col = col0 + c;
    if (a.A == 1) return col;
    const int64_t aa = (ncols >> 32) ? col / a.B : (int64_t)((uint32_t)col / (uint32_t)a.B);
    return aa * m * a.B + (col - aa * a.B);
  };
  // a thread keeps its column through the phases (blockDim is a multiple of Ct)
  const int c = tid & (Ct - 1), jstep = bd >> logCt;

  if constexpr (TAB)  // read from step 2 on; the parts are multiples of 16 bytes
    for (int i = tid; i < T.words / 4; i += bd)
      reinterpret_cast<uint4 *>(sm)[i] = __ldg(reinterpret_cast<const uint4 *>(gtab) + i);
  if (a.rows) {
    const uint32_t *src = in + col0 * m;
    for (int k = tid >> 5; k < ncol; k += bd >> 5)
      for (int r = tid & 31; r < m; r += 32) Y[k * mp + r] = src[(int64_t)k * m + r];
    __syncthreads();
  }
  // the column's node values: node r at src[r * sstep]
  const uint32_t *src = a.rows ? Y + c * mp : in + word0(c < ncol ? c : 0);
  const int64_t sstep = a.rows ? 1 : a.B;
  // 1. inverse DFT of each whole coset, twisted
  {
    const uint32_t *sj = src + (int64_t)(tid >> logCt) * L * sstep;
    const uint32_t *tw = gtab + T.tw1 + (tid >> logCt) * L;
    uint32_t *qj = Qv + ((tid >> logCt) << logCt) + c;
    for (int j = tid >> logCt; j < Jf; j += jstep) {
      uint32_t x[L];
#pragma unroll
      for (int t = 0; t < L; ++t) x[t] = c < ncol ? sj[t * sstep] : 0u;
      small_dft<L>(x, gtab + T.rk, p, pinv);
#pragma unroll
      for (int r = 0; r < L; ++r) qj[(r * JJ) << logCt] = mmul(x[r], __ldg(tw + r), p, pinv);
      sj += (int64_t)jstep * L * sstep;
      tw += jstep * L;
      qj += jstep << logCt;
    }
  }
  // the last coset's values: where a chain bounds the pass and there are
  // several, loaded ahead and all at once
  constexpr bool AHEAD = U == 1 && L > 2;
  uint32_t last[L];
  if constexpr (AHEAD) {
#pragma unroll
    for (int t = 0; t + 1 < L; ++t) last[t] = (t < s && c < ncol) ? src[(Jf * L + t) * sstep] : 0u;
  }
  __syncthreads();
  if (s > 0) {  // 2. the last coset
    for (int r = tid >> logCt; r < L; r += jstep)
      Es[(r << logCt) + c] = dot_strided<TAB>(tab + T.ell, Qv + ((r * JJ) << logCt) + c, Ct, Jf, p, pinv);
    __syncthreads();
    for (int r = tid >> logCt; r < L; r += jstep) {
      uint32_t lam = 0u;
      if (r < s && c < ncol) {
        lam = dot_strided<TAB>(tab + T.nx + r * L, Es + c, Ct, L, p, pinv);
        if constexpr (AHEAD) {
#pragma unroll
          for (int t = 0; t + 1 < L; ++t)
            if (t < s) lam = addm(lam, mmul(ci_ld<TAB>(tab + T.bm + r * s + t), last[t], p, pinv), p);
        } else {
          for (int t = 0; t < s; ++t)
            lam = addm(lam, mmul(ci_ld<TAB>(tab + T.bm + r * s + t), src[(Jf * L + t) * sstep], p, pinv), p);
        }
      }
      Qv[((r * JJ + Jf) << logCt) + c] = lam;
    }
    __syncthreads();
  }
  // 3. coefficient e = L u + r of columns c2 and c2 + Ct / 2, u = u0 .. u0 + U - 1
  const int half = Ct >> 1, c2 = tid & (half - 1);
  const int chunks = (Jf + U - 1) / U;
  uint32_t *dst[2];
  const int64_t dstep = a.rows ? 1 : a.B;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int ch = c2 + h * half;
    dst[h] = a.rows ? Y + ch * mp : out + word0(ch < ncol ? ch : 0);
  }
  for (int ru = tid >> (logCt - 1); ru < chunks * L; ru += bd >> (logCt - 1)) {
    const int r = ru % L, u0 = ru / L * U;
    const uint32_t *V = tab + T.vt + u0;  // U == 4: 16-byte aligned, every table offset is a multiple of 4 words
    const uint32_t *y = Qv + ((r * JJ) << logCt) + c2;
    const int vstep = T.jp;
    uint32_t acc[U][2];
#pragma unroll
    for (int i = 0; i < U; ++i) acc[i][0] = acc[i][1] = 0u;
    auto group = [&](auto count) {  // up to four products per REDC
      constexpr int N = decltype(count)::value;
      uint64_t t[U][2];
#pragma unroll
      for (int k = 0; k < N; ++k) {
        uint32_t v[U];
        if constexpr (U == 4) {
          const uint4 v4 = __ldg(reinterpret_cast<const uint4 *>(V + k * vstep));
          v[0] = v4.x, v[1] = v4.y, v[2] = v4.z, v[3] = v4.w;
        } else {
          v[0] = ci_ld<TAB>(V + k * vstep);
        }
        const uint32_t y0 = y[k << logCt], y1 = y[(k << logCt) + half];
#pragma unroll
        for (int i = 0; i < U; ++i) {
          t[i][0] = (uint64_t)v[i] * y0 + (k ? t[i][0] : 0ull);
          t[i][1] = (uint64_t)v[i] * y1 + (k ? t[i][1] : 0ull);
        }
      }
      V += N * vstep;
      y += N << logCt;
#pragma unroll
      for (int i = 0; i < U; ++i) {
        acc[i][0] = addm(acc[i][0], redc4(t[i][0], p, pinv), p);
        acc[i][1] = addm(acc[i][1], redc4(t[i][1], p, pinv), p);
      }
    };
    int j = JJ;
    for (; j >= 4; j -= 4) group(std::integral_constant<int, 4>());
    if (j == 3) group(std::integral_constant<int, 3>());
    if (j == 2) group(std::integral_constant<int, 2>());
    if (j == 1) group(std::integral_constant<int, 1>());
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (c2 + h * half >= ncol) continue;
      uint32_t *d = dst[h] + (L * u0 + r) * dstep;
#pragma unroll
      for (int i = 0; i < U; ++i) {
        if (u0 + i < Jf) *d = acc[i][h];
        d += L * dstep;
      }
    }
  }
  // the top coefficients lambda_r: e = L Jf + r, r < s
  for (int f = tid; f < s << logCt; f += bd) {
    const int r = f >> logCt, k = f & (Ct - 1);
    if (k >= ncol) continue;
    const uint32_t lam = Qv[((r * JJ + Jf) << logCt) + k];
    if (a.rows)
      Y[k * mp + L * Jf + r] = lam;
    else
      out[word0(k) + (L * Jf + r) * a.B] = lam;
  }
  if (a.rows) {
    __syncthreads();
    uint32_t *o = out + col0 * m;
    for (int k = tid >> 5; k < ncol; k += bd >> 5)
      for (int r = tid & 31; r < m; r += 32) o[(int64_t)k * m + r] = Y[k * mp + r];
  }
}

// Shared-memory words of a cinterp CTA of ct columns.
static size_t cinterp_words(int m, int L, int ct, bool rows) {
  const int Jf = m / L, s = m % L;
  return (size_t)ct * ((size_t)L * (Jf + (s > 0)) + (s > 0 ? L : 0) + (rows ? (m | 1) : 0));
}

static int interp_nodes(polydet_plan_t pl, const uint32_t *detvals, int lo, int hi,
                        uint32_t *residues, uint32_t *ws, cudaStream_t st) {
  const int k = pl->nvars, np = hi - lo;
  const uint64_t slot = pl->interp_ws_words / 2;
  constexpr size_t kMaxSmem = 200 * 1024;
  int dev = 0, sms = 0;
  PD_CUDA(cudaGetDevice(&dev));
  PD_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  static PdPerDevice attr;
  const int arc = pd_once_per_device(attr, [] {
    int rc = POLYDET_OK;
    auto allow = [&](auto kern) {
      if (rc == POLYDET_OK)
        rc = [&] {
          PD_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
          return POLYDET_OK;
        }();
    };
    allow(cinterp_kernel<1, kCiU, false>), allow(cinterp_kernel<1, 1, false>), allow(cinterp_kernel<1, 1, true>);
    allow(cinterp_kernel<2, kCiU, false>), allow(cinterp_kernel<2, 1, false>), allow(cinterp_kernel<2, 1, true>);
    allow(cinterp_kernel<4, kCiU, false>), allow(cinterp_kernel<4, 1, false>), allow(cinterp_kernel<4, 1, true>);
    allow(cinterp_kernel<8, kCiU, false>), allow(cinterp_kernel<8, 1, false>), allow(cinterp_kernel<8, 1, true>);
    return rc;
  });
  if (arc) return arc;
  const uint32_t *cur = detvals;
  int64_t cur_prime = pl->G;
  int t = 0;
  for (int v = k - 1; v >= 0; --v, ++t) {
    CiArgs a = {};
    a.A = 1;
    for (int u = 0; u < v; ++u) a.A *= pl->M[u];
    a.B = 1;
    for (int u = v + 1; u < k; ++u) a.B *= pl->M[u];
    const int L = pl->LPo[v];
    a.m = pl->M[v];
    a.Jf = a.m / L;
    a.s = a.m % L;
    a.rows = a.B == 1;
    const int64_t ncols = a.A * a.B;
    int ct = 32;
    while (ct > 2 && cinterp_words(a.m, L, ct, a.rows) * sizeof(uint32_t) > 56 * 1024) ct >>= 1;
    while (ct > 2 && ct / 2 >= ncols) ct >>= 1;
    // small passes (a job's few columns): fewer columns per CTA, so that the
    // grid still spreads over the SMs (two CTAs each) and every CTA's
    // phases, which run one after another, are short
    while (ct > 4 && (ncols + ct - 1) / ct * np < 2 * sms) ct >>= 1;
    // fewer columns still, while every CTA has an SM to itself
    while (ct > 2 && (ncols + ct / 2 - 1) / (ct / 2) * np <= sms) ct >>= 1;
    const int64_t ctas = (ncols + ct - 1) / ct * np;
    int items = std::max(1, (a.Jf + kCiU - 1) / kCiU) * L * (ct / 2);
    const bool small = ctas * items < 256 * sms;
    if (small) items = std::max(1, a.Jf) * L * (ct / 2);
    // threads: a multiple of the columns, no more than step 3 has items for.
    // Small CTAs, so that those of an SM are in different phases (73^3 nodes,
    // 18 primes: 172 us with 128 threads, 180 with 192, 207 with 512; 64
    // columns and 320 threads 186), larger ones where the grid is short of
    // four CTAs per SM (193^2 nodes, 24 primes: 34.8 us with 256, 36.9 with 128)
    // and the largest where it is short of one
    const int most = ctas >= 4 * sms ? 128 : small && ctas <= sms ? kCiSmallThreads : 256;
    const int th = std::min((items + 63) / 64 * 64, most);
    size_t smem = cinterp_words(a.m, L, ct, a.rows) * sizeof(uint32_t);
    const int tab_words = CiTab(a.m, L).words;
    const bool staged =
        small && a.Jf > 8 && tab_words <= kCiTabWords && smem + tab_words * sizeof(uint32_t) <= kMaxSmem;
    if (staged) smem += tab_words * sizeof(uint32_t);
    if (smem > kMaxSmem) return POLYDET_EINVAL;
    a.Ct = ct;
    a.logCt = ilog2(ct);
    a.in = cur;
    a.in_prime_stride = cur_prime;
    if (v == 0) {
      a.out = residues;
      a.out_prime_stride = pl->C;
    } else {
      a.out = ws + (uint64_t)(t % 2) * slot * (uint64_t)np;
      a.out_prime_stride = (int64_t)slot;
    }
    a.prime_lo = lo;
    a.mod = pl->d_mod;
    a.tab = pl->d_itab + pl->itab_off[v];
    a.tab_len = pl->itab_len;
    dim3 grid((unsigned)((ncols + ct - 1) / ct), 1, (unsigned)np);
    auto launch = [&](auto len) {
      constexpr int LL = decltype(len)::value;
      if (staged)
        cinterp_kernel<LL, 1, true><<<grid, th, smem, st>>>(a);
      else if (small)
        cinterp_kernel<LL, 1, false><<<grid, th, smem, st>>>(a);
      else
        cinterp_kernel<LL, kCiU, false><<<grid, th, smem, st>>>(a);
    };
    switch (L) {
      case 1: launch(std::integral_constant<int, 1>()); break;
      case 2: launch(std::integral_constant<int, 2>()); break;
      case 4: launch(std::integral_constant<int, 4>()); break;
      default: launch(std::integral_constant<int, 8>()); break;
    }
    PD_CUDA(cudaGetLastError());
    cur = a.out;
    cur_prime = a.out_prime_stride;
  }
  return POLYDET_OK;
}

extern "C" int polydet_interp(polydet_plan_t pl, const uint32_t *detvals, int lo, int hi,
                              uint32_t *residues, uint32_t *ws, void *stream) {
  if (check_range(pl, lo, hi) || !detvals || !residues) return POLYDET_EINVAL;
  if (pl->interp_ws_words && !ws) return POLYDET_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  if (!pl->full) return interp_nodes(pl, detvals, lo, hi, residues, ws, st);
  const int k = pl->nvars, np = hi - lo;
  const uint64_t slot = pl->interp_ws_words / 2;
  const void *cur_in = detvals;
  int64_t cur_prime = pl->G;
  int t = 0;
  for (int v = k - 1; v >= 0; --v, ++t) {
    TxArgs a = {};
    a.A = 1;
    for (int u = 0; u < v; ++u) a.A *= pl->N[u];
    a.B = 1;
    for (int u = v + 1; u < k; ++u) a.B *= pl->D[u] + 1;
    a.Lin = pl->N[v];
    a.N = pl->N[v];
    a.logN = pl->logN[v];
    a.Lout = pl->D[v] + 1;
    a.in = cur_in;
    a.in_item_stride = 0;
    a.in_prime_stride = cur_prime;
    a.in_is_i32 = 0;
    if (v == 0) {
      a.out = residues;
      a.out_prime_stride = pl->C;
    } else {
      a.out = ws + (uint64_t)(t % 2) * slot * (uint64_t)np;
      a.out_prime_stride = (int64_t)slot;
    }
    a.out_item_stride = 0;
    a.inverse = 1;
    a.prime_lo = lo;
    a.mod = pl->d_mod;
    a.tw = pl->d_tw_inv;
    a.tw_len = pl->tw_len;
    a.tw_off = pl->tw_off[v];
    a.ninv = pl->d_ninv;
    a.nvars = k;
    a.var = v;
    a.status = pl->d_status;
    int rc = launch_pass(a, 1, np, st);
    if (rc) return rc;
    cur_in = a.out;
    cur_prime = a.out_prime_stride;
  }
  return POLYDET_OK;
}

// Words per entry of the tensor after the passes of x_k, ..., x_{v+1}:
// prod_{u<=v} L_u * prod_{u>v} M_u (0-based v; L_u = d_u + 1).
static uint64_t words_after(const polydet_plan_s *pl, int v) {
  uint64_t s = 1;
  for (int u = 0; u < pl->nvars; ++u) s *= (u <= v) ? (uint64_t)(pl->d[u] + 1) : (uint64_t)pl->M[u];
  return s;
}

uint64_t pd_head_words(const polydet_plan_s *pl) { return words_after(pl, 0); }

uint64_t pd_head_ws_words(const polydet_plan_s *pl) {
  // passes v >= 2 with v even land in the scratch (so that v = 1 lands in head)
  uint64_t best = 0;
  for (int v = 2; v < pl->nvars; v += 2) best = std::max(best, words_after(pl, v - 1));
  return best * (uint64_t)pl->nitems;
}

__global__ void reduce_kernel(const int32_t *__restrict__ in, uint32_t *__restrict__ out, int64_t len,
                              const ModP *__restrict__ mod, int lo) {
  const uint32_t p = mod[lo + blockIdx.y].p;
  for (int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; f < len;
       f += (int64_t)gridDim.x * blockDim.x)
    out[(int64_t)blockIdx.y * len + f] = reduce_i32(in[f], p);
}

static TxArgs forward_pass(const polydet_plan_s *pl, int v, int lo) {
  TxArgs a = {};
  a.A = 1;
  for (int u = 0; u < v; ++u) a.A *= pl->d[u] + 1;
  a.B = 1;
  for (int u = v + 1; u < pl->nvars; ++u) a.B *= pl->M[u];
  a.Lin = pl->d[v] + 1;
  a.N = pl->N[v];
  a.logN = pl->logN[v];
  a.Lout = pl->M[v];
  a.olp = pl->LPo[v];
  a.inverse = 0;
  a.prime_lo = lo;
  a.mod = pl->d_mod;
  a.tw = pl->d_tw_fwd;
  a.tws = pl->d_tw_shoup;
  a.tw_len = pl->tw_len;
  a.tw_off = pl->tw_off[v];
  a.ninv = pl->d_ninv;
  a.nvars = pl->nvars;
  a.var = v;
  a.status = pl->d_status;
  return a;
}

int pd_eval_head(const polydet_plan_s *pl, const int32_t *coeffs, int lo, int hi, uint32_t *head,
                 uint32_t *ws, cudaStream_t st) {
  if (check_range(pl, lo, hi)) return POLYDET_EINVAL;
  const int k = pl->nvars;
  const int64_t items = pl->nitems;
  if (items == 0) return POLYDET_OK;
  if (k == 1) {
    const int64_t len = items * pl->E;
    const unsigned blocks = (unsigned)std::min<int64_t>((len + 255) / 256, 4096);
    reduce_kernel<<<dim3(blocks, hi - lo), 256, 0, st>>>(coeffs, head, len, pl->d_mod, lo);
    PD_CUDA(cudaGetLastError());
    return POLYDET_OK;
  }
  const int64_t S1 = (int64_t)pd_head_words(pl);
  int64_t S2 = 0;
  for (int v = 2; v < k; v += 2) S2 = std::max<int64_t>(S2, (int64_t)words_after(pl, v - 1));
  const void *cur_in = coeffs;
  int64_t cur_item = pl->E, cur_prime = 0;
  int cur_i32 = 1;
  for (int v = k - 1; v >= 1; --v) {
    TxArgs a = forward_pass(pl, v, lo);
    a.in = cur_in;
    a.in_item_stride = cur_item;
    a.in_prime_stride = cur_prime;
    a.in_is_i32 = cur_i32;
    a.out = (v % 2) ? head : ws;
    a.out_item_stride = (v % 2) ? S1 : S2;
    a.out_prime_stride = items * a.out_item_stride;
    int rc = launch_pass(a, (int)items, hi - lo, st);
    if (rc) return rc;
    cur_in = a.out;
    cur_item = a.out_item_stride;
    cur_prime = a.out_prime_stride;
    cur_i32 = 0;
  }
  return POLYDET_OK;
}

EvLayout pd_tail_layout(const polydet_plan_s *pl, int rows) {
  const int64_t B = pl->G / pl->M[0];  // nodes of the other variables: one row
  const int64_t Bs = B >= 1024 ? (B + 31) / 32 * 32 : B;  // padding <= 3 % of a row
  return EvLayout{B, Bs, (int64_t)(rows > 0 ? rows : pl->M[0]) * Bs};
}

int pd_eval_tail(const polydet_plan_s *pl, const uint32_t *head, int head_q0, int lo, int hi,
                 int row_lo, int row_hi, uint32_t *evals, EvLayout lay, cudaStream_t st) {
  if (check_range(pl, lo, hi) || !head || !evals || lo < head_q0) return POLYDET_EINVAL;
  const int64_t items = pl->nitems, nent = pl->nent;
  const int64_t S1 = (int64_t)pd_head_words(pl);
  TxArgs a = forward_pass(pl, 0, lo);
  if (row_lo < 0 || row_hi > pl->M[0] || row_lo >= row_hi) return POLYDET_EINVAL;
  if (lay.rowlen != a.B || lay.entry != (int64_t)(row_hi - row_lo) * lay.rowstride) return POLYDET_EINVAL;
  if (row_lo > 0 || row_hi < pl->M[0]) {
    a.row_lo = row_lo;
    a.row_hi = row_hi;
  }
  if (nent > items) a.zero_item_plus1 = (int)items + 1;  // the zero entry's slot (entry map)
  a.in = head + (int64_t)(lo - head_q0) * items * S1;
  a.in_item_stride = S1;
  a.in_prime_stride = items * S1;
  a.in_is_i32 = 0;
  a.out = evals;
  a.out_row = lay.rowstride;
  a.out_item_stride = lay.entry;
  a.out_prime_stride = nent * lay.entry;
  return launch_pass(a, (int)nent, hi - lo, st);
}

uint64_t pd_partial_ws_words(const polydet_plan_s *pl) {
  // pass v >= 1 output per entry: prod_{u<v} L_u * prod_{v<=u<k-1} N_u * L_{k-1}
  const int k = pl->nvars;
  uint64_t best = 0;
  for (int v = 1; v <= k - 2; ++v) {
    uint64_t s = (uint64_t)(pl->d[k - 1] + 1);
    for (int u = 0; u < k - 1; ++u) s *= (u < v) ? (uint64_t)(pl->d[u] + 1) : (uint64_t)pl->M[u];
    if (s > best) best = s;
  }
  return 2 * best * (uint64_t)pl->n * pl->n;
}

int pd_eval_partial(const polydet_plan_s *pl, const int32_t *coeffs, int lo, int hi, uint32_t *out,
                    int Lp, uint32_t *ws, cudaStream_t st) {
  const int k = pl->nvars, np = hi - lo;
  if (k < 2) return POLYDET_EINVAL;
  const int64_t n2 = (int64_t)pl->n * pl->n;
  const int Lk = pl->d[k - 1] + 1;
  int64_t rows = 1;
  for (int u = 0; u < k - 1; ++u) rows *= pl->M[u];
  const uint64_t slot = pd_partial_ws_words(pl) / (2 * (uint64_t)n2);
  const void *cur_in = coeffs;
  int64_t cur_item = pl->E, cur_prime = 0;
  int cur_i32 = 1;
  int t = 0;
  for (int v = k - 2; v >= 0; --v, ++t) {
    TxArgs a = {};
    a.A = 1;
    for (int u = 0; u < v; ++u) a.A *= pl->d[u] + 1;
    a.B = Lk;
    for (int u = v + 1; u < k - 1; ++u) a.B *= pl->M[u];
    a.Lin = pl->d[v] + 1;
    a.N = pl->N[v];
    a.logN = pl->logN[v];
    a.Lout = pl->M[v];
    a.olp = pl->LPo[v];
    a.in = cur_in;
    a.in_item_stride = cur_item;
    a.in_prime_stride = cur_prime;
    a.in_is_i32 = cur_i32;
    if (v == 0) {
      a.out = out;
      a.out_prime_stride = rows * n2 * Lp;
      a.il_L = Lk;
      a.il_Lp = Lp;
      a.il_n2 = n2;
    } else {
      a.out = ws + (uint64_t)(t % 2) * slot * (uint64_t)n2 * (uint64_t)np;
      a.out_item_stride = (int64_t)slot;
      a.out_prime_stride = n2 * (int64_t)slot;
    }
    a.prime_lo = lo;
    a.mod = pl->d_mod;
    a.tw = pl->d_tw_fwd;
    a.tws = pl->d_tw_shoup;
    a.tw_len = pl->tw_len;
    a.tw_off = pl->tw_off[v];
    a.ninv = pl->d_ninv;
    a.nvars = k;
    a.var = v;
    a.status = pl->d_status;
    int rc = launch_pass(a, (int)n2, np, st);
    if (rc) return rc;
    cur_in = a.out;
    cur_item = a.out_item_stride;
    cur_prime = a.out_prime_stride;
    cur_i32 = 0;
  }
  return POLYDET_OK;
}

extern "C" int polydet_condense_batch(polydet_plan_t pl, const uint32_t *evals, int lo, int hi,
                                      uint32_t *detvals, void *stream) {
  if (check_range(pl, lo, hi) || !evals || !detvals) return POLYDET_EINVAL;
  const EvLayout lay = {pl->G, pl->G, pl->G};
  return pd_launch_condense(pl, evals, lay, lo, hi - lo, detvals, (cudaStream_t)stream);
}

// Streamed evaluation + condensation (multi-round evaluation of Sec. 3.1):
// the workspace holds one prime's head tensor (every variable but x_1
// evaluated) and, after it, the head passes' scratch, which the slabs of
// evaluated matrices reuse once the head is complete.
static int stream_quantum(const polydet_plan_s *pl) {
  return pl->full ? 1 : pl->LPo[0];  // slab starts on a coset of x_1 (node grid)
}

static uint64_t stream_head_words(const polydet_plan_s *pl) {
  return ((uint64_t)pl->nitems * pd_head_words(pl) + 63) / 64 * 64;
}

extern "C" uint64_t polydet_stream_ws_words(polydet_plan_t pl, int rows) {
  if (!pl || rows < 1) return 0;
  const int qn = stream_quantum(pl);
  rows = std::min(pl->M[0], (rows + qn - 1) / qn * qn);
  const uint64_t slab = (uint64_t)pl->nent * (uint64_t)pd_tail_layout(pl, rows).entry;
  return stream_head_words(pl) + std::max<uint64_t>(pd_head_ws_words(pl), slab);
}

extern "C" int polydet_eval_condense(polydet_plan_t pl, const int32_t *coeffs, int lo, int hi,
                                     uint32_t *detvals, uint32_t *ws, uint64_t ws_words, void *stream) {
  if (check_range(pl, lo, hi) || !coeffs || !detvals || !ws) return POLYDET_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  const int qn = stream_quantum(pl), M0 = pl->M[0];
  const uint64_t hw = stream_head_words(pl);
  if (ws_words < polydet_stream_ws_words(pl, 1)) return POLYDET_EINVAL;
  // slab rows: as many as the workspace holds, a multiple of the coset size
  const uint64_t row_words = (uint64_t)pl->nent * (uint64_t)pd_tail_layout(pl, 1).entry;
  int R = (int)std::min<uint64_t>((uint64_t)M0, (ws_words - hw) / std::max<uint64_t>(row_words, 1));
  if (R < M0) R = std::max(qn, R / qn * qn);
  uint32_t *head = ws, *rest = ws + hw;
  const int64_t B = pl->G / M0;
  for (int q = lo; q < hi; ++q) {
    int rc = pd_eval_head(pl, coeffs, q, q + 1, head, rest, st);
    if (rc) return rc;
    for (int r0 = 0; r0 < M0; r0 += R) {
      const int r1 = std::min(M0, r0 + R);
      const EvLayout lay = pd_tail_layout(pl, r1 - r0);
      rc = pd_eval_tail(pl, head, q, q, q + 1, r0, r1, rest, lay, st);
      if (rc) return rc;
      rc = pd_launch_condense_nodes(pl, rest, lay, (int64_t)(r1 - r0) * B, pl->G, q, 1,
                                    detvals + (int64_t)(q - lo) * pl->G + (int64_t)r0 * B, st);
      if (rc) return rc;
    }
  }
  return POLYDET_OK;
}
