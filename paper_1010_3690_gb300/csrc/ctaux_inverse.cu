// Blocked Gauss-Jordan inversion in place (see ctaux_inverse.cuh).
//
// Unblocked column step c (pivot row pr) maps X to
//   X[pr][j] / X[pr][c] (j != c), 1 / X[pr][c] at (pr, c),
//   -X[i][c] / X[pr][c] at (i, c), X[i][j] - X[i][c] X[pr][j] / X[pr][c] elsewhere.
// Blocked: for a panel C of 32 columns with pivot rows R, the column steps are
// applied to the panel alone, giving P' = X'[:, C]; every other column then
// follows in one rank-32 product
//   X'[:, J] = Z[:, J] + P' X[R, J],  Z = X with the rows R set to zero.
// After all panels, inv[c][perm[j]] = X[perm[c]][j].
// Pivots: the largest |value| over rows not yet pivoted, by a key of the upper
// half of the float64 magnitude (ties to the lower row).
//
// Three launches per panel:
//   k_inv_panel   one thread-block cluster per matrix holds the panel in its
//     distributed shared memory.  A column step costs one exchange of candidate
//     pivot rows (a grid barrier per column, the alternative, is 5-7 us on 152
//     SMs): every CTA pushes its own to all CTAs with stores that count at the
//     receivers' mbarriers, and the previous step's update of the other columns
//     runs while they travel.
//   k_inv_rows    the pivot rows of the other columns, sliced (ctaux_oz.cuh).
//   k_inv_update  the rank-32 product on the float16 tensor cores.
// Balance.  The product's error is relative to the largest element of a row of P'
// and of a column of X[R, J].  A pivot row's own scale r goes into its inner index
// as 1 / r in P' and as r in X[R, J], so in a matrix whose rows differ in scale the
// index with the largest multipliers loses the digits of exactly its own pivot row
// (rows scaled by 2^-27 to 2^27, order 64: error 1e-8 in place of 2e-14).  Inner
// index k is therefore scaled by the power of two 2^s_k, s_k = max_i (exponent of
// P'[i][k] - largest exponent in row i) <= 0, taken off P' and put on X[R, J]: the
// least that keeps every row's largest element, so that what an index adds to the
// error is bounded by its own terms.  It costs an exchange per panel in the cluster
// (order 310: 773 -> 794 us).
// N^{-1} = [e^V / (e^V - 1) - G0] (e^V - 1) has rows of one scale and goes without;
// scaled columns cancel by themselves.
// From order kInvTwoLevel on, two levels: the rank-32 products of four panels stay
// inside 128 columns, the rest of the matrix follows with one rank-128 product
// (k_inv_cols slices the 128 columns).  That reads and writes X, and runs the
// float64 epilogue, once per 128 columns instead of four times.
//
// One chain (two matrices), ms per recomputation, against the float64-pipe
// elimination with a grid barrier per column that this replaces: 2.8 -> 1.2 at
// order 431, 44 -> 8.0 at 2000, 1150 -> 79 at 6800 (where 1.06 TFLOP/s of
// float64 was the bound; now 16 TFLOP/s).
#include <cooperative_groups.h>

#include "ctaux_dev.cuh"
#include "ctaux_inverse.cuh"
#include "ctaux_oz.cuh"

namespace ctaux {

namespace {

constexpr int kMaxWidth = oz::kK;
constexpr int kMaxCluster = 16;
constexpr int kNoShift = -(1 << 16);   // below every difference of exponents

// Pivot key: the upper 32 bits of the float64 pattern of a magnitude (sign 0,
// the whole exponent, 20 significand bits) order like the magnitude for every
// non-negative double, so a normal entry, however small, beats an exact zero;
// ties within 2^-20 go to the lower row.
struct PivotKey {
  uint32_t mag, row;   // row complemented: the larger key has the lower row
};
__device__ __forceinline__ uint32_t magnitude(double v) {
  return (uint32_t)__double2hiint(v) & 0x7fffffffu;
}
__device__ __forceinline__ void key_max(PivotKey& a, uint32_t mag, uint32_t row) {
  if (mag > a.mag || (mag == a.mag && row > a.row)) {
    a.mag = mag;
    a.row = row;
  }
}
__device__ __forceinline__ PivotKey warp_key_max(PivotKey k) {
  PivotKey r;
  r.mag = __reduce_max_sync(0xffffffffu, k.mag);
  r.row = __reduce_max_sync(0xffffffffu, k.mag == r.mag ? k.row : 0u);
  return r;
}

// 1 / p by two Newton-Raphson steps y += y (1 - x y) on 64-bit fixed-point
// numbers, from a float32 reciprocal of the significand: within one unit in
// the last place, in about 350 clocks.  The same steps on the float64 pipe take
// 274 alone, but 900 to 1600 behind the other warps' updates, which hold that
// pipe 19 clocks per warp operation.  Zero, subnormal, infinite, NaN and
// extreme p divide.
__device__ __forceinline__ double reciprocal(double p) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(p);
  const int ex = (int)(bits >> 52) & 0x7ff;
  if (ex < 2 || ex > 2044) return 1.0 / p;
  const unsigned long long x = (bits << 11) | 0x8000000000000000ull;   // 2^64 x, x in [1/2, 1)
  float y0;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y0) : "f"((float)(uint32_t)(x >> 32) * 2.3283064365386963e-10f));
  unsigned long long y = (unsigned long long)__float2uint_rn(y0 * 1073741824.f) << 32;   // 2^62 / x
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const long long err = (long long)(0x4000000000000000ull - __umul64hi(x, y));   // 2^62 (1 - x y)
    y += (unsigned long long)__mul64hi((long long)(y >> 1), err * 8);   // |err| < 2^42
  }
  // y in [2^62, 2^63]: the power of two itself, or 53 bits after rounding
  const int top = (int)(y >> 63);
  const unsigned long long m = (y + (512ull << top)) >> (10 + top);   // [2^52, 2^53]
  const unsigned long long r = ((unsigned long long)(2044 - ex + top) << 52) + m;
  return __longlong_as_double((long long)(r | (bits & 0x8000000000000000ull)));
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_rank(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
// Store to another CTA's shared memory that counts 8 bytes at its mbarrier.
__device__ __forceinline__ void st_async(uint32_t addr, unsigned long long v, uint32_t mbar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(addr), "l"(v),
               "r"(mbar)
               : "memory");
}

// Column steps of panel [c0, c0 + width) of every matrix, one cluster per
// matrix, rows dealt to the CTAs in contiguous runs.  Step k makes column k its
// multipliers F[:, k] (-X[i][k] / pivot, and 1 / pivot in the pivot row) and
// updates only the columns to its right: with the pivot rows' multipliers
// L[k][l] = F[R_k][l], l < k, every column of the matrix, the panel's own ones
// included, follows as X'[:, j] = Z[:, j] + F y (k_inv_rows, k_inv_update).  F is
// written as slices, zero in a pivot row before its own step.
// Shared memory: the CTA's panel rows [column][row] and three generations of
// every CTA's candidate (key and row values): a CTA may push step k + 2's while
// another still updates with step k's.
// A step's critical chain is about 2500 clocks (exchange 540, selection 250,
// reciprocal 500, new column and key 600, candidate 400); beside it the update
// takes 19 clocks of the float64 pipe per column and 32 rows of a CTA, which
// bounds the step from about 200 rows per CTA on.  Keeping the update to the
// columns on the right halves that part.
template <int THREADS, bool BALANCE>
__global__ void __launch_bounds__(THREADS, THREADS == 512 ? 1 : 3)
k_inv_panel(const InvView* views, const int* orders, int c0, int width, int rows_cap) {
  constexpr int kWarps = THREADS / 32;
  const uint32_t rank = cluster_rank(), ncta = cluster_size();
  const int item = blockIdx.x / ncta;
  const int m = orders[item];
  if (c0 >= m) return;   // the whole cluster
  const InvView v = views[item];
  const int bw = min(width, m - c0);
  const int per = (m + (int)ncta - 1) / (int)ncta;
  const int r0 = min(m, (int)rank * per), nr = min(m, r0 + per) - r0, groups = (nr + 31) >> 5;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rs = rows_cap;   // row stride of a panel column

  extern __shared__ __align__(16) unsigned char panel_smem[];
  double* Ps = reinterpret_cast<double*>(panel_smem);          // [width][rs]
  double* crow = Ps + (size_t)width * rs;                      // [3][kMaxCluster][kMaxWidth]
  unsigned long long* ckey = reinterpret_cast<unsigned long long*>(crow + 3 * kMaxCluster * kMaxWidth);
  int8_t* us = reinterpret_cast<int8_t*>(ckey + 3 * kMaxCluster);   // [rs] 0 free, 1 pivoted before, 2 + k in step k
  int* shifts = reinterpret_cast<int*>(us + ((rs + 15) & ~15));     // with balance: [kMaxCluster][kMaxWidth]
  __shared__ uint32_t wmag[kWarps], wrow[kWarps];
  __shared__ double cand_row[kMaxWidth];
  __shared__ int shift[kMaxWidth];
  __shared__ uint64_t landed[3];   // candidates of a generation: one local arrival and their bytes
  __shared__ volatile int gave_up;
  const uint32_t bytes = ncta * (uint32_t)(sizeof(double) * kMaxWidth + sizeof(unsigned long long));

  for (int k = 0; k < bw; ++k)
    for (int r = tid; r < nr; r += THREADS) Ps[(size_t)k * rs + r] = v.X[(size_t)(c0 + k) * v.ld + r0 + r];
  for (int r = tid; r < nr; r += THREADS) us[r] = v.used[r0 + r];
  if (tid == 0) {
    gave_up = 0;
    for (int g = 0; g < 3; ++g) tc::mbar_init(tc::smem_u32(landed + g), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // remote shared memory may be written once every CTA of the cluster runs
  __syncthreads();
  cluster_arrive();
  cluster_wait();

  PivotKey key{0u, 0u};
  for (int r = tid; r < nr; r += THREADS)
    if (!us[r]) key_max(key, magnitude(Ps[r]), 0xffffffffu - (uint32_t)(r0 + r));

  int prl = -1;             // the previous pivot row, local (outside [0, nr) when another CTA's)
  const double* prow = nullptr;   // its values before the step

  for (int k = 0; k < bw; ++k) {
    // ---- the CTA's candidate
    const PivotKey wk = warp_key_max(key);
    if (lane == 0) {
      wmag[warp] = wk.mag;
      wrow[warp] = wk.row;
    }
    __syncthreads();
    const int gen = k % 3;
    const uint32_t bar = tc::smem_u32(landed + gen);
    const double* f = k > 0 ? Ps + (size_t)(k - 1) * rs : Ps;   // the previous step's multipliers
    PivotKey cand{0u, 0u};
    if (warp == 0) {
      double x = 0.0;
      if (lane < kWarps) cand = PivotKey{wmag[lane], wrow[lane]};
      cand = warp_key_max(cand);
      if (cand.row && lane < bw && lane >= k) {   // otherwise no row is left here
        const int lr = (int)(0xffffffffu - cand.row) - r0;
        x = Ps[(size_t)lane * rs + lr];
        if (k > 0 && lane != k) x = fma(f[lr], prow[lane], x);
      }
      cand_row[lane] = x;
      if (lane == 0) tc::mbar_expect_tx(bar, bytes);
    }
    __syncthreads();   // the candidate row is read before the update below changes it
    const uint32_t slot = (uint32_t)(gen * kMaxCluster + (int)rank);
    for (uint32_t w = (uint32_t)warp; w < ncta; w += kWarps)   // the row to every CTA, a warp each
      st_async(map_rank(tc::smem_u32(crow + slot * kMaxWidth + lane), w),
               (unsigned long long)__double_as_longlong(cand_row[lane]), map_rank(bar, w));
    if (warp == 0 && lane < (int)ncta)   // its key, a lane each
      st_async(map_rank(tc::smem_u32(ckey + slot), (uint32_t)lane),
               ((unsigned long long)cand.mag << 32) | cand.row, map_rank(bar, (uint32_t)lane));
    // ---- the previous step's update of the columns to its right, while the
    // candidates travel.  In the pivot row the multiplier is the reciprocal
    // pivot and the old value counts as zero: X[pr][j] / pivot comes from the
    // same multiply-add.
    if (k > 0) {
      if (k + 1 < bw) {   // column k + 1 by the threads that own its rows in this step
        const double pn = prow[k + 1];
        double* Pn = Ps + (size_t)(k + 1) * rs;
        for (int r = tid; r < nr; r += THREADS) Pn[r] = fma(f[r], pn, r == prl ? 0.0 : Pn[r]);
      }
      // the others a column per warp, a row per lane; warp 0 goes on to wait
      for (int j = warp == 0 ? bw : k + 1 + warp; j < bw; j += kWarps - 1) {
        const double pj = prow[j];
        double* Pj = Ps + (size_t)j * rs;
        // groups of 32 rows, four at a time; branches, not predicates: a float64
        // operation whose lanes are all masked holds the pipe as long as a real one
        int g = 0;
        for (; g + 4 <= groups; g += 4) {
          double x[4], y[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int r = (g + q) * 32 + lane;
            x[q] = r < nr && r != prl ? Pj[r] : 0.0;
            y[q] = r < nr ? f[r] : 0.0;
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) x[q] = fma(y[q], pj, x[q]);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if ((g + q) * 32 + lane < nr) Pj[(g + q) * 32 + lane] = x[q];
        }
#pragma unroll 1
        for (; g < groups; ++g) {
          const int r = g * 32 + lane;
          const double x = fma(r < nr ? f[r] : 0.0, pj, r < nr && r != prl ? Pj[r] : 0.0);
          if (r < nr) Pj[r] = x;
        }
      }
    }
    if (!__all_sync(0xffffffffu, tc::mbar_wait(bar, (uint32_t)(k / 3) & 1, gave_up ? 1u : tc::kWaitLimit))) {
      if (lane == 0) {   // the remaining steps run without waiting and without pivots
        atomicOr(v.status, DS_TIMEOUT);
        gave_up = 1;
      }
    }
    // ---- the pivot of column k, its column and the next one
    uint32_t mag = 0u, row = 0u;
    if (lane < (int)ncta) {
      const unsigned long long kk = ckey[gen * kMaxCluster + lane];
      mag = (uint32_t)(kk >> 32);
      row = (uint32_t)kk;
    }
    // ties go to the lower rank, which holds the lower rows
    const uint32_t best = __reduce_max_sync(0xffffffffu, row ? mag : 0u);
    const uint32_t winners = __ballot_sync(0xffffffffu, row != 0u && mag == best);
    const int who = winners ? __ffs(winners) - 1 : 0;
    const int pr = (int)(0xffffffffu - __shfl_sync(0xffffffffu, row, who));
    prow = crow + (size_t)(gen * kMaxCluster + who) * kMaxWidth;
    prl = pr - r0;
    if (rank == 0 && tid == 0 && pr >= 0 && pr < m) {
      const double piv = prow[k];
      v.perm[c0 + k] = pr;
      v.pcol[pr] = c0 + k;
      v.used[pr] = 1;
      v.piv[c0 + k] = piv;
      if (!(fabs(piv) > 0.0) || !isfinite(piv)) atomicOr(v.status, DS_SINGULAR);
    }
    key = PivotKey{0u, 0u};
    const double ipiv = warp * 32 < nr ? reciprocal(prow[k]) : 0.0;   // warps that own rows
    const bool next = k + 1 < bw;
    const double pn = next ? prow[k + 1] : 0.0;
    for (int r = tid; r < nr; r += THREADS) {
      const bool piv_row = r == prl;
      const double fr = (piv_row ? 1.0 : -Ps[(size_t)k * rs + r]) * ipiv;
      Ps[(size_t)k * rs + r] = fr;
      if (piv_row) us[r] = (int8_t)(2 + k);
      if (next) {
        const double xn = fma(fr, pn, piv_row ? 0.0 : Ps[(size_t)(k + 1) * rs + r]);
        Ps[(size_t)(k + 1) * rs + r] = xn;
        if (!us[r]) key_max(key, magnitude(xn), 0xffffffffu - (uint32_t)(r0 + r));
      }
    }
  }
  __syncthreads();
  if constexpr (BALANCE) {
    // ---- balance of the inner index: the CTA's rows, then all CTAs'
    if (tid < kMaxWidth) shift[tid] = kNoShift;
    __syncthreads();
    for (int e = tid; e < ((nr + 31) & ~31) * 4; e += THREADS) {   // the whole warp
      const int r = (e >> 7) * 32 + lane, ch = (e >> 5) & 3;
      const int step = r < nr ? max((int)us[r] - 2, 0) : bw;
      int mx = 0;
      for (int k = step; k < bw; ++k) mx = max(mx, oz::exp_field((uint32_t)__double2hiint(Ps[(size_t)k * rs + r])));
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const int k = ch * 8 + t;
        const int f = k >= step && k < bw ? oz::exp_field((uint32_t)__double2hiint(Ps[(size_t)k * rs + r])) : 0;
        // a row that is not finite has products that are not finite in any case
        const int s = __reduce_max_sync(0xffffffffu, f != 0 && mx != 0x7ff ? f - mx : kNoShift);
        if (lane == 0) atomicMax(shift + k, s);
      }
    }
    __syncthreads();
    for (uint32_t w = (uint32_t)warp; w < ncta; w += kWarps)
      asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(map_rank(tc::smem_u32(shifts + rank * kMaxWidth + lane), w)),
                   "r"(shift[lane])
                   : "memory");
    __syncwarp();
    cluster_arrive();
    cluster_wait();
    if (tid < kMaxWidth) {
      int s = kNoShift;
      for (uint32_t w = 0; w < ncta; ++w) s = max(s, shifts[w * kMaxWidth + tid]);
      shift[tid] = s == kNoShift ? 0 : s;
      if (rank == 0) v.balance[tid] = shift[tid];
    }
    __syncthreads();
  }
  cluster_arrive();   // no CTA exits while another may still store to it
  // ---- L, and the slices of F: four threads per row, 8 columns (one 16-byte
  // chunk of every slice) each
  for (int e = tid; e < ((nr + 31) & ~31) * 4; e += THREADS) {
    const int r = (e >> 7) * 32 + lane, ch = (e >> 5) & 3;
    if (r >= nr) continue;
    const int step = (int)us[r] - 2;   // of a pivot row of this panel
    if (step >= 0)
      for (int k = ch * 8; k < min(step, ch * 8 + 8); ++k) v.L[step * kMaxWidth + k] = Ps[(size_t)k * rs + r];
    int mx = 0, top = 0;   // the largest exponent field, balanced, and as it is
    for (int k = max(step, 0); k < bw; ++k) {
      const int f = oz::exp_field((uint32_t)__double2hiint(Ps[(size_t)k * rs + r]));
      top = max(top, f);
      if (BALANCE && f) mx = max(mx, f - shift[k]);
    }
    if (!BALANCE || top == 0x7ff) mx = top;
    const int row = r0 + r;
    unsigned char* img = v.As + (size_t)(row >> 7) * v.chunks * oz::kImageA + oz::chunk_offset(row & 127, ch);
    long long y[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int k = ch * 8 + t;
      y[t] = oz::biased_digits(k < bw && k >= step ? Ps[(size_t)k * rs + r] : 0.0, mx, BALANCE && top != 0x7ff ? -shift[k] : 0);
    }
    oz::store_chunk(img, oz::kRowsA, y);
    if (ch == 0) v.ea[row] = oz::row_exponent(mx);
  }
  __syncwarp();
  cluster_wait();
}

// A product's columns: [j0, j1), of rank 32 with the panel [c0, c0 + width)
// itself, of rank 128 without it (its columns are final then).
struct InvRange {
  int c0, width, j0, j1;
};
// The columns of a matrix of order m in the product of rank 32 with the panel from c0
// on: all, or the panel's own 128 in two levels.
__device__ __forceinline__ InvRange inv_range(int m, int c0, int width) {
  const bool two = m >= kInvTwoLevel;
  const int j0 = two ? c0 & ~127 : 0;
  return InvRange{c0, width, j0, two ? min(m, j0 + 128) : m};
}
// Whether it takes part in the product of rank 128.
__device__ __forceinline__ bool inv_wide(int m, int c0) { return m > c0 && m >= kInvTwoLevel; }

// The pivot rows of the panel, in the columns of the range, as slice images: a
// warp per column, a lane per pivot row.  Rank 32: y_k, the column at pivot row k
// just before step k, y_k = X[R_k][j] + sum_{l<k} L[k][l] y_l; the panel's own
// column c0 + k starts from the unit vector e_k.
template <bool BALANCE>
__global__ void __launch_bounds__(256) k_inv_rows(const InvView* views, const int* orders, int items, int width,
                                                  int c0, bool wide) {
  __shared__ int off[2 * kMaxChains + 1];
  for (int i = threadIdx.x; i < items; i += blockDim.x) {
    const int m = orders[i];
    const InvRange g = inv_range(m, c0, width);
    off[i] = wide ? (inv_wide(m, c0) ? (m + 7) / 8 : 0) : m > c0 ? (g.j1 - g.j0 + 7) / 8 : 0;
  }
  __syncthreads();
  block_exclusive_scan(off, items);
  const int total = off[items], lane = threadIdx.x & 31;
  for (int u = blockIdx.x; u < total; u += gridDim.x) {
    const int it = find_chain(off, items, u);
    const InvView& v = views[it];
    const int m = orders[it];
    const InvRange g = wide ? InvRange{c0, 128, 0, m} : inv_range(m, c0, width);
    const int bw = min(g.width, m - g.c0);
    const int j = g.j0 + (u - off[it]) * 8 + (threadIdx.x >> 5);
    const bool own = j >= g.c0 && j < g.c0 + bw;
    if (j >= g.j1 || (wide && own)) continue;   // the whole warp
    const int nc = (bw + oz::kK - 1) / oz::kK;
    double x[4];
    int mx = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int k = c * oz::kK + lane;
      x[c] = k >= bw ? 0.0 : own ? (j == g.c0 + k ? 1.0 : 0.0) : v.X[(size_t)j * v.ld + v.perm[g.c0 + k]];
    }
    if (!wide) {
      // forward substitution, a lane per row; eight multipliers in flight
      for (int l0 = 0; l0 < bw - 1; l0 += 8) {
        double lk[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) lk[t] = lane < bw && l0 + t < lane ? v.L[lane * kMaxWidth + l0 + t] : 0.0;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          if (l0 + t >= bw - 1) break;
          const double yl = __shfl_sync(0xffffffffu, x[0], l0 + t);
          x[0] = fma(lk[t], yl, x[0]);
        }
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) mx = max(mx, oz::exp_field((uint32_t)__double2hiint(x[c])));
    mx = __reduce_max_sync(0xffffffffu, mx);
    int shift = 0;
    if (BALANCE && mx != 0 && mx != 0x7ff) {   // (rank 32: x[0] alone)
      shift = lane < bw ? v.balance[lane] : 0;
      const int f = oz::exp_field((uint32_t)__double2hiint(x[0]));
      mx = __reduce_max_sync(0xffffffffu, f ? f + shift : kNoShift);
    }
    unsigned char* img = v.Bs + (size_t)(j >> 6) * v.chunks * oz::kImageB +
                         oz::chunk_offset(j & 63, lane >> 3) + (lane & 7) * 2;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (c >= nc) break;
      const long long y = oz::biased_digits(x[c], mx, shift);
#pragma unroll
      for (int i = 0; i < oz::kSlices; ++i)
        *reinterpret_cast<uint16_t*>(img + (size_t)c * oz::kImageB + (size_t)i * oz::kRowsB * 64) =
            oz::digit_half(oz::digit_u(y, i));
    }
    if (lane == 0) v.eb[j] = oz::row_exponent(mx);
  }
}

// The columns [c0, c0 + 128) of X as slice images, one exponent per row: a CTA
// stages 16 rows in shared memory, a thread then writes a 16-byte chunk of
// every slice of a row.
__global__ void __launch_bounds__(256) k_inv_cols(const InvView* views, const int* orders, int items, int c0) {
  __shared__ int off[2 * kMaxChains + 1];
  __shared__ double xs[128][17];
  __shared__ int mxs[16];
  for (int i = threadIdx.x; i < items; i += blockDim.x)
    off[i] = inv_wide(orders[i], c0) ? (orders[i] + 15) / 16 : 0;
  __syncthreads();
  block_exclusive_scan(off, items);
  const int total = off[items], r = threadIdx.x & 15, ch = threadIdx.x >> 4;
  for (int u = blockIdx.x; u < total; u += gridDim.x) {
    const int it = find_chain(off, items, u);
    const InvView& v = views[it];
    const int m = orders[it], bw = min(128, m - c0), row = (u - off[it]) * 16 + r;
    __syncthreads();   // the previous unit's readers are done
    if (threadIdx.x < 16) mxs[r] = 0;
    __syncthreads();
    int mx = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int k = ch + 16 * q;
      const double x = k < bw && row < m ? v.X[(size_t)(c0 + k) * v.ld + row] : 0.0;
      xs[k][r] = x;
      mx = max(mx, oz::exp_field((uint32_t)__double2hiint(x)));
    }
    atomicMax(&mxs[r], mx);
    __syncthreads();
    mx = mxs[r];
    if (row < m && ch < (bw + oz::kK - 1) / oz::kK * 4) {
      long long y[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) y[t] = oz::biased_digits(xs[ch * 8 + t][r], mx);
      oz::store_chunk(v.As + ((size_t)(row >> 7) * v.chunks + (ch >> 2)) * oz::kImageA +
                          oz::chunk_offset(row & 127, ch & 3), oz::kRowsA, y);
    }
    if (row < m && ch == 0) v.ea[row] = oz::row_exponent(mx);
  }
}

// X'[:, J] = Z[:, J] + F Y (rank 32; Z = 0 in the panel's own columns) or
// Z[:, J] + P' X[R, J] (rank 128) in 128 x 64 tiles: one persistent CTA per
// SM, warp 0 bulk copies (two stages of one image pair each), warp 1 the 68
// MMAs of a tile into the eight group accumulators (all 512 TMEM columns),
// warps 2-17 the epilogue (TMEM lane quarter w % 4, 16 columns each), which empties
// the accumulators into 64-bit integers first, so that the next tile's MMAs
// run while it adds to X on the float64 pipe.  Per tile: 34 x 2 MMAs of 48
// clocks (128 x 64 x 16, bound by shared-memory reads of A and B) against 8192
// float64 additions, 19 clocks per warp.  X's loads and additions hide behind
// the next tile's MMAs once the tile has been sent for (830 -> 741 us per rank-128
// product at order 6760, both spins, caches cold); what is left open is the
// emptying of the accumulators, with its conversions to integers (741 -> 732 us
// with four of them per element in place of six).  With the emptying cut to a
// quarter it took 590 us: shared memory, reads for the MMAs and writes of the bulk
// copies, is the bound there.
constexpr int kUpdStages = 2, kUpdThreads = 576;
constexpr int kUpdCols = 16;   // columns of an epilogue warp
constexpr int kUpdStageBytes = oz::kImageA + oz::kImageB;

struct UpdTile {
  int it, m, i0, j0;
};
template <bool WIDE>
__device__ __forceinline__ UpdTile upd_tile(const int* off, const int* orders, int items, int w, int c0) {
  UpdTile t;
  t.it = find_chain(off, items, w);
  t.m = orders[t.it];
  const int tm = (t.m + 127) / 128, l = w - off[t.it];
  t.i0 = (l % tm) * 128;
  t.j0 = (WIDE ? 0 : inv_range(t.m, c0, 0).j0) + (l / tm) * 64;
  return t;
}

// WIDE: rank 128 (up to four image pairs per tile), else rank 32.
template <bool WIDE>
__global__ void __launch_bounds__(kUpdThreads, 1)
k_inv_update(const InvView* views, const int* orders, int items, int width, int c0) {
  using namespace tc;
  __shared__ int off[2 * kMaxChains + 1];
  for (int i = threadIdx.x; i < items; i += blockDim.x) {
    const int m = orders[i], tm = (m + 127) / 128;
    const InvRange g = inv_range(m, c0, width);
    off[i] = WIDE ? (inv_wide(m, c0) ? tm * ((m + 63) / 64) : 0)
                  : m > c0 ? tm * ((g.j1 - g.j0 + 63) / 64) : 0;
  }
  __syncthreads();
  block_exclusive_scan(off, items);
  const int total = off[items];
  if ((int)blockIdx.x >= total) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  extern __shared__ __align__(1024) unsigned char upd_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>(((uintptr_t)upd_raw + 1023) & ~(uintptr_t)1023);
  __shared__ uint64_t full[kUpdStages], empty[kUpdStages], accfull, accempty, drain;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int err_s;

  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < kUpdStages; ++s) {
      mbar_init(smem_u32(full + s), 1);
      mbar_init(smem_u32(empty + s), 1);
    }
    mbar_init(smem_u32(&accfull), 1);
    mbar_init(smem_u32(&accempty), 16);
    mbar_init(smem_u32(&drain), 1);
    err_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  uint32_t issued = 0;
  auto fail = [&]() {   // tiles of any matrix may stay undone
    err_s = 1;
    for (int i = 0; i < items; ++i)
      if (orders[i] > 0) atomicOr(views[i].status, DS_TIMEOUT);
  };

  if (warp == 0 && lane == 0) {
    for (int w = blockIdx.x; w < total && !err_s; w += gridDim.x) {
      const UpdTile t = upd_tile<WIDE>(off, orders, items, w, c0);
      const InvView& v = views[t.it];
      const int nc = WIDE ? (min(128, t.m - c0) + oz::kK - 1) / oz::kK : 1;
      const unsigned char* sa = v.As + (size_t)(t.i0 >> 7) * v.chunks * oz::kImageA;
      const unsigned char* sb = v.Bs + (size_t)(t.j0 >> 6) * v.chunks * oz::kImageB;
      bool ok = true;
      for (int c = 0; c < nc && ok; ++c) {
        const uint32_t s = issued % kUpdStages, use = issued / kUpdStages;
        ok = use == 0 || mbar_wait(smem_u32(empty + s), (use - 1) & 1);
        if (!ok) break;
        const uint32_t fb = smem_u32(full + s), dst = smem_u32(base + s * kUpdStageBytes);
        mbar_expect_tx(fb, kUpdStageBytes);
        oz::bulk_load(dst, sa + (size_t)c * oz::kImageA, oz::kImageA, fb);
        oz::bulk_load(dst + oz::kImageA, sb + (size_t)c * oz::kImageB, oz::kImageB, fb);
        ++issued;
      }
      if (!ok) {
        fail();
        break;
      }
    }
    // every copy issued lands before the CTA may exit
    for (uint32_t i = issued > kUpdStages ? issued - kUpdStages : 0; i < issued; ++i)
      mbar_wait(smem_u32(full + i % kUpdStages), (i / kUpdStages) & 1);
  } else if (warp == 1) {   // all lanes wait, one issues
    uint32_t q = 0, taken = 0;
    for (int w = blockIdx.x; w < total; w += gridDim.x, ++q) {
      if (__any_sync(0xffffffffu, err_s != 0)) break;
      const UpdTile t = upd_tile<WIDE>(off, orders, items, w, c0);
      const int nc = WIDE ? (min(128, t.m - c0) + oz::kK - 1) / oz::kK : 1;
      bool ok = __all_sync(0xffffffffu, q == 0 || mbar_wait(smem_u32(&accempty), (q - 1) & 1));
      for (int c = 0; c < nc && ok; ++c, ++taken) {
        const uint32_t s = taken % kUpdStages;
        ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(full + s), (taken / kUpdStages) & 1));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t a = smem_u32(base + s * kUpdStageBytes);
        if (oz::elect_one()) {
          if (c == 0) oz::mma_images<true>(tmem, a, a + oz::kImageA);
          else oz::mma_images<false>(tmem, a, a + oz::kImageA);
          mma_commit(smem_u32(empty + s));
        }
        __syncwarp();
      }
      if (!ok) {
        if (lane == 0) fail();
        break;
      }
      if (oz::elect_one()) mma_commit(smem_u32(&accfull));
      __syncwarp();
    }
    if (oz::elect_one()) mma_commit(smem_u32(&drain));   // every MMA issued completes before the TMEM is freed
    __syncwarp();
    mbar_wait(smem_u32(&drain), 0);
  } else if (warp >= 2) {
    const int quarter = warp & 3, group = (warp - 2) >> 2;
    uint32_t q = 0;
    for (int w = blockIdx.x; w < total; w += gridDim.x, ++q) {
      const UpdTile t = upd_tile<WIDE>(off, orders, items, w, c0);
      const InvView& v = views[t.it];
      const InvRange g = WIDE ? InvRange{c0, 128, 0, t.m} : inv_range(t.m, c0, width);
      const int ld = v.ld, i = t.i0 + quarter * 32 + lane, jb = t.j0 + group * kUpdCols;
      const int cn = min(g.c0 + g.width, t.m), je = g.j1;
      const bool row_ok = i < t.m;
      const int pci = row_ok ? v.pcol[i] : -1;
      const bool load = row_ok && !(pci >= g.c0 && pci < cn);   // pivot rows start from zero
      const int ea = row_ok ? v.ea[i] - (WIDE ? 54 : 56) : 0;
      double* Xi = v.X + (size_t)jb * ld + i;
      {   // the warp's share of X towards L2 while the products run, a 128-byte line per lane
        const int pi = t.i0 + quarter * 32 + (lane & 1) * 16, pj = jb + (lane >> 1);
        if (pi < t.m && pj < je)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(v.X + (size_t)pj * ld + pi));
      }
      if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&accfull), q & 1, err_s ? 1u : kWaitLimit))) {
        if (lane == 0) fail();
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      long long S[kUpdCols];
      const uint32_t ta = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(group * kUpdCols);
#pragma unroll
      for (int cc = 0; cc < kUpdCols / 4; ++cc) {
        uint32_t r[oz::kGroups][4];
#pragma unroll
        for (int x = 0; x < oz::kGroups; ++x) oz::tmem_ld4(ta + (uint32_t)(64 * x + cc * 4), r[x]);
        oz::tmem_wait_ld();
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          uint32_t sums[oz::kGroups];
#pragma unroll
          for (int x = 0; x < oz::kGroups; ++x) sums[x] = r[x][e];
          S[cc * 4 + e] = WIDE ? oz::combine128(sums) : oz::combine(sums);
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&accempty));
      const int* eb = v.eb + jb;
      double z[kUpdCols];
#pragma unroll
      for (int e = 0; e < kUpdCols; ++e) {
        const int j = jb + e;
        z[e] = load && j < je && !(j >= g.c0 && j < cn) ? Xi[(size_t)e * ld] : 0.0;
      }
#pragma unroll
      for (int e = 0; e < kUpdCols; ++e) {
        const int j = jb + e;
        if (row_ok && j < je && !(WIDE && j >= g.c0 && j < cn))
          Xi[(size_t)e * ld] = z[e] + oz::scaled_double(S[e], ea + eb[e]);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

constexpr int kPanelSmem = 220 * 1024;
constexpr int upd_smem() { return kUpdStages * kUpdStageBytes + 1024; }

int panel_smem_bytes(int width, int rows, bool balance) {
  return (int)(sizeof(double) * ((size_t)width * rows + 3 * kMaxCluster * kMaxWidth) +
               sizeof(unsigned long long) * 3 * kMaxCluster + (size_t)((rows + 15) & ~15) +
               (balance ? sizeof(int) * kMaxCluster * kMaxWidth : 0));
}

}  // namespace

cudaError_t inv_device(int sm_count, bool balance, InvDevice* out) {
  *out = InvDevice{sm_count, 16, balance};
  auto attrs = [&](auto* fn, int bytes) {
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  };
  auto* panel512 = balance ? k_inv_panel<512, true> : k_inv_panel<512, false>;
  auto* panel256 = balance ? k_inv_panel<256, true> : k_inv_panel<256, false>;
  cudaError_t e = cudaFuncSetAttribute(panel512, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess) e = attrs(panel512, kPanelSmem);
  if (e == cudaSuccess) e = attrs(panel256, kPanelSmem);
  if (e == cudaSuccess) e = attrs(k_inv_update<false>, upd_smem());
  if (e == cudaSuccess) e = attrs(k_inv_update<true>, upd_smem());
  if (e != cudaSuccess) return e;
  // 16 CTAs need a GPC with that many free SMs
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(16);
  cfg.blockDim = dim3(512);
  cfg.dynamicSmemBytes = kPanelSmem;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = 16;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  int n = 0;
  e = cudaOccupancyMaxActiveClusters(&n, panel512, &cfg);
  if (n == 0) out->largest = 8;
  return e;
}

int inv_width(int ld, const InvDevice& dev) {
  int width = kMaxWidth;
  while (width > 4 && panel_smem_bytes(width, (ld + dev.largest - 1) / dev.largest, dev.balance) > kPanelSmem) width /= 2;
  return width;
}

// Cluster size per panel, from the matrices that can still reach it: 16 CTAs for
// a few (a GPC holds one such cluster; order 431 alone: 1.23 ms, against 1.35 with
// 8 and 1.48 with 4; order 2000: 8.3, 9.8, 13.2), 8 in batches (192 matrices of up
// to order 1084: 13.0 ms, 14.3 with 4; larger clusters pay where a batch's last,
// largest matrices are left), 4 beyond 256 matrices, whose rows fill the float64
// pipes of all SMs anyway.
std::vector<InvShape> inv_shapes(const std::vector<int>& lds, const InvDevice& dev) {
  std::vector<InvShape> out;
  for (int width = kMaxWidth; width >= 4; width /= 2) {
    InvShape s{dev, width, {}};
    int max_ld = 0;
    for (int ld : lds)
      if (inv_width(ld, dev) == width && ld > max_ld) max_ld = ld;
    if (max_ld == 0) continue;
    auto smem_of = [&](int cluster) { return panel_smem_bytes(width, (max_ld + cluster - 1) / cluster, dev.balance); };
    for (int c0 = 0; c0 < max_ld; c0 += width) {
      int active = 0;
      for (int ld : lds) active += ld > c0 && inv_width(ld, dev) == width;
      int cl = active <= 8 ? dev.largest : active <= 256 ? 8 : 4;
      while (cl < dev.largest && smem_of(cl) > kPanelSmem) cl *= 2;
      s.panels.push_back(InvPanel{cl, cl == 16 ? 512 : 256, (max_ld + cl - 1) / cl, smem_of(cl)});
    }
    out.push_back(s);
  }
  return out;
}

int launch_inverse(const InvView* views, const int* orders, int items, int max_order,
                   const InvShape& sh, cudaStream_t st, cudaError_t* err) {
  int n = 0;
  const int reach = (int)sh.panels.size() * sh.width;   // no order of this set is above it
  max_order = max_order < reach ? max_order : reach;
  auto grid = [&](long units, long most) { return (int)(units < most ? units : most); };
  const long rb = (max_order + 127) / 128, sms = sh.dev.sm_count;
  // the product of the panel from c0 on with up to `cols` columns of a matrix
  auto update = [&](int c0, bool wide, long cols) {
    auto* rows = sh.dev.balance ? k_inv_rows<true> : k_inv_rows<false>;
    rows<<<grid(items * ((cols + 7) / 8), 8 * sms), 256, 0, st>>>(views, orders, items, sh.width, c0, wide);
    const int ug = grid(items * rb * ((cols + 63) / 64), sms);
    if (wide) k_inv_update<true><<<ug, kUpdThreads, upd_smem(), st>>>(views, orders, items, sh.width, c0);
    else k_inv_update<false><<<ug, kUpdThreads, upd_smem(), st>>>(views, orders, items, sh.width, c0);
    n += 2;
  };
  for (int c0 = 0; c0 < max_order; c0 += sh.width) {
    const InvPanel& pn = sh.panels[c0 / sh.width];
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(items * pn.cluster));
    cfg.blockDim = dim3((unsigned)pn.threads);
    cfg.dynamicSmemBytes = (size_t)pn.smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)pn.cluster;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    auto* fn = pn.threads == 512 ? (sh.dev.balance ? k_inv_panel<512, true> : k_inv_panel<512, false>)
                                 : (sh.dev.balance ? k_inv_panel<256, true> : k_inv_panel<256, false>);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, fn, views, orders, c0, sh.width, pn.rows);
    n += 1;
    if (e != cudaSuccess) {
      *err = e;
      return n;
    }
    const int o0 = c0 / 128 * 128, next = c0 + sh.width;
    // (some order may be below the line also where the largest is above it)
    update(c0, false, max_order < kInvTwoLevel ? max_order : kInvTwoLevel);
    if (max_order >= kInvTwoLevel && (next % 128 == 0 || next >= max_order)) {
      k_inv_cols<<<grid(items * ((max_order + 15) / 16), 8 * sms), 256, 0, st>>>(views, orders, items, o0);
      n += 1;
      update(o0, true, max_order);
    }
  }
  *err = cudaGetLastError();
  return n;
}

}  // namespace ctaux
