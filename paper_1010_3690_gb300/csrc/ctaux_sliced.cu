// Prep and flush products of the float64 form on the float16 tensor cores
// (sliced operands, ctaux_oz.cuh):
//   prep 0: R~^T[j][a] = sum_{l<n} N[l][j] C[a][l]      -> N_ext[n + a][j]
//   prep 1: G[i][a]    = sum_{l<n} N[i][l] B[l][a]      -> Gcol[a][i]
//   prep 2: G[n+a][b]  = sum_{l<n} C[a][l] G[l][b] + G0 -> Gcol[b][n + a]
//   Y:      Y[a][r]    = sum_q (G - 1)[S_a][P_q] Gamma^{-1}[q][r]
//   flush:  N'[a][b]   = N[S_a][S_b] + sum_q (-Y)[a][q] N[P_q][S_b]
// On the float64 pipe (1/64 of the float32 rate) these were nine tenths of a
// block at 100 sites (per block of two chains: prep 86 -> 5.8 ms, Y 2.67 -> 0.25, flush 69 -> 2.6; at the
// 6 x 6 cluster 2.8 -> 0.41, 0.16 -> 0.06 and 1.33 -> 0.10).  Relative error of N after 8 blocks without recomputation,
// 6 x 6 cluster, sliced / on the float64 pipe: 2.1e-14 / 4.5e-14.
// Bound by the MMAs (68 per chunk of 32, 48 clocks each: shared-memory reads at
// N = 64) and, exposed between parts, by the 4 conversions per output of the
// eight accumulators that fill the TMEM.  The matrix side (N, N^T or Y) is the tensor cores' A
// operand, 128 rows per tile; the insertions or surviving columns are B, 64
// per tile.  Long inner dimensions are summed in parts of 128: within a part
// the integer sums are exact, every part has its own exponents per row, and
// the parts' float64 values are added in order.
#include "ctaux_dev.cuh"
#include "ctaux_kernels.h"
#include "ctaux_oz.cuh"
#include "ctaux_sliced.cuh"

namespace ctaux {

namespace {

using namespace tc;
static_assert(kSlicedImageA == oz::kImageA && kSlicedImageB == oz::kImageB, "image sizes of the host's layout");

// Four consecutive elements of a row (inner index 4 lane of a part) into every
// slice: 8 bytes per slice, a warp per row and part.
__device__ __forceinline__ void store_four(unsigned char* img, int image_rows, int image_bytes, int r, int lane,
                                           const double* x, int mx) {
  unsigned char* dst = img + (size_t)(lane >> 3) * image_bytes + oz::chunk_offset(r, (lane & 7) >> 1) + (lane & 1) * 8;
  long long y[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) y[t] = oz::biased_digits(x[t], mx);
#pragma unroll
  for (int i = 0; i < oz::kSlices; ++i) {
    uint2 q;
    q.x = oz::digits_half2(oz::digit_u(y[0], i), oz::digit_u(y[1], i));
    q.y = oz::digits_half2(oz::digit_u(y[2], i), oz::digit_u(y[3], i));
    *reinterpret_cast<uint2*>(dst + (size_t)i * image_rows * 64) = q;
  }
}

__device__ __forceinline__ int max_field4(const double* x) {
  int mx = 0;
#pragma unroll
  for (int t = 0; t < 4; ++t) mx = max(mx, oz::exp_field((uint32_t)__double2hiint(x[t])));
  return __reduce_max_sync(0xffffffffu, mx);
}

// A part of a contiguous row: elements [p 128 + 4 lane, + 4), zero from n on.
__device__ __forceinline__ void load_four(const double* row, int p, int lane, int n, double* x) {
  const int k = p * 128 + lane * 4;
#pragma unroll
  for (int t = 0; t < 4; ++t) x[t] = k + t < n ? row[k + t] : 0.0;
}

// Balance of the inner index.  N = D^{-1} (D^{-1} + 1 - G0)^{-1} with D = e^V - 1,
// so its rows differ by the factor D of their spins (320 at K = 1), which C (and
// Y) carry the other way round.  A row's slices resolve its largest element, so
// the matrix with the old vertices' rows along the inner index is scaled by the
// power of two of D and the other operand by its inverse (exact): every inner
// index then has the same scale, and the error stays relative to the largest
// terms of the sum, as in float64.
struct Balance {
  double up, down;   // for s = +1, -1
  __device__ __forceinline__ Balance(const Chain<double>& c, int spin, bool inverse)
      : up(scale(c.ev[spin][3] - 1.0, inverse)), down(scale(c.ev[spin][1] - 1.0, inverse)) {}
  __device__ __forceinline__ static double scale(double d, bool inverse) {
    const int ex = oz::exp_field((uint32_t)__double2hiint(d));
    if (ex < 64 || ex > 1982) return 1.0;
    return __hiloint2double((inverse ? 2046 - ex : ex) << 20, 0);
  }
  __device__ __forceinline__ double of(int s) const { return s > 0 ? up : s < 0 ? down : 1.0; }
};

// Sixteen rows x 128 inner elements val(k, r), zero for k >= kn and r >= rn, into
// images of ROWS rows: staged in shared memory, then a thread per row and 16-byte
// chunk.  256 threads.
struct StageRows {
  double xs[128][17];
  int mxs[16];
};
template <int ROWS, class F>
__device__ __forceinline__ void slice_rows(StageRows& st, int rn, int kn, F val, unsigned char* img, int r_in_image,
                                           int* exps, int exp_stride) {
  const int r = threadIdx.x & 15, ch = threadIdx.x >> 4;
  __syncthreads();   // the previous unit's readers are done
  if (threadIdx.x < 16) st.mxs[r] = 0;
  __syncthreads();
  int mx = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int k = ch + 16 * q;
    const double x = k < kn && r < rn ? val(k, r) : 0.0;
    st.xs[k][r] = x;
    mx = max(mx, oz::exp_field((uint32_t)__double2hiint(x)));
  }
  atomicMax(&st.mxs[r], mx);
  __syncthreads();
  mx = st.mxs[r];
  if (r < rn && ch < (kn + oz::kK - 1) / oz::kK * 4) {
    long long y[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) y[t] = oz::biased_digits(st.xs[ch * 8 + t][r], mx);
    oz::store_chunk(img + (size_t)(ch >> 2) * oz::kSlices * ROWS * 64 + oz::chunk_offset(r_in_image + r, ch & 3), ROWS, y);
  }
  if (r < rn && ch == 0) exps[(size_t)r * exp_stride] = oz::row_exponent(mx);
}

__device__ __forceinline__ void balance_four(double* x, const Chain<double>& c, const Balance& b, int p, int lane, int n) {
  const int k = p * 128 + lane * 4;
#pragma unroll
  for (int t = 0; t < 4; ++t)
    if (k + t < n) x[t] *= b.of(c.s0[k + t]);
}

// The panels C (rows) and B (columns) of every chain, a warp per (row, part).
__global__ void __launch_bounds__(256) k_slice_panels(const Chain<double>* chains, int n_chains,
                                                      const SlicedView* views) {
  __shared__ int off[kMaxChains + 1];
  for (int ci = threadIdx.x; ci < n_chains; ci += blockDim.x) {
    const Dyn& d = *chains[ci].dyn;
    off[ci] = d.status || !chains[ci].sliced ? 0 : 4 * ((d.k_ins + 7) / 8) * ((d.n + 127) / 128);
  }
  __syncthreads();
  block_exclusive_scan(off, n_chains);
  const int total = off[n_chains], warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int u = blockIdx.x; u < total; u += gridDim.x) {
    const int ci = find_chain(off, n_chains, u);
    const Chain<double>& c = chains[ci];
    const int n = c.dyn->n, k_ins = c.dyn->k_ins, parts = (n + 127) / 128;
    int l = u - off[ci];
    const int p = l % parts;
    l /= parts;
    const int job = l & 3, a = (l >> 2) * 8 + warp, spin = job >> 1, prod = job & 1;
    if (a >= k_ins) continue;
    const SlicedView& v = views[2 * ci + spin];
    double x[4];
    load_four((prod == 0 ? c.Cpan[spin] : c.Bpan[spin]) + (size_t)a * c.ld, p, lane, n, x);
    if (prod == 0) balance_four(x, c, Balance(c, spin, true), p, lane, n);
    const int mx = max_field4(x);
    store_four(v.cs[prod] + ((size_t)(a >> 6) * v.pl + p) * 4 * oz::kImageB, oz::kRowsB, oz::kImageB, a & 63, lane, x, mx);
    if (lane == 0) v.ce[prod][(size_t)a * v.pl + p] = oz::row_exponent(mx);
  }
}

// The columns of G_{old,new} of every chain, a warp per (column, part); their inner
// index is balanced against C's.
__global__ void __launch_bounds__(256) k_slice_g(const Chain<double>* chains, int n_chains, const SlicedView* views) {
  __shared__ int off[kMaxChains + 1];
  for (int ci = threadIdx.x; ci < n_chains; ci += blockDim.x) {
    const Dyn& d = *chains[ci].dyn;
    off[ci] = d.status || !chains[ci].sliced_new ? 0 : 2 * ((d.k_ins + 7) / 8) * ((d.n + 127) / 128);
  }
  __syncthreads();
  block_exclusive_scan(off, n_chains);
  const int total = off[n_chains], warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int u = blockIdx.x; u < total; u += gridDim.x) {
    const int ci = find_chain(off, n_chains, u);
    const Chain<double>& c = chains[ci];
    const int n = c.dyn->n, k_ins = c.dyn->k_ins, parts = (n + 127) / 128;
    int l = u - off[ci];
    const int p = l % parts;
    l /= parts;
    const int spin = l & 1, b = (l >> 1) * 8 + warp;
    if (b >= k_ins) continue;
    const SlicedView& v = views[2 * ci + spin];
    double x[4];
    load_four(c.Gcol[spin] + (size_t)b * c.ld, p, lane, n, x);
    balance_four(x, c, Balance(c, spin, false), p, lane, n);
    const int mx = max_field4(x);
    store_four(v.gs + ((size_t)(b >> 7) * v.pl + p) * 4 * oz::kImageA, oz::kRowsA, oz::kImageA, b & 127, lane, x, mx);
    if (lane == 0) v.ge[(size_t)b * v.pl + p] = oz::row_exponent(mx);
  }
}

// N (rows i, product 1) or N^T (rows j, product 0) of a strip's jobs: a CTA
// per 16 rows, all parts.
__global__ void __launch_bounds__(256) k_slice_n(const Chain<double>* chains, const SlicedView* views,
                                                 const SlicedJob* jobs, int n_jobs, unsigned char* pool, int* pool_exp) {
  extern __shared__ int joff[];
  __shared__ StageRows st;
  for (int i = threadIdx.x; i < n_jobs; i += blockDim.x) {
    const Dyn& d = *chains[jobs[i].ci].dyn;
    joff[i] = d.status || d.k_ins == 0 ? 0 : (d.n + 15) / 16;
  }
  __syncthreads();
  block_exclusive_scan(joff, n_jobs);
  const int total = joff[n_jobs], warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int u = blockIdx.x; u < total; u += gridDim.x) {
    const int ji = find_chain(joff, n_jobs, u);
    const SlicedJob jb = jobs[ji];
    const Chain<double>& c = chains[jb.ci];
    const int n = c.dyn->n, pl = views[2 * jb.ci].pl, parts = (n + 127) / 128, r0 = (u - joff[ji]) * 16;
    const double* N = c.N[c.dyn->buf][jb.spin];
    unsigned char* img = pool + jb.img + (size_t)(r0 >> 7) * pl * 4 * oz::kImageA;
    int* exps = pool_exp + jb.exps + (size_t)r0 * pl;
    if (jb.prod == 0) {
      const Balance bal(c, jb.spin, false);
      for (int e = warp; e < 16 * parts; e += 8) {
        const int r = e & 15, p = e >> 4;
        if (r0 + r >= n) continue;
        double x[4];
        load_four(N + (size_t)(r0 + r) * c.ld, p, lane, n, x);
        balance_four(x, c, bal, p, lane, n);
        const int mx = max_field4(x);
        store_four(img + (size_t)p * 4 * oz::kImageA, oz::kRowsA, oz::kImageA, (r0 + r) & 127, lane, x, mx);
        if (lane == 0) exps[(size_t)r * pl + p] = oz::row_exponent(mx);
      }
    } else {
      for (int p = 0; p < parts; ++p) {
        const double* src = N + (size_t)p * 128 * c.ld + r0;
        slice_rows<oz::kRowsA>(st, n - r0, n - p * 128, [&](int k, int r) { return src[(size_t)k * c.ld + r]; },
                               img + (size_t)p * 4 * oz::kImageA, r0 & 127, exps + p, pl);
      }
    }
  }
}

__device__ __forceinline__ int flush_rows(const Chain<double>& c) {
  const Dyn& d = *c.dyn;
  return !c.sliced || d.status || d.flush_noop || d.k_acc == 0 ? 0 : d.n_new;
}

// -Y (16 rows per CTA unit) and N[P, S] (16 columns per CTA unit) of every chain.
__global__ void __launch_bounds__(256) k_slice_flush(const Chain<double>* chains, int n_chains, const SlicedView* views) {
  __shared__ int off[kMaxChains + 1];
  __shared__ StageRows st;
  __shared__ double ys[kMaxK];   // minus the inverse balance of the touched slots
  for (int ci = threadIdx.x; ci < n_chains; ci += blockDim.x)
    off[ci] = 4 * ((flush_rows(chains[ci]) + 15) / 16);
  __syncthreads();
  block_exclusive_scan(off, n_chains);
  const int total = off[n_chains], warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int u = blockIdx.x; u < total; u += gridDim.x) {
    const int ci = find_chain(off, n_chains, u);
    const Chain<double>& c = chains[ci];
    const Dyn& d = *c.dyn;
    const int l = u - off[ci], spin = (l >> 1) & 1, r0 = (l >> 2) * 16, nn = d.n_new, ka = d.k_acc;
    const SlicedView& v = views[2 * ci + spin];
    if ((l & 1) == 0) {
      const Balance bal(c, spin, true);
      __syncthreads();
      for (int q = threadIdx.x; q < kMaxK; q += blockDim.x) ys[q] = q < ka ? -bal.of(c.s0[c.P[q]]) : 0.0;
      for (int p = 0; p * 128 < ka; ++p)   // starts with a barrier
      {
        const double* src = c.Y[spin] + (size_t)p * 128 * c.ld + r0;
        slice_rows<oz::kRowsA>(st, nn - r0, ka - p * 128,
                               [&](int k, int r) { return src[(size_t)k * c.ld + r] * ys[p * 128 + k]; },
                               v.ys + ((size_t)(r0 >> 7) * v.yc + p * 4) * oz::kImageA, r0 & 127,
                               v.ye + (size_t)r0 * 2 + p, 2);
      }
    } else {
      const double* N = c.N[d.buf][spin];
      const Balance bal(c, spin, false);
      for (int r = r0 + warp; r < min(nn, r0 + 16); r += 8) {
        const double* col = N + (size_t)c.S[r] * c.ld;
        for (int p = 0; p * 128 < ka; ++p) {
          double x[4];
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const int q = p * 128 + lane * 4 + t;
            x[t] = q < ka ? col[c.P[q]] * bal.of(c.s0[c.P[q]]) : 0.0;
          }
          const int mx = max_field4(x);
          // only the chunks that the product reads exist
          if (p * 4 + (lane >> 3) < (ka + oz::kK - 1) / oz::kK)
            store_four(v.xs + ((size_t)(r >> 6) * v.yc + p * 4) * oz::kImageB, oz::kRowsB, oz::kImageB, r & 63, lane, x, mx);
          if (lane == 0) v.xe[(size_t)r * 2 + p] = oz::row_exponent(mx);
        }
      }
    }
  }
}

// Balance of Y's inner index: the columns of G - 1 and the rows of Gamma^{-1} carry
// a slot's e^V inversely (a factor of 400 between the spins at K = 1; without a
// balance N lost three digits there in a block), and Gamma^{-1} is graded where it is
// nearly singular.  Column q is scaled by the power of two that brings its largest
// element and that of row q to the same size.  A CTA per q.
__global__ void __launch_bounds__(256) k_balance_y(const Chain<double>* chains, int n_chains, const SlicedView* views) {
  __shared__ int off[kMaxChains + 1], most[2];
  for (int ci = threadIdx.x; ci < n_chains; ci += blockDim.x)
    off[ci] = chains[ci].sliced_y && flush_rows(chains[ci]) ? 2 * chains[ci].dyn->k_acc : 0;
  __syncthreads();
  block_exclusive_scan(off, n_chains);
  const int total = off[n_chains];
  for (int u = blockIdx.x; u < total; u += gridDim.x) {
    const int ci = find_chain(off, n_chains, u);
    const Chain<double>& c = chains[ci];
    const Dyn& d = *c.dyn;
    const int l = u - off[ci], spin = l & 1, q = l >> 1, nn = d.n_new, ka = d.k_acc;
    if (threadIdx.x < 2) most[threadIdx.x] = 0;
    __syncthreads();
    const double *N = c.N[d.buf][spin], *Gc = c.Gcol[spin], *Gi = c.Ginv[spin] + (size_t)q * (c.k_max + 1);
    const int j = c.P[q];
    int mg = 0, mi = 0;
#pragma unroll 4
    for (int a = threadIdx.x; a < nn; a += blockDim.x) {
      const int i = c.S[a];
      mg = max(mg, oz::exp_field((uint32_t)__double2hiint(g_int<double>(c, N, Gc, d.n, spin, i, j) - (i == j ? 1.0 : 0.0))));
    }
    for (int r = threadIdx.x; r < ka; r += blockDim.x) mi = max(mi, oz::exp_field((uint32_t)__double2hiint(Gi[r])));
    mg = __reduce_max_sync(0xffffffffu, mg);
    mi = __reduce_max_sync(0xffffffffu, mi);
    if ((threadIdx.x & 31) == 0) {
      atomicMax(&most[0], mg);
      atomicMax(&most[1], mi);
    }
    __syncthreads();
    mg = most[0];
    mi = most[1];
    // zero, subnormal and non-finite rows and columns stay as they are
    if (threadIdx.x == 0) views[2 * ci + spin].qe[q] = mg == 0 || mg == 0x7ff || mi == 0 || mi == 0x7ff ? 0 : (mi - mg) / 2;
    __syncthreads();   // both read before the next unit clears them
  }
}

// G - 1 at the surviving rows and touched columns (16 rows per CTA unit) and the
// columns of Gamma^{-1} (16 per CTA unit) of every chain, in the images of -Y and
// N[P, S], which follow once Y is there.
__global__ void __launch_bounds__(256) k_slice_y(const Chain<double>* chains, int n_chains, const SlicedView* views) {
  __shared__ int off[kMaxChains + 1];
  __shared__ StageRows st;
  __shared__ int ps[kMaxK], si[16];
  __shared__ double bs[kMaxK];
  for (int ci = threadIdx.x; ci < n_chains; ci += blockDim.x) {
    const int nn = chains[ci].sliced_y ? flush_rows(chains[ci]) : 0;
    off[ci] = nn ? 2 * ((nn + 15) / 16 + (chains[ci].dyn->k_acc + 15) / 16) : 0;
  }
  __syncthreads();
  block_exclusive_scan(off, n_chains);
  const int total = off[n_chains];
  for (int u = blockIdx.x; u < total; u += gridDim.x) {
    const int ci = find_chain(off, n_chains, u);
    const Chain<double>& c = chains[ci];
    const Dyn& d = *c.dyn;
    const int l = u - off[ci], spin = l & 1, nn = d.n_new, ka = d.k_acc, rb = (nn + 15) / 16;
    const bool rows = (l >> 1) < rb;
    const int r0 = (rows ? l >> 1 : (l >> 1) - rb) * 16;
    const SlicedView& v = views[2 * ci + spin];
    __syncthreads();
    for (int q = threadIdx.x; q < ka; q += blockDim.x) {
      ps[q] = c.P[q];
      // |qe| <= 1023: a power of two within the normal range, or next to it
      bs[q] = __hiloint2double((1023 + max(-1022, min(1023, rows ? v.qe[q] : -v.qe[q]))) << 20, 0);
    }
    if (rows) {
      if (threadIdx.x < 16) si[threadIdx.x] = r0 + threadIdx.x < nn ? c.S[r0 + threadIdx.x] : 0;
    }
    for (int p = 0; p * 128 < ka; ++p) {   // starts with a barrier
      if (rows) {
        const double *N = c.N[d.buf][spin], *Gc = c.Gcol[spin];
        slice_rows<oz::kRowsA>(st, nn - r0, ka - p * 128,
                               [&](int k, int r) {
                                 const int i = si[r], j = ps[p * 128 + k];
                                 return (g_int<double>(c, N, Gc, d.n, spin, i, j) - (i == j ? 1.0 : 0.0)) * bs[p * 128 + k];
                               },
                               v.ys + ((size_t)(r0 >> 7) * v.yc + p * 4) * oz::kImageA, r0 & 127,
                               v.ye + (size_t)r0 * 2 + p, 2);
      } else {
        const double* Gi = c.Ginv[spin] + (size_t)p * 128 * (c.k_max + 1) + r0;
        slice_rows<oz::kRowsB>(st, ka - r0, ka - p * 128,
                               [&](int k, int r) { return Gi[(size_t)k * (c.k_max + 1) + r] * bs[p * 128 + k]; },
                               v.xs + ((size_t)(r0 >> 6) * v.yc + p * 4) * oz::kImageB, r0 & 63,
                               v.xe + (size_t)r0 * 2 + p, 2);
      }
    }
  }
}

// ------------------------------------------------------------- products
// One persistent CTA per SM: warp 0 bulk copies (two stages of one image
// pair), warp 1 the MMAs of a part into the eight group accumulators (all 512
// TMEM columns), warps 2-17 the epilogue, which empties them into 64-bit
// integers and adds the part's float64 values while the next part's MMAs run.
constexpr int kProdStages = 2, kProdThreads = 576, kProdCols = 16;
constexpr int kProdStageBytes = oz::kImageA + oz::kImageB;

struct ProdItem {
  const unsigned char *a, *b;   // first chunk's images
  const int *ea, *eb;           // exponents of the tile's rows and columns, first part
  int es_a, es_b;               // exponent strides between rows
  int chunks;                   // of this item (its parts' chunks, four each but the last)
  int m0, n0, M, N;             // tile origin and output sizes
  int ci, spin, prod, tile, slice, slices;
};

struct PrepSrc {
  const Chain<double>* chains;
  const SlicedView* views;
  const SlicedJob* jobs;
  int n;
  const unsigned char* pool;
  const int* pool_exp;
  __device__ __forceinline__ int chain(int i) const { return jobs[i].ci; }
  __device__ __forceinline__ bool takes(int) const { return true; }
  __device__ __forceinline__ int count(int i) const {
    const Dyn& d = *chains[jobs[i].ci].dyn;
    if (d.status || d.k_ins == 0 || d.n == 0) return 0;
    return ((d.n + 127) / 128) * ((d.k_ins + 63) / 64) * sliced_slices(d.n, d.k_ins);
  }
  __device__ __forceinline__ ProdItem item(int i, int l) const {
    const SlicedJob& jb = jobs[i];
    const Dyn& d = *chains[jb.ci].dyn;
    const SlicedView& v = views[2 * jb.ci + jb.spin];
    ProdItem t;
    t.ci = jb.ci;
    t.spin = jb.spin;
    t.prod = jb.prod;
    t.M = d.n;
    t.N = d.k_ins;
    t.slices = sliced_slices(d.n, d.k_ins);
    const int ct = (t.N + 63) / 64, parts = (d.n + 127) / 128;
    // consecutive items share the matrix rows (column tiles, then slices, then row blocks)
    const int c = l % ct, r = l / ct / t.slices;
    t.slice = l / ct % t.slices;
    t.tile = r * ct + c;
    const int p0 = (int)((long)parts * t.slice / t.slices), p1 = (int)((long)parts * (t.slice + 1) / t.slices);
    t.m0 = r * 128;
    t.n0 = c * 64;
    t.chunks = min(p1 * 4, (d.n + oz::kK - 1) / oz::kK) - p0 * 4;
    t.a = pool + jb.img + ((size_t)r * v.pl + p0) * 4 * oz::kImageA;
    t.b = v.cs[jb.prod] + ((size_t)c * v.pl + p0) * 4 * oz::kImageB;
    t.ea = pool_exp + jb.exps + (size_t)t.m0 * v.pl + p0;
    t.eb = v.ce[jb.prod] + (size_t)t.n0 * v.pl + p0;
    t.es_a = t.es_b = v.pl;
    return t;
  }
};

// G_{new,new}: rows are the columns b of G_{old,new}, columns the rows a of C.
struct NewSrc {
  const Chain<double>* chains;
  const SlicedView* views;
  int n;
  __device__ __forceinline__ int chain(int i) const { return i; }
  __device__ __forceinline__ bool takes(int i) const { return chains[i].sliced_new; }
  __device__ __forceinline__ int count(int i) const {
    const Dyn& d = *chains[i].dyn;
    if (!chains[i].sliced_new || d.status || d.k_ins == 0 || d.n == 0) return 0;
    return 2 * ((d.k_ins + 127) / 128) * ((d.k_ins + 63) / 64) * sliced_new_slices(d.n);
  }
  __device__ __forceinline__ ProdItem item(int i, int l) const {
    const Dyn& d = *chains[i].dyn;
    ProdItem t;
    t.ci = i;
    t.spin = l & 1;
    l >>= 1;
    const SlicedView& v = views[2 * i + t.spin];
    t.prod = 3;
    t.M = t.N = d.k_ins;
    t.slices = sliced_new_slices(d.n);
    const int ct = (t.N + 63) / 64, parts = (d.n + 127) / 128;
    t.slice = l % t.slices;
    t.tile = l / t.slices;
    const int r = t.tile / ct, c = t.tile % ct;
    const int p0 = (int)((long)parts * t.slice / t.slices), p1 = (int)((long)parts * (t.slice + 1) / t.slices);
    t.m0 = r * 128;
    t.n0 = c * 64;
    t.chunks = min(p1 * 4, (d.n + oz::kK - 1) / oz::kK) - p0 * 4;
    t.a = v.gs + ((size_t)r * v.pl + p0) * 4 * oz::kImageA;
    t.b = v.cs[0] + ((size_t)c * v.pl + p0) * 4 * oz::kImageB;
    t.ea = v.ge + (size_t)t.m0 * v.pl + p0;
    t.eb = v.ce[0] + (size_t)t.n0 * v.pl + p0;
    t.es_a = t.es_b = v.pl;
    return t;
  }
};

struct FlushSrc {
  const Chain<double>* chains;
  const SlicedView* views;
  int n;
  __device__ __forceinline__ int chain(int i) const { return i; }
  __device__ __forceinline__ bool takes(int i) const { return chains[i].sliced; }
  __device__ __forceinline__ int count(int i) const {
    const int nn = flush_rows(chains[i]);
    return 2 * ((nn + 127) / 128) * ((nn + 63) / 64);
  }
  __device__ __forceinline__ ProdItem item(int i, int l) const {
    const Dyn& d = *chains[i].dyn;
    ProdItem t;
    t.ci = i;
    t.M = t.N = d.n_new;
    const int tm = (t.M + 127) / 128, tn = (t.N + 63) / 64;
    t.spin = l / (tm * tn);
    l -= t.spin * tm * tn;
    const SlicedView& v = views[2 * i + t.spin];
    t.m0 = (l % tm) * 128;
    t.n0 = (l / tm) * 64;
    t.chunks = (d.k_acc + oz::kK - 1) / oz::kK;
    t.a = v.ys + (size_t)(t.m0 >> 7) * v.yc * oz::kImageA;
    t.b = v.xs + (size_t)(t.n0 >> 6) * v.yc * oz::kImageB;
    t.ea = v.ye + (size_t)t.m0 * 2;
    t.eb = v.xe + (size_t)t.n0 * 2;
    t.es_a = t.es_b = 2;
    t.prod = t.tile = t.slice = 0;
    t.slices = 1;
    return t;
  }
};

struct YSrc {
  const Chain<double>* chains;
  const SlicedView* views;
  int n;
  __device__ __forceinline__ int chain(int i) const { return i; }
  __device__ __forceinline__ bool takes(int i) const { return chains[i].sliced_y; }
  __device__ __forceinline__ int count(int i) const {
    const int nn = chains[i].sliced_y ? flush_rows(chains[i]) : 0;
    return nn ? 2 * ((nn + 127) / 128) * ((chains[i].dyn->k_acc + 63) / 64) : 0;
  }
  __device__ __forceinline__ ProdItem item(int i, int l) const {
    const Dyn& d = *chains[i].dyn;
    ProdItem t;
    t.ci = i;
    t.M = d.n_new;
    t.N = d.k_acc;
    const int tm = (t.M + 127) / 128, tn = (t.N + 63) / 64;
    t.spin = l / (tm * tn);
    l -= t.spin * tm * tn;
    const SlicedView& v = views[2 * i + t.spin];
    t.m0 = (l / tn) * 128;
    t.n0 = (l % tn) * 64;
    t.chunks = (d.k_acc + oz::kK - 1) / oz::kK;
    t.a = v.ys + (size_t)(t.m0 >> 7) * v.yc * oz::kImageA;
    t.b = v.xs + (size_t)(t.n0 >> 6) * v.yc * oz::kImageB;
    t.ea = v.ye + (size_t)t.m0 * 2;
    t.eb = v.xe + (size_t)t.n0 * 2;
    t.es_a = t.es_b = 2;
    t.prod = 2;
    t.tile = t.slice = 0;
    t.slices = 1;
    return t;
  }
};

// A wait of more than wl polls gives up: the CTA stops, and every chain of the launch
// gets DS_TIMEOUT, since the CTA may leave items of any of them undone and a CTA that
// starts later finds other work lists (split-K arrivals are then incomplete;
// ctaux_set_config clears them with the status).  With `stall` set (a test of this
// path) the MMA issuer of CTA 0 first waits on a barrier that nothing completes, until
// the chain of its first item has been recomputed twice.
template <class Src, bool FLUSH>
__global__ void __launch_bounds__(kProdThreads, 1) k_sliced_product(Src src, uint32_t wl, int stall) {
  extern __shared__ __align__(1024) unsigned char prod_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>(((uintptr_t)prod_raw + 1023) & ~(uintptr_t)1023);
  int* off = reinterpret_cast<int*>(base + kProdStages * kProdStageBytes);
  __shared__ uint64_t full[kProdStages], empty[kProdStages], accfull, accempty, drain, never;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int err_s;
  for (int i = threadIdx.x; i < src.n; i += blockDim.x) off[i] = src.count(i);
  __syncthreads();
  block_exclusive_scan(off, src.n);
  const int total = off[src.n];
  if ((int)blockIdx.x >= total) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto item = [&](int w) {
    const int i = find_chain(off, src.n, w);
    return src.item(i, w - off[i]);
  };
  auto fail = [&]() {
    err_s = 1;
    for (int i = 0; i < src.n; ++i)
      if (src.takes(i)) atomicOr(&src.chains[src.chain(i)].dyn->status, DS_TIMEOUT);
  };

  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < kProdStages; ++s) {
      mbar_init(smem_u32(full + s), 1);
      mbar_init(smem_u32(empty + s), 1);
    }
    mbar_init(smem_u32(&accfull), 1);
    mbar_init(smem_u32(&accempty), 16);
    mbar_init(smem_u32(&drain), 1);
    mbar_init(smem_u32(&never), 1);
    err_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;

  if (warp == 0 && lane == 0) {
    uint32_t issued = 0;
    for (int w = blockIdx.x; w < total && !err_s; w += gridDim.x) {
      const ProdItem t = item(w);
      bool ok = true;
      for (int c = 0; c < t.chunks; ++c) {
        const uint32_t s = issued % kProdStages, use = issued / kProdStages;
        ok = use == 0 || mbar_wait(smem_u32(empty + s), (use - 1) & 1, wl);
        if (!ok) break;
        const uint32_t fb = smem_u32(full + s), dst = smem_u32(base + s * kProdStageBytes);
        mbar_expect_tx(fb, kProdStageBytes);
        oz::bulk_load(dst, t.a + (size_t)c * oz::kImageA, oz::kImageA, fb);
        oz::bulk_load(dst + oz::kImageA, t.b + (size_t)c * oz::kImageB, oz::kImageB, fb);
        ++issued;
      }
      if (!ok) {
        fail();
        break;
      }
    }
    // every copy issued lands before the CTA may exit
    for (uint32_t i = issued > kProdStages ? issued - kProdStages : 0; i < issued; ++i)
      mbar_wait(smem_u32(full + i % kProdStages), (i / kProdStages) & 1);
  } else if (warp == 1) {   // all lanes wait, one issues
    uint32_t q = 0, taken = 0;
    bool ok = true;
    if (stall && blockIdx.x == 0 && src.chains[item(0).ci].dyn->refreshes < 2)
      ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&never), 0, wl));
    if (!ok && lane == 0) fail();
    __syncwarp();
    for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
      if (__any_sync(0xffffffffu, err_s != 0)) break;
      const ProdItem t = item(w);
      for (int c0 = 0; c0 < t.chunks && ok; c0 += 4, ++q) {
        ok = __all_sync(0xffffffffu, q == 0 || mbar_wait(smem_u32(&accempty), (q - 1) & 1, wl));
        for (int c = c0; c < min(t.chunks, c0 + 4) && ok; ++c, ++taken) {
          const uint32_t s = taken % kProdStages;
          ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(full + s), (taken / kProdStages) & 1, wl));
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t a = smem_u32(base + s * kProdStageBytes);
          if (oz::elect_one()) {
            if (c == c0) oz::mma_images<true>(tmem, a, a + oz::kImageA);
            else oz::mma_images<false>(tmem, a, a + oz::kImageA);
            mma_commit(smem_u32(empty + s));
          }
          __syncwarp();
        }
        if (ok && oz::elect_one()) mma_commit(smem_u32(&accfull));
        __syncwarp();
      }
      if (!ok && lane == 0) fail();
      __syncwarp();
    }
    if (oz::elect_one()) mma_commit(smem_u32(&drain));   // every MMA issued completes before the TMEM is freed
    __syncwarp();
    mbar_wait(smem_u32(&drain), 0);
  } else if (warp >= 2) {
    const int quarter = warp & 3, group = (warp - 2) >> 2, rl = quarter * 32 + lane, cl = group * kProdCols;
    uint32_t q = 0;
    for (int w = blockIdx.x; w < total; w += gridDim.x) {
      const ProdItem t = item(w);
      const Chain<double>& c = src.chains[t.ci];
      const Dyn& d = *c.dyn;
      const int i = t.m0 + rl, ld = c.ld;
      const bool row_ok = i < t.M;
      double z[kProdCols];
      if constexpr (FLUSH) {   // N[S_i][S_j]
        const double* Ni = c.N[d.buf][t.spin] + (row_ok ? c.S[i] : 0);
#pragma unroll
        for (int e = 0; e < kProdCols; ++e) {
          const int j = t.n0 + cl + e;
          z[e] = row_ok && j < t.N ? Ni[(size_t)c.S[j] * ld] : 0.0;
        }
      } else {
#pragma unroll
        for (int e = 0; e < kProdCols; ++e) z[e] = 0.0;
      }
      const uint32_t ta = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)cl;
      const int* pa = t.ea + (size_t)(row_ok ? rl : 0) * t.es_a;
      const int* pb = t.eb + (size_t)cl * t.es_b;
      bool ok = true;
      for (int c0 = 0; c0 < t.chunks; c0 += 4, ++q, ++pa, ++pb) {
        const int ea = *pa - 54;
        ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&accfull), q & 1, err_s ? 1u : wl));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        long long S[kProdCols];
#pragma unroll
        for (int cc = 0; cc < kProdCols / 4; ++cc) {
          uint32_t r[oz::kGroups][4];
#pragma unroll
          for (int x = 0; x < oz::kGroups; ++x) oz::tmem_ld4(ta + (uint32_t)(64 * x + cc * 4), r[x]);
          oz::tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            uint32_t sums[oz::kGroups];
#pragma unroll
            for (int x = 0; x < oz::kGroups; ++x) sums[x] = r[x][e];
            S[cc * 4 + e] = oz::combine128(sums);
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&accempty));
#pragma unroll
        for (int e = 0; e < kProdCols; ++e) z[e] += oz::scaled_double(S[e], ea + pb[(size_t)e * t.es_b]);
      }
      if (!ok) {
        if (lane == 0) fail();
        break;
      }
      if constexpr (!FLUSH) {
        if (t.slices > 1) {   // partial tiles, added in slice order by the last to arrive
          const SlicedView& v = src.views[2 * t.ci + t.spin];
          // (a warp's 32 x 16 share of the tile by itself: no barrier)
          double* part = (t.prod == 3 ? v.gpart : v.part[t.prod]) + (size_t)t.tile * t.slices * 8192 + cl * 128 + rl;
#pragma unroll
          for (int e = 0; e < kProdCols; ++e) part[(size_t)t.slice * 8192 + e * 128] = z[e];
          __threadfence();
          __syncwarp();
          int* ticket = (t.prod == 3 ? v.gticket : v.ticket[t.prod]) + t.tile * 16 + warp - 2;
          int arrived = 0;
          if (lane == 0) arrived = atomicAdd(ticket, 1);
          if (__shfl_sync(0xffffffffu, arrived, 0) != t.slices - 1) continue;
          __threadfence();
#pragma unroll
          for (int e = 0; e < kProdCols; ++e) z[e] = 0.0;
          for (int x = 0; x < t.slices; ++x) {
#pragma unroll
            for (int e = 0; e < kProdCols; ++e) z[e] += __ldcg(part + (size_t)x * 8192 + e * 128);
          }
          if (lane == 0) *ticket = 0;
        }
      }
      if (!row_ok) continue;
      if constexpr (FLUSH) {
        double* out = c.N[1 - d.buf][t.spin] + i;
#pragma unroll
        for (int e = 0; e < kProdCols; ++e)
          if (t.n0 + cl + e < t.N) out[(size_t)(t.n0 + cl + e) * ld] = z[e];
      } else {
        double* out = t.prod == 0   ? c.N[d.buf][t.spin] + (size_t)i * ld + d.n
                      : t.prod == 1 ? c.Gcol[t.spin] + i
                      : t.prod == 2 ? c.Y[t.spin] + i
                                    : c.Gcol[t.spin] + (size_t)i * ld + d.n;
        const size_t cs = t.prod == 0 || t.prod == 3 ? 1 : (size_t)ld;
        if (t.prod == 3) {   // onto G0(new, new)
#pragma unroll
          for (int e = 0; e < kProdCols; ++e)
            if (t.n0 + cl + e < t.N) z[e] += out[t.n0 + cl + e];
        }
#pragma unroll
        for (int e = 0; e < kProdCols; ++e)
          if (t.n0 + cl + e < t.N) out[(size_t)(t.n0 + cl + e) * cs] = z[e];
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

int prod_smem(int n) { return kProdStages * kProdStageBytes + 1024 + (int)sizeof(int) * (n + 1); }

}  // namespace

// The limits hold for the process: for the most chains and jobs (four per chain).
cudaError_t configure_sliced() {
  const cudaFuncAttribute dyn = cudaFuncAttributeMaxDynamicSharedMemorySize;
  constexpr int kMaxJobs = 4 * kMaxChains;
  cudaError_t e = cudaFuncSetAttribute(k_sliced_product<PrepSrc, false>, dyn, prod_smem(kMaxJobs));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_slice_n, dyn, (int)sizeof(int) * (kMaxJobs + 1));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_sliced_product<NewSrc, false>, dyn, prod_smem(kMaxChains));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_sliced_product<YSrc, false>, dyn, prod_smem(kMaxChains));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_sliced_product<FlushSrc, true>, dyn, prod_smem(kMaxChains));
  return e;
}

namespace {
template <class Src, bool FLUSH>
void launch_product(const Src& src, const LaunchShape& ls, cudaStream_t st) {
  const int lim = ls.tc_wait_limit;
  const uint32_t wl = lim > 0 ? (uint32_t)lim : lim < 0 ? (uint32_t)(-(int64_t)lim) : kWaitLimit;
  k_sliced_product<Src, FLUSH><<<ls.tc_ctas, kProdThreads, prod_smem(src.n), st>>>(src, wl, lim < 0 ? 1 : 0);
}
}  // namespace

int launch_sliced_prep(const Chain<double>* dchains, const LaunchShape& ls, cudaStream_t st) {
  const SlicedPlan& p = ls.sliced;
  int n = 1;
  k_slice_panels<<<ls.persist_ctas, 256, 0, st>>>(dchains, ls.n_chains, p.views);
  for (int s = 0; s < p.n_strips; ++s, n += 2) {
    const SlicedStrip& sp = p.strips[s];
    const SlicedJob* jobs = p.jobs + sp.first;
    k_slice_n<<<ls.persist_ctas, 256, sizeof(int) * (sp.count + 1), st>>>(dchains, p.views, jobs, sp.count, p.pool,
                                                                         p.pool_exp);
    const PrepSrc src{dchains, p.views, jobs, sp.count, p.pool, p.pool_exp};
    launch_product<PrepSrc, false>(src, ls, st);
  }
  if (ls.any_sliced_new) {
    k_slice_g<<<ls.persist_ctas, 256, 0, st>>>(dchains, ls.n_chains, p.views);
    const NewSrc src{dchains, p.views, ls.n_chains};
    launch_product<NewSrc, false>(src, ls, st);
    n += 2;
  }
  return n;
}

int launch_sliced_y(const Chain<double>* dchains, const LaunchShape& ls, cudaStream_t st) {
  k_balance_y<<<ls.persist_ctas, 256, 0, st>>>(dchains, ls.n_chains, ls.sliced.views);
  k_slice_y<<<ls.persist_ctas, 256, 0, st>>>(dchains, ls.n_chains, ls.sliced.views);
  const YSrc src{dchains, ls.sliced.views, ls.n_chains};
  launch_product<YSrc, false>(src, ls, st);
  return 3;
}

int launch_sliced_flush(const Chain<double>* dchains, const LaunchShape& ls, cudaStream_t st) {
  k_slice_flush<<<ls.persist_ctas, 256, 0, st>>>(dchains, ls.n_chains, ls.sliced.views);
  const FlushSrc src{dchains, ls.sliced.views, ls.n_chains};
  launch_product<FlushSrc, true>(src, ls, st);
  return 2;
}

}  // namespace ctaux
