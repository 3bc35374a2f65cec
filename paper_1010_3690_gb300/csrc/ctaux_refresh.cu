// From-scratch FP64 recomputation of N for every chain: build
// N^{-1} = e^V - G0 (e^V - 1) (Eq. Nmatrix) of both spins from the
// configuration, invert it (ctaux_inverse.cu), report the drift of the running
// N and replace it.  Both precision forms eliminate in float64 accuracy on the
// tensor cores, which is also the fastest form: the double-float elimination
// that the mixed form offered as an option took 20 ms at n = 2085.
#include "ctaux_inverse.cuh"
#include "ctaux_refresh.cuh"

namespace ctaux {

namespace {

// Orders of the matrices (chain, spin) that take part: all chains, or one.  With
// several panel widths, those of each as well.
struct InvWidths {
  int count, w[4];
};
template <typename T>
__global__ void k_refresh_orders(const Chain<T>* chains, int n_chains, int only_chain, int* orders,
                                 const InvView* views, InvWidths widths, RefreshOrders ro) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 2 * n_chains) return;
  const int ci = i >> 1;
  Dyn& d = *chains[ci].dyn;
  bool take = (only_chain < 0 || only_chain == ci) && !(d.status & ~DS_SINGULAR);
  if (take && d.n > ro.bound) {
    atomicOr(&d.status, DS_NUMERIC);
    take = false;
  }
  if (ro.seen && !(i & 1)) ro.seen[ci] = ((unsigned long long)ro.number << 32) | (unsigned)d.n;
  orders[i] = take ? d.n : 0;
  for (int s = 0; s < widths.count; ++s)
    orders[(size_t)(1 + s) * 2 * n_chains + i] = take && views[i].width == widths.w[s] ? d.n : 0;
}

// N^{-1} into X: kBuildCols columns by kBuildRows rows per CTA and unit, so that
// a thread's conversion of its row's time serves kBuildCols entries.
// Bounded by the FP64 pipe and the table gathers: 2.46 -> 0.82 ms at n = 6760 (both spins).
constexpr int kBuildCols = 8, kBuildRows = 1024;

template <typename T>
__global__ void __launch_bounds__(256) k_refresh_build(const Chain<T>* chains, const InvView* views,
                                                       const int* orders, int items) {
  __shared__ int off[2 * kMaxChains + 1];
  __shared__ long long tj[kBuildCols];
  __shared__ double emj[kBuildCols];
  __shared__ int sj[kBuildCols];
  for (int i = threadIdx.x; i < items; i += blockDim.x) {
    const int m = orders[i];
    off[i] = ((m + kBuildCols - 1) / kBuildCols) * ((m + kBuildRows - 1) / kBuildRows);
  }
  __syncthreads();
  block_exclusive_scan(off, items);
  const int total = off[items];
  for (int u = blockIdx.x; u < total; u += gridDim.x) {
    const int it = find_chain(off, items, u), m = orders[it], spin = it & 1, w = u - off[it];
    const Chain<T>& c = chains[it >> 1];
    const InvView& v = views[it];
    const double* tau = c.tau[c.dyn->buf];
    const int* site = c.site[c.dyn->buf];
    const int8_t* s = c.s[c.dyn->buf];
    const int groups = (m + kBuildCols - 1) / kBuildCols;
    const int j0 = w % groups * kBuildCols, i0 = w / groups * kBuildRows;
    __syncthreads();   // the previous unit's readers are done
    if (threadIdx.x < kBuildCols && j0 + threadIdx.x < m) {
      const int j = j0 + threadIdx.x;
      tj[threadIdx.x] = tau_fix(c, tau[j]);
      sj[threadIdx.x] = site[j];
      emj[threadIdx.x] = c.ev[spin][s[j] + 2] - 1.0;
      if (i0 == 0) {
        v.used[j] = 0;
        v.pcol[j] = -1;
      }
    }
    __syncthreads();
    const int nj = min(kBuildCols, m - j0);
    for (int i = i0 + threadIdx.x; i < min(m, i0 + kBuildRows); i += blockDim.x) {
      const long long ti = tau_fix(c, tau[i]);
      const int si = site[i];
#pragma unroll
      for (int q = 0; q < kBuildCols; ++q) {
        if (q >= nj) break;
        const int j = j0 + q;
        double g;
        if (!g0_fixed(c, g0_row(c, spin, si, sj[q]), ti - tj[q], g)) g = g0_eval(c, spin, tau[i], si, tau[j], sj[q]);
        double x = -g * emj[q];
        if (i == j) x += c.ev[spin][s[j] + 2];
        v.X[(size_t)j * v.ld + i] = x;
      }
    }
  }
}

// The inverse into N, with the drift; the pivot flags cleared for the next user.
template <typename T>
__global__ void __launch_bounds__(256) k_refresh_store(const Chain<T>* chains, const InvView* views,
                                                       const int* orders, int items) {
  __shared__ int off[2 * kMaxChains + 1];
  __shared__ double red[3][8];
  for (int i = threadIdx.x; i < items; i += blockDim.x) {
    const bool ok = !(chains[i >> 1].dyn->status & ~DS_SINGULAR);   // no wait gave up
    off[i] = ok ? orders[i] : 0;
  }
  __syncthreads();
  block_exclusive_scan(off, items);
  const int total = off[items];
  for (int u = blockIdx.x; u < total; u += gridDim.x) {
    const int it = find_chain(off, items, u), j = u - off[it];
    const InvView& v = views[it];
    if (threadIdx.x == 0) {
      v.used[j] = 0;
      v.pcol[j] = -1;
    }
    refresh_store_column(chains[it >> 1], it & 1, j, orders[it], v.X, (double*)nullptr, red);
  }
}

// Log-determinants (sum of log|pivot|, in a fixed order) and the stats of
// every refreshed chain, one CTA per chain.
template <typename T>
__global__ void __launch_bounds__(256) k_refresh_finish(const Chain<T>* chains, const InvView* views,
                                                        const int* orders, int only_chain) {
  const int ci = only_chain >= 0 ? only_chain : (int)blockIdx.x;
  const Chain<T>& c = chains[ci];
  if (c.dyn->status & ~DS_SINGULAR) return;
  __shared__ double part[8];
  for (int spin = 0; spin < 2; ++spin) {
    const double* piv = views[2 * ci + spin].piv;
    const int m = orders[2 * ci + spin];
    double s = 0.0;
    for (int k = threadIdx.x; k < m; k += blockDim.x) s += log(fabs(piv[k]));
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < 8; ++w) t += part[w];
      c.work_logdet[spin] = t;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) refresh_finish_one(c);
}

}  // namespace

template <typename T>
cudaError_t launch_refresh(Chain<T>* dchains, const LaunchShape& ls, int only_chain, const RefreshOrders& ro,
                           cudaStream_t st, PhaseTimer* pt) {
  pt->begin(6, st);
  const int max_order = ro.bound;
  const int items = 2 * ls.n_chains, nch = ls.n_chains;
  InvWidths widths{};
  if (only_chain < 0 && ls.inv_all.size() > 1)
    for (const InvShape& sh : ls.inv_all) widths.w[widths.count++] = sh.width;
  k_refresh_orders<T><<<(items + 127) / 128, 128, 0, st>>>(dchains, nch, only_chain, ls.inv_orders, ls.inv_views, widths,
                                                        ro);
  // one chain: only its two matrices
  const int first = only_chain >= 0 ? 2 * only_chain : 0, count = only_chain >= 0 ? 2 : items;
  const InvView* views = ls.inv_views + first;
  const int* orders = ls.inv_orders + first;
  const Chain<T>* chains = dchains + first / 2;
  k_refresh_build<T><<<ls.persist_ctas, 256, 0, st>>>(chains, views, orders, count);
  cudaError_t e = cudaSuccess;
  int n = 0;
  if (only_chain >= 0) {
    n = launch_inverse(views, orders, count, max_order, ls.inv_one[ls.inv_one_of[only_chain]], st, &e);
  } else {
    for (size_t s = 0; s < ls.inv_all.size() && e == cudaSuccess; ++s)
      n += launch_inverse(views, widths.count ? orders + (1 + s) * items : orders, count, max_order, ls.inv_all[s], st, &e);
  }
  if (e == cudaSuccess) {
    k_refresh_store<T><<<ls.persist_ctas, 256, 0, st>>>(chains, views, orders, count);
    k_refresh_finish<T><<<only_chain >= 0 ? 1 : nch, 256, 0, st>>>(dchains, ls.inv_views, ls.inv_orders, only_chain);
    e = cudaGetLastError();
  }
  pt->end(6, st, 4 + n);
  return e;
}

template cudaError_t launch_refresh<double>(Chain<double>*, const LaunchShape&, int, const RefreshOrders&,
                                            cudaStream_t, PhaseTimer*);
template cudaError_t launch_refresh<float>(Chain<float>*, const LaunchShape&, int, const RefreshOrders&,
                                           cudaStream_t, PhaseTimer*);
size_t refresh_work_doubles(int ld) { return 2 * refresh_work_per_spin(ld); }
size_t refresh_work_one(int ld) { return refresh_work_per_spin(ld); }

}  // namespace ctaux
