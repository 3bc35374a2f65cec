// The k_max proposals of a block with Gamma^{-1} spread over a thread-block
// cluster: one cluster per chain, half of its CTAs per spin.
//
// The single-CTA form (ctaux_block.cu) is bound by one SM: at k = 256 its
// float64 matrix-vector products and rank-one updates took 48 us per proposal.
// Here a proposal takes about 3.4 us at k = 64 (the chain: exchange, gather of
// G^0 from L2, float64 latencies of 60 clocks in the dot and the decision) and
// 7.3 us at k = 256.  Every CTA keeps the rows r = rank (mod CTAs per spin) of
// Gamma^{-1} and, as a second copy, the same columns, in shared memory.  A
// proposal then needs one exchange: each CTA forms its share of y = Gamma^{-1} s
// (rows) and of w^T Gamma^{-1} (columns, before the decision is known), sends
// both to the other CTAs with stores that count at the receivers' mbarriers,
// and every CTA takes the same decision from the whole vectors and updates its
// two shares.  A slot touched twice sends column and row q of Gamma^{-1}
// instead.  The bookkeeping (alive vertices, P, lambda) is kept by every CTA;
// rank 0 writes the chain's state.
//
// Every sum is taken in the order of the single-CTA form (the partial sums of
// a row belong to fixed threads of that row), so the results are the same bits
// for any cluster size.
#include <type_traits>

#include "ctaux_dev.cuh"
#include "ctaux_kernels.h"
#include "ctaux_tc.cuh"

namespace ctaux {

namespace {

constexpr int kGammaThreads = 256;

__device__ __forceinline__ uint32_t gc_map(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void gc_send(uint32_t addr, double v, uint32_t mbar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(addr),
               "l"(__double_as_longlong(v)), "r"(mbar)
               : "memory");
}
__device__ __forceinline__ void gc_send(uint32_t addr, float v, uint32_t mbar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr),
               "r"(__float_as_uint(v)), "r"(mbar)
               : "memory");
}
__device__ __forceinline__ void gc_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <typename A>
__device__ __forceinline__ A gc_warp_sum(A v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Detection-only guard of the near-tie count (as in the single-CTA form).
constexpr double kGammaTieGuard = 1e-4;

// Sum of a row (or column) share, elements g[i] x[i], i < n, by four adjacent
// lanes.  float64: each every fourth element.  float32: even and odd elements
// (each pair of lanes the same), or every fourth element of whole groups of four
// with the rest in the first lane's sum.  All four lanes get the result.
template <typename A, int PARTS>
__device__ __forceinline__ A share_sum(const A* g, const A* x, int n, int part) {
  constexpr int kStep = sizeof(A) == 8 ? 4 : PARTS;
  const int first = kStep == 2 ? part & 1 : part;
  const int end = (sizeof(A) == 8 || PARTS == 2) ? n : n & ~3;
  A acc = (A)0;
  int i = first;
  // the loads of eight elements at once: one shared-memory latency for all
#pragma unroll 1
  for (; i + 7 * kStep < end; i += 8 * kStep) {
    A a[8], b[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      a[u] = g[i + u * kStep];
      b[u] = x[i + u * kStep];
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) acc += a[u] * b[u];
  }
  {
    A a[7], b[7];
#pragma unroll
    for (int u = 0; u < 7; ++u) {
      const bool in = i + u * kStep < end;
      a[u] = in ? g[i + u * kStep] : (A)0;
      b[u] = in ? x[i + u * kStep] : (A)0;
    }
#pragma unroll
    for (int u = 0; u < 7; ++u) {
      if (i - first + u * kStep >= end) break;   // the same in the row's lanes; zeros add nothing
      acc += a[u] * b[u];
    }
  }
  if (sizeof(A) == 4 && PARTS == 4 && part == 0)
    for (int r = end; r < n; ++r) acc += g[r] * x[r];
  acc += __shfl_xor_sync(0xffffffffu, acc, 1);
  if constexpr (kStep == 4) acc += __shfl_xor_sync(0xffffffffu, acc, 2);
  return acc;
}

// The idx-th set bit of the mask, by every warp for itself: the 1024-bit group
// from the groups' counts, the word, the bit.
__device__ __forceinline__ int warp_select_bit(const uint32_t* mask, const int* group_count, int n_words, int idx,
                                               int lane) {
  auto pick = [&](int cnt, int& rest) -> int {   // the lane whose elements hold number `rest`
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    const uint32_t over = __ballot_sync(0xffffffffu, incl > rest);
    if (!over) return -1;
    const int who = __ffs(over) - 1;
    rest -= __shfl_sync(0xffffffffu, incl - cnt, who);
    return who;
  };
  int rest = idx;
  const int grp = pick(lane * 32 < n_words ? group_count[lane] : 0, rest);
  if (grp < 0) return -1;
  const int w = grp * 32 + lane;
  const uint32_t word = w < n_words ? mask[w] : 0u;
  const int who = pick(__popc(word), rest);
  if (who < 0) return -1;
  uint32_t x = __shfl_sync(0xffffffffu, word, who);
  int pos = 0;
#pragma unroll
  for (int h = 16; h > 0; h >>= 1) {
    const int cnt = __popc(x & ((1u << h) - 1u));
    if (rest >= cnt) {
      rest -= cnt;
      x >>= h;
      pos += h;
    }
  }
  return (grp * 32 + who) * 32 + pos;
}

// PARTS: lanes per row of y in float32 (2 where the single-CTA form holds
// Gamma^{-1} in shared memory, else 4).
template <typename T, int PARTS>
__global__ void __launch_bounds__(kGammaThreads, 1) k_proposals_cluster(Chain<T>* chains, int max_k, int max_cap) {
  using A = T;
  uint32_t rank, ncta;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(ncta));
  const Chain<T>& c = chains[blockIdx.x / ncta];
  Dyn& d = *c.dyn;
  if (d.status) return;   // the whole cluster
  const int per = (int)ncta >> 1, spin = (int)rank / per, own = (int)rank % per;   // CTAs per spin, this one's place
  const int tid = threadIdx.x, half = tid >> 7, ht = tid & 127, hw = ht >> 5, lane = tid & 31;
  const int KM = c.k_max, LG = KM + 1, ld = c.ld;
  const int n_old = d.n, m = d.m, buf = d.buf;
  const int64_t t0 = d.t;
  int8_t* s_glob = c.s[buf];
  const int64_t* birth = c.birth[buf];

  // shared memory, sized for max_k and max_cap (gamma_cluster_smem)
  const int lg = __ffs(per) - 1, pm = per - 1;          // CTAs per spin: a power of two
  const int kr = (max_k + per - 1) >> lg, ls = gamma_share_stride(max_k, sizeof(A)), krp = kr | 1;
  extern __shared__ __align__(16) unsigned char gsm[];
  A* rows = reinterpret_cast<A*>(gsm);                  // [kr][ls]: row own + per lr
  A* cols = rows + (size_t)kr * ls;                     // [kr][ls]: column own + per lc
  A* yin = cols + (size_t)kr * ls;                      // [2][2 spins][per][krp] received y
  A* zin = yin + (size_t)4 * per * krp;                 // [2][per][krp] received z, this spin
  A* tok = zin + (size_t)2 * per * krp;                 // [2][16] a token of every CTA
  A* sv = tok + 32;                                     // [max_k] column of G^0 over P, this spin
  A* wv = sv + max_k;                                   // [2][max_k] row of G^0 over P, both spins
  A* ysv = wv + 2 * max_k;                              // [max_k] y and z / beta of an accepted
  A* zsv = ysv + max_k;                                 // [max_k] first touch, this spin
  double* lam = reinterpret_cast<double*>(gsm + (((size_t)(zsv + max_k - rows) * sizeof(A) + 15) & ~(size_t)15));
  double* ilam = lam + 2 * max_k;
  int* P_s = reinterpret_cast<int*>(ilam + 2 * max_k);
  uint32_t* alive = reinterpret_cast<uint32_t*>(P_s + max_k);
  short* pmap = reinterpret_cast<short*>(alive + (max_cap + 31) / 32);
  int8_t* s0_s = reinterpret_cast<int8_t*>(pmap + ((max_cap + 7) & ~7));
  int8_t* sc_s = s0_s + ((max_cap + 15) & ~15);
  const int n_words = (m + 31) / 32;

  __shared__ A red[2][4];
  __shared__ A dd_s[2];         // G^0_pp - (1 + lambda) / lambda
  __shared__ A ratio_s[2];
  __shared__ A scal_s;          // this spin's 1/beta, Sherman-Morrison coefficient or Schur pivot
  __shared__ double ev_s[2][5], iem1_s[2][5], lam_s[2][5];
  __shared__ A glam_s[2][5];
  __shared__ int dec_s, fin_s;  // 0 reject, 1 accept, 2 near tie (stop), 3 gave up
  __shared__ double R_s;
  __shared__ A f_s;             // move factor
  __shared__ A nlam_s[2][5];    // -lambda in A
  __shared__ int group_count[32], idx3_s[3];
  __shared__ volatile int gave_up;
  __shared__ uint64_t landed[2];
  __shared__ BlockDraw bd_s[kMaxK];

  for (int i = tid; i < m; i += kGammaThreads) {
    pmap[i] = -1;
    s0_s[i] = c.s0[i];
    sc_s[i] = s_glob[i];
  }
  if (tid < 32) group_count[tid] = 0;
  __syncthreads();
  for (int w = tid; w < n_words; w += kGammaThreads) {
    uint32_t bits = 0;
    for (int b = 0; b < 32; ++b) {
      const int i = w * 32 + b;
      if (i < m && s_glob[i] != 0) bits |= (1u << b);
    }
    alive[w] = bits;
    atomicAdd(&group_count[w >> 5], __popc(bits));
  }
  if (tid < 10) {
    const int sp_ = tid / 5, k_ = tid % 5;
    ev_s[sp_][k_] = c.ev[sp_][k_];
    lam_s[sp_][k_] = c.ev[sp_][k_] - 1.0;
    nlam_s[sp_][k_] = -(A)lam_s[sp_][k_];
    iem1_s[sp_][k_] = c.inv_em1[sp_][k_];
    glam_s[sp_][k_] = c.glam[sp_][k_];
  }
  for (int e = tid; e < KM; e += kGammaThreads) bd_s[e] = c.draws[e];
  if (tid == 0) {
    gave_up = 0;
    tc::mbar_init(tc::smem_u32(landed), 1);
    tc::mbar_init(tc::smem_u32(landed + 1), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // replicated bookkeeping (every thread of every CTA)
  int j = 0, n_cur = n_old;
  // rank 0, threads 0 and 64
  int sign = d.sign;
  int prop0 = 0, prop1 = 0, prop2 = 0, acc0 = 0, acc1 = 0, acc2 = 0, numeric = 0, ties = 0;   // by move
  long long flops2 = 0;
  // read once: the decision of a near tie taken in FP64 after the previous block
  const int64_t forced_t = (sizeof(T) == 4) ? d.forced_t : -1;
  const bool forced_accept = (sizeof(T) == 4) && d.forced_accept != 0;
  const double forced_R = (sizeof(T) == 4) ? d.forced_R : 0.0;
  const double tie_guard = (sizeof(T) == 4 && c.tie_guard > 0.0) ? d.guard_eff : 0.0;
  const float guard_f = (float)(tie_guard > 0.0 ? tie_guard : kGammaTieGuard);
  const int trace_cap = c.trace_cap;
  const int64_t trace_base = d.trace_written;
  __syncthreads();
  gc_barrier();   // every CTA has read the chain's state, and its barriers exist
  int consumed = KM;
  uint32_t round = 0;

  // ---- the exchange: y (to every CTA) and z (to this spin's CTAs)
  auto y_at = [&](uint32_t g, int sp, int r) -> A { return yin[((g * 2 + sp) * per + (r & pm)) * krp + (r >> lg)]; };
  auto z_at = [&](uint32_t g, int r) -> A { return zin[(g * per + (r & pm)) * krp + (r >> lg)]; };
  // offsets from this CTA's shared memory to that of a lane's destinations:
  // CTA lane % 4 + 4 i of the cluster, and of this spin's half
  const uint32_t here = tc::smem_u32(gsm);
  uint32_t to_all[4], to_spin[2];
#pragma unroll
  for (int i = 0; i < 4; ++i) to_all[i] = gc_map(here, min((uint32_t)((lane & 3) + 4 * i), ncta - 1)) - here;
#pragma unroll
  for (int i = 0; i < 2; ++i) to_spin[i] = gc_map(here, (uint32_t)(spin * per + min((lane & 3) + 4 * i, per - 1))) - here;
  // the value of row (column) r from four lanes that hold it and share the destinations
  auto send_y = [&](int r, A v, uint32_t bar, uint32_t g) {
    const uint32_t a = tc::smem_u32(yin + ((g * 2 + spin) * per + own) * krp + (r >> lg));
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if ((lane & 3) + 4 * i < (int)ncta) gc_send(a + to_all[i], v, bar + to_all[i]);
  };
  auto send_z = [&](int r, A v, uint32_t bar, uint32_t g) {
    const uint32_t a = tc::smem_u32(zin + (g * per + own) * krp + (r >> lg));
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if ((lane & 3) + 4 * i < per) gc_send(a + to_spin[i], v, bar + to_spin[i]);
  };
  // Every CTA sends a token every round, also without rows: none runs ahead by
  // more than the two buffers.
  auto open_round = [&](int jn, uint32_t bar, uint32_t g) {
    if (tid == 0) tc::mbar_expect_tx(bar, (uint32_t)((3 * jn + (int)ncta) * sizeof(A)));
    if (tid >= kGammaThreads - 32 && lane < (int)ncta)
      gc_send(gc_map(tc::smem_u32(tok + g * 16 + rank), (uint32_t)lane), (A)0, gc_map(bar, (uint32_t)lane));
  };
  auto close_round = [&](uint32_t bar) {
    if (!tc::mbar_wait(bar, (round >> 1) & 1, gave_up ? 1u : tc::kWaitLimit)) gave_up = 1;
    ++round;
  };
  // column (row) k of the shares of Gamma^{-1}, below jn
  auto send_line = [&](int k, int jn, uint32_t bar, uint32_t g) {
#pragma unroll 1
    for (int l = ht >> 2; own + per * l < jn; l += 32) {
      if (half == 0) send_y(own + per * l, rows[(size_t)l * ls + k], bar, g);
      else send_z(own + per * l, cols[(size_t)l * ls + k], bar, g);
    }
  };

  // ---- the vertex of a proposal, and its row and column of G^0 over P
  int p = -1, s_new = 0, q = -1;   // slot, proposed spin, place in P
  auto choose = [&](int jj, int idx) {   // idx: place among the n_cur vertices, < 0 where not at hand
    p = -1;
    if (jj >= KM) return;
    const int move = bd_s[jj].move;
    if (move == MV_INSERT) {
      p = bd_s[jj].slot;
      s_new = bd_s[jj].s_new;
    } else if (n_cur > 0) {
      if (idx < 0) idx = min((int)floor(bd_s[jj].u_idx * (double)n_cur), n_cur - 1);
      p = warp_select_bit(alive, group_count, n_words, idx, lane);
      if (p >= 0 && p < m) s_new = (move == MV_REMOVE) ? 0 : -(int)sc_s[p];
      else p = -2;
    }
    q = p >= 0 ? (int)pmap[p] : -1;
  };
  // Items of the gather of vertex p over jn entries of P: s of this spin, w of
  // spin 0 and 1, G^0_pp of both; a thread takes items tid + 256 i.  The loads
  // are issued while the previous proposal's update runs, the arithmetic
  // follows: G = (N e^V - 1)/(e^V - 1) for old columns (Eq. NfromG), the prep
  // columns for new ones.
  const T *N0 = c.N[buf][0], *N1 = c.N[buf][1], *G0 = c.Gcol[0], *G1 = c.Gcol[1];
  T raw[4];
  auto item = [&](int e, int jn, int& sp, int& i, int& col, int& kind) {
    kind = e < jn ? 0 : e < 2 * jn ? 1 : e < 3 * jn ? 2 : 3;
    const int r = e - kind * jn;
    sp = kind == 0 ? spin : kind == 3 ? r : kind - 1;
    const int pr = kind == 3 ? p : P_s[r];
    i = kind == 0 ? pr : p;
    col = kind == 0 ? p : pr;
    return r;
  };
  auto issue = [&](int jn) {
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      if (x * kGammaThreads >= 3 * jn + 2) break;   // the whole CTA
      const int e = tid + x * kGammaThreads;
      if (e < 3 * jn + 2) {
        int sp, i, col, kind;
        item(e, jn, sp, i, col, kind);
        const T* src = col < n_old ? (sp == 0 ? N0 : N1) : (sp == 0 ? G0 : G1);
        raw[x] = src[(long)(col < n_old ? col : col - n_old) * ld + i];
      }
    }
  };
  auto finish = [&](int jn, int dk) {
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      if (x * kGammaThreads >= 3 * jn + 2) break;
      const int e = tid + x * kGammaThreads;
      if (e < 3 * jn + 2) {
        int sp, i, col, kind;
        const int r = item(e, jn, sp, i, col, kind);
        A v = (A)raw[x];
        if (col < n_old) {
          const int kc = s0_s[col] + 2;
          v = (v * (A)ev_s[sp][kc] - (kind == 3 ? (A)1 : (A)0)) * (A)iem1_s[sp][kc];
        }
        if (kind == 0) sv[r] = v;
        else if (kind == 3) dd_s[sp] = v - glam_s[sp][dk];
        else wv[sp * max_k + r] = v;
      }
    }
  };

  choose(0, -1);
  if (p >= 0 && q < 0) issue(0);
  for (int jj = 0; jj < KM; ++jj) {
    const int64_t t = t0 + jj;
    const BlockDraw dr = bd_s[jj];
    const int move = dr.move, nc = n_cur;
    if (p < 0) {
      if (p == -2) {
        if (rank == 0 && tid == 0) atomicOr(&d.status, DS_INDEX);
        break;
      }
      // removal or flip with no vertex: automatic rejection
      if (rank == 0 && tid == 0) {
        prop1 += move == MV_REMOVE;
        prop2 += move == MV_FLIP;
        if (trace_cap > 0) {
          TraceRec& r = c.trace[(trace_base + jj) % trace_cap];
          r.t = t; r.move = move; r.n = nc; r.birth = -1; r.s_new = 0; r.accept = 0;
          r.ratio[0] = r.ratio[1] = 0.0; r.R = 0.0; r.u = dr.u_acc;
        }
      }
      choose(jj + 1, -1);
      if (p >= 0 && q < 0) issue(j);
      continue;
    }
    const float u_f = (float)dr.u_acc;
    const int dk = s_new - s0_s[p] + 2;             // index of lambda_new in the tables
    const bool to_start = (s_new == s0_s[p]);       // lambda_new = 0
    const uint32_t g = round & 1, bar = tc::smem_u32(landed + g);
    if (q < 0) finish(j, dk);
    __syncthreads();   // s, w in place; the previous update of the shares is done
    open_round(j, bar, g);
    // off the critical path, read after the exchange: the move factor, and the
    // place of the next removal or flip for the three orders it may meet
    if (tid == 192)
      f_s = (A)((move == MV_INSERT) ? c.K / (double)(nc + 1) : (move == MV_REMOVE ? (double)nc / c.K : 1.0));
    if (tid >= 224 && tid < 227 && jj + 1 < KM) {
      const int n1 = nc + tid - 225;
      if (n1 > 0) idx3_s[tid - 224] = min((int)floor(bd_s[jj + 1].u_idx * (double)n1), n1 - 1);
    }
    if (q < 0) {
      // this CTA's rows of y = Gamma^{-1} s (first half) and columns of
      // w^T Gamma^{-1} (second half)
      if (half == 0) {
#pragma unroll 1
        for (int l0 = 0; own + per * (l0 + hw * 8) < j; l0 += 32) {   // warps with rows
          const int lr = l0 + (ht >> 2), r = own + per * lr;
          const A y = share_sum<A, PARTS>(rows + (size_t)(r < j ? lr : 0) * ls, sv, r < j ? j : 0, ht & 3);
          if (r < j) send_y(r, y, bar, g);
        }
      } else {
        const A* w = wv + spin * max_k;
#pragma unroll 1
        for (int l0 = 0; own + per * (l0 + hw * 8) < j; l0 += 32) {
          const int lc = l0 + (ht >> 2), cc = own + per * lc;
          const A z = share_sum<A, 4>(cols + (size_t)(cc < j ? lc : 0) * ls, w, cc < j ? j : 0, ht & 3);
          if (cc < j) send_z(cc, z, bar, g);
        }
      }
    } else {
      send_line(q, j, bar, g);   // a slot of P again: column and row q of Gamma^{-1}
    }
    __syncwarp();
    close_round(bar);
    if (q < 0) {
      // w . y of both spins, a half each, in the order of the single-CTA form
      const A* w = wv + half * max_k;
      A part = (A)0;
      bool has_rows;
      if constexpr (sizeof(A) == 8) {
        has_rows = hw * 8 < j;
        if ((ht & 3) == 0)
#pragma unroll 1
          for (int r = ht >> 2; r < j; r += 32) part += w[r] * y_at(g, half, r);
        if (has_rows) {   // the other lanes hold zeros: their additions are exact
#pragma unroll
          for (int o = 16; o > 2; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        }
      } else {
        has_rows = hw * 32 < j;
#pragma unroll 1
        for (int r = ht; r < j; r += 128) part += w[r] * y_at(g, half, r);
        if (has_rows) part = gc_warp_sum(part);
      }
      if (lane == 0) red[half][hw] = has_rows ? part : (A)0;
    }
    __syncthreads();
    // beta of a first touch
    auto beta_of = [&](int sp) -> A {
      return dd_s[sp] - ((red[sp][0] + red[sp][1]) + (red[sp][2] + red[sp][3]));
    };
    if (tid == 0) {
      A ratio[2];
#pragma unroll
      for (int sp = 0; sp < 2; ++sp) {
        const A nlam = nlam_s[sp][dk];
        if (q < 0) {
          ratio[sp] = nlam * beta_of(sp);
        } else {
          const A ilo = (A)ilam[sp * max_k + q];  // 1 / lambda of the slot's first change
          const A gqq = y_at(g, sp, q);
          if (!to_start) {
            const A delta = ilo - (A)iem1_s[sp][dk];  // 1/lambda_old - 1/lambda_new
            ratio[sp] = (-nlam * ilo) * ((A)1 + delta * gqq);
          } else {
            ratio[sp] = -gqq * ilo;
          }
        }
        ratio_s[sp] = ratio[sp];
      }
      double R;
      bool accept, finite, near;
      // float32 form: the decision in float32 unless the product overflows
      // (near ties lie inside the guard band, which is decided in FP64)
      const float Rf = (sizeof(T) == 4) ? (float)f_s * (float)ratio[0] * (float)ratio[1] : 0.f;
      if (sizeof(T) == 4 && isfinite(Rf)) {
        const float uf = u_f, aR = fabsf(Rf);
        R = (double)Rf;
        finite = true;
        accept = uf < fminf(1.f, aR);
        near = fabsf(uf - aR) < guard_f * fmaxf(uf, aR);
      } else {
        // u < min(1, |R|) is u < |R| (u < 1), and doubles of one sign compare
        // like their bits: integer comparisons, a float64 one costs 60 clocks
        const double f = sizeof(T) == 8 ? (double)f_s
                         : (move == MV_INSERT) ? c.K / (double)(nc + 1) : (move == MV_REMOVE ? (double)nc / c.K : 1.0);
        R = f * (double)ratio[0] * (double)ratio[1];
        const long long aR = __double_as_longlong(R) & 0x7fffffffffffffffll;
        finite = aR < 0x7ff0000000000000ll;
        accept = __double_as_longlong(dr.u_acc) < aR;
        near = (sizeof(T) == 4) && finite &&
               fabs(dr.u_acc - fabs(R)) < (tie_guard > 0.0 ? tie_guard : kGammaTieGuard) * fmax(dr.u_acc, fabs(R));
      }
      if (!finite) accept = false;
      const bool forced = (sizeof(T) == 4) && forced_t == t;
      int dec;
      if (forced) {
        // decided in FP64 after the previous block stopped here (k_tie_refine)
        accept = forced_accept;
        R = forced_R;
        finite = true;
        dec = accept ? 1 : 0;
      } else if (sizeof(T) == 4 && tie_guard > 0.0 && finite && near) {
        // near tie in the float32 form: the block ends before this proposal,
        // which is decided in FP64 after the flush
        if (rank == 0) {
          d.tie_pending = 1;
          d.tie_jj = jj;
          d.tie_R32 = R;
        }
        ties++;
        dec = 2;
      } else {
        dec = accept ? 1 : 0;
        if (sizeof(T) == 4 && tie_guard == 0.0 && finite && near) ties++;  // detection only
      }
      if (dec != 2) {
        if (!finite) numeric++;
        if (accept && __double2hiint(R) < 0) sign = -sign;
        if (forced && rank == 0) d.forced_t = -1;
      }
      R_s = R;
      fin_s = forced ? 1 : 0;
      dec_s = gave_up ? 3 : dec;
    } else if (tid == 32) {   // needed only on acceptance, beside the decision
      if (q < 0) {
        scal_s = (A)1 / beta_of(spin);
      } else {
        const A gqq = y_at(g, spin, q);
        if (!to_start) {
          const A delta = (A)ilam[spin * max_k + q] - (A)iem1_s[spin][dk];
          scal_s = delta / ((A)1 + delta * gqq);  // Sherman-Morrison coefficient
        } else {
          scal_s = (A)1 / gqq;  // Schur complement pivot
        }
      }
    }
    __syncthreads();
    const int dec = dec_s;
    if (dec >= 2) {
      consumed = jj;
      if (dec == 3 && tid == 0) atomicOr(&d.status, DS_TIMEOUT);
      break;
    }
    if (rank == 0 && tid == 64) {
      // counters and the trace record, off the critical path
      const bool accept = dec == 1;
      prop0 += move == MV_INSERT;
      prop1 += move == MV_REMOVE;
      prop2 += move == MV_FLIP;
      acc0 += accept && move == MV_INSERT;
      acc1 += accept && move == MV_REMOVE;
      acc2 += accept && move == MV_FLIP;
      // algorithmic flops, both spins: y GEMV and the dot (first touch); on
      // acceptance the z GEMV and the bordered update, or the rank-one update
      int fl = (q < 0) ? (2 * j * j + 2 * j) : 4;
      if (accept) fl += (q < 0) ? 2 * j * j + 3 * (j + 1) * (j + 1) : 3 * j * j;
      flops2 += fl;
      if (trace_cap > 0) {
        const bool forced = fin_s != 0;
        TraceRec& rr = c.trace[(trace_base + jj) % trace_cap];
        rr.t = t; rr.move = move; rr.n = nc;
        rr.birth = birth[p]; rr.s_new = s_new; rr.accept = (accept ? 1 : 0) | (forced ? 2 : 0);
        rr.ratio[0] = forced ? d.forced_ratio[0] : (double)ratio_s[0];
        rr.ratio[1] = forced ? d.forced_ratio[1] : (double)ratio_s[1];
        rr.R = R_s; rr.u = dr.u_acc;
      }
    }
    const int jo = j, qo = q, last = j - 1;   // of this proposal: the next one is chosen below
    if (dec == 1) {
      if (q < 0) {   // once, not per element of the shares
        const A sc = scal_s;
        for (int r = ht; r < j; r += 128) {
          if (half == 0) ysv[r] = y_at(g, spin, r);
          else zsv[r] = z_at(g, r) * sc;
        }
      }
      if (tid == 0) {
        if (q < 0) {
          P_s[j] = p;
          pmap[p] = (short)j;
        } else if (to_start) {
          if (q != last) {
            const int pl = P_s[last];
            P_s[q] = pl;
            pmap[pl] = (short)q;
          }
          pmap[p] = -1;
        }
      } else if (tid == 32) {
        sc_s[p] = (int8_t)s_new;
        if (rank == 0) s_glob[p] = (int8_t)s_new;
        const uint32_t bit = 1u << (p & 31), w = alive[p >> 5];
        const uint32_t w1 = s_new == 0 ? w & ~bit : w | bit;
        alive[p >> 5] = w1;
        group_count[p >> 10] += __popc(w1) - __popc(w);
      } else if (tid == 64 || tid == 65) {   // lambda of both spins
        const int sp = tid - 64;
        double* lm = lam + sp * max_k;
        double* il = ilam + sp * max_k;
        if (q < 0) {
          lm[j] = lam_s[sp][dk];
          il[j] = iem1_s[sp][dk];
        } else if (!to_start) {
          lm[q] = lam_s[sp][dk];
          il[q] = iem1_s[sp][dk];
        } else if (q != last) {
          lm[q] = lm[last];
          il[q] = il[last];
        }
      }
      if (move == MV_INSERT) n_cur = nc + 1;
      else if (move == MV_REMOVE) n_cur = nc - 1;
      if (q < 0) j += 1;
      else if (to_start) j = last;
      __syncthreads();
    }
    // ---- the next proposal's vertex, its loads in flight during the update
    choose(jj + 1, n_cur > 0 ? idx3_s[n_cur - nc + 1] : -1);
    if (p >= 0 && q < 0) issue(j);
    if (dec != 1) continue;
    // ---- accepted: both shares of Gamma^{-1}, a row or column per 16 threads
    const A sc = scal_s;
    if (qo < 0) {
      // [[G + y z / beta, -y / beta], [-z / beta, 1 / beta]]: row (column) a of the
      // share per 16 threads; `mine` is its y (z / beta), `o` the others' z / beta (y)
      const int jn = jo + 1;
      A* sh = half == 0 ? rows : cols;
      const A* o = half == 0 ? zsv : ysv;
#pragma unroll 1
      for (int l = ht >> 4; own + per * l < jn; l += 8) {
        const int a = own + per * l;
        A* x = sh + (size_t)l * ls;
        if (a < jo) {
          const A mine = half == 0 ? ysv[a] : zsv[a];
#pragma unroll 4
          for (int b = ht & 15; b < jo; b += 16) x[b] += mine * o[b];
          if ((ht & 15) == 0) x[jo] = half == 0 ? -mine * sc : -mine;
        } else {
#pragma unroll 1
          for (int b = ht & 15; b < jn; b += 16) x[b] = b == jo ? sc : half == 0 ? -o[b] : -o[b] * sc;
        }
      }
    } else {
      A* sh = half == 0 ? rows : cols;
#pragma unroll 1
      for (int l = ht >> 4; own + per * l < jo; l += 8) {
        const int a = own + per * l;
        A* x = sh + (size_t)l * ls;
#pragma unroll 1
        for (int b = ht & 15; b < jo; b += 16) {
          const A y = y_at(g, spin, half == 0 ? a : b), z = z_at(g, half == 0 ? b : a);
          x[b] = to_start ? x[b] - y * z * sc : x[b] - sc * y * z;
        }
      }
      if (to_start && qo != last) {
        // the last entry of P moves into position q: row and column `last` to everyone
        __syncthreads();
        const uint32_t g2 = round & 1, bar2 = tc::smem_u32(landed + g2);
        open_round(jo, bar2, g2);
        send_line(last, jo, bar2, g2);
        __syncthreads();   // every share is read before it changes
        close_round(bar2);
        // y: G[e][last], z: G[last][e]
        for (int e = tid; e < last; e += kGammaThreads) {
          if ((e & pm) == own) {
            rows[(size_t)(e >> lg) * ls + qo] = y_at(g2, spin, e);   // G[e][q]; row q itself follows
            cols[(size_t)(e >> lg) * ls + qo] = z_at(g2, e);         // G[q][e]
          }
        }
        __syncthreads();
        if ((qo & pm) == own)
          for (int e = tid; e < last; e += kGammaThreads) {
            rows[(size_t)(qo >> lg) * ls + e] = z_at(g2, e == qo ? last : e);
            cols[(size_t)(qo >> lg) * ls + e] = e == qo ? z_at(g2, last) : y_at(g2, spin, e);
          }
      }
    }
  }
  __syncthreads();
  // Gamma^{-1}, lambda, P
  T* dst = c.Ginv[spin];
  for (int l = tid >> 5; own + per * l < j; l += kGammaThreads / 32)
    for (int cc = lane; cc < j; cc += 32) dst[(size_t)(own + per * l) * LG + cc] = rows[(size_t)l * ls + cc];
  if (own == 0)
    for (int r = tid; r < j; r += kGammaThreads) c.lam[spin][r] = lam[spin * max_k + r];
  if (rank == 0) {
    for (int r = tid; r < j; r += kGammaThreads) c.P[r] = P_s[r];
    // thread 64 counted the decisions, thread 0 the automatic rejections
    auto add_counts = [&]() {
      d.proposals[0] += prop0;
      d.proposals[1] += prop1;
      d.proposals[2] += prop2;
      d.accepted[0] += acc0;
      d.accepted[1] += acc1;
      d.accepted[2] += acc2;
      d.work_gamma += 2.0 * (double)flops2;
    };
    if (tid == 64) add_counts();
    __syncthreads();
    if (tid == 0) {
      d.k_acc = j;
      d.sign = sign;
      add_counts();
      d.numeric_rejects += numeric;
      d.near_ties += ties;
      if (c.trace_cap > 0) d.trace_written += consumed;
    }
  }
  __syncwarp();
  gc_barrier();   // no CTA exits while another may still send to it
}

template <typename T>
size_t gamma_cluster_smem(int max_k, int max_cap, int per) {
  const size_t kr = (max_k + per - 1) / per, ls = gamma_share_stride(max_k, sizeof(T));
  size_t el = 2 * kr * ls + 6 * per * (kr | 1) + 32 + 5 * (size_t)max_k;
  size_t b = (el * sizeof(T) + 15) & ~(size_t)15;
  b += sizeof(double) * 4 * max_k + sizeof(int) * max_k + sizeof(uint32_t) * ((max_cap + 31) / 32);
  b += sizeof(short) * ((max_cap + 7) & ~7) + 2 * (size_t)((max_cap + 15) & ~15) + 64;
  return b;
}

template <typename T>
const void* gamma_kernel(const LaunchShape& ls) {
  return ls.gamma_in_smem ? (const void*)k_proposals_cluster<T, 2> : (const void*)k_proposals_cluster<T, 4>;
}

}  // namespace

// Cluster size for the proposals of a context, 0 for the single-CTA form: 16
// CTAs, or as many as give every chain its own SMs, at least 2 in float64 and 4 in
// float32; none for short blocks, whose few rows do not pay for the exchange.
// Proposal phase of one chain, us per block, one CTA / clusters of 4 / 8 / 16:
//   float64  k = 16 (impurity) 53 / 56 / 56 / 56, k = 20 (4 sites) 72 / 70 / 70 / 70,
//            k = 32 (2x2x2) 128 / 112 / 109 / 109, k = 64 335 / 247 / 227 / 220,
//            k = 96 654 / 435 / 369 / 347, k = 128 (6x6) 1703 / 762 / 601 / 538
//   float32  k = 20 62 / 64 / 63 / 64, k = 32 105 / 98 / 97 / 98, k = 64 227 / 200 / 188 / 186,
//            k = 128 669 / 470 / 412 / 383
// and at k = 256 (100 sites) 12.4 ms -> 1.9 ms in float64, 6.5 -> 1.2 in float32.
template <typename T>
cudaError_t configure_gamma_cluster(LaunchShape& ls, int max_cap, int sm_count) {
  ls.gamma_cluster = 0;
  ls.max_cap = max_cap;
  if (ls.gamma_lu) return cudaSuccess;
  cudaError_t e = cudaSuccess;
  for (int cl = ls.max_k <= 24 ? 0 : 16; cl >= (sizeof(T) == 8 ? 2 : 4); cl /= 2) {
    if (ls.n_chains * cl > sm_count) continue;
    const size_t smem = gamma_cluster_smem<T>(ls.max_k, max_cap, cl / 2);
    if (smem > 220 * 1024) break;
    const void* fn = gamma_kernel<T>(ls);
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)cl);
    cfg.blockDim = dim3(kGammaThreads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)cl;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int fit = 0;
    e = cudaOccupancyMaxActiveClusters(&fit, fn, &cfg);
    if (e != cudaSuccess) return e;
    if (fit == 0) continue;
    ls.gamma_cluster = cl;
    ls.gamma_cluster_smem = (int)smem;
    break;
  }
  return e;
}

template <typename T>
cudaError_t launch_gamma_cluster(Chain<T>* dchains, const LaunchShape& ls, cudaStream_t st) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(ls.n_chains * ls.gamma_cluster));
  cfg.blockDim = dim3(kGammaThreads);
  cfg.dynamicSmemBytes = (size_t)ls.gamma_cluster_smem;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)ls.gamma_cluster;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return ls.gamma_in_smem ? cudaLaunchKernelEx(&cfg, k_proposals_cluster<T, 2>, dchains, ls.max_k, ls.max_cap)
                          : cudaLaunchKernelEx(&cfg, k_proposals_cluster<T, 4>, dchains, ls.max_k, ls.max_cap);
}

template cudaError_t configure_gamma_cluster<double>(LaunchShape&, int, int);
template cudaError_t configure_gamma_cluster<float>(LaunchShape&, int, int);
template cudaError_t launch_gamma_cluster<double>(Chain<double>*, const LaunchShape&, cudaStream_t);
template cudaError_t launch_gamma_cluster<float>(Chain<float>*, const LaunchShape&, cudaStream_t);

}  // namespace ctaux
