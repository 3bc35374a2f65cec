// Host-side interface between the C ABI (ctaux_api.cu) and the kernels.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include "ctaux_dev.cuh"
#include "ctaux_inverse.cuh"
#include "ctaux_sliced.cuh"

namespace ctaux {

constexpr int kMaxPartials = 4096;  // split-K partial tiles per (chain, spin) and product
constexpr int kMaxMatsFreq = 64;    // Matsubara frequencies of the G(iw) measurement
constexpr int kMaxMatsSites = 1024; // cluster sites of the G(iw) measurement
constexpr int kTieSlices = 64;   // column slices of the near-tie matrix-vector products
// vertices per measurement evaluation chunk: small orders get short chunks
// (more work items for the GPU), large ones longer chunks (fewer partial sums)
constexpr int kMeasChunk = 16;      // the shortest chunk (sizes the partial-sum buffers)
constexpr int kMeasChunkMax = 32;
__host__ __device__ inline int meas_chunk(int n) { return n <= 1024 ? kMeasChunk : kMeasChunkMax; }

// Measurement product v_b = N g_b (k_meas_v): items of kMeasRows rows, up to
// kMeasAnchors anchors and one slice of the columns.  The slices are narrow
// where an order alone has few row blocks (order 415: 7 blocks x 7 slices for
// each spin in float64), wide where partial sums would cost more than they
// spread: float32, which is bound by its reads of N, four times as wide (96
// uneven mixed chains: 0.40 -> 0.346 ms per measurement).  One float64 chain of
// order 415, whose measurement runs beside the next block, takes 64 rather than
// 32 columns: twice the CTAs slowed that block by half a percent.  They depend on
// the order and the anchors only, so a chain gives the same bits alone or in a
// batch.
constexpr int kMeasRows = 64, kMeasAnchors = 8;
__host__ __device__ inline int meas_v_groups(int anchors) { return (anchors + kMeasAnchors - 1) / kMeasAnchors; }
__host__ __device__ inline int meas_v_width(int n, int anchors, bool fp64) {
  return (n <= 1024 ? 64 : n <= 4096 ? 128 : n <= 16384 ? 256 : 512) * meas_v_groups(anchors) *
         (fp64 ? 1 : 4);
}
__host__ __device__ inline int meas_v_slices(int n, int anchors, bool fp64) {
  const int w = meas_v_width(n, anchors, fp64);
  return (n + w - 1) / w;
}
// partial sums [slice][anchor][row] and tickets [row block][anchor group] of a spin
inline size_t meas_v_partials(int cap, int anchors, bool fp64) {
  size_t most = 1;   // the largest order of each width
  for (int n : {1024, 4096, 16384, cap}) {
    const int m = n < cap ? n : cap, s = meas_v_slices(m, anchors, fp64);
    const size_t need = s > 1 ? (size_t)s * anchors * m : 1;
    most = need > most ? need : most;
  }
  return most;
}
inline size_t meas_v_tickets(int cap, int anchors) {
  return (size_t)((cap + kMeasRows - 1) / kMeasRows) * meas_v_groups(anchors);
}

// tensor-core flush (mixed form): 128 x 128 output tiles, K chunks of 16 float32;
// the gathered N[S_m][S_n] input of a tile is staged as 128 column segments of
// kTcNsRows source rows
constexpr int kTcBM = 128, kTcBN = 128, kTcBK = 16, kTcStages = 4, kTcThreads = 384;
constexpr int kTcNsRows = 160;

// TMA descriptors of one (chain, spin): split Y (rows a), split X (rows b) and
// both buffers of N, as column segments of kTcNsRows rows, one column (nb1)
// or kTcNsGroup adjacent columns (nbg) per box
constexpr int kTcNsGroup = 8;
struct TcMaps {
  CUtensorMap yh, yl, xh, xl;
  CUtensorMap nb1[2], nbg[2];
  // tensor-core prep: the panels' rows and N, N^T as K-major rows (boxes of
  // 128 rows x kTcBK float32, 64-byte swizzle)
  CUtensorMap cpan, bpan, nb[2], nt[2];
};

enum { PH_RTILDE = 0, PH_GCOL_OLD = 1, PH_GCOL_NEW = 2, PH_FLUSH = 3, PH_MEAS = 4, PH_COUNT = 5 };

// Output tile of each product (rows x columns, per thread TM x TN; 256
// threads).  float64 (FP64-pipe bound, so padding costs time): skinny where
// one dimension is the number of insertions (R~: rows, G_{old,new}: columns),
// 32 x 32 otherwise.  float32 (the faster pipe makes re-reads of N and per-item
// overheads matter more): 64 x 64.  The measurement product has a kernel of its
// own (k_meas_v), without variants.
struct GemmTile {
  int bm, bn, tm, tn;
};
constexpr GemmTile gemm_tile(bool fp64, int phase) {
  return !fp64                  ? GemmTile{64, 64, 4, 4}
         : phase == PH_RTILDE   ? GemmTile{16, 64, 1, 4}
         : phase == PH_GCOL_OLD ? GemmTile{64, 16, 4, 1}
                                : GemmTile{32, 32, 2, 2};
}

// Compiled tile variants of each product (the autotuner's choices):
// 0 = the default above; 1 and 2 trade re-reads of the operands against
// padding and per-item overhead.  Every variant keeps 256 threads per tile.
constexpr int kTileVariants = 3;
constexpr GemmTile tile_variant(bool fp64, int phase, int v) {
  return v == 0 ? gemm_tile(fp64, phase)
         : !fp64 ? (v == 1 ? GemmTile{32, 32, 2, 2} : GemmTile{128, 64, 8, 4})
         : phase == PH_RTILDE   ? (v == 1 ? GemmTile{32, 32, 2, 2} : GemmTile{16, 128, 1, 8})
         : phase == PH_GCOL_OLD ? (v == 1 ? GemmTile{32, 32, 2, 2} : GemmTile{128, 16, 8, 1})
                                : (v == 1 ? GemmTile{64, 64, 4, 4} : GemmTile{64, 32, 4, 2});
}

// Tile-variant table of a context (the autotuner's cache): one byte per
// (product, octave of the expansion order, octave of k_max), read by the
// product kernels on the device for each chain's current order.
constexpr int kTileOct = 16, kTileKOct = 9;
constexpr int kTileTable = PH_COUNT * kTileOct * kTileKOct;
static_assert(kTileTable == 720 && kTileVariants == 3, "table size and variants in include/ctaux.h");
__host__ __device__ inline int tile_table_index(int phase, int n, int k) {
  int o = 0, ko = 0;
  while (o + 1 < kTileOct && (2 << o) <= n) ++o;
  while (ko + 1 < kTileKOct && (2 << ko) <= k) ++ko;
  return (phase * kTileOct + o) * kTileKOct + ko;
}

// Fixed launch shapes of one context (derived from capacities at init, so
// that a sweep needs no host-side knowledge of the current orders).
struct LaunchShape {
  int n_chains;
  int gather_slices;
  int kchunk;            // slice width of the inner dimension (while partial tiles fit)
  int persist_ctas;      // grid of the persistent batched kernels
  int tie_grid;          // cooperative grid of the near-tie refinement
  int tie_iters;         // most refinement iterations (0: every near tie takes the fallback)
  int prop_smem;
  int gamma_in_smem;
  int meas_lchunks;      // vertex chunks of the measurement evaluation
  int meas_cb_blocks;
  int meas_acc_blocks;   // one warp per (class, bin) output
  const InvView* inv_views;   // [chain][spin] matrices of the from-scratch recomputation (device)
  int* inv_orders;            // [chain][spin] their orders, written by each recomputation; then,
                              // for each of several shapes, the orders of its matrices
  std::vector<InvShape> inv_all;  // its launch shapes for every chain
  std::vector<InvShape> inv_one;  // and for one chain alone, by leading dimension
  std::vector<int> inv_one_of;    // [chain] place in inv_one
  int use_tc;            // mixed form: flush on the tensor cores
  int tc_ctas;           // persistent grid of the tensor-core flush (one CTA per SM)
  int split_x_blocks;
  int mats;              // Matsubara-frequency measurement on (n_matsubara > 0)
  int tc_wait_limit;     // polls of a tensor-core flush pipeline wait (0: 2^24)
  int prep_tc;           // mixed form: prep products on the tensor cores
  int gamma_lu;          // Gamma kept as L U (CTAUX_GAMMA_LU)
  int gamma_cluster, gamma_cluster_smem;  // CTAs per chain of the proposals, 0: one CTA (ctaux_block.cu)
  int max_cap;           // largest capacity + k_max of the chains
  int max_k;             // largest k_max of the context's chains
  int any_sliced, any_plain;  // float64 form: chains with sliced prep and flush products, and without
  int any_sliced_y, any_plain_y;  // the same for the flush coefficients
  int any_sliced_new, any_plain_new;  // and for G_{new,new}
  SlicedPlan sliced;
  int tile_mask[PH_COUNT];  // tile variants in the context's table, per product (bit v)
};

// Largest dynamic shared memory of the proposals of one CTA.  A kernel's limit holds
// for the process, not for a context: every configure_* sets one that no context
// exceeds, and the launches ask for what their context needs.
constexpr int kPropSmem = 200 * 1024;

// Row stride of a CTA's share of Gamma^{-1} in the cluster form: four lanes per
// row read consecutive elements of a warp's eight rows without bank conflicts.
__host__ __device__ inline int gamma_share_stride(int k, size_t element) {
  const int unit = element == 8 ? 16 : 32;
  return k <= 4 ? 4 : (k - 4 + unit - 1) / unit * unit + 4;
}

// CUDA-event timing of the sweep phases and kernel launch counts.  Phases:
// 0 plan + G0 gather, 1 prep products, 2 proposals (Gamma growth), 3 flush
// product, 4 flush support (survivors, Y, end of block), 5 measurement,
// 6 FP64 refresh.  Events are recorded only while profiling is on; launch
// counts are always kept.
struct PhaseTimer {
  static constexpr int kPhases = 8;
  static constexpr int kPool = 1024;
  cudaEvent_t ev[kPool];
  int phase_of[kPool / 2];
  int used = 0;
  int open_slot[kPhases];
  double ms[kPhases] = {0, 0, 0, 0, 0, 0, 0, 0};
  long long timed[kPhases] = {0, 0, 0, 0, 0, 0, 0, 0};
  long long kernels[kPhases] = {0, 0, 0, 0, 0, 0, 0, 0};
  bool created = false;
  bool on = false;
  void begin(int ph, cudaStream_t st) {
    if (!on) return;
    if (used + 2 > kPool) collect();
    open_slot[ph] = used;
    cudaEventRecord(ev[used], st);
    used += 1;
  }
  void end(int ph, cudaStream_t st, int n_kernels) {
    kernels[ph] += n_kernels;
    if (!on) return;
    const int s = open_slot[ph];
    cudaEventRecord(ev[used], st);
    phase_of[s / 2] = ph;
    used += 1;
  }
  // Sums the durations of recorded pairs (synchronises on the last event).
  void collect() {
    if (used == 0) return;
    cudaEventSynchronize(ev[used - 1]);
    for (int s = 0; s + 1 < used; s += 2) {
      float t = 0.f;
      if (cudaEventElapsedTime(&t, ev[s], ev[s + 1]) == cudaSuccess) {
        ms[phase_of[s / 2]] += t;
        timed[phase_of[s / 2]] += 1;
      }
    }
    used = 0;
  }
};

// Work run beside a block on a second stream: forked before the block's
// proposals, joined before its end (k_finish_block).
struct BlockFork {
  cudaStream_t side;
  cudaEvent_t ev_fork, ev_join;
  void (*fn)(void* arg, cudaStream_t side);
  void* arg;
};

template <typename T>
void launch_block(Chain<T>* dchains, const LaunchShape& ls, cudaStream_t st, PhaseTimer* pt,
                  const TcMaps* maps, const BlockFork* fork = nullptr);
template <typename T>
cudaError_t configure_block_kernels();
size_t refresh_work_doubles(int ld);
size_t refresh_work_one(int ld);
template <typename T>
void launch_measure(Chain<T>* dchains, const LaunchShape& ls, cudaStream_t st, PhaseTimer* pt);
// The measurement in two parts: the head (counters, G0 panels and the copy of
// the spins) must run before the next block's proposals change the spins; the
// tail reads only what the next block leaves alone until its end.
template <typename T>
int launch_measure_head(Chain<T>* dchains, const LaunchShape& ls, cudaStream_t st);
template <typename T>
int launch_measure_tail(Chain<T>* dchains, const LaunchShape& ls, cudaStream_t st);
// What a recomputation is launched for: no chain's order is above `bound` (a chain for
// which that does not hold stops with DS_NUMERIC); `number` and each chain's order go to
// `seen` (mapped host memory) when it begins, unless null.
struct RefreshOrders {
  int bound;
  uint32_t number;
  unsigned long long* seen;
};
template <typename T>
cudaError_t launch_refresh(Chain<T>* dchains, const LaunchShape& ls, int only_chain, const RefreshOrders& ro,
                           cudaStream_t st, PhaseTimer* pt);
// scratch: each chain's refresh work area (both spins)
cudaError_t launch_tie_refine(Chain<float>* dchains, const LaunchShape& ls, cudaStream_t st);
template <typename T>
void launch_reset_measure(Chain<T>* dchains, const LaunchShape& ls, cudaStream_t st);
template <typename T>
void launch_matsubara(Chain<T>* dchains, const LaunchShape& ls, cudaStream_t st);
// (value, step to the next value) of every table entry, the last step of a row 0;
// the same in float32 into g0f, unless null (it may take the plain table's place).
void launch_g0_pairs(const double* plain, int n_tau, long entries, double2* g0, float2* g0f, cudaStream_t st);
void launch_g0_matsubara(const double2* table, int n_classes, int n_tau, double beta, int n_freq,
                         double2* out, cudaStream_t st);
int tc_smem_bytes();
cudaError_t configure_prep_tc();
void launch_prep_tc(Chain<float>* dchains, const TcMaps* maps, const LaunchShape& ls,
                    cudaStream_t st);
cudaError_t encode_prep_maps(TcMaps* out, float* cpan, float* bpan, int panel_rows,
                             float* n0, float* n1, float* nt0, float* nt1, int ld);
cudaError_t configure_flush_tc();
void launch_flush_tc(Chain<float>* dchains, const TcMaps* maps, const LaunchShape& ls,
                     cudaStream_t st);
void launch_transpose_n(Chain<float>* dchains, const LaunchShape& ls, cudaStream_t st);
cudaError_t encode_tc_maps(TcMaps* out, float* yh, float* yl, float* xh, float* xl, int rows,
                           int kp, float* n0, float* n1, int ld);
// Proposals with Gamma^{-1} spread over a cluster (ctaux_gamma.cu).
template <typename T>
cudaError_t configure_gamma_cluster(LaunchShape& ls, int max_cap, int sm_count);
template <typename T>
cudaError_t launch_gamma_cluster(Chain<T>* dchains, const LaunchShape& ls, cudaStream_t st);
cudaError_t configure_sliced();
// The prep products R~ and G_{old,new}, and the flush product, of the sliced
// chains; return the kernels launched.
int launch_sliced_prep(const Chain<double>* dchains, const LaunchShape& ls, cudaStream_t st);
int launch_sliced_y(const Chain<double>* dchains, const LaunchShape& ls, cudaStream_t st);
int launch_sliced_flush(const Chain<double>* dchains, const LaunchShape& ls, cudaStream_t st);
void launch_philox_test(uint64_t seed, uint32_t chain, int64_t t0, int count, int purpose,
                        double* out, cudaStream_t st);

}  // namespace ctaux
