// Prep and flush products of the float64 form as sliced float16 tensor-core
// products (ctaux_oz.cuh): descriptors shared by the host and the kernels in
// ctaux_sliced.cu.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace ctaux {

// Slice images of one (chain, spin).  A "part" is 128 elements of the inner
// dimension (four 32-element chunks); every operand row has an exponent per part.
struct SlicedView {
  unsigned char* cs[2];   // C rows (product 0) and B columns (product 1): [64 rows][chunk] images
  int* ce[2];             // their exponents, [row][pl]
  unsigned char* ys;      // -Y rows: [128 rows][chunk] images
  unsigned char* xs;      // N[P, S] columns: [64 rows][chunk] images
  int *ye, *xe;           // exponents, [row][2]
  int* qe;                // balance of Y's inner index, exponents
  unsigned char* gs;      // columns of G_{old,new}: [128 rows][chunk] images
  int* ge;                // their exponents, [row][pl]
  double* gpart;          // split-K partial tiles of G_{new,new}
  int* gticket;           // arrivals per tile and epilogue warp
  double* part[2];        // split-K partial tiles of the prep products (128 x 64)
  int* ticket[2];         // arrivals per tile and epilogue warp
  int pl;                 // parts of the inner dimension at the capacity
  int yc;                 // chunks of ys and xs
};

// One prep product of one (chain, spin): its operand N (product 1) or N^T
// (product 0) is sliced into the pool of the strip that the job belongs to.
struct SlicedJob {
  int ci, spin, prod, pad;
  size_t img;   // byte offset of its images in the pool, [128 rows][chunk]
  size_t exps;  // offset of its exponents, [row][pl]
};
struct SlicedStrip {
  int first, count;
};

// Work list of a context (device pointers; strips on the host).
struct SlicedPlan {
  const SlicedView* views = nullptr;   // [chain][spin]
  const SlicedJob* jobs = nullptr;
  unsigned char* pool = nullptr;
  int* pool_exp = nullptr;
  const SlicedStrip* strips = nullptr;
  int n_strips = 0;
};

constexpr size_t kSlicedImageA = 7 * 128 * 64, kSlicedImageB = 7 * 64 * 64;   // oz::kImageA, oz::kImageB

// Split of a prep product's inner dimension, from its own sizes only (so that a
// chain gives the same bits alone or in a batch): enough slices that the
// chain's four products make about 600 items (four per SM), at least two parts
// per slice.
constexpr int kSlicedItems = 600;
__host__ __device__ inline int sliced_slices(int n, int k_ins) {
  const int parts = (n + 127) / 128, tiles = 4 * ((n + 127) / 128) * ((k_ins + 63) / 64);
  if (tiles == 0) return 1;
  int s = (kSlicedItems + tiles - 1) / tiles;
  if (s > (parts + 1) / 2) s = (parts + 1) / 2;
  return s < 1 ? 1 : s;
}
// Partial tiles of one product of a chain, the most over the orders n <= cap.
inline size_t sliced_partials(int cap, int k) {
  size_t most = 0;
  for (int rb = 1; rb <= (cap + 127) / 128; ++rb)
    for (int ct = 1; ct <= (k + 63) / 64; ++ct) {
      const int s = sliced_slices(rb * 128, ct * 64);
      if (s > 1 && (size_t)rb * ct * s > most) most = (size_t)rb * ct * s;
    }
  return most;
}

// Capacity (with the insertions) from which a chain's products are sliced.  One
// chain alone, us per block, float64 pipe against sliced: 187 / 193 at order 100,
// 212 / 220 at 200, 435 / 410 at 300, 513 / 451 at 415; in batches the float64
// pipe saturates, so that the line lies below the crossover of one chain.
constexpr int kSlicedMinOrder = 256;
// k_max from which a sliced chain's flush coefficients Y are a sliced product too:
// us per block of the flush support, float64 pipe against sliced, 53 / 71 for 40
// chains of k_max 32, 37.3 / 36.4 for one of 64 at order 415, 164 / 57 for one of 128
// at order 2085, 2670 / 254 for two of 256 at order 6760.
constexpr int kSlicedYMinK = 64;
// k_max from which G_{new,new} is one: us per block of the prep, float64 pipe against
// sliced, 87 / 108 for one chain of 64 at order 415, 465 / 412 for one of 128 at
// order 2085, 7480 / 5800 for two of 256 at order 6760.
constexpr int kSlicedNewMinK = 128;
// Split of G_{new,new} = C G_{old,new} over its inner dimension: a part or two per
// slice, since it has few tiles (at most eight per spin).
__host__ __device__ inline int sliced_new_slices(int n) { return ((n + 127) / 128 + 1) / 2; }
// Bytes of the strip pool, unless one job needs more; and what its allocation leaves
// for the stacks of kernels, which are allocated when they are first launched.
constexpr size_t kSlicedPool = (size_t)8 << 30, kSlicedReserve = (size_t)256 << 20;

}  // namespace ctaux
