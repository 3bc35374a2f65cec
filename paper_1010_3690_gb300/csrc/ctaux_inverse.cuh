// Blocked Gauss-Jordan inversion in place, with partial pivoting, of many
// matrices at once: the from-scratch recomputation of N and the inversion
// entry point without allocation (kernels in ctaux_inverse.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

namespace ctaux {

// One matrix and its work area (device pointers).
struct InvView {
  double* X;            // the matrix, column-major, leading dimension ld
  int ld;
  int chunks;           // images per row block: 1, or 4 (panels of 128 columns in two levels)
  unsigned char* As;    // slice images of the panel's columns: ceil(ld / 128) x chunks x oz::kImageA
  unsigned char* Bs;    // slice images of the pivot rows: ceil(ld / 64) x chunks x oz::kImageB
  int* ea;              // row exponents of the images
  int* eb;
  int* perm;            // pivot row of each column
  int8_t* used;         // row already pivoted
  int* pcol;            // column at which a row was pivoted, -1 if not yet
  double* piv;          // pivots, in column order
  double* L;            // [32][32] multipliers of the current panel's pivot rows
  int* balance;         // [32] balance of the current panel (ctaux_inverse.cu); null where the
                        // matrix is known to have rows of one scale
  int* status;          // DS_SINGULAR and DS_TIMEOUT bits
};

// Panels of 128 columns in two levels (see ctaux_inverse.cu) where the largest
// leading dimension of a launch is at least this: the five extra launches per
// 128 columns against three of four passes over the matrix.  One level against
// two, ms per recomputation of one chain: 2.29 / 2.49 at order 700, 3.19 / 3.29
// at 900, 4.44 / 4.46 at 1100, 6.51 / 6.23 at 1500, 10.9 / 9.6 at 2000 (leading
// dimensions a quarter above the order).
constexpr int kInvTwoLevel = 1408;
inline int inv_chunks(int max_ld) { return max_ld >= kInvTwoLevel ? 4 : 1; }

// Doubles of As, Bs, ea, eb and piv for a leading dimension (the matrix itself
// comes first and takes ld^2 doubles).
__host__ __device__ inline size_t inv_extra_doubles(int ld, int chunks = 4) {
  const size_t lp = (size_t)((ld + 127) / 128 * 128);
  return lp * (112 * (size_t)chunks + 2) + 1024;   // 2 x 448 bytes of slices per chunk; L
}
__host__ __device__ inline void inv_layout(double* work, int ld, int chunks, InvView& v) {
  const size_t lp = (size_t)((ld + 127) / 128 * 128), slices = lp * 448 * (size_t)chunks;
  v.X = work;
  v.ld = ld;
  v.chunks = chunks;
  unsigned char* p = reinterpret_cast<unsigned char*>(work + (size_t)ld * ld);
  v.As = p;
  v.Bs = p + slices;
  v.ea = reinterpret_cast<int*>(p + 2 * slices);
  v.eb = v.ea + lp;
  v.piv = reinterpret_cast<double*>(v.eb + lp);
  v.L = v.piv + lp;
}

// Column of the inverse that column j of X holds.  After a bounded wait gave up
// (status beyond `singular`, a zero pivot's bit), perm may hold rows of an earlier,
// larger matrix, and what X holds is of no use: every column then stays in its place,
// inside the caller's matrix.
__host__ __device__ inline int inv_column(int status, int singular, const int* perm, int j) {
  return (status & ~singular) ? j : perm[j];
}

// Launch parameters of the inversion of a set of matrices.
struct InvPanel {
  int cluster;     // CTAs of a matrix's cluster (2 to 16)
  int threads;     // of a CTA: 512 in clusters of 16, else 256
  int rows;        // panel rows per CTA at the largest leading dimension
  int smem;        // dynamic shared memory
};
struct InvShape {
  int width;                     // panel width (32; 16 or 8 where a panel would not fit)
  int chunks;                    // 4: two levels
  int sm_count;
  bool balance;
  std::vector<InvPanel> panels;  // of each panel: fewer matrices reach the later ones
};
// lds: the leading dimension of every matrix.  balance: for matrices whose rows may
// differ in scale (one level only); their views then have room for it.
cudaError_t inv_configure(const std::vector<int>& lds, int sm_count, bool balance, InvShape* out);

// Inverts the matrices views[0..items) of orders orders[0..items) (device; 0 =
// leave out), none above max_order: afterwards inv[c][perm[j]] = X[perm[c]][j].
// `used` must be zero and `pcol` -1 on entry.  Returns the kernels launched.
int launch_inverse(const InvView* views, const int* orders, int items, int max_order,
                   const InvShape& sh, cudaStream_t st, cudaError_t* err);

}  // namespace ctaux
