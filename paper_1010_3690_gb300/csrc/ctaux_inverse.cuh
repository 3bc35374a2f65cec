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
  int chunks;           // images per row block that there is room for: 1, or 4 (two levels)
  int width;            // panel width
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

// Panels of 128 columns in two levels (see ctaux_inverse.cu) for matrices of this order
// on, whatever else is in the launch (a chain gives the same bits alone or in a batch):
// the five extra launches per 128 columns against three of four passes over the matrix.
// One level against two, ms per recomputation of one chain: 2.29 / 2.49 at order 700,
// 3.19 / 3.29 at 900, 4.44 / 4.46 at 1100, 6.51 / 6.23 at 1500, 10.9 / 9.6 at 2000.  In a
// batch the passes cost more and the launches less: 96 chains of order 58 to 1084, 8
// blocks with one recomputation, 33.7 ms with the line at 1060, 32.2 at 768, 32.7 at 512
// (31.1 with all of them in two levels, where one chain of order 431 alone takes a tenth
// longer).
constexpr int kInvTwoLevel = 768;
inline int inv_chunks(int ld) { return ld >= kInvTwoLevel ? 4 : 1; }   // images, at the largest order

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

// What the launches need to know of the device; sets the kernels up.  balance: for
// matrices whose rows may differ in scale (one level only); their views then have
// room for it.
struct InvDevice {
  int sm_count;
  int largest;     // CTAs of the largest cluster
  bool balance;
};
cudaError_t inv_device(int sm_count, bool balance, InvDevice* out);
int inv_width(int ld, const InvDevice& dev);   // 32; less where a panel would not fit

// Launch parameters of the inversion of a set of matrices.
struct InvPanel {
  int cluster;     // CTAs of a matrix's cluster (2 to 16)
  int threads;     // of a CTA: 512 in clusters of 16, else 256
  int rows;        // panel rows per CTA at the largest leading dimension
  int smem;        // dynamic shared memory
};
struct InvShape {
  InvDevice dev;
  int width;                     // panel width
  std::vector<InvPanel> panels;  // of each panel: fewer matrices reach the later ones
};
// lds: the leading dimension of every matrix.  One shape for each panel width among them,
// nearly always one in all.
std::vector<InvShape> inv_shapes(const std::vector<int>& lds, const InvDevice& dev);

// Inverts the matrices views[0..items) of orders orders[0..items) (device; 0 =
// leave out), none above max_order: afterwards inv[c][perm[j]] = X[perm[c]][j].
// `used` must be zero and `pcol` -1 on entry.  Returns the kernels launched.
int launch_inverse(const InvView* views, const int* orders, int items, int max_order,
                   const InvShape& sh, cudaStream_t st, cudaError_t* err);

}  // namespace ctaux
