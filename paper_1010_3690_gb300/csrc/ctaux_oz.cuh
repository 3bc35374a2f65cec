// Float64 products on the float16 tensor cores, by error-free slicing (Ozaki,
// Ogita, Oishi & Rump, Numer. Algorithms 59 (2012) 95; Mukunoki et al., ISC 2020).
//
// GB300 runs float64 at 1/64 of its float32 rate (2 multiply-adds per SM and
// clock) and float16 tensor products at 4096.  Each row of an operand (32
// consecutive elements of the inner dimension) is scaled by a power of two and
// rounded to a fixed-point number of 7 balanced base-256 digits (|digit| <=
// 128, exact in float16):
//   x = 2^(e - 55) sum_{i<7} d_i 256^(6 - i) + r,  |r| <= 2^(e - 56),  |x| < 2^e.
// A product of two such rows is sum_g 256^(12 - g) sum_{i+j=g} <a_i, b_j>, and
// every inner product of digit rows is a sum of integers that float32
// accumulates exactly: K <= 32 elements, at most 7 digit pairs per group g and
// |d_i d_j| <= 2^14 give |sum| < 2^22.  Groups g = 0..7 are kept (34 digit
// products); what is dropped is below 2^(ea + eb - 61) per element.  The eight
// group sums are combined as one 64-bit integer S with
//   <a, b> = S 2^(ea + eb - 56)
// rounded once in its last place.  That is below the rounding of a chain of 32 float64
// multiply-adds, which is relative to the running sum, where the elements of a row (and
// of a column of the other operand) are of one scale: an element 2^t below its row's
// largest keeps 55 - t bits.  Where they are not, the caller balances the inner index by
// powers of two first (ctaux_sliced.cu, ctaux_inverse.cu).
//
// Slice images: an operand block of R rows (128 for A, 64 for B) and 32 inner
// elements is stored as 7 consecutive [R][32] float16 tiles (64-byte rows,
// 64-byte swizzle), in the layout the tensor cores read, so that one
// contiguous bulk copy fills a shared-memory stage.
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

#include "ctaux_tc.cuh"

namespace ctaux {
namespace oz {

constexpr int kSlices = 7, kGroups = 8;
constexpr int kK = 32;                                   // inner elements of an image
constexpr int kRowsA = 128, kRowsB = 64;
constexpr int kImageA = kSlices * kRowsA * 64;           // bytes
constexpr int kImageB = kSlices * kRowsB * 64;
constexpr int kRowBytes = kSlices * 64;                  // slice bytes of one operand row
constexpr int kNonFinite = 1 << 20;                      // exponent of a row holding inf or NaN

// Biased exponent field of x's upper word.
__device__ __forceinline__ int exp_field(uint32_t hi) { return (int)((hi >> 20) & 0x7ffu); }

// Exponent e of a row from its largest exponent field: |x| < 2^e.
__device__ __forceinline__ int row_exponent(int max_field) {
  return max_field == 0x7ff ? kNonFinite : max_field - 1022;
}

// x 2^shift as a fixed-point integer, ~ q 2^(e - 55), |q| <= 2^55, plus the bias
// that makes the six low bytes the digits + 128 (the digits are balanced); the
// seventh digit is the (signed) rest.  max_field: the row's largest exponent
// field, its shift added.  Subnormal x count as zero.
__device__ __forceinline__ long long biased_digits(double x, int max_field, int shift = 0) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)(bits >> 52) & 0x7ff;
  const int t = max_field - ex - shift;   // >= 0
  unsigned long long q = 0;
  if (ex != 0 && t < 56) {
    const unsigned long long v = ((bits & 0xfffffffffffffull) | 0x10000000000000ull) << 2;
    q = (v + ((1ull << t) >> 1)) >> t;
  }
  const long long s = (long long)bits < 0 ? -(long long)q : (long long)q;
  return s + 0x808080808080ll;
}

// Digit i (0 = most significant) of a biased value, plus 128: 0..256.
__device__ __forceinline__ uint32_t digit_u(long long y, int i) {
  return i == 0 ? (uint32_t)((int)(y >> 48) + 128) : (uint32_t)(y >> (8 * (6 - i))) & 0xffu;
}
// Two digits as float16 integers: 1024 + u has the bits 0x6400 + u.
__device__ __forceinline__ uint32_t digits_half2(uint32_t u0, uint32_t u1) {
  const uint32_t p = (0x6400u + u0) | ((0x6400u + u1) << 16);
  __half2 h;
  *reinterpret_cast<uint32_t*>(&h) = p;
  h = __hsub2(h, __half2half2(__ushort_as_half(0x6480)));   // 1152
  return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ uint16_t digit_half(uint32_t u) {
  return __half_as_ushort(__hsub(__ushort_as_half((unsigned short)(0x6400u + u)), __ushort_as_half(0x6480)));
}
// Byte offset of the 16-byte chunk `c` (8 inner elements) of row r in a tile
// with the 64-byte swizzle.
__device__ __forceinline__ uint32_t chunk_offset(int r, int c) {
  return (uint32_t)(r * 64 + ((c ^ ((r >> 1) & 3)) << 4));
}

// Eight elements of a row (biased values y) into every slice of an image, at
// the byte offset `dst` of its first slice.
__device__ __forceinline__ void store_chunk(unsigned char* dst, int image_rows, const long long* y) {
#pragma unroll
  for (int i = 0; i < kSlices; ++i) {
    uint4 q;
    q.x = digits_half2(digit_u(y[0], i), digit_u(y[1], i));
    q.y = digits_half2(digit_u(y[2], i), digit_u(y[3], i));
    q.z = digits_half2(digit_u(y[4], i), digit_u(y[5], i));
    q.w = digits_half2(digit_u(y[6], i), digit_u(y[7], i));
    *reinterpret_cast<uint4*>(dst + (size_t)i * image_rows * 64) = q;
  }
}

// kind::f16 instruction descriptor: D float32, A and B float16, both K-major, M = 128, N = 64.
constexpr uint32_t kIdesc = (1u << 4) | ((uint32_t)(64 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);

// One thread of a converged warp (the same one every time).
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}

// Shared-memory descriptors of K-major tiles with 64-byte rows (tc::smem_desc):
// the lower word holds the address, the upper one is constant.
constexpr uint32_t kDescHigh = (512u >> 4) | (1u << 14) | (4u << 29);

template <bool ACC>
__device__ __forceinline__ void mma_f16(uint32_t tmem, uint32_t a_low, uint32_t b_low) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b64 da, db;\n mov.b64 da, {%1, %3};\n mov.b64 db, {%2, %3};\n"
      " setp.ne.b32 p, %5, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n}\n" ::"r"(tmem),
      "r"(a_low), "r"(b_low), "n"(kDescHigh), "n"(kIdesc), "n"(ACC ? 1 : 0)
      : "memory");
}

// All digit products of one pair of images into the eight group accumulators
// (64 TMEM columns each), FIRST clearing them; by the elected thread of a
// converged warp.  With addresses that are uniform in the warp and 32-bit
// arithmetic an MMA issues every 48 clocks also beside busy epilogue warps; from
// one thread in a divergent branch with 64-bit descriptors it took 75 there.
template <bool FIRST>
__device__ __forceinline__ void mma_images(uint32_t tmem, uint32_t a, uint32_t b) {
  const uint32_t al = (a >> 4) | (1u << 16), bl = (b >> 4) | (1u << 16);
#pragma unroll
  for (int kk = 0; kk < 2; ++kk) {
#pragma unroll
    for (int i = 0; i < kSlices; ++i) {
#pragma unroll
      for (int j = 0; j < kSlices; ++j) {
        const int g = i + j;
        if (g >= kGroups) continue;
        const uint32_t x = al + (uint32_t)((i * kRowsA * 64 + kk * 32) >> 4), y = bl + (uint32_t)((j * kRowsB * 64 + kk * 32) >> 4);
        // the first product of group g is digit 0 of A (g = 7: digit 1)
        if (FIRST && kk == 0 && i == (g == 7 ? 1 : 0)) mma_f16<false>(tmem + 64 * g, x, y);
        else mma_f16<true>(tmem + 64 * g, x, y);
      }
    }
  }
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(mbar)
      : "memory");
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Exact float32 integer a of magnitude below 2^22 as the bits 0x4b400000 + a.
__device__ __forceinline__ uint32_t small_bits(uint32_t f) {
  return __float_as_uint(__uint_as_float(f) + 12582912.f);
}

// The same for sums over up to 128 elements (|a| < 2^24, exact in float32 too):
// unit 2^(ea + eb - 54), |S| < 2^62.  Only the first two groups stay below 2^22.
__device__ __forceinline__ long long combine128(const uint32_t* g) {
  constexpr uint32_t kB = 0x4b400000u;
  auto num = [&](int i) { return __float2int_rn(__uint_as_float(g[i])); };
  const uint32_t high = small_bits(g[1]) + small_bits(g[0]) * 256u - 257u * kB;
  // the last two are rounded to the next unit in float32 (a conversion to an
  // integer issues at a quarter of the rate); every sum here is below 2^24
  auto round8 = [](float a) { return fmaf(a, 1.f / 256.f, 12582912.f) - 12582912.f; };
  auto f = [&](int i) { return __uint_as_float(g[i]); };
  const int low = __float2int_rn(f(5) + round8(f(6) + round8(f(7))));
  long long s = (long long)num(2) * (1 << 24) + (long long)low;
  s += (long long)num(3) * (1 << 16);
  s += (long long)num(4) * (1 << 8);
  return (long long)((unsigned long long)s + ((unsigned long long)high << 32));
}

// The group sums of one output element as S (see above): unit 2^(ea + eb - 56).
// The biases of the eight conversions are taken off together.
__device__ __forceinline__ long long combine(const uint32_t* g) {
  constexpr uint32_t kB = 0x4b400000u;
  const uint32_t b0 = small_bits(g[0]), b1 = small_bits(g[1]), b2 = small_bits(g[2]), b3 = small_bits(g[3]),
                 b4 = small_bits(g[4]), b5 = small_bits(g[5]), b6 = small_bits(g[6]), b7 = small_bits(g[7]);
  // 32-bit arithmetic modulo 2^32 is exact for what fits
  const int low = (int)((b5 - kB) * 4u) + ((int)(b6 * 256u + b7 + ((1u << 13) - 257u * kB)) >> 14);
  const uint32_t high = b1 * 4u + b0 * 1024u - 1028u * kB;
  constexpr unsigned long long kBias = (unsigned long long)kB * ((1ull << 26) + (1ull << 18) + (1ull << 10));
  unsigned long long s = (unsigned long long)b2 * (1u << 26) + ((unsigned long long)(long long)low - kBias);
  s += (unsigned long long)b3 * (1u << 18);
  s += (unsigned long long)b4 * (1u << 10);
  return (long long)(s + ((unsigned long long)high << 32));
}

// S 2^E rounded to float64 (|S| < 2^62); float64 conversions run on the slow
// float64 pipe, so this is integer arithmetic.  Results below the normal
// range are zero, above it infinite; E of a non-finite operand row gives NaN.
__device__ __forceinline__ double scaled_double(long long s, int E) {
  const unsigned long long u = (unsigned long long)(s < 0 ? -s : s);
  const int lz = __clzll((long long)u);
  const unsigned long long v = u << lz;                       // leading one at bit 63
  const unsigned long long mant = (v >> 11) + ((v >> 10) & 1ull);   // [2^52, 2^53]
  const int be = 1023 + 63 - lz + E;                          // biased exponent
  unsigned long long bits = mant + ((unsigned long long)(uint32_t)(be - 1) << 52);
  if (be <= 0 || u == 0) bits = 0;
  if (be >= 0x7ff && u != 0) bits = 0x7ff0000000000000ull;
  if (E > 4096) bits = 0x7ff8000000000000ull;
  return __longlong_as_double((long long)(bits | ((unsigned long long)s & 0x8000000000000000ull)));
}

}  // namespace oz
}  // namespace ctaux
