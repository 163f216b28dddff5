// Fixed-point arithmetic of the exactly sliced FP64 products (apply_tc64.cu).
//
// GB300 runs FP64 arithmetic at 1/64 of its FP32 rate, so the pointwise work
// around the tensor-core products uses 64-bit integers at a scale that a whole
// row shares: a double v with |v| < 2^E is the integer v 2^{59-E}, an element's
// coefficient c with |c| < 2^e the integer c 2^{62-e}, and their product needs
// two 32-bit high multiplications and one wide one (a float-float product and
// its conversions took about five times the instructions).
//
// A tensor-core operand is an integer of 56 bits and a sign, cut into seven
// base-256 digits x = sum_k d_k 256^k, balanced (-128 <= d_k <= 127) but for
// the leading one (|d_6| <= 257): adding 128 to every lower digit position turns
// them into the bytes of x + kBias, each byte becomes the FP16 number 1024 + byte
// by a byte permutation, and subtracting 1152 leaves the digit, exactly; the
// leading one keeps ten bits. Two values share every permutation and
// subtraction, so a value costs nine instructions for its seven digits. (Eight
// 7-bit sign-magnitude slices in BF16, the former form, took 32 and 36 slice
// products instead of 34.) Digit products are at most 2^14 (2^15 and 2^16 with
// leading digits), so FP32 accumulators hold sums of several hundred exactly.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#include <cuda_fp16.h>

#include "tc05.cuh"
#define DGX_HD __host__ __device__ __forceinline__
#else
#define DGX_HD inline
#endif

namespace dgx {
namespace fx {

constexpr int kDigits = 7;                       // of each operand
constexpr int kSums = 8;                         // digit sums i + j kept: 0 .. 7
constexpr long long kBias = 0x0200808080808080ll;  // 128 in the six lower digits' bytes, 512 above them
constexpr int kZeroExp = -1100;                  // exponent of an all-zero row
constexpr int kBadExp = 1025;                    // exponent of a row with an infinity or a NaN

DGX_HD long long bits_of(double v) {
  long long b;
#ifdef __CUDA_ARCH__
  b = __double_as_longlong(v);
#else
  std::memcpy(&b, &v, 8);
#endif
  return b;
}
DGX_HD double double_of(long long b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(b);
#else
  double v;
  std::memcpy(&v, &b, 8);
  return v;
#endif
}
DGX_HD int imin(int a, int b) { return a < b ? a : b; }
DGX_HD int imax(int a, int b) { return a > b ? a : b; }

// e with |v| < 2^e (kZeroExp for zero and denormals, kBadExp for inf and NaN)
DGX_HD int exp_bound(double v) {
  const int E = int((bits_of(v) >> 52) & 0x7ff);
  return E == 0 ? kZeroExp : E - 1022;
}

// v 2^{B-E} for |v| < 2^E, truncated towards zero (53 < B <= 62)
template <int B>
DGX_HD long long fix(double v, int E) {
  const long long b = bits_of(v);
  const int Eb = int((b >> 52) & 0x7ff);
  unsigned long long m = ((b & 0xFFFFFFFFFFFFFll) | 0x10000000000000ll);
  m = Eb ? m << (B - 53) : 0ull;
  m >>= imin(imax(E - (Eb - 1022), 0), 63);
  return b < 0 ? -(long long)m : (long long)m;
}

// Arithmetic right shift by any count >= 0.
DGX_HD long long sar(long long x, int n) { return x >> imin(n, 63); }

// A 64-bit integer as h 2^32 + l with both halves signed.
struct Split {
  int h, l;
};
DGX_HD Split split(long long x) {
  const unsigned lo = unsigned(x);
  return Split{int(unsigned(x >> 32) + (lo >> 31)), int(lo)};
}
DGX_HD long long join(Split s) { return (long long)((unsigned long long)(long long)s.h << 32) + s.l; }

DGX_HD long long madwide(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (long long)a * b + c;
#endif
}

// a c / 2^64 to nearest (the product of the low halves, below a quarter, left
// out). Truncation would not do: where neighbours agree the jumps are zero, and a
// bias that every face shares is a smooth source that the inverse amplifies.
DGX_HD long long mul(Split a, Split c) {
  const long long mid = madwide(a.l, c.h, madwide(a.h, c.l, 0x80000000ll));
  return madwide(a.h, c.h, (long long)int(mid >> 32));
}

// I 2^S as a double (rounded to nearest, halves up); below the normal range 0, above it infinity.
DGX_HD double to_double(long long I, int S) {
  const unsigned s = unsigned(I >> 63);
  unsigned long long a = (unsigned long long)((I ^ (I >> 63)) - (I >> 63));
  if (a == 0) return 0.0;
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)a);
#else
  const int lz = __builtin_clzll(a);
#endif
  a <<= lz;
  const int e = S + 63 - lz + 1023;  // biased exponent
  if (e < 1) return 0.0;
  if (e > 2046) return double_of((long long)((unsigned long long)s << 63) | 0x7ff0000000000000ll);
  a = (a >> 11) + ((a >> 10) & 1ull);  // 53 bits, the hidden one adds 1 to the exponent field
  const unsigned long long b = a + ((unsigned long long)(e - 1) << 52);
  return double_of((long long)(b | ((unsigned long long)s << 63)));
}

DGX_HD int round_int(float x) {
#ifdef __CUDA_ARCH__
  return __float2int_rn(x);
#else
  return int(std::nearbyint(x));
#endif
}

// Digit sums of a product, s-th weight 2^{-8s}: sum_s a_s 2^{40-8s}. The last two
// weigh 2^{-8} and 2^{-16} of the result's unit and are added in FP32.
DGX_HD long long from_sums(const float (&a)[kSums]) {
  const int a5 = round_int(fmaf(fmaf(a[7], 0.00390625f, a[6]), 0.00390625f, a[5]));
  long long r = madwide(round_int(a[4]), 256, (long long)a5);
  r = madwide(round_int(a[3]), 65536, r);
  r = madwide(round_int(a[2]), 16777216, r);
  return r + (long long)((unsigned long long)(unsigned)(round_int(a[1]) + round_int(a[0]) * 256) << 32);
}

// The digit sums times 2^S as a double. A small result (a smooth field's, whose
// terms cancel) has room for six more bits of the last sums: rounded to the unit, it
// differs from what the neighbour's takes up, and that was the largest error of an
// element's balance (pressure solve, N = 8, 524,288 triangles: 1.8e-13 against 64
// bits, 0.94e-13 with them).
DGX_HD double sums_to_double(const float (&a)[kSums], int S) {
  const int t = round_int(a[1]) + round_int(a[0]) * 256;
  const bool small = (t < 0 ? -t : t) < (1 << 23);  // the result is below 2^56
  const int n = small ? 6 : 0;
  const int a5 = round_int(fmaf(fmaf(a[7], 0.00390625f, a[6]), 0.00390625f, a[5]) * (small ? 64.0f : 1.0f));
  long long r = madwide(round_int(a[4]), 256 << n, (long long)a5);
  r = madwide(round_int(a[3]), 65536 << n, r);
  r = madwide(round_int(a[2]), 16777216 << n, r);
  return to_double(r + (long long)((unsigned long long)(unsigned)(t << n) << 32), S - n);
}

#ifdef __CUDACC__
// The digits of values x (|x| <= 2^56) as FP16 pairs, slice j = 0 the leading
// digit: eight values are 16 bytes of each slice, four are eight.
__device__ __forceinline__ uint32_t half2_minus(uint32_t h, unsigned short c) {
  const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&h), __half2half2(__ushort_as_half(c)));
  return *reinterpret_cast<const uint32_t*>(&d);
}
__device__ __forceinline__ uint32_t digit_pair(uint32_t bytes, uint32_t sel) {  // 1024 + byte - 1152
  return half2_minus(__byte_perm(bytes, 0x64646464u, sel), 0x6480);
}
// two values' digits: w[j] = slice j
__device__ __forceinline__ void digits2(long long x, long long y, uint32_t (&w)[kDigits]) {
  const unsigned long long p = (unsigned long long)(x + kBias), q = (unsigned long long)(y + kBias);
  const uint32_t pl = uint32_t(p), ql = uint32_t(q), ph = uint32_t(p >> 32), qh = uint32_t(q >> 32);
  const uint32_t t01 = __byte_perm(pl, ql, 0x5140), t23 = __byte_perm(pl, ql, 0x7362);
  const uint32_t t45 = __byte_perm(ph, qh, 0x5140), t6 = __byte_perm(ph, qh, 0x7632);
  w[6] = digit_pair(t01, 0x4140);
  w[5] = digit_pair(t01, 0x4342);
  w[4] = digit_pair(t23, 0x4140);
  w[3] = digit_pair(t23, 0x4342);
  w[2] = digit_pair(t45, 0x4140);
  w[1] = digit_pair(t45, 0x4342);
  w[0] = half2_minus(t6 | 0x64006400u, 0x6600);  // 1024 + ten bits - 1536
}
__device__ __forceinline__ void digits8(const long long (&x)[8], uint8_t* dst, int slice_stride) {
  uint32_t w[4][kDigits];
#pragma unroll
  for (int i = 0; i < 4; ++i) digits2(x[2 * i], x[2 * i + 1], w[i]);
#pragma unroll
  for (int j = 0; j < kDigits; ++j)
    *reinterpret_cast<uint4*>(dst + j * slice_stride) = make_uint4(w[0][j], w[1][j], w[2][j], w[3][j]);
}
__device__ __forceinline__ void digits4(const long long (&x)[4], uint8_t* dst, int slice_stride) {
  uint32_t w[2][kDigits];
#pragma unroll
  for (int i = 0; i < 2; ++i) digits2(x[2 * i], x[2 * i + 1], w[i]);
#pragma unroll
  for (int j = 0; j < kDigits; ++j)
    *reinterpret_cast<uint2*>(dst + j * slice_stride) = make_uint2(w[0][j], w[1][j]);
}

// accumulator columns d .. d + rows += data digit x the operator's stacked rows
// (ROW bytes of shared memory apart: 32 for blocks 16 columns wide, 64 for 32)
template <int ROW>
__device__ __forceinline__ void issue_rows(uint32_t d, uint64_t a, uint64_t b, int rows, uint32_t acc) {
  const int n0 = rows <= 256 ? rows : ((rows / 2 + 15) & ~15);
  tc::mma_ss(d, a, b, tc::idesc_f16(128, n0, false), acc);
  if (n0 < rows) tc::mma_ss(d + n0, a, b + ((n0 * ROW) >> 4), tc::idesc_f16(128, rows - n0, false), acc);
}
// The digit products i + j <= 7 of 16 columns: data digits (slices of `aslice`
// bytes at a) with the operator's (nc stacked rows each at b); `first` starts the sums.
template <int ROW>
__device__ __forceinline__ void issue_step(uint32_t d, uint64_t a, int aslice, uint64_t b, int nc, bool first) {
  issue_rows<ROW>(d, a, b, kDigits * nc, first ? 0u : 1u);  // sums 0 .. 6
  a += aslice >> 4;
  if (first) {  // sums 1 .. 6 are there, sum 7 starts here
    issue_rows<ROW>(d + nc, a, b, (kDigits - 1) * nc, 1u);
    issue_rows<ROW>(d + kDigits * nc, a, b + (((kDigits - 1) * nc * ROW) >> 4), nc, 0u);
  } else {
    issue_rows<ROW>(d + nc, a, b, kDigits * nc, 1u);
  }
#pragma unroll 1
  for (int j = 2; j < kDigits; ++j) {
    a += aslice >> 4;
    issue_rows<ROW>(d + j * nc, a, b, (kSums - j) * nc, 1u);
  }
}
#endif

// ------------------------------------------------------------------ operators (host)
inline int ceil_log2(double x) {  // e with x < 2^e (0 for zero)
  int e = 0;
  std::frexp(x, &e);
  return e;
}
// A row's exponent: its entries below 2^e, and its absolute sum below 2^{e+6}, so
// that a product's digit sums stay below 2^62 where from_sums joins them.
inline int row_exp(double mx, double l1) { return imax(ceil_log2(mx), ceil_log2(l1) - 6); }

inline uint16_t fp16_int(int d) {  // exact for |d| <= 2048
  if (d == 0) return 0;
  const int m = d < 0 ? -d : d;
  int e = 0;
  while ((m >> e) > 1) ++e;
  return uint16_t((d < 0 ? 0x8000 : 0) | ((e + 15) << 10) | (((m << 10) >> e) & 0x3ff));
}
// The digits of an integer (|x| <= 2^56 + 1), leading one first.
inline void digits_of(long long x, int (&out)[kDigits]) {
  for (int i = kDigits - 1; i >= 0; --i) {  // last digit first
    const int d = i == 0 ? int(x) : int((x + 128) & 255) - 128;
    x = (x - d) >> 8;
    out[i] = d;
  }
}

// An operator row's digits, for the bound on its products' digit sums. Sums 0 .. 4
// have to be integers below 2^24, which FP32 holds exactly, whatever the data (whose
// leading digit is at most 257 in size, the others 128). Sum 5 weighs one unit of the
// result, 2^-56 of its bound, 6 and 7 less: where digits of one sign in every place take
// them past 2^24 (1.12 of it at degree 9, 1.28 at degree 10) a step's rounding is one
// unit of the result or less.
struct ExactSums {
  double l1[5] = {};
  void add(const int (&d)[kDigits]) {
    for (int i = 0; i < 5; ++i) l1[i] += d[i] < 0 ? -d[i] : d[i];
  }
  bool exact() const {
    for (int s = 0; s < 5; ++s) {
      double most = 257.0 * l1[s];
      for (int i = 0; i < s; ++i) most += 128.0 * l1[i];
      if (most >= 16777216.0) return false;
    }
    return true;
  }
};

}  // namespace fx
}  // namespace dgx
