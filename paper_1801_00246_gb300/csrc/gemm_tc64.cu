// Dense FP64 products on the Blackwell tensor cores (tcgen05) for the tetrahedral
// apply and the advection: out[row] = A X[row] for 128 rows per tile, exact to
// FP64 accuracy by integer slicing (the error-free splitting of Ozaki et al.,
// Numer. Algorithms 59, 2012). Every operator row is scaled by a power of two and
// cut into 8 signed 7-bit slices on the host, every data row the same way on the
// device (integer operations on the double's bits); the 36 slice products with
// i + j <= 7 run as tcgen05.mma (BF16 operands from shared memory, FP32
// accumulators in tensor memory, one accumulator per slice exponent i + j: integer
// sums below 2^24 for K <= 256 and up to 4 products, exact); the accumulators are
// recombined by Horner's rule in float-float and rebuilt as doubles from the
// exponent bits. Data slices are written by the threads into a double-buffered
// shared-memory chunk (32 columns) while the previous chunk's products run;
// operator blocks (48 rows x 32 columns, 8 slices) arrive by bulk copy.
// Accuracy: relative error near 2^-44 of |A||X| (the slicing's).
#include <cmath>
#include <cstring>
#include <vector>

#include "dg_internal.h"
#include "tc05.cuh"

namespace dgx {
namespace {

constexpr int kT = 128;                      // rows per tile (MMA M)
constexpr int kKC = 32;                      // data columns per chunk
constexpr int kNC = 48;                      // output columns per pass (MMA N)
constexpr int kSl = 8;                       // slices of 7 bits
// Longest sum: a slice product is below 127^2 in magnitude, and an accumulator
// group with up to 4 products over 256 terms stays below 4 * 256 * 127^2 <
// 2^24, an integer FP32 represents exactly; groups with more products carry
// weights below 2^-28 of the leading one (the fifth group stays exact up to
// 208 terms: 5 * 208 * 127^2 < 2^24).
constexpr int kMaxDepth = 256;
constexpr int kABytes = kSl * kT * kKC * 2;  // one data chunk, 8 slices: 64 KB
constexpr int kBBytes = kSl * kNC * kKC * 2; // one operator block, 8 slices: 24 KB
constexpr int kASlice = kT * kKC * 2, kBSlice = kNC * kKC * 2;
constexpr int kSmem = 2 * kABytes + 2 * kBBytes + 4 * kT * 4 + 12 * 8;  // the tail: 10 mbarriers, slot, 2 flags

__device__ int g_tc64_err;

// exponent e with |v| < 2^e (-1100 for zero)
__device__ __forceinline__ int exp_bound64(double v) {
  const int E = int((__double_as_longlong(v) >> 52) & 0x7ff);
  return E == 0 ? -1100 : E - 1022;
}

// |v| 2^{56 - E} as a 56-bit integer (|v| < 2^E) and its sign
__device__ __forceinline__ uint64_t fixed56(double v, int E, uint32_t& sgn) {
  const unsigned long long b = __double_as_longlong(v);
  const int Eb = int((b >> 52) & 0x7ff);
  sgn = uint32_t(b >> 63);
  if (Eb == 0) return 0ull;
  const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  const int sh = Eb - 1075 + 56 - E;  // <= 3 whenever |v| < 2^E
  if (sh >= 0) return sh < 11 ? (m << sh) : 0ull;
  return sh > -63 ? (m >> (-sh)) : 0ull;
}
// exact double of (h + l) 2^sc for a float-float pair with |l| small against h
__device__ __forceinline__ double ff_to_double(float h, float l, int sc) {
  const float s = __fadd_rn(h, l);
  l = __fsub_rn(l, __fsub_rn(s, h));
  h = s;
  const uint32_t uh = __float_as_uint(h), ul = __float_as_uint(l);
  const int eh = int((uh >> 23) & 0xffu), el = int((ul >> 23) & 0xffu);
  if (eh == 0) return 0.0;
  long long M = (long long)((uh & 0x7fffffu) | 0x800000u) << 29;  // h in a 53-bit frame
  if (el != 0) {
    const int sh = 29 - (eh - el);
    const long long ml = (long long)((ul & 0x7fffffu) | 0x800000u);
    long long Ml = sh >= 0 ? (ml << sh) : (sh > -40 ? (ml >> (-sh)) : 0ll);
    if ((uh ^ ul) >> 31) Ml = -Ml;
    M += Ml;
  }
  int e = eh;
  if (M >= (1ll << 53)) {
    M >>= 1;
    ++e;
  } else if (M < (1ll << 52)) {
    M <<= 1;
    --e;
  }
  const unsigned long long bits = ((unsigned long long)(uh >> 31) << 63) |
                                  ((unsigned long long)(e - 127 + 1023 + sc) << 52) |
                                  ((unsigned long long)M & 0xFFFFFFFFFFFFFull);
  return __longlong_as_double((long long)bits);
}

// ------------------------------------------------------------------ float-float
struct ff {
  float h, l;
};
__device__ __forceinline__ ff ff_renorm(float s, float e) {
  const float h = __fadd_rn(s, e);
  return ff{h, __fsub_rn(e, __fsub_rn(h, s))};
}
// ------------------------------------------------------------------ the GEMM
// Horner's rule over the 8 slice sums of one output column: (h, l) with
// h + l = sum_s acc_s 2^{-7 s} (float-float)
__device__ __forceinline__ ff horner8(const uint32_t (&acc)[kSl][4], int c) {
  float h = __uint_as_float(acc[kSl - 1][c]), l = 0.f;
#pragma unroll
  for (int s = kSl - 2; s >= 0; --s) {
    const float a = __uint_as_float(acc[s][c]);
    const float hs = h * 0.0078125f, ls = l * 0.0078125f;
    const float sum = __fadd_rn(a, hs);
    const float bb = __fsub_rn(sum, a);
    const float err = __fadd_rn(__fsub_rn(a, __fsub_rn(sum, bb)), __fsub_rn(hs, bb));
    h = sum;
    l = __fadd_rn(ls, err);
  }
  return ff_renorm(h, l);
}

// out[r][c] = sum_k A[c][k] X[r][k] for r < rows, c < M, k < Kd (A sliced in
// blocks of kNC rows x kKC columns: block (nc, kc) at (nc KCH + kc) kBBytes).
//
// Warp-specialised pipeline over a stream of data chunks (tile, output pass
// nc, column chunk kc), chunk g using shared-memory buffer g & 1:
//  * warps 0-15 (four threads per row of the 128-row tile) find each row's
//    scale exponent, slice chunk g into buffer g & 1 once the products of
//    chunk g - 2 have released it (mbarrier `empty`), signal `full`, and after
//    a pass's last chunk wait for its accumulators (`acc_full`), drain them
//    (Horner's rule, epilogue) and release them (`acc_empty`);
//  * warp 16 loads operator block g by bulk copy, waits for `full`, issues the
//    36 slice products per 16 columns from one lane and commits to `empty`
//    (and to `acc_full` after a pass's last chunk); before a pass's first
//    chunk it waits until the previous pass has been drained.
// No CTA-wide barrier in the steady state; every wait is bounded in time.
constexpr int kSlicers = 512;  // threads of warps 0-15
__global__ void __launch_bounds__(kSlicers + 32, 1) tc64_gemm(int64_t rows, int M, int Kd, int NCH, int KCH,
                                                              const double* __restrict__ X, int64_t ldx, int vec2,
                                                              const int* __restrict__ ex_given,
                                                              const uint8_t* __restrict__ Bops,
                                                              const int* __restrict__ ea, double* __restrict__ out,
                                                              int64_t ldo, int accum) {
  extern __shared__ __align__(1024) uint8_t sm[];
  uint8_t* sA = sm;                        // [2][8 slices][128 rows][32] canonical
  uint8_t* sB = sm + 2 * kABytes;          // [2][8 slices][48 rows][32] canonical
  int* pmax = reinterpret_cast<int*>(sB + 2 * kBBytes);  // [4][kT]
  // full[2], empty[2], bfull[2], acc_full, acc_empty, bempty[2]
  uint64_t* bars = reinterpret_cast<uint64_t*>(pmax + 4 * kT);
  uint64_t *full = bars, *empty = bars + 2, *bfull = bars + 4, *acc_full = bars + 6, *acc_empty = bars + 7,
           *bempty = bars + 8;
  uint32_t* slot = reinterpret_cast<uint32_t*>(bars + 10);
  int* abort_flag = reinterpret_cast<int*>(slot + 1);
  int* tile_abort = abort_flag + 1;  // the slicers' common copy of abort_flag at a tile's start
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t ntiles = (rows + kT - 1) / kT;
  // with at most two data chunks per row, both stay in the two buffers for all
  // output passes of a tile: sliced once per tile instead of once per pass
  const bool resident = KCH <= 2 && NCH > 1;
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(full + i, kSlicers / 32);  // one arrival per slicing warp
      tc::mbar_init(empty + i, 1);             // the products' commit
      tc::mbar_init(bfull + i, 1);             // the bulk copy
    }
    tc::mbar_init(acc_full, 1);
    tc::mbar_init(acc_empty, kSlicers / 32);
    for (int i = 0; i < 2; ++i) tc::mbar_init(bempty + i, 1);  // an operator stage's products completed
    *abort_flag = 0;
    tc::mbar_init_fence();
  }
  if (warp == 0) tc::tmem_alloc(slot, 512);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tb = *slot;
  constexpr uint32_t idesc = tc::idesc_f16(128, kNC, true);

  if (warp == kSlicers / 32) {
    // ================= products
    uint32_t g = 0, pass = 0, it = 0;
    const uint64_t adesc0 = tc::smem_desc(tc::smem_addr(sA), 128, (kKC / 8) * 128);
    const uint64_t bdesc0 = tc::smem_desc(tc::smem_addr(sB), 128, (kKC / 8) * 128);
    for (int64_t tile = blockIdx.x; tile < ntiles && !*abort_flag; tile += gridDim.x, ++it) {
      for (int nc = 0; nc < NCH; ++nc, ++pass) {
        // the accumulators are free once the previous pass has been drained
        if (pass > 0 && !tc::mbar_wait(acc_empty, (pass - 1) & 1u)) *abort_flag = 1;
        tc::fence_after();
        for (int kc = 0; kc < KCH; ++kc, ++g) {
          const uint32_t bs = g & 1u;                 // operator stage
          const uint32_t bd = resident ? kc : bs;     // data buffer
          // the operator stage is free once chunk g - 2's products completed
          if (g >= 2 && !tc::mbar_wait(bempty + bs, ((g - 2) >> 1) & 1u)) *abort_flag = 1;
          if (lane == 0) {
            tc::mbar_expect_tx(bfull + bs, kBBytes);
            tc::bulk_g2s(sB + bs * kBBytes, Bops + size_t(nc * KCH + kc) * kBBytes, kBBytes, bfull + bs);
          }
          __syncwarp();
          // the data chunk: sliced once per chunk, or (resident) once per tile for all passes
          if (!resident && !tc::mbar_wait(full + bd, (g >> 1) & 1u)) *abort_flag = 1;
          if (resident && nc == 0 && !tc::mbar_wait(full + bd, it & 1u)) *abort_flag = 1;
          if (!tc::mbar_wait(bfull + bs, (g >> 1) & 1u)) *abort_flag = 1;
          tc::fence_after();
          if (lane == 0) {
            const uint64_t ab = adesc0 + ((bd * kABytes) >> 4), bb = bdesc0 + ((bs * kBBytes) >> 4);
            uint32_t started = kc > 0 ? 0xffu : 0u;
#pragma unroll
            for (int ks = 0; ks < kKC / 16; ++ks)
#pragma unroll
              for (int i = 0; i < kSl; ++i)
#pragma unroll
                for (int j = 0; j < kSl - i; ++j) {
                  const int s = i + j;
                  tc::mma_ss(tb + s * kNC, ab + ((j * kASlice + ks * 256) >> 4), bb + ((i * kBSlice + ks * 256) >> 4),
                             idesc, (started >> s) & 1u);
                  started |= 1u << s;
                }
            tc::mma_commit(bempty + bs);
            if (!resident || nc == NCH - 1) tc::mma_commit(empty + bd);  // the data buffer is free
            if (kc == KCH - 1) tc::mma_commit(acc_full);
          }
          __syncwarp();
        }
      }
    }
  } else {
    // ================= slicing and epilogue
    const int e = (warp & 3) * 32 + lane;
    const int q = warp >> 2;
    const uint32_t lanebase = uint32_t((warp & 3) * 32) << 16;
    uint32_t g = 0, pass = 0, it = 0;
    auto load8 = [&](const double* xr, bool live, int k0, double (&v)[8]) {
      if (live && vec2 && k0 + 8 <= Kd) {
        const double2* p2 = reinterpret_cast<const double2*>(xr + k0);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const double2 w = __ldg(p2 + t);
          v[2 * t] = w.x;
          v[2 * t + 1] = w.y;
        }
      } else {
#pragma unroll
        for (int t = 0; t < 8; ++t) v[t] = (live && k0 + t < Kd) ? __ldg(xr + k0 + t) : 0.0;
      }
    };
    // output product (row exponents given): the last chunk of a tile requests the
    // next tile's first chunk and exponent (vn, En), so that their latency overlaps
    // the drain
    bool have_next = false;
    int En = 0;
    double vn[8];  // the next chunk's values (loaded one chunk ahead)
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it) {
      // every slicer takes the same decision to stop (they meet at named barriers below)
      asm volatile("bar.sync 1, %0;\n" ::"r"(kSlicers) : "memory");
      if (tid == 0) *reinterpret_cast<volatile int*>(tile_abort) = *reinterpret_cast<volatile int*>(abort_flag);
      asm volatile("bar.sync 1, %0;\n" ::"r"(kSlicers) : "memory");
      if (*reinterpret_cast<volatile int*>(tile_abort)) break;
      const int64_t row = tile * kT + e;
      const bool live = row < rows;
      const double* xr = X + (live ? row : 0) * ldx;
      // scale exponent of the row: a bound |X[row][k]| < 2^E, given by the producer
      // of X or found here
      int E;
      if (ex_given) {
        E = have_next ? En : (live ? __ldg(ex_given + row) : 0);
        if (E == -1100) E = 0;
      } else {
        int em = -1100;
        if (live) {
          double v[2][8];
          for (int kc = 0; kc < KCH; kc += 2) {
            load8(xr, live, kc * kKC + 8 * q, v[0]);
            load8(xr, live && kc + 1 < KCH, (kc + 1) * kKC + 8 * q, v[1]);
#pragma unroll
            for (int t = 0; t < 8; ++t) em = max(em, max(exp_bound64(v[0][t]), exp_bound64(v[1][t])));
          }
        }
        asm volatile("bar.sync 1, %0;\n" ::"r"(kSlicers) : "memory");  // pmax free (previous tile read it)
        pmax[q * kT + e] = em;
        asm volatile("bar.sync 1, %0;\n" ::"r"(kSlicers) : "memory");
        E = max(max(pmax[e], pmax[kT + e]), max(pmax[2 * kT + e], pmax[3 * kT + e]));
        if (E == -1100) E = 0;
      }
      if (!have_next) load8(xr, live, 8 * q, vn);
      have_next = false;
      for (int nc = 0; nc < NCH; ++nc, ++pass) {
        for (int kc = 0; kc < KCH; ++kc, ++g) {
          if (resident && nc > 0) continue;  // the tile's chunks are still in the buffers
          const uint32_t b = resident ? uint32_t(kc) : (g & 1u);
          double v[8];
#pragma unroll
          for (int t = 0; t < 8; ++t) v[t] = vn[t];
          {  // request the next chunk of this row (the next pass starts again at chunk 0)
            const int kn = kc + 1 < KCH ? kc + 1 : 0;
            if (kc + 1 < KCH || (nc + 1 < NCH && !resident)) {
              load8(xr, live, kn * kKC + 8 * q, vn);
            } else if (ex_given && nc + 1 == NCH && tile + gridDim.x < ntiles) {
              const int64_t nrow = row + int64_t(gridDim.x) * kT;
              const bool nlive = nrow < rows;
              load8(X + (nlive ? nrow : 0) * ldx, nlive, 8 * q, vn);
              En = nlive ? __ldg(ex_given + nrow) : 0;
              have_next = true;
            }
          }
          // each value's 56-bit fixed-point magnitude as two 28-bit halves, and its sign
          // as the pair (s, c) with fma(2^23 + x, s, c) = +-x exactly for 0 <= x < 2^23
          uint32_t hi[8], lo[8];
          float sm[8], sc[8];
#pragma unroll
          for (int t = 0; t < 8; ++t) {
            uint32_t sgn;
            const uint64_t I = fixed56(v[t], E, sgn);
            hi[t] = uint32_t(I >> 28);
            lo[t] = uint32_t(I) & 0xFFFFFFFu;
            sm[t] = sgn ? -1.0f : 1.0f;
            sc[t] = sgn ? 8388608.0f : -8388608.0f;
          }
          // buffer b is free once the products that read it completed: chunk g - 2's, or
          // (resident) the previous tile's last pass
          if (!resident && g >= 2 && !tc::mbar_wait(empty + b, ((g - 2) >> 1) & 1u)) *abort_flag = 1;
          if (resident && it >= 1 && !tc::mbar_wait(empty + b, (it - 1) & 1u)) *abort_flag = 1;
          uint8_t* dst = sA + b * kABytes + (e >> 3) * 512 + q * 128 + (e & 7) * 16;
#pragma unroll
          for (int j = 0; j < kSl; ++j) {
            // slice j: 7 bits of the magnitude below bit 56 - 7j, as a signed float,
            // whose upper 16 bits are its BF16 pattern (at most 8 significant bits)
            uint32_t fb[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) {
              const uint32_t x = ((j < 4 ? hi[t] : lo[t]) >> (21 - 7 * (j & 3))) & 127u;
              fb[t] = __float_as_uint(__fmaf_rn(__uint_as_float(0x4B000000u | x), sm[t], sc[t]));
            }
            uint4 w;  // value 2i in the low half of word i, value 2i + 1 in the high half
            w.x = __byte_perm(fb[0], fb[1], 0x7632);
            w.y = __byte_perm(fb[2], fb[3], 0x7632);
            w.z = __byte_perm(fb[4], fb[5], 0x7632);
            w.w = __byte_perm(fb[6], fb[7], 0x7632);
            *reinterpret_cast<uint4*>(dst + j * kASlice) = w;
          }
          tc::fence_async_smem();
          __syncwarp();
          if (lane == 0) asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" ::"r"(
                                          tc::smem_addr(full + b))
                                      : "memory");
        }
        // drain: output columns [12q, 12q + 12) of this pass
        if (!tc::mbar_wait(acc_full, pass & 1u)) *abort_flag = 1;
        tc::fence_after();
#pragma unroll 1
        for (int p = 0; p < 3; ++p) {
          const int c0 = 12 * q + 4 * p;
          uint32_t acc[kSl][4];
#pragma unroll
          for (int s = 0; s < kSl; ++s) {
            uint32_t vv[4];
            tc::tmem_ld4(tb + lanebase + s * kNC + c0, vv);
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[s][c] = vv[c];
          }
          tc::tmem_wait_ld();
          if (p == 2) {  // the accumulators are read: release them to the next pass
            tc::fence_before();
            __syncwarp();
            if (lane == 0) asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" ::"r"(
                                            tc::smem_addr(acc_empty))
                                        : "memory");
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const int col = nc * kNC + c0 + c;
            if (live && col < M) {
              // value = 2^{ea + E - 14} sum_s acc_s 2^{-7 s}
              const ff hl = horner8(acc, c);
              const double v = ff_to_double(hl.h, hl.l, __ldg(ea + col) + E - 14);
              if (accum) out[row * ldo + col] += v;
              else out[row * ldo + col] = v;
            }
          }
        }
      }
    }
  }
  if (*abort_flag && tid == 0) atomicExch(&g_tc64_err, 1);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_dealloc(tb, 512);
}

// ------------------------------------------------------------------ host side
int row_exp(const double* row, int K) {
  double mx = 0.0;
  for (int k = 0; k < K; ++k) mx = std::max(mx, std::fabs(row[k]));
  if (mx == 0.0) return 0;
  int e = 0;
  std::frexp(mx, &e);  // mx < 2^e
  return e;
}

uint16_t bf16_int(int x) {  // exact for |x| <= 256
  const float f = float(x);
  uint32_t b;
  std::memcpy(&b, &f, 4);
  return uint16_t(b >> 16);
}

}  // namespace

// A (M x K, row-major FP64) into the block layout of tc64_gemm.
cudaError_t tc64_op_create(const std::vector<double>& A, int M, int K, Tc64Op* op) {
  op->M = M;
  op->K = K;
  op->NCH = (M + kNC - 1) / kNC;
  op->KCH = (K + kKC - 1) / kKC;
  if (K > kMaxDepth) return cudaErrorInvalidValue;  // longer sums would leave the FP32 group sums inexact
  std::vector<uint8_t> img(size_t(op->NCH) * op->KCH * kBBytes, 0);
  std::vector<int> ea(size_t(op->NCH) * kNC, 0);
  for (int r = 0; r < M; ++r) {
    const int er = row_exp(&A[size_t(r) * K], K);
    ea[r] = er;
    for (int k = 0; k < K; ++k) {
      const double v = A[size_t(r) * K + k];
      if (v == 0.0 || !std::isfinite(v)) continue;
      int e2 = 0;
      const double fr = std::frexp(std::fabs(v), &e2);
      const int sh = e2 + 56 - er;
      if (sh <= 0) continue;
      const unsigned long long I = (unsigned long long)std::ldexp(fr, sh);
      const int sgn = v < 0 ? -1 : 1;
      const int nc = r / kNC, rl = r % kNC, kc = k / kKC, kl = k % kKC;
      uint8_t* blk = img.data() + size_t(nc * op->KCH + kc) * kBBytes;
      const size_t off = size_t(rl / 8) * ((kKC / 8) * 128) + size_t(kl / 8) * 128 + size_t(rl % 8) * 16 + size_t(kl % 8) * 2;
      for (int i = 0; i < kSl; ++i) {
        const int x = sgn * int((I >> (49 - 7 * i)) & 127ull);
        const uint16_t b = bf16_int(x);
        std::memcpy(blk + size_t(i) * kBSlice + off, &b, 2);
      }
    }
  }
  cudaError_t e = cudaMalloc(&op->blocks, img.size());
  if (e == cudaSuccess) e = cudaMemcpy(op->blocks, img.data(), img.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMalloc(&op->ea, ea.size() * sizeof(int));
  if (e == cudaSuccess) e = cudaMemcpy(op->ea, ea.data(), ea.size() * sizeof(int), cudaMemcpyHostToDevice);
  return e;
}

void tc64_op_free(Tc64Op* op) {
  cudaFree(op->blocks);
  cudaFree(op->ea);
  op->blocks = nullptr;
  op->ea = nullptr;
}

cudaError_t tc64_gemm_launch(const Tc64Op& op, int64_t rows, const double* X, int64_t ldx, double* out, int64_t ldo,
                             cudaStream_t st, int accum, const int* ex) {
  if (rows <= 0) return cudaSuccess;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  static int grid[64];
  {
    std::lock_guard<std::mutex> lk(table_mutex());
    if (!grid[dev & 63]) {
      e = cudaFuncSetAttribute(tc64_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
      int sms = 0;
      if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
      if (e != cudaSuccess) return e;
      grid[dev & 63] = sms;  // one CTA per SM (all of tensor memory, most of shared memory)
    }
  }
  const int vec2 = (ldx % 2 == 0 && (reinterpret_cast<uintptr_t>(X) & 15u) == 0) ? 1 : 0;
  const int64_t tiles = (rows + kT - 1) / kT;
  const unsigned g = unsigned(std::min<int64_t>(tiles, grid[dev & 63]));
  tc64_gemm<<<g, kSlicers + 32, kSmem, st>>>(rows, op.M, op.K, op.NCH, op.KCH, X, ldx, vec2, ex, op.blocks, op.ea, out,
                                             ldo, accum);
  note_launch();
  return cudaGetLastError();
}

cudaError_t tc64_gemm_error(int* flag) {
  int zero = 0;
  cudaError_t e = cudaMemcpyFromSymbol(flag, g_tc64_err, sizeof(int));
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_tc64_err, &zero, sizeof(int));
  return e;
}

}  // namespace dgx
