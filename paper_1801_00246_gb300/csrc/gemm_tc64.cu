// Dense FP64 products on the Blackwell tensor cores (tcgen05) for the tetrahedral
// apply and the advection: out[row] = A X[row] for 128 rows per tile, exact to
// FP64 accuracy by integer slicing (the error-free splitting of Ozaki et al.,
// Numer. Algorithms 59, 2012). Operator rows (on the host) and data rows (on the
// device, in integer arithmetic on the double's bits) are scaled by powers of two
// to 56 bits and cut into seven base-256 digits (fix64.cuh); the 34 digit products
// with i + j <= 7 run as tcgen05.mma (FP16 operands from shared memory, FP32
// accumulators in tensor memory, one per digit sum), the operator's digits
// stacked along N; the sums are joined and rebuilt as doubles with integers. Data
// digits are written by the threads into a double-buffered shared-memory chunk
// (32 columns) while the previous chunk's products run; operator blocks (48 rows
// x 32 columns, 7 digits) arrive by bulk copy.
#include <cmath>
#include <cstring>
#include <vector>

#include "dg_internal.h"
#include "fix64.cuh"
#include "tc05.cuh"

namespace dgx {
namespace {

using fx::kDigits;
using fx::kSums;

constexpr int kT = 128;                      // rows per tile (MMA M)
constexpr int kKC = 32;                      // data columns per chunk
constexpr int kNC = 48;                      // output columns per pass (MMA N)
constexpr int kASlice = kT * kKC * 2, kABytes = kDigits * kASlice;   // one data chunk, 7 digits: 56 KB
constexpr int kBSlice = kNC * kKC * 2, kBBytes = kDigits * kBSlice;  // one operator block, 7 digits: 21 KB
constexpr int kSmem = 2 * kABytes + 2 * kBBytes + 4 * kT * 4 + 12 * 8;  // the tail: 10 mbarriers, slot, 2 flags

__device__ int g_tc64_err;

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
  uint8_t* sA = sm;                        // [2][7 digits][128 rows][32] canonical
  uint8_t* sB = sm + 2 * kABytes;          // [2][7 digits x 48 rows][32] canonical
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
#pragma unroll
            for (int ks = 0; ks < kKC / 16; ++ks)
              fx::issue_step<kKC * 2>(tb, ab + ((ks * 256) >> 4), kASlice, bb + ((ks * 256) >> 4), kNC,
                                      kc == 0 && ks == 0);
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
            for (int t = 0; t < 8; ++t) em = max(em, max(fx::exp_bound(v[0][t]), fx::exp_bound(v[1][t])));
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
          long long x[8];
#pragma unroll
          for (int t = 0; t < 8; ++t) x[t] = fx::fix<56>(v[t], E);
          // buffer b is free once the products that read it completed: chunk g - 2's, or
          // (resident) the previous tile's last pass
          if (!resident && g >= 2 && !tc::mbar_wait(empty + b, ((g - 2) >> 1) & 1u)) *abort_flag = 1;
          if (resident && it >= 1 && !tc::mbar_wait(empty + b, (it - 1) & 1u)) *abort_flag = 1;
          fx::digits8(x, sA + b * kABytes + (e >> 3) * 512 + q * 128 + (e & 7) * 16, kASlice);
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
          float acc[4][kSums];
#pragma unroll
          for (int s = 0; s < kSums; ++s) {
            uint32_t vv[4];
            tc::tmem_ld4(tb + lanebase + s * kNC + c0, vv);
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[c][s] = __uint_as_float(vv[c]);
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
              const double v = fx::to_double(fx::from_sums(acc[c]), __ldg(ea + col) + E - 56);
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
}  // namespace

// A (M x K, row-major FP64) into the block layout of tc64_gemm; cudaErrorInvalidValue if
// its sums are too long to stay exact (beyond some 400 terms).
cudaError_t tc64_op_create(const std::vector<double>& A, int M, int K, Tc64Op* op) {
  op->M = M;
  op->K = K;
  op->NCH = (M + kNC - 1) / kNC;
  op->KCH = (K + kKC - 1) / kKC;
  std::vector<uint8_t> img(size_t(op->NCH) * op->KCH * kBBytes, 0);
  std::vector<int> ea(size_t(op->NCH) * kNC, 0);
  for (int r = 0; r < M; ++r) {
    double mx = 0.0, l1 = 0.0;
    for (int k = 0; k < K; ++k) {
      mx = std::max(mx, std::fabs(A[size_t(r) * K + k]));
      l1 += std::fabs(A[size_t(r) * K + k]);
    }
    ea[r] = fx::row_exp(mx, l1);
    double l1d[4] = {};  // absolute sums of the row's four leading digits
    for (int k = 0; k < K; ++k) {
      const double v = A[size_t(r) * K + k];
      if (v == 0.0 || !std::isfinite(v)) continue;
      int d[kDigits];
      fx::digits_of(v, ea[r], d);
      for (int i = 0; i < 4; ++i) l1d[i] += std::abs(d[i]);
      uint8_t* blk = img.data() + size_t(r / kNC * op->KCH + k / kKC) * kBBytes;
      for (int i = 0; i < kDigits; ++i) {
        const int R = i * kNC + r % kNC, c = k % kKC;
        const uint16_t h = fx::fp16_int(d[i]);
        std::memcpy(blk + size_t(R / 8) * ((kKC / 8) * 128) + size_t(c / 8) * 128 + size_t(R % 8) * 16 + size_t(c % 8) * 2,
                    &h, 2);
      }
    }
    // The sums that carry the result (s <= 3) have to stay integers below 2^24, which
    // FP32 holds exactly, whatever the data: its leading digit is at most 257, the others 128.
    for (int s4 = 0; s4 < 4; ++s4) {
      double most = 257.0 * l1d[s4];
      for (int i = 0; i < s4; ++i) most += 128.0 * l1d[i];
      if (most >= 16777216.0) return cudaErrorInvalidValue;
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
