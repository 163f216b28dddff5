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
constexpr int kASlice = kT * kKC * 2, kABytes = kDigits * kASlice;  // one data chunk, 7 digits: 56 KB
constexpr int kStages = 4;                   // operator blocks in flight
__host__ __device__ constexpr int block_bytes(int nc) { return kDigits * nc * kKC * 2; }
// the tail: row exponents, 20 mbarriers, slot, flag
__host__ __device__ constexpr int gemm_smem(int nc) {
  return 2 * kABytes + kStages * block_bytes(nc) + 4 * kT * 4 + 20 * 8 + 16;
}
// Output columns per pass (MMA N): 32, with two accumulator sets in tensor memory so
// that a pass's products run under the drain of the one before, where all of a row's
// data stays in shared memory for its passes (two chunks) or one pass is enough;
// else 48 in one set, so that a deep row is sliced once (more than 48 columns of
// output: once per pass).
int pass_columns(int M, int K) { return K <= 2 * kKC || M <= 32 ? 32 : 48; }

__device__ int g_tc64_err;

// out[r][c] = sum_k A[c][k] X[r][k] for r < rows, c < M, k < Kd; X row-major, or with
// xcol, out with ocol (COLS only), column-major (ldx, ldo then lie between columns: a warp's 32
// rows read and write 256 contiguous bytes a column, where rows of an odd length cost
// 32 sectors an access) (A sliced in
// blocks of NC rows x kKC columns: block (nc, kc) at (nc KCH + kc) block_bytes).
//
// Warp-specialised pipeline over a stream of data chunks (tile, output pass
// nc, column chunk kc), chunk g using shared-memory buffer g & 1:
//  * warps 0-15 (four threads per row of the 128-row tile) find each row's
//    scale exponent, slice chunk g into buffer g & 1 once the products of
//    chunk g - 2 have released it (mbarrier `empty`), signal `full`, and after
//    a pass's last chunk wait for its accumulators (`accf`), drain them and
//    release them (`acce`);
//  * warp 16 waits for `full`, issues the 34 digit products per 16 columns from
//    one lane and commits to `empty` (and to `accf` after a pass's last chunk);
//  * warp 17 keeps a ring of operator blocks filled by bulk copies (loaded by
//    warp 16 only when a chunk needed them, their latency was in every chunk:
//    16,384 rows of 208 outputs, 45 deep, took 44 us).
// Four products of a tetrahedral apply (196,608 elements, N = 3): 920 us with eight
// 7-bit digits in BF16 (36 products, each its own instruction, and a float-float
// recombination) -> 563 us, bound by the slicing and the drain of thin tiles.
// No CTA-wide barrier in the steady state; every wait is bounded in time.
constexpr int kSlicers = 512;  // threads of warps 0-15
template <int NC, bool COLS>
__global__ void __launch_bounds__(kSlicers + 64, 1) tc64_gemm(int64_t rows, int M, int Kd, int NCH, int KCH,
                                                              const double* __restrict__ X, int64_t ldx, int vec2,
                                                              int xcol, const int* __restrict__ ex_given,
                                                              const uint8_t* __restrict__ Bops,
                                                              const int* __restrict__ ea, double* __restrict__ out,
                                                              int64_t ldo, int ocol, int accum) {
  extern __shared__ __align__(1024) uint8_t sm[];
  constexpr int kBBytes = block_bytes(NC);
  constexpr int kAcc = 2 * kSums * NC <= 512 ? 2 : 1;  // accumulator sets
  uint8_t* sA = sm;                        // [2][7 digits][128 rows][32] canonical
  uint8_t* sB = sm + 2 * kABytes;          // [kStages][7 digits x NC rows][32] canonical
  int* pmax = reinterpret_cast<int*>(sB + kStages * kBBytes);  // [4][kT]
  uint64_t* bars = reinterpret_cast<uint64_t*>(pmax + 4 * kT);
  uint64_t *full = bars, *empty = bars + 2, *accf = bars + 4, *acce = bars + 6, *bfull = bars + 8,
           *bempty = bars + 8 + kStages, *done = bars + 8 + 2 * kStages;
  uint32_t* slot = reinterpret_cast<uint32_t*>(bars + 20);
  volatile int* abort_flag = reinterpret_cast<int*>(slot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t ntiles = (rows + kT - 1) / kT;
  // with at most two data chunks per row, both stay in the two buffers for all
  // output passes of a tile: sliced once per tile instead of once per pass
  const bool resident = KCH <= 2 && NCH > 1;
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(full + i, kSlicers / 32);  // one arrival per slicing warp
      tc::mbar_init(empty + i, 1);             // the products' commit
      tc::mbar_init(accf + i, 1);
      tc::mbar_init(acce + i, kSlicers / 32);
    }
    for (int i = 0; i < kStages; ++i) {
      tc::mbar_init(bfull + i, 1);   // the bulk copy
      tc::mbar_init(bempty + i, 1);  // the block's products completed
    }
    tc::mbar_init(done, 1);
    *abort_flag = 0;
    tc::mbar_init_fence();
  }
  if (warp == 0) tc::tmem_alloc(slot, 512);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tb = *slot;

  if (warp == kSlicers / 32 + 1) {
    // ================= operator blocks
    uint32_t g = 0;
    for (int64_t tile = blockIdx.x; tile < ntiles && !tc::aborted(abort_flag); tile += gridDim.x)
      for (int s = 0; s < NCH * KCH; ++s, ++g) {
        const uint32_t b = g % kStages, use = g / kStages;
        if (use > 0) tc::wait_or_abort(bempty + b, (use - 1) & 1u, abort_flag);
        if (tc::aborted(abort_flag)) break;
        if (lane == 0) {
          tc::mbar_expect_tx(bfull + b, kBBytes);
          tc::bulk_g2s(sB + b * kBBytes, Bops + size_t(s) * kBBytes, kBBytes, bfull + b);
        }
        __syncwarp();
      }
    // every copy has landed before the block ends
    for (uint32_t k = g < kStages ? 0 : g - kStages; k < g; ++k)
      tc::wait_done(bfull + k % kStages, (k / kStages) & 1u, abort_flag);
  } else if (warp == kSlicers / 32) {
    // ================= products
    uint32_t g = 0, pass = 0, it = 0;
    const uint64_t adesc0 = tc::smem_desc(tc::smem_addr(sA), 128, (kKC / 8) * 128);
    const uint64_t bdesc0 = tc::smem_desc(tc::smem_addr(sB), 128, (kKC / 8) * 128);
    for (int64_t tile = blockIdx.x; tile < ntiles && !tc::aborted(abort_flag); tile += gridDim.x, ++it) {
      for (int nc = 0; nc < NCH; ++nc, ++pass) {
        // the accumulators are free once the pass that last used them has been drained
        const uint32_t ab = pass % kAcc, ause = pass / kAcc;
        if (ause > 0) tc::wait_or_abort(acce + ab, (ause - 1) & 1u, abort_flag);
        for (int kc = 0; kc < KCH; ++kc, ++g) {
          const uint32_t bs = g % kStages;                      // operator stage
          const uint32_t bd = resident ? kc : (g & 1u);         // data buffer
          // the data chunk: sliced once per chunk, or (resident) once per tile for all passes
          if (!resident) tc::wait_or_abort(full + bd, (g >> 1) & 1u, abort_flag);
          else if (nc == 0) tc::wait_or_abort(full + bd, it & 1u, abort_flag);
          tc::wait_or_abort(bfull + bs, (g / kStages) & 1u, abort_flag);
          tc::fence_after();
          if (lane == 0) {
            const uint64_t a0 = adesc0 + ((bd * kABytes) >> 4), b0 = bdesc0 + ((bs * kBBytes) >> 4);
#pragma unroll
            for (int ks = 0; ks < kKC / 16; ++ks)
              fx::issue_step<kKC * 2>(tb + ab * kSums * NC, a0 + ((ks * 256) >> 4), kASlice, b0 + ((ks * 256) >> 4), NC,
                                      kc == 0 && ks == 0);
            tc::mma_commit(bempty + bs);
            if (!resident || nc == NCH - 1) tc::mma_commit(empty + bd);  // the data buffer is free
            if (kc == KCH - 1) tc::mma_commit(accf + ab);
          }
          __syncwarp();
        }
      }
    }
    if (lane == 0) tc::mma_commit(done);
    __syncwarp();
    tc::wait_done(done, 0, abort_flag);
  } else {
    // ================= slicing and epilogue
    const int e = (warp & 3) * 32 + lane;
    const int q = warp >> 2;
    const uint32_t lanebase = uint32_t((warp & 3) * 32) << 16;
    uint32_t g = 0, pass = 0, it = 0;
    auto load8 = [&](const double* xr, bool live, int k0, double (&v)[8]) {
      if (COLS && xcol) {
#pragma unroll
        for (int t = 0; t < 8; ++t) v[t] = (live && k0 + t < Kd) ? __ldg(xr + int64_t(k0 + t) * ldx) : 0.0;
      } else if (live && vec2 && k0 + 8 <= Kd) {
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
      const int64_t row = tile * kT + e;
      const bool live = row < rows;
      const double* xr = X + (live ? row : 0) * (COLS && xcol ? 1 : ldx);
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
        tc::bar_sync(1, kSlicers);  // pmax free (previous tile read it)
        pmax[q * kT + e] = em;
        tc::bar_sync(1, kSlicers);
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
              load8(X + (nlive ? nrow : 0) * (COLS && xcol ? 1 : ldx), nlive, 8 * q, vn);
              En = nlive ? __ldg(ex_given + nrow) : 0;
              have_next = true;
            }
          }
          long long x[8];
#pragma unroll
          for (int t = 0; t < 8; ++t) x[t] = fx::fix<56>(v[t], E);
          // buffer b is free once the products that read it completed: chunk g - 2's, or
          // (resident) the previous tile's last pass
          if (!resident && g >= 2) tc::wait_or_abort(empty + b, ((g - 2) >> 1) & 1u, abort_flag);
          if (resident && it >= 1) tc::wait_or_abort(empty + b, (it - 1) & 1u, abort_flag);
          fx::digits8(x, sA + b * kABytes + (e >> 3) * 512 + q * 128 + (e & 7) * 16, kASlice);
          tc::fence_async_smem();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(full + b);
        }
        // drain: output columns [NC/4 q, NC/4 (q + 1)) of this pass
        const uint32_t ab = pass % kAcc;
        tc::wait_or_abort(accf + ab, (pass / kAcc) & 1u, abort_flag);
        tc::fence_after();
#pragma unroll 1
        for (int p = 0; p < NC / 16; ++p) {
          const int c0 = NC / 4 * q + 4 * p;
          __syncwarp();
          if (nc * NC + c0 >= M) break;
          float acc[4][kSums];
#pragma unroll
          for (int s = 0; s < kSums; ++s) {
            uint32_t vv[4];
            tc::tmem_ld4(tb + lanebase + (ab * kSums + s) * NC + c0, vv);
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[c][s] = __uint_as_float(vv[c]);
          }
          tc::tmem_wait_ld();
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const int col = nc * NC + c0 + c;
            if (live && col < M) {
              const double v = fx::to_double(fx::from_sums(acc[c]), __ldg(ea + col) + E - 56);
              double* o = out + (COLS && ocol ? col * ldo + row : row * ldo + col);
              *o = accum ? *o + v : v;
            }
          }
        }
        tc::fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(acce + ab);
      }
    }
  }
  if (*abort_flag && tid == 0) atomicExch(&g_tc64_err, 1);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_dealloc(tb, 512);
}

template <int NC>
cudaError_t allow_smem() {
  const auto a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  const cudaError_t e = cudaFuncSetAttribute(tc64_gemm<NC, false>, a, gemm_smem(NC));
  return e == cudaSuccess ? cudaFuncSetAttribute(tc64_gemm<NC, true>, a, gemm_smem(NC)) : e;
}
}  // namespace

// A (M x K, row-major FP64) into the block layout of tc64_gemm; cudaErrorInvalidValue if
// its sums are too long to stay exact (beyond some 350 terms).
cudaError_t tc64_op_create(const std::vector<double>& A, int M, int K, Tc64Op* op) {
  op->M = M;
  op->K = K;
  const int nc = pass_columns(M, K), bytes = block_bytes(nc);
  op->nc = nc;
  op->NCH = (M + nc - 1) / nc;
  op->KCH = (K + kKC - 1) / kKC;
  std::vector<uint8_t> img(size_t(op->NCH) * op->KCH * bytes, 0);
  std::vector<int> ea(size_t(op->NCH) * nc, 0);
  for (int r = 0; r < M; ++r) {
    double mx = 0.0, l1 = 0.0;
    for (int k = 0; k < K; ++k) {
      mx = std::max(mx, std::fabs(A[size_t(r) * K + k]));
      l1 += std::fabs(A[size_t(r) * K + k]);
    }
    ea[r] = fx::row_exp(mx, l1);
    fx::ExactSums sums;
    for (int k = 0; k < K; ++k) {
      const double v = A[size_t(r) * K + k];
      if (v == 0.0 || !std::isfinite(v)) continue;
      int d[kDigits];
      fx::digits_of(std::llround(std::ldexp(v, 56 - ea[r])), d);
      sums.add(d);
      uint8_t* blk = img.data() + size_t(r / nc * op->KCH + k / kKC) * bytes;
      for (int i = 0; i < kDigits; ++i) {
        const int R = i * nc + r % nc, c = k % kKC;
        const uint16_t h = fx::fp16_int(d[i]);
        std::memcpy(blk + size_t(R / 8) * ((kKC / 8) * 128) + size_t(c / 8) * 128 + size_t(R % 8) * 16 + size_t(c % 8) * 2,
                    &h, 2);
      }
    }
    if (!sums.exact()) return cudaErrorInvalidValue;
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
                             cudaStream_t st, int accum, const int* ex, int xcol, int ocol) {
  if (rows <= 0) return cudaSuccess;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  static int grid[64];
  {
    std::lock_guard<std::mutex> lk(table_mutex());
    if (!grid[dev & 63]) {
      e = allow_smem<32>();
      if (e == cudaSuccess) e = allow_smem<48>();
      int sms = 0;
      if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
      if (e != cudaSuccess) return e;
      grid[dev & 63] = sms;  // one CTA per SM (all of tensor memory, most of shared memory)
    }
  }
  const int vec2 = (ldx % 2 == 0 && (reinterpret_cast<uintptr_t>(X) & 15u) == 0) ? 1 : 0;
  const int64_t tiles = (rows + kT - 1) / kT;
  const unsigned g = unsigned(std::min<int64_t>(tiles, grid[dev & 63]));
  // (the layouts of a product with a column-major side stay run-time choices: the
  // specialised forms measured 8 ms slower in a flow step of 70 ms)
  auto go = [&](auto kernel) {
    kernel<<<g, kSlicers + 64, gemm_smem(op.nc), st>>>(rows, op.M, op.K, op.NCH, op.KCH, X, ldx, vec2, xcol, ex, op.blocks,
                                                       op.ea, out, ldo, ocol, accum);
  };
  if (op.nc == 32) xcol || ocol ? go(tc64_gemm<32, true>) : go(tc64_gemm<32, false>);
  else xcol || ocol ? go(tc64_gemm<48, true>) : go(tc64_gemm<48, false>);
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
