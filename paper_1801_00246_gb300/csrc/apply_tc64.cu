// SIPDG apply in FP64 on the Blackwell tensor cores (tcgen05), without the
// FP64 pipe (GB300 runs FP64 arithmetic at 1/64 of its FP32 rate).
//
// The operator of Eq. ellipticOp3, element by element, is one dense product of
// a reference matrix with a column X of the element's own and its neighbours'
// data, Au = OB X with
//   X  = [Grr u, Grs u, Gss u | 1/2 nr sJ [u], 1/2 ns sJ [u], -sJ ({n.grad u} + tau [u]) (| lambda J u)]
//   OB = [S_rr, S_rs + S_sr, S_ss | Dr_f^T Mf, Ds_f^T Mf, E_f Mf (| M)],   S_ab = D_a^T M D_b,
// so that the volume term needs no gradient; the only derivative left is
// n.grad u at the face nodes. Two kernels:
//  * t64_trace: per 128 elements the rows of [Dr; Ds] at the 3N boundary nodes
//    times u, from which q = sJ n.grad u at every face node; writes u and q as
//    fixed-point integers at the element's own scale, column-major (entry i of
//    element e at [i][e], so that a warp's 32 elements are contiguous);
//  * t64_output: forms X chunk by chunk in registers from those integers (own
//    and neighbours'), cuts it into digits in shared memory and multiplies; X
//    never reaches memory.
// Constants are in the kernel of D_a and S_ab, so both kernels work on v = u - u0,
// u0 the element's first node, and add the difference of the two u0 to a jump:
// a smooth field's columns are as small as its gradient's, which keeps the
// digits for the result (on u itself an apply to a smooth field had 20 times
// the error: S_ab is N^2 times larger than what it yields there).
// Both products are exact to FP64 accuracy by integer slicing (Ozaki et al.,
// Numer. Algorithms 59, 2012) into seven base-256 digits (fix64.cuh): the 34
// digit products with i + j <= 7 run as tcgen05.mma in FP16 with FP32
// accumulators in tensor memory, one accumulator per digit sum i + j. The
// operator's digits are stacked along N, so one instruction multiplies data
// digit j with the operator's digits 0 .. 7 - j into the accumulators j .. 7:
// 7 to 12 instructions per 16 columns in place of 34, each reading the data
// digit once.
// Accuracy: columns of X carry 56 bits of a bound on the row, rounded to nearest
// (a bias that all elements share would be a smooth source, which a solve
// amplifies), and the digit products left out weigh 2^-60 of the largest. Against
// 64-bit arithmetic the relative error of an apply is 0.9e-15 (N = 3) to 1.2e-14
// (N = 10) on random fields, 1.5 times the FP64-pipe kernel's. What an apply yields
// summed over an element (its flux balance) matters more to a solve than any entry:
// the operator's columns sum to what the basis says exactly (tables64.cpp), so a
// column's rounding drops out of that sum.
// 524,288 triangles, N = 8: 1714 us and 2.6 GB of traffic with the pointwise stage
// in float-float between two generic products and X in memory; 780 us and 1.0 GB now.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "dg_internal.h"
#include "fix64.cuh"
#include "tables64.h"
#include "tc05.cuh"

namespace dgx {
namespace {

using fx::kDigits;
using fx::kSums;
using fx::Split;

constexpr int kT = 128;       // rows (elements x right-hand sides) per tile: MMA M
constexpr int kItems = 16;    // items of X per chunk, three columns each
constexpr int kChunkSlice = kT * 3 * kItems * 2;       // one digit of a chunk: 12 KB
constexpr int kChunkBytes = kDigits * kChunkSlice;     // 84 KB
constexpr int kTraceN = 32;                            // output columns (16 boundary nodes) per pass of t64_trace
constexpr int kTraceStep = kDigits * kTraceN * 16 * 2; // operator block of one pass and 16 columns
constexpr int trace_smem(int ks) {
  return kDigits * kT * ks * 32 + (ks != 3 ? 2 : 1) * ks * kTraceStep + 6 * kT * 4 + 7 * 8;
}
constexpr int kCoefs = 12;    // Grr, Grs, Gss | per face nr sJ, ns sJ | per face -sJ tau0

__device__ int g_t64_err;

using tc::aborted;
using tc::bar_sync;
using tc::mbar_arrive;
__device__ __forceinline__ bool wait(uint64_t* b, uint32_t parity, volatile int* abort_flag) {
  return tc::wait_or_abort(b, parity, abort_flag);
}
__device__ __forceinline__ int64_t elem_of(int64_t row, int64_t K) { return row < K ? row : row % K; }

__device__ __forceinline__ int node_of(int N, int f, int j) {  // local node of face f's j-th node
  auto rs = [N](int row) { return row * (N + 1) - row * (row - 1) / 2; };
  return f == 0 ? j : (f == 1 ? rs(j) + (N - j) : rs(N - j));
}

// Per-element coefficients in fixed point, one exponent for each kind (|c| < 2^e):
// word i of element e at tab[i K + e], exponents in ex (G, n sJ, sJ tau0).
__global__ void k_fix_geometry(int64_t K, const double* __restrict__ gx, int2* __restrict__ tab,
                               short4* __restrict__ ex) {
  const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (e >= K) return;
  const double* g = gx + 16 * e;
  double c[kCoefs];
  for (int i = 0; i < 3; ++i) c[i] = g[1 + i];
  for (int f = 0; f < 3; ++f) {
    const double sJ = g[4 + 4 * f + 2];
    c[3 + 2 * f] = g[4 + 4 * f] * sJ;
    c[4 + 2 * f] = g[4 + 4 * f + 1] * sJ;
    c[9 + f] = -g[4 + 4 * f + 3] * sJ;
  }
  int eg = fx::kZeroExp, ec = fx::kZeroExp, et = fx::kZeroExp;
  for (int i = 0; i < 3; ++i) eg = max(eg, fx::exp_bound(c[i]));
  for (int i = 3; i < 9; ++i) ec = max(ec, fx::exp_bound(c[i]));
  for (int i = 9; i < 12; ++i) et = max(et, fx::exp_bound(c[i]));
  for (int i = 0; i < kCoefs; ++i) {
    const Split s = fx::split(fx::fix<62>(c[i], i < 3 ? eg : (i < 9 ? ec : et)));
    tab[int64_t(i) * K + e] = make_int2(s.h, s.l);
  }
  ex[e] = make_short4(short(eg), short(ec), short(et), 0);
}

__device__ __forceinline__ Split coef(const int2* p) {
  const int2 v = __ldg(p);
  return Split{v.x, v.y};
}

// ------------------------------------------------------------------ boundary derivatives
struct TraceArgs {
  int N, passes, aligned;
  int64_t K, rows, row0;   // rows of this launch, the first one's global index
  const double* u;         // this launch's first row
  const int2* tab;
  const short4* tex;
  const uint8_t* ops;      // [pass][16 columns][7 digits x 32 rows][16]
  int ea;                  // common exponent of the operator
  long long* Iu;           // [Np][ldc], first row of this launch
  long long* Iq;           // [3 (N + 1)][ldc]
  int64_t ldc;
  int4* ex;                // per row: exponents of v, q's scale, q, u
  double* u0;              // per row: u at the first node
};

// KS: 16-column steps of u (Np <= 16 KS). Eight warps (two threads per row)
// slice a tile and drain its products, one warp issues copies and products;
// two blocks per SM up to KS = 3 (shared memory 110 KB, tensor memory 256
// columns each), so one block's slicing runs under the other's products. The
// tile's rows arrive by one bulk copy into the space that then takes their
// digits (each thread reads its values before the first digit is written), so
// the row-major u is read with full sectors. 524,288 triangles, N = 8: 223 us (70
// of it the 0.48 GB at the copy rate), bound by the slicing and the drain, whose
// 64-bit integer work the two blocks overlap with each other's waits; the product
// of all gradient rows that it replaces took 808 us.
template <int KS>
__global__ void __launch_bounds__(288, KS <= 3 ? 2 : 1) t64_trace(const TraceArgs a) {
  extern __shared__ __align__(1024) uint8_t sm[];
  constexpr int kSlice = kT * KS * 16 * 2;
  constexpr bool kResident = KS != 3;  // all passes' operator blocks stay in shared memory (KS = 3: one at a time)
  constexpr int kPass = KS * kTraceStep;
  uint8_t* sB = sm + kDigits * kSlice;
  int* pmax = reinterpret_cast<int*>(sB + (kResident ? 2 : 1) * kPass);  // [2 halves][exponent of v, of u, bits of q][kT]
  uint64_t* bars = reinterpret_cast<uint64_t*>(pmax + 6 * kT);
  uint64_t *ufull = bars, *full = bars + 1, *accf = bars + 2, *acce = bars + 3, *bfull = bars + 4,
           *done = bars + 5;
  uint32_t* slot = reinterpret_cast<uint32_t*>(bars + 6);
  volatile int* abort_flag = reinterpret_cast<int*>(slot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int N = a.N, Np = (N + 1) * (N + 2) / 2;
  const int64_t ntiles = (a.rows + kT - 1) / kT;
  if (tid == 0) {
    tc::mbar_init(ufull, 1);
    tc::mbar_init(full, 8);
    tc::mbar_init(accf, 1);
    tc::mbar_init(acce, 8);
    tc::mbar_init(bfull, 1);
    tc::mbar_init(done, 1);
    *abort_flag = 0;
    tc::mbar_init_fence();
  }
  if (warp == 0) tc::tmem_alloc(slot, 256);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tb = *slot;
  // a tile's rows arrive by bulk copy where address and size are multiples of 16 bytes
  auto bulk_rows = [&](int64_t tile) -> uint32_t {
    const int64_t left = a.rows - tile * kT;
    const uint32_t bytes = uint32_t(left < kT ? left : kT) * uint32_t(Np) * 8u;
    return a.aligned && (bytes & 15u) == 0 ? bytes : 0u;
  };

  if (warp == 8) {
    const uint64_t ad = tc::smem_desc(tc::smem_addr(sm), 128, KS * 256);
    const uint64_t bd = tc::smem_desc(tc::smem_addr(sB), 128, 256);
    uint32_t loads = 0, bulks = 0, it = 0, pc = 0;
    auto load_ops = [&](int pass0, int n) {
      if (lane == 0) {
        tc::mbar_expect_tx(bfull, n * kPass);
        tc::bulk_g2s(sB, a.ops + size_t(pass0) * kPass, n * kPass, bfull);
      }
      ++loads;
    };
    auto load_u = [&](int64_t tile) {
      const uint32_t bytes = bulk_rows(tile);
      if (bytes && lane == 0) {
        tc::mbar_expect_tx(ufull, bytes);
        tc::bulk_g2s(sm, a.u + tile * kT * Np, bytes, ufull);
      }
      bulks += bytes != 0;
    };
    load_ops(0, kResident ? a.passes : 1);
    if (int64_t(blockIdx.x) < ntiles) load_u(blockIdx.x);
    for (int64_t tile = blockIdx.x; tile < ntiles && !aborted(abort_flag); tile += gridDim.x, ++it) {
      wait(full, it & 1u, abort_flag);
      for (int p = 0; p < a.passes; ++p, ++pc) {
        wait(bfull, (loads - 1) & 1u, abort_flag);
        if (pc > 0) wait(acce, (pc - 1) & 1u, abort_flag);
        tc::fence_after();
        if (lane == 0) {
          const uint64_t b0 = bd + ((kResident ? p * kPass : 0) >> 4);
#pragma unroll 1
          for (int ks = 0; ks < KS; ++ks)
            fx::issue_step<32>(tb, ad + ((ks * 256) >> 4), kSlice, b0 + ((ks * kTraceStep) >> 4), kTraceN, ks == 0);
          tc::mma_commit(accf);
        }
        __syncwarp();
        const bool last = p + 1 == a.passes;
        if (!kResident || last) {  // the products are done: their operands' space is free
          if (!wait(accf, pc & 1u, abort_flag)) continue;
          if (!kResident && a.passes > 1 && (!last || tile + gridDim.x < ntiles)) load_ops(last ? 0 : p + 1, 1);
          if (last && tile + gridDim.x < ntiles) load_u(tile + gridDim.x);
        }
      }
    }
    // nothing is left in flight when the block ends
    tc::wait_done(bfull, (loads - 1) & 1u, abort_flag);
    if (bulks > 0) tc::wait_done(ufull, (bulks - 1) & 1u, abort_flag);
    if (lane == 0) tc::mma_commit(done);
    __syncwarp();
    tc::wait_done(done, 0, abort_flag);
  } else {
    const int e = (warp & 3) * 32 + lane, half = warp >> 2;
    const uint32_t lanebase = uint32_t((warp & 3) * 32) << 16;
    const double* su = reinterpret_cast<const double*>(sm);
    uint32_t it = 0, pc = 0, bulks = 0;
    int* pm = pmax + half * 3 * kT + e;
    int4 xprev{};
    // a row's exponents are complete once both its threads have seen their part of q:
    // written behind the next barrier (the next tile's, or the last one)
    auto write_exponents = [&](int64_t row) {
      if (half != 0 || row >= a.rows) return;
      const int bits = pmax[2 * kT + e] | pmax[5 * kT + e];  // of |q|'s upper words
      xprev.z = xprev.y + 7 - __clz(bits);                   // |q| < 2^{64 - clz} at scale 2^{57-eq}
      a.ex[row] = xprev;
    };
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it) {
      const int64_t row = tile * kT + e;
      const bool live = row < a.rows;
      if (bulk_rows(tile)) {
        wait(ufull, bulks & 1u, abort_flag);
        ++bulks;
      } else {  // every product that read the space has completed (accf below)
        const int64_t left = a.rows - tile * kT;
        const int n = int(left < kT ? left : kT) * Np;
        for (int i = tid; i < n; i += 256) reinterpret_cast<double*>(sm)[i] = __ldg(a.u + tile * kT * Np + i);
        bar_sync(1, 256);
      }
      // this thread's columns: 8-column groups half, half + 2, ...
      double v[KS * 8];
      const double u0 = live ? su[e * Np] : 0.0;
      int ev = fx::kZeroExp, eu = fx::kZeroExp;
#pragma unroll
      for (int ks = 0; ks < KS; ++ks)
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          const int n = (2 * ks + half) * 8 + t;
          const double u = live && n < Np ? su[e * Np + n] : u0;
          v[ks * 8 + t] = u - u0;
          eu = max(eu, fx::exp_bound(u));
          ev = max(ev, fx::exp_bound(v[ks * 8 + t]));
        }
      pm[0] = ev;
      pm[kT] = eu;
      bar_sync(1, 256);  // exponents written, and the rows read before digits overwrite them
      if (it > 0) write_exponents(row - int64_t(gridDim.x) * kT);
      ev = max(pmax[e], pmax[3 * kT + e]);
      eu = max(pmax[kT + e], pmax[4 * kT + e]);
      if (ev >= fx::kBadExp) eu = fx::kBadExp;
      const int64_t el = live ? elem_of(a.row0 + row, a.K) : 0;
      const int eq = a.ea + ev + __ldg(reinterpret_cast<const short*>(a.tex + el) + 1) + 3;
      xprev = make_int4(ev, eq, 0, eu);
      if (live && half == 0) a.u0[row] = u0;
      int qbits = 0;
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        long long x[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          const int n = (2 * ks + half) * 8 + t;
          x[t] = fx::fix<59>(v[ks * 8 + t], ev);
          if (live && n < Np) a.Iu[int64_t(n) * a.ldc + row] = x[t];
          x[t] = (x[t] + 4) >> 3;
        }
        fx::digits8(x, sm + (e >> 3) * (KS * 256) + (2 * ks + half) * 128 + (e & 7) * 16, kSlice);
      }
      tc::fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(full);
      for (int p = 0; p < a.passes; ++p, ++pc) {
        wait(accf, pc & 1u, abort_flag);
        tc::fence_after();
        const int b0 = 16 * p + 8 * half;  // this warp's boundary nodes of the pass
        int f = b0 / N, j = b0 - f * N;    // node b is the j-th of face f; a corner also ends the face before it
#pragma unroll 1
        for (int i = 0; i < 4; ++i) {
          const int b = b0 + 2 * i;
          if (b >= 3 * N) break;
          float acc[2][2][kSums];
          __syncwarp();
#pragma unroll
          for (int s = 0; s < kSums; ++s) {
            uint32_t w[4];
            tc::tmem_ld4(tb + lanebase + s * kTraceN + 16 * half + 4 * i, w);
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[c >> 1][c & 1][s] = __uint_as_float(w[c]);
          }
          tc::tmem_wait_ld();
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            if (b + k >= 3 * N) break;
            const Split ur = fx::split(fx::from_sums(acc[k][0])), us = fx::split(fx::from_sums(acc[k][1]));
            if (live) {
              const int2* c = a.tab + el;
              const long long q = fx::mul(ur, coef(c + (3 + 2 * f) * a.K)) + fx::mul(us, coef(c + (4 + 2 * f) * a.K));
              a.Iq[int64_t(f * (N + 1) + j) * a.ldc + row] = q;
              qbits |= int(q >> 32) ^ int(q >> 63);
              if (j == 0) {
                const int g = f == 0 ? 2 : f - 1;
                const long long p2 = fx::mul(ur, coef(c + (3 + 2 * g) * a.K)) + fx::mul(us, coef(c + (4 + 2 * g) * a.K));
                a.Iq[int64_t(g * (N + 1) + N) * a.ldc + row] = p2;
                qbits |= int(p2 >> 32) ^ int(p2 >> 63);
              }
            }
            if (++j == N) ++f, j = 0;
          }
        }
        tc::fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acce);
      }
      pm[2 * kT] = qbits;
    }
    bar_sync(1, 256);
    if (it > 0) write_exponents((blockIdx.x + int64_t(it - 1) * gridDim.x) * kT + e);
  }
  if (*abort_flag && tid == 0) atomicExch(&g_t64_err, 1);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_dealloc(tb, 256);
}

// ------------------------------------------------------------------ output product
constexpr int kOutStages = 2;  // operator blocks in flight (three measured the same)
struct OutArgs {
  int N, chunks, M;         // chunks of two item groups, output columns of this launch
  int gvol, gface;          // groups of eight items: [0, gvol) volume, [gvol, gface) face, then mass
  int cpen, lpen;           // (N+1)(N+2)/2 <= 2^lpen
  int k1, k2, km;           // data columns carry 2^-k (k1: flux, k2: jumps, km: mass), operator columns 2^k
  int helm;
  double lambda;
  int64_t K, rows, row0;
  const long long* Iu;      // all rows
  const long long* Iq;
  int64_t ldc;
  const int4* ex;
  const double* u0;
  const int2* tab;
  const short4* tex;
  const double* gx;
  const int32_t* conn;
  const uint8_t* ops;       // [chunk][3 kinds of columns][7 digits x NC rows][16]
  const int* ea;            // [NC]
  double* out;              // this launch's first row, first column
  int64_t ldo;
};

constexpr int kWorkers = 512;
constexpr int kOutThreads = kWorkers + 128;
constexpr int kLut = 3 * (kMaxN + 1);          // local nodes of the face nodes
constexpr int kScaleWords = 2 * kCoefs + 6 + 7;  // a row's scale: coefficients, differences of u0, E, neighbours, shifts
constexpr int kBadScale = 1 << 20;             // E of a row with an infinity or a NaN among its data
__host__ __device__ constexpr int out_sets(int nc) { return nc <= 48 ? 2 : 1; }
__host__ __device__ constexpr int out_smem(int nc) {
  return 2 * kChunkBytes + kOutStages * kDigits * nc * 32 + out_sets(nc) * kScaleWords * kT * 4 + 24 * 8 + 16 + kLut * 8;
}

// NC: output columns (a multiple of 16). Sixteen warps in two groups of eight:
// group p forms the chunks of buffer p (two threads per row, eight items each)
// while the products of the other buffer run; all sixteen drain a tile's
// accumulators after the first chunk of the next one, so neither the products
// nor the copies wait for the drain. Warp 16 issues the products, warp 17 the
// operator's copies (a ring of 16-column blocks); warps 18 and 19 run a tile
// ahead and work out each row's scale: a bound on its columns from its own and
// its neighbours' exponents, the coefficients at that scale and the shifts that
// bring both sides of a face to a common one (done by every thread that forms
// columns, this took a third of the kernel's instructions).
// 524,288 triangles, N = 8: 553 us, in place of 234 (face terms) and 667 (product).
// Nothing is near its limit: without the loads about 485, without the stores 495, without
// the products 390, with none of them 275 and as an empty pipeline 170 us; a chunk's
// forming, slicing and products follow each other and only two chunks fit in shared
// memory. Handing over every 16 columns in place of a chunk gave 520 at N = 8 but
// 6 % more at N = 5 and 9 % at N = 6.
template <int NC>
__global__ void __launch_bounds__(kOutThreads, 1) t64_output(const OutArgs a) {
  extern __shared__ __align__(1024) uint8_t sm[];
  constexpr int kStages = kOutStages;
  constexpr int kSets = out_sets(NC);
  constexpr int kStage = kDigits * NC * 32;
  constexpr int kAcc = 2 * kSums * NC <= 512 ? 2 : 1;  // accumulator sets
  uint8_t* sB = sm + 2 * kChunkBytes;
  int2* scoef = reinterpret_cast<int2*>(sB + kStages * kStage);        // [sets][kCoefs][kT], at the row's scale
  long long* sdiff = reinterpret_cast<long long*>(scoef + kSets * kCoefs * kT);  // [sets][3][kT]: u0+ - u0- at the jump's scale
  int* sinfo = reinterpret_cast<int*>(sdiff + kSets * 3 * kT);         // [sets][E | 3 neighbours | 3 shifts][kT]
  long long* lut = reinterpret_cast<long long*>(sinfo + kSets * 7 * kT);   // [3][N + 1]: offset of face f's j-th node in Iu
  uint64_t* bars = reinterpret_cast<uint64_t*>(lut + kLut);
  uint64_t *full = bars, *empty = bars + 2, *accf = bars + 4, *acce = bars + 6, *sfull = bars + 8, *sempty = bars + 10,
           *bfull = bars + 12, *bempty = bars + 12 + kStages, *done = bars + 12 + 2 * kStages;
  uint32_t* slot = reinterpret_cast<uint32_t*>(bars + 24);
  volatile int* abort_flag = reinterpret_cast<int*>(slot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t ntiles = (a.rows + kT - 1) / kT;
  if (tid < 3 * (a.N + 1)) lut[tid] = node_of(a.N, tid / (a.N + 1), tid % (a.N + 1)) * a.ldc;
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(full + i, 8);
      tc::mbar_init(empty + i, 1);
      tc::mbar_init(accf + i, 1);
      tc::mbar_init(acce + i, 16);
      tc::mbar_init(sfull + i, 2);
      tc::mbar_init(sempty + i, 16);
    }
    for (int i = 0; i < kStages; ++i) {
      tc::mbar_init(bfull + i, 1);
      tc::mbar_init(bempty + i, 1);
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

  if (warp == 17) {
    // ================= operator blocks
    uint32_t n = 0;
    const int steps = 3 * a.chunks;
    for (int64_t tile = blockIdx.x; tile < ntiles && !aborted(abort_flag); tile += gridDim.x)
      for (int s = 0; s < steps; ++s, ++n) {
        const uint32_t b = n % kStages, use = n / kStages;
        if (use > 0) wait(bempty + b, (use - 1) & 1u, abort_flag);
        if (aborted(abort_flag)) break;
        if (lane == 0) {
          tc::mbar_expect_tx(bfull + b, kStage);
          tc::bulk_g2s(sB + b * kStage, a.ops + size_t(s) * kStage, kStage, bfull + b);
        }
        __syncwarp();
      }
    // every copy has landed before the block ends
    for (uint32_t k = n < kStages ? 0 : n - kStages; k < n; ++k)
      tc::wait_done(bfull + k % kStages, (k / kStages) & 1u, abort_flag);
  } else if (warp == 16) {
    // ================= products
    const uint64_t ad = tc::smem_desc(tc::smem_addr(sm), 128, 6 * 128);
    const uint64_t bd = tc::smem_desc(tc::smem_addr(sB), 128, 256);
    uint32_t n = 0, g = 0, it = 0;
    for (int64_t tile = blockIdx.x; tile < ntiles && !aborted(abort_flag); tile += gridDim.x, ++it) {
      const uint32_t ab = it % kAcc, use = it / kAcc;
      if (use > 0) wait(acce + ab, (use - 1) & 1u, abort_flag);
      for (int kc = 0; kc < a.chunks; ++kc, ++g) {
        wait(full + (g & 1u), (g >> 1) & 1u, abort_flag);
        for (int c = 0; c < 3; ++c, ++n) {
          const uint32_t b = n % kStages;
          wait(bfull + b, (n / kStages) & 1u, abort_flag);
          tc::fence_after();
          if (lane == 0) {
            fx::issue_step<32>(tb + ab * kSums * NC, ad + (((g & 1u) * kChunkBytes + c * 256) >> 4), kChunkSlice,
                       bd + ((b * kStage) >> 4), NC, kc == 0 && c == 0);
            tc::mma_commit(bempty + b);
            if (c == 2) tc::mma_commit(empty + (g & 1u));
            if (c == 2 && kc + 1 == a.chunks) tc::mma_commit(accf + ab);
          }
          __syncwarp();
        }
      }
    }
    if (lane == 0) tc::mma_commit(done);
    __syncwarp();
    tc::wait_done(done, 0, abort_flag);
  } else if (warp >= 18) {
    // ================= scales
    uint32_t it = 0;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it) {
      const uint32_t set = it % kSets;
      if (it >= kSets) wait(sempty + set, (it / kSets - 1) & 1u, abort_flag);
#pragma unroll 1
      for (int k = 0; k < 2; ++k) {
        const int e = (warp - 18) * 32 + lane + 64 * k;
        const int64_t row = tile * kT + e, be = a.row0 + (row < a.rows ? row : 0), el = elem_of(be, a.K);
        const int boff = int(be - el);
        int code[3];
#pragma unroll
        for (int f = 0; f < 3; ++f) code[f] = __ldg(a.conn + 3 * el + f);
        const int4 x = __ldg(a.ex + be);
        const short4 t = __ldg(a.tex + el);
        const double u0 = __ldg(a.u0 + be);
        long long c[kCoefs];
#pragma unroll
        for (int i = 0; i < kCoefs; ++i) c[i] = fx::join(coef(a.tab + el + int64_t(i) * a.K));
        int4 y[3];
        double d[3];  // the jump without its v parts
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          const int64_t nb = boff + (code[f] >> 2);
          y[f] = code[f] >= 0 ? __ldg(a.ex + nb) : x;
          d[f] = code[f] >= 0 ? __ldg(a.u0 + nb) - u0 : (code[f] == -2 ? -2.0 * u0 : 0.0);
        }
        const int et = t.z + a.lpen;
        int E = x.x + t.x;
        bool bad = x.w >= fx::kBadExp;
        int ej[3];  // each of the jump's three parts is below 2^ej
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          ej[f] = max(max(x.x, y[f].x), fx::exp_bound(d[f]));
          bad = bad || y[f].w >= fx::kBadExp;
          E = max(E, max(max(ej[f] + t.y + 1 - a.k2, ej[f] + et + 3 - a.k1), max(x.z, y[f].z) + 1 - a.k1));
          E = max(E, max(x.y, y[f].y) - 2 - a.k1);  // q is only shifted down
        }
        if (a.helm) E = max(E, x.w + fx::exp_bound(a.lambda * __ldg(a.gx + 16 * el)) - a.km);
        int2* sc = scoef + set * kCoefs * kT + e;
        int* si = sinfo + set * 7 * kT + e;
        // columns at scale 2^{56-E}, from v 2^{59-ev} and a coefficient c 2^{62-e}
        auto put = [&](int i, long long v, int sh) {
          const Split q = fx::split(fx::sar(v, sh));
          sc[i * kT] = make_int2(q.h, q.l);
        };
#pragma unroll
        for (int i = 0; i < 3; ++i) put(i, c[i], E - x.x - t.x + 1);
        si[0] = bad ? kBadScale : E;
        const int sq = E + 2 + a.k1;  // half of q 2^{57-eq} at 2^{56-E}
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          const int sj = E - ej[f] - t.y + 2 + a.k2;  // half the jump
          put(3 + 2 * f, c[3 + 2 * f], sj);
          put(4 + 2 * f, c[4 + 2 * f], sj);
          put(9 + f, (c[9 + f] >> a.lpen) * a.cpen, E - ej[f] - et + 1 + a.k1);
          sdiff[(set * 3 + f) * kT + e] = fx::fix<59>(d[f], ej[f]);
          si[(1 + f) * kT] = code[f] >= 0 ? boff + (code[f] >> 2) : code[f];
          si[(4 + f) * kT] = (code[f] & 3) | (min(ej[f] - x.x, 63) << 2) | (min(ej[f] - y[f].x, 63) << 8) |
                             (min(sq - x.y, 63) << 14) | (min(sq - y[f].y, 63) << 20);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(sfull + set);
    }
  } else {
    // ================= columns and drain
    const int grp = warp >> 3, half = (warp >> 2) & 1, e = (warp & 3) * 32 + lane;
    const uint32_t lanebase = uint32_t((warp & 3) * 32) << 16;
    const int N = a.N, Np = (N + 1) * (N + 2) / 2, Nfp = N + 1, nface = 3 * Nfp;
    uint32_t it = 0, g0 = 0;
    int Eprev = 0;

    auto drain = [&](uint32_t t, int64_t row, int E) {
      const uint32_t ab = t % kAcc;
      wait(accf + ab, (t / kAcc) & 1u, abort_flag);
      tc::fence_after();
      const int c0 = (warp >> 2) * (NC / 4);
#pragma unroll 1
      for (int p = 0; p < NC / 16; ++p) {
        const int col = c0 + 4 * p;
        if (col < a.M) {
          float acc[4][kSums];
          __syncwarp();
#pragma unroll
          for (int s = 0; s < kSums; ++s) {
            uint32_t w[4];
            tc::tmem_ld4(tb + lanebase + (ab * kSums + s) * NC + col, w);
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[c][s] = __uint_as_float(w[c]);
          }
          tc::tmem_wait_ld();
          if (row < a.rows) {
            double* o = a.out + row * a.ldo + col;
#pragma unroll
            for (int c = 0; c < 4; ++c)
              if (col + c < a.M) {
                const double v = fx::sums_to_double(acc[c], __ldg(a.ea + col + c) + E - 56);
                o[c] = E == kBadScale ? fx::double_of(0x7ff8000000000000ll) : v;
              }
          }
        }
      }
      tc::fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acce + ab);
    };

    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it, g0 += a.chunks) {
      const int64_t row = tile * kT + e, be = a.row0 + (row < a.rows ? row : 0);
      const long long *uo = a.Iu + be, *qo = a.Iq + be;
      const uint32_t set = it % kSets;
      const int2* sc = scoef + set * kCoefs * kT + e;
      const long long* sd = sdiff + set * 3 * kT + e;
      const int* si = sinfo + set * 7 * kT + e;
      wait(sfull + set, (it / kSets) & 1u, abort_flag);
      const int E = si[0];
      bool drained = it == 0;
      for (int kc = 0; kc < a.chunks; ++kc) {
        const uint32_t g = g0 + kc;
        if ((g & 1u) != uint32_t(grp)) continue;
        if (g >= 2) wait(empty + grp, ((g >> 1) - 1) & 1u, abort_flag);
        const int gr = 2 * kc + half;  // this warp's group of eight items
        uint8_t* dst = sm + grp * kChunkBytes + (e >> 3) * 768 + half * 128 + (e & 7) * 16;
        auto cf = [&](int k) {
          const int2 q = sc[k * kT];
          return Split{q.x, q.y};
        };
        if (gr < a.gvol) {  // Grr u, Grs u, Gss u at eight nodes
          long long v[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) v[i] = 8 * gr + i < Np ? __ldg(uo + (8 * gr + i) * a.ldc) : 0;
#pragma unroll 1
          for (int c = 0; c < 3; ++c) {
            const Split k = cf(c);
            long long x[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = fx::mul(fx::split(v[i]), k);
            fx::digits8(x, dst + c * 256, kChunkSlice);
          }
        } else if (gr < a.gface) {
#pragma unroll 1
          for (int hb = 0; hb < 2; ++hb) {  // four face nodes at a time: their sixteen loads are in flight together
            const int i0 = 8 * (gr - a.gvol) + 4 * hb;
            long long v[4], w[4], y[4], z[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int t = i0 + i, f = t >= 2 * Nfp ? 2 : (t >= Nfp ? 1 : 0);
              v[i] = w[i] = y[i] = z[i] = 0;
              if (t < nface) {
                const int nb = si[(1 + f) * kT], fn = si[(4 + f) * kT] & 3;
                v[i] = __ldg(uo + lut[t]);
                y[i] = __ldg(qo + t * a.ldc);
                if (nb >= 0) {
                  const int tn = fn * Nfp + N - (t - f * Nfp);
                  w[i] = __ldg(a.Iu + nb + lut[tn]);
                  z[i] = __ldg(a.Iq + nb + tn * a.ldc);
                }
              }
            }
            long long x[3][4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int t = i0 + i, f = t >= 2 * Nfp ? 2 : (t >= Nfp ? 1 : 0);
              const int nb = si[(1 + f) * kT], info = si[(4 + f) * kT];
              const long long um = v[i] >> ((info >> 2) & 63), qm = y[i] >> ((info >> 14) & 63);
              long long up = w[i] >> ((info >> 8) & 63), qp = z[i] >> ((info >> 20) & 63);
              if (nb < 0) {  // Dirichlet: u+ = -u-, grad u+ = grad u-; Neumann: no terms
                up = nb == -2 ? -um : um;
                qp = nb == -2 ? ~qm : qm;  // ~: the shifts' roundings cancel, as two neighbours' do
              }
              const Split s = fx::split(up - um + sd[f * kT]);
              x[0][i] = fx::mul(s, cf(3 + 2 * f));
              x[1][i] = fx::mul(s, cf(4 + 2 * f));
              x[2][i] = qp - qm + fx::mul(s, cf(9 + f));
            }
#pragma unroll
            for (int c = 0; c < 3; ++c)
              fx::digits4(x[c], dst + c * 256 + hb * 8, kChunkSlice);
          }
        } else {  // lambda J u, three nodes an item (zero past the last group)
          const int n0 = 24 * (gr - a.gface);
          Split k{0, 0};
          long long k0 = 0;  // lambda J u0
          if (a.helm) {
            const double lj = a.lambda * __ldg(a.gx + 16 * elem_of(be, a.K)), l0 = lj * __ldg(a.u0 + be);
            const int elj = fx::exp_bound(lj), e0 = fx::exp_bound(l0);
            k = fx::split(fx::sar(fx::fix<62>(lj, elj), E - __ldg(a.ex + be).x - elj + 1 + a.km));
            k0 = fx::sar(fx::fix<59>(l0, e0), E - e0 + 3 + a.km);
          }
#pragma unroll 1
          for (int c = 0; c < 3; ++c) {
            long long x[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const int n = n0 + 3 * i + c;
              x[i] = a.helm && n < Np ? fx::mul(fx::split(__ldg(uo + n * a.ldc)), k) + k0 : 0;
            }
            fx::digits8(x, dst + c * 256, kChunkSlice);
          }
        }
        tc::fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(full + grp);
        if (!drained) {
          drain(it - 1, row - int64_t(gridDim.x) * kT, Eprev);
          drained = true;
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(sempty + set);  // the tile's columns are formed
      if (!drained) drain(it - 1, row - int64_t(gridDim.x) * kT, Eprev);
      Eprev = E;
    }
    if (it > 0) drain(it - 1, (blockIdx.x + int64_t(it - 1) * gridDim.x) * kT + e, Eprev);
  }
  if (*abort_flag && tid == 0) atomicExch(&g_t64_err, 1);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_dealloc(tb, 512);
}

// ------------------------------------------------------------------ host side
// An operator block image: the integers A(r, k) (a row's entries 2^{56 - its exponent}),
// r < M <= nc, k < K, cut into digits (fix64.cuh), digit i of row r at stacked row
// i nc + r, in 16-column steps of the canonical layout (columns past K are zero).
// False if a row's digit sums could leave the integers that FP32 holds.
template <typename F>
bool slice_block(const F& A, int M, int nc, int K, std::vector<uint8_t>& img) {
  const int steps = (K + 15) / 16;
  const size_t step_bytes = size_t(kDigits) * nc * 32;
  const size_t base = img.size();
  img.resize(base + steps * step_bytes, 0);
  for (int r = 0; r < M; ++r) {
    fx::ExactSums sums;
    for (int k = 0; k < K; ++k) {
      const long long x = A(r, k);
      if (x == 0) continue;
      int d[kDigits];
      fx::digits_of(x, d);
      sums.add(d);
      uint8_t* blk = img.data() + base + size_t(k / 16) * step_bytes;
      for (int i = 0; i < kDigits; ++i) {
        const int R = i * nc + r, c = k % 16;
        const uint16_t h = fx::fp16_int(d[i]);
        std::memcpy(blk + size_t(R / 8) * 256 + (c / 8) * 128 + (R % 8) * 16 + (c % 8) * 2, &h, 2);
      }
    }
    if (!sums.exact()) return false;
  }
  return true;
}

struct OutOp {
  int M = 0, c0 = 0;  // output columns [c0, c0 + M)
  uint8_t* ops = nullptr;
  int* ea = nullptr;
};
struct OutSet {  // one form of the operator: Poisson, or with the Helmholtz columns
  int gvol = 0, gface = 0, chunks = 0, nc = 0, parts = 0;
  OutOp part[2];
};
struct Tc64Apply {
  bool ready = false;
  int trace_ea = 0, passes = 0, ks = 0, k1 = 0, k2 = 0, km = 0;
  uint8_t* trace = nullptr;
  OutSet out[2];  // [helmholtz]
};
Tc64Apply g_t64[64][kMaxN + 1];  // [device][degree]

cudaError_t upload(const void* p, size_t n, void** d) {
  cudaError_t e = cudaMalloc(d, n);
  if (e == cudaSuccess) e = cudaMemcpy(*d, p, n, cudaMemcpyHostToDevice);
  return e;
}

cudaError_t build_t64(const RefElem& R, Tc64Apply& o) {
  const int N = R.N, Np = R.Np;
  // boundary derivatives: rows 2b, 2b + 1 = d/dr, d/ds at the b-th node counter-clockwise
  auto trace = [&](int r, int k) {
    const int b = r / 2, n = face_node(N, b / N, b % N);
    return (r & 1) ? R.Ds[size_t(n) * Np + k] : R.Dr[size_t(n) * Np + k];
  };
  double mx = 0.0, l1 = 0.0;
  for (int r = 0; r < 6 * N; ++r) {
    double s = 0.0;
    for (int k = 0; k < Np; ++k) {
      mx = std::max(mx, std::fabs(trace(r, k)));
      s += std::fabs(trace(r, k));
    }
    l1 = std::max(l1, s);
  }
  o.trace_ea = fx::row_exp(mx, l1);
  o.passes = (6 * N + kTraceN - 1) / kTraceN;
  o.ks = (Np + 15) / 16;
  std::vector<uint8_t> img;
  bool exact = true;
  for (int p = 0; p < o.passes; ++p)
    exact &= slice_block([&](int r, int k) { return k < Np ? std::llround(std::ldexp(trace(p * kTraceN + r, k), 56 - o.trace_ea)) : 0ll; },
                         std::min(kTraceN, 6 * N - p * kTraceN), kTraceN, 16 * o.ks, img);
  cudaError_t e = exact ? cudaSuccess : cudaErrorInvalidValue;
  if (exact) e = upload(img.data(), img.size(), reinterpret_cast<void**>(&o.trace));
  OutTable tables[2];
  build_out_tables(R, tables);
  for (int helm = 0; helm < 2; ++helm) {
    OutSet& w = o.out[helm];
    const OutTable& t = tables[helm];
    o.k1 = t.k1;
    o.k2 = t.k2;
    o.km = t.km;
    w.gvol = t.gvol;
    w.gface = t.gface;
    w.chunks = t.chunks;
    w.parts = Np > 64 ? 2 : 1;
    const int M = (Np + w.parts - 1) / w.parts;
    w.nc = (M + 15) & ~15;
    for (int q = 0; q < w.parts; ++q) {
      OutOp& p = w.part[q];
      p.c0 = q * M;
      p.M = std::min(M, Np - p.c0);
      std::vector<int> ea(w.nc, 0);
      std::copy(t.ea.begin() + p.c0, t.ea.begin() + p.c0 + p.M, ea.begin());
      std::vector<uint8_t> im;
      if (!slice_block([&](int r, int k) { return t.x[size_t(p.c0 + r) * t.cols + k]; }, p.M, w.nc, t.cols, im))
        return cudaErrorInvalidValue;
      if (e == cudaSuccess) e = upload(im.data(), im.size(), reinterpret_cast<void**>(&p.ops));
      if (e == cudaSuccess) e = upload(ea.data(), ea.size() * sizeof(int), reinterpret_cast<void**>(&p.ea));
    }
  }
  o.ready = e == cudaSuccess;
  return e;
}

// The degree's sliced operators on the current device, built on first use
// when `build` is set (null if not built, or if building failed: *err says why).
const Tc64Apply* t64_ops(dg_mesh* m, int degree, bool build, cudaError_t* err) {
  *err = cudaSuccess;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) {
    *err = e;
    return nullptr;
  }
  std::lock_guard<std::mutex> lk(table_mutex());
  Tc64Apply& o = g_t64[dev & 63][degree];
  if (!o.ready) {
    if (!build) return nullptr;
    const RefElem R = m->ref[degree].N ? m->ref[degree] : build_reference(degree);
    Tc64Apply built;
    e = build_t64(R, built);
    if (e != cudaSuccess) {
      *err = e;
      return nullptr;
    }
    o = built;
  }
  return &o;
}
int64_t t64_ldc(int64_t nE) { return (nE + 31) & ~int64_t(31); }

// Shared memory of the kernels, once per device; returns the SM count.
cudaError_t t64_launch_setup(int* sms) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  static int count[64];
  std::lock_guard<std::mutex> lk(table_mutex());
  if (!count[dev & 63]) {
    auto allow = [&](const void* f, int bytes) {
      if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    };
    allow(reinterpret_cast<const void*>(t64_trace<1>), trace_smem(1));
    allow(reinterpret_cast<const void*>(t64_trace<2>), trace_smem(2));
    allow(reinterpret_cast<const void*>(t64_trace<3>), trace_smem(3));
    allow(reinterpret_cast<const void*>(t64_trace<4>), trace_smem(4));
    allow(reinterpret_cast<const void*>(t64_trace<5>), trace_smem(5));
    allow(reinterpret_cast<const void*>(t64_output<16>), out_smem(16));
    allow(reinterpret_cast<const void*>(t64_output<32>), out_smem(32));
    allow(reinterpret_cast<const void*>(t64_output<48>), out_smem(48));
    allow(reinterpret_cast<const void*>(t64_output<64>), out_smem(64));
    int n = 0;
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    count[dev & 63] = n;
  }
  *sms = count[dev & 63];
  return cudaSuccess;
}

cudaError_t launch_trace(const TraceArgs& a, int ks, int sms, cudaStream_t st) {
  const int64_t tiles = (a.rows + kT - 1) / kT;
  const unsigned g = unsigned(std::min<int64_t>(tiles, int64_t(sms) * (ks <= 3 ? 2 : 1)));
  switch (ks) {
    case 1: t64_trace<1><<<g, 288, trace_smem(1), st>>>(a); break;
    case 2: t64_trace<2><<<g, 288, trace_smem(2), st>>>(a); break;
    case 3: t64_trace<3><<<g, 288, trace_smem(3), st>>>(a); break;
    case 4: t64_trace<4><<<g, 288, trace_smem(4), st>>>(a); break;
    default: t64_trace<5><<<g, 288, trace_smem(5), st>>>(a); break;
  }
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_output(const OutArgs& a, int nc, int sms, cudaStream_t st) {
  const unsigned g = unsigned(std::min<int64_t>((a.rows + kT - 1) / kT, sms));
  switch (nc) {
    case 16: t64_output<16><<<g, kOutThreads, out_smem(16), st>>>(a); break;
    case 32: t64_output<32><<<g, kOutThreads, out_smem(32), st>>>(a); break;
    case 48: t64_output<48><<<g, kOutThreads, out_smem(48), st>>>(a); break;
    default: t64_output<64><<<g, kOutThreads, out_smem(64), st>>>(a); break;
  }
  note_launch();
  return cudaGetLastError();
}

// The largest forward distance from an element to one of its neighbours (rows),
// from the host copy of the connectivity; kept with the mesh.
int64_t t64_reach(dg_mesh* m) {
  if (m->nb_reach < 0) {
    int64_t r = 0;
    for (int64_t e = 0; e < m->K; ++e)
      for (int f = 0; f < 3; ++f) {
        const int32_t code = m->conn_h[size_t(3 * e + f)];
        if (code >= 0) r = std::max<int64_t>(r, int64_t(code >> 2) - e);
      }
    m->nb_reach = r;
  }
  return m->nb_reach;
}
}  // namespace

bool tc64_supported(int degree) { return degree >= 1 && degree <= kMaxN; }

// The scratch a caller that brings its own has to hold: u and q in fixed point
// and each row's exponents and u0 need Np + 3 (N + 1) + 3 words per row; the size
// stays the published one (include/dg.h), which is larger.
size_t tc64_scratch_words(int degree, int64_t nE, bool helm) {
  const int Np = (degree + 1) * (degree + 2) / 2, NFN = 3 * (degree + 1);
  return size_t(t64_ldc(nE)) * (2 * Np + 5 * NFN + (helm ? Np : 0)) + 2 * (size_t(nE + 1) / 2) + 2;
}

cudaError_t ensure_tc64_ops(dg_mesh* m, int degree) {
  if (!tc64_supported(degree)) return cudaSuccess;
  cudaError_t e;
  t64_ops(m, degree, true, &e);
  return e;
}

bool tc64_ops_ready(int degree) {
  if (!tc64_supported(degree)) return false;
  cudaError_t e;
  return t64_ops(nullptr, degree, false, &e) != nullptr;
}

cudaError_t build_fixed_geometry(dg_mesh* m) {
  cudaError_t e = cudaMalloc(&m->gfix, sizeof(int2) * kCoefs * m->K);
  if (e == cudaSuccess) e = cudaMalloc(&m->gfix_ex, sizeof(short4) * m->K);
  if (e != cudaSuccess) return e;
  k_fix_geometry<<<unsigned((m->K + 255) / 256), 256>>>(m->K, m->geox, m->gfix, m->gfix_ex);
  note_launch();
  e = cudaGetLastError();
  return e == cudaSuccess ? cudaStreamSynchronize(nullptr) : e;
}

cudaError_t launch_apply_tc64(dg_mesh* m, int degree, int B, double lambda, const double* u, double* Au,
                              cudaStream_t st, double* scratch, const ApplyChunks* chunks) {
  if (B < 1) return cudaSuccess;
  if (!tc64_supported(degree)) return cudaErrorInvalidValue;
  cudaError_t e;
  const Tc64Apply* ops = t64_ops(m, degree, scratch == nullptr, &e);
  if (!ops) return e != cudaSuccess ? e : cudaErrorNotReady;
  int sms = 0;
  e = t64_launch_setup(&sms);
  if (e != cudaSuccess) return e;
  const int N = degree, Np = (N + 1) * (N + 2) / 2, nface = 3 * (N + 1);
  const bool helm = lambda != 0.0;
  const int64_t nE = int64_t(B) * m->K;
  if (nE > 0x7fffffff) return cudaErrorInvalidValue;  // rows are addressed in 32 bits (their scratch is above 160 GB)
  const int64_t ldc = t64_ldc(nE);
  // scratch: u and q in fixed point [Np + 3 (N + 1)][ldc], the rows' exponents and u0;
  // every word read is written first by this call
  const size_t words = size_t(ldc) * (Np + nface + 3);
  if (!scratch && m->t64_cap < words) {
    cudaFree(m->t64_scratch);
    m->t64_scratch = nullptr;
    m->t64_cap = 0;
    e = cudaMalloc(&m->t64_scratch, words * sizeof(double));
    if (e == cudaSuccess) e = poison(m->t64_scratch, words * sizeof(double), POISON_APPLY);
    if (e != cudaSuccess) return e;
    m->t64_cap = words;
    ++m->scratch_gen;
  }
  // (a given scratch may start at any double; its size has room for the rounding)
  uintptr_t base = reinterpret_cast<uintptr_t>(scratch ? scratch : m->t64_scratch);
  long long* Iu = reinterpret_cast<long long*>((base + 15) & ~uintptr_t(15));
  long long* Iq = Iu + size_t(ldc) * Np;
  int4* ex = reinterpret_cast<int4*>(Iq + size_t(ldc) * nface);  // 16-byte aligned: ldc is a multiple of 32
  double* u0 = reinterpret_cast<double*>(ex + ldc);
  const OutSet& w = ops->out[helm ? 1 : 0];
  const bool chunked = chunks && chunks->n > 0 && chunks->bounds && chunks->bounds[chunks->n] == nE;
  const int nch = chunked ? chunks->n : 1;
  const int64_t whole[2] = {0, nE};
  const int64_t* bnd = chunked ? chunks->bounds : whole;
  // a chunk's output product needs the boundary derivatives of every chunk that
  // holds one of its rows' neighbours: rows up to (last row + reach)
  const int64_t reach = nch > 1 ? t64_reach(m) : nE;
  auto ready_after = [&](int c) {  // the last chunk whose first phase chunk c's output product needs
    const int64_t last = std::min<int64_t>(nE - 1, bnd[c + 1] - 1 + reach);
    int j = c;
    while (j + 1 < nch && bnd[j + 1] <= last) ++j;
    return j;
  };
  auto finish = [&](int c) -> cudaError_t {  // output product of chunk c
    const int64_t r0 = bnd[c], n = bnd[c + 1] - r0;
    const int cpen = (N + 1) * (N + 2) / 2;
    OutArgs a{};
    a.N = N;
    a.gvol = w.gvol;
    a.gface = w.gface;
    a.chunks = w.chunks;
    a.cpen = cpen;
    while ((1 << a.lpen) < cpen) ++a.lpen;
    a.k1 = ops->k1;
    a.k2 = ops->k2;
    a.km = ops->km;
    a.helm = helm;
    a.lambda = lambda;
    a.K = m->K;
    a.rows = n;
    a.row0 = r0;
    a.Iu = Iu;
    a.Iq = Iq;
    a.ldc = ldc;
    a.ex = ex;
    a.u0 = u0;
    a.tab = m->gfix;
    a.tex = m->gfix_ex;
    a.gx = m->geox;
    a.conn = m->conn;
    a.ldo = Np;
    cudaError_t err = cudaSuccess;
    for (int q = 0; q < w.parts && err == cudaSuccess; ++q) {
      a.M = w.part[q].M;
      a.ops = w.part[q].ops;
      a.ea = w.part[q].ea;
      a.out = Au + r0 * Np + w.part[q].c0;
      err = launch_output(a, w.nc, sms, st);
    }
    if (err == cudaSuccess && chunked && chunks->after) err = chunks->after(chunks->ctx, c, r0, r0 + n);
    return err;
  };
  int done = 0;  // chunks whose output product is issued
  for (int c = 0; c < nch; ++c) {  // boundary derivatives, element-local
    const int64_t r0 = bnd[c], r1 = bnd[c + 1];
    if (chunked && chunks->before && (e = chunks->before(chunks->ctx, c, r0, r1)) != cudaSuccess) return e;
    TraceArgs a{};
    a.N = N;
    a.passes = ops->passes;
    a.u = u + r0 * Np;
    a.aligned = (reinterpret_cast<uintptr_t>(a.u) & 15u) == 0;
    a.K = m->K;
    a.rows = r1 - r0;
    a.row0 = r0;
    a.tab = m->gfix;
    a.tex = m->gfix_ex;
    a.ops = ops->trace;
    a.ea = ops->trace_ea;
    a.Iu = Iu + r0;
    a.Iq = Iq + r0;
    a.ldc = ldc;
    a.ex = ex + r0;
    a.u0 = u0 + r0;
    e = launch_trace(a, ops->ks, sms, st);
    if (e != cudaSuccess) return e;
    while (done < nch && ready_after(done) <= c)
      if ((e = finish(done++)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t tc64_error(int* flag) {
  int zero = 0, gemm = 0;
  cudaError_t e = cudaMemcpyFromSymbol(flag, g_t64_err, sizeof(int));
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_t64_err, &zero, sizeof(int));
  if (e == cudaSuccess) e = tc64_gemm_error(&gemm);
  *flag |= gemm;
  return e;
}

}  // namespace dgx
