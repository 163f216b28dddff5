// The tile kernel's FP32 form at degrees 9 and 10 (DG_KERNEL_TILE), where the
// tensor-memory kernel's operands no longer fit: small dense products from shared
// memory, eight elements per thread.
//
// One thread per (element, node) would read two operator entries and one field value
// from shared memory for every two multiply-adds. Here a thread has one row of an
// operator and eight elements of the tile; fields lie [node][element], so eight values
// come as two wide reads at one address for all lanes: two operator entries and two wide
// reads for sixteen multiply-adds, which go two to an instruction (fma.f32x2, the same
// roundings; 162 -> 153 us). A neighbour's normal derivative needs the operator rows of
// the face that the neighbour has there; the tile's faces are therefore sorted by that
// local face into groups of eight which share their rows. Nothing is kept outside the
// block, so the apply needs no scratch. Two blocks per SM: their barriers and loads
// interleave. 32,768 triangles, N = 10, Helmholtz: 348 -> 139 us, of which the
// multiply-adds are about 30; latency of the shared reads and the barriers between the
// stages take the rest (four elements per thread and twice the warps: 152).
#include <algorithm>

#include "dg_internal.h"
#include "fma2.cuh"

namespace dgx {
namespace {

constexpr int kE = 16;               // elements per tile
constexpr int kG = 8;                // elements per thread
constexpr int kLd = kE + 4;          // row pitch of a tile's fields: 16-byte rows, 4-way conflicts in the transposes
constexpr int kBatch = 9;            // gathered values in flight per thread: three rounds at most
constexpr int kSlots = 3 * kE + 16;  // faces with a neighbour in groups of kG by its local face
constexpr int kLdN = kSlots + 4;     // row pitch of the neighbours' values
constexpr int kTables = 3 * kE + kSlots + kSlots / kG + kE + 2 * kE + 2 * 3 * kE;

__host__ __device__ constexpr int row_start(int N, int row) { return row * (N + 1) - row * (row - 1) / 2; }
__device__ __forceinline__ int fnode(int N, int f, int j) {
  return f == 0 ? j : (f == 1 ? row_start(N, j) + (N - j) : row_start(N, N - j));
}

template <int N>
struct Sz {
  static constexpr int Np = (N + 1) * (N + 2) / 2, Nfp = N + 1, NFN = 3 * Nfp;
  static constexpr int LD = Np | 1;  // odd: a warp's 32 operator rows fall into different banks
  static constexpr int items = Np * (kE / kG);
  static constexpr int threads = (items + 31) / 32 * 32;
  // words of shared memory: fields, face data, geometry, tile tables, operators
  static constexpr int fields = 3 * Np * kLd + 3 * NFN * kLd;
  static constexpr int words(bool helm) {
    return fields + 16 * kE + kTables + (helm ? 5 : 4) * Np * LD + Nfp * Nfp;
  }
  static_assert(Np * kLdN <= 3 * Np * kLd + NFN * kLd, "the neighbours' values fit over u, w and F1");
};

// x[e] += a, y[e] += b times the values at p of a thread's elements
__device__ __forceinline__ void fma_g(float (&x)[kG], float (&y)[kG], float a, float b, const float* p) {
  float w[kG];
  load_vec(w, p);
  fma_vec(x, a, w);
  fma_vec(y, b, w);
}
__device__ __forceinline__ void fma_g(float (&x)[kG], float a, const float* p) {
  float w[kG];
  load_vec(w, p);
  fma_vec(x, a, w);
}

template <int N, bool HELM>
__global__ void __launch_bounds__(Sz<N>::threads, 2)
    t32_apply(int64_t K, int64_t nE, const float* __restrict__ gx, const int32_t* __restrict__ conn,
              const float* __restrict__ ops, float lambda, const float* __restrict__ u, float* __restrict__ Au) {
  using S = Sz<N>;
  constexpr int Np = S::Np, Nfp = S::Nfp, NFN = S::NFN, LD = S::LD, T = S::threads;
  constexpr float cpen = float((N + 1) * (N + 2)) * 0.5f;
  extern __shared__ __align__(16) float sm[];
  float* sup = sm;                  // [Np][kLdN] neighbours' values, until their face data are taken
  float* su = sm;                   // [Np][kLd]
  float* swr = su + Np * kLd;       // then the result
  float* sws = swr + Np * kLd;
  float* sf = sws + Np * kLd;       // [NFN][kLd]: own n.grad u, then F1
  float* sj = sf + NFN * kLd;       // u+, jump, F2r
  float* sa = sj + NFN * kLd;       // n.grad u+, average + tau jump, F2s
  float* sg = sa + NFN * kLd;       // [16 words][kE] geometry
  int64_t* sbase = reinterpret_cast<int64_t*>(sg + 16 * kE);  // first element of the right-hand side
  float2* snn = reinterpret_cast<float2*>(sbase + kE);        // neighbour's n.grad r, n.grad s [f kE + e]
  int* sel = reinterpret_cast<int*>(snn + 3 * kE);            // element of the mesh
  int* scode = sel + kE;                                      // [f kE + e]
  int* sslot = scode + 3 * kE;                                // [slot] -> f kE + e or -1
  int* sgrp = sslot + kSlots;                                 // [group] -> the neighbours' local face
  float* sDr = sg + 16 * kE + kTables;  // [Np][LD] each
  float* sDs = sDr + Np * LD;
  float* sBr = sDs + Np * LD;
  float* sBs = sBr + Np * LD;
  float* sM = sBs + Np * LD;
  float* sMf = sM + (HELM ? Np * LD : 0);
  for (int k = threadIdx.x; k < Np * Np; k += T) {
    const int i = k / Np, o = i * LD + k - i * Np;
    sDr[o] = ops[k];
    sDs[o] = ops[Np * Np + k];
    sBr[o] = ops[2 * Np * Np + k];
    sBs[o] = ops[3 * Np * Np + k];
    if (HELM) sM[o] = ops[4 * Np * Np + k];
  }
  for (int k = threadIdx.x; k < Nfp * Nfp; k += T) sMf[k] = ops[5 * Np * Np + k];
  const int64_t ntiles = (nE + kE - 1) / kE;
  const int tid = threadIdx.x, g = tid / Np, i = tid - g * Np;  // this thread's elements g kG .. and node
  const bool mine = g < kE / kG;
  int onf[3] = {-1, -1, -1};  // the node's rows among the face nodes
  {
    int row = 0, rs = 0;
    while (i >= rs + (N + 1 - row)) rs += N + 1 - row++;
    const int col = i - rs;
    if (row == 0) onf[0] = col;
    if (col == N - row) onf[1] = Nfp + row;
    if (col == 0) onf[2] = 2 * Nfp + N - row;
  }
  constexpr int kOwn = (kE * Np + T - 1) / T;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t e0 = tile * kE;
    const int ne = int(nE - e0 < kE ? nE - e0 : kE);
    __syncthreads();  // the previous tile's result has been read
    float own[kOwn];  // the tile's own values, in flight until their place is free
#pragma unroll
    for (int t = 0; t < kOwn; ++t) {
      const int k = tid + t * T;
      own[t] = k < ne * Np ? __ldg(u + e0 * Np + k) : 0.f;
    }
    if (tid < kE) {
      const int64_t be = e0 + (tid < ne ? tid : 0), el = be < K ? be : be % K;
      sel[tid] = int(el);
      sbase[tid] = be - el;
    }
    if (tid >= 64 && tid < 64 + kSlots) sslot[tid - 64] = -1;
    __syncthreads();
    for (int k = tid; k < 16 * kE; k += T) sg[(k & 15) * kE + (k >> 4)] = __ldg(gx + 16 * int64_t(sel[k >> 4]) + (k & 15));
    if (tid < 3 * kE) scode[tid] = tid % kE < ne ? __ldg(conn + 3 * int64_t(sel[tid % kE]) + tid / kE) : -1;
    __syncthreads();
    int ng = 0;
    {  // sort the faces by the neighbour's local face (the counts give every thread the number of groups)
      const int mycode = tid < 3 * kE ? scode[tid] : -1;
      int n[3] = {0, 0, 0}, rank = 0;
#pragma unroll 12
      for (int k = 0; k < 3 * kE; ++k) {
        const int c = scode[k], l = c < 0 ? -1 : c & 3;
        if (k == tid && c >= 0) rank = l == 0 ? n[0] : (l == 1 ? n[1] : n[2]);
        n[0] += l == 0;
        n[1] += l == 1;
        n[2] += l == 2;
      }
      const int g0 = (n[0] + kG - 1) / kG, g1 = g0 + (n[1] + kG - 1) / kG;
      ng = g1 + (n[2] + kG - 1) / kG;
      if (mycode >= 0) {
        const int l = mycode & 3;
        sslot[(l == 0 ? 0 : (l == 1 ? g0 : g1)) * kG + rank] = tid;
        const float* nb = gx + 16 * int64_t(mycode >> 2) + 4 + 4 * l;
        snn[tid] = make_float2(__ldg(nb), __ldg(nb + 1));
      }
      if (tid < ng) sgrp[tid] = tid < g0 ? 0 : (tid < g1 ? 1 : 2);
    }
    __syncthreads();
    for (int k0 = tid; k0 < ng * kG * Np; k0 += kBatch * T) {  // kBatch loads in flight
      float v[kBatch];
#pragma unroll
      for (int t = 0; t < kBatch; ++t) {
        const int k = k0 + t * T, s = k / Np, m = k - s * Np;
        const int ef = k < ng * kG * Np ? sslot[s] : -1;
        v[t] = ef >= 0 ? __ldg(u + (sbase[ef % kE] + (scode[ef] >> 2)) * Np + m) : 0.f;
      }
#pragma unroll
      for (int t = 0; t < kBatch; ++t) {
        const int k = k0 + t * T, s = k / Np, m = k - s * Np;
        if (k < ng * kG * Np) sup[m * kLdN + s] = v[t];
      }
    }
    __syncthreads();
    for (int it = tid; it < ng * Nfp; it += T) {  // u+ and n+.grad u+, in the order of the element's own face
      const int q = it / Nfp, j = it - q * Nfp, n = fnode(N, sgrp[q], j);
      float a[kG] = {}, b[kG] = {};
#pragma unroll 6
      for (int m = 0; m < Np; ++m) fma_g(a, b, sDr[n * LD + m], sDs[n * LD + m], sup + m * kLdN + q * kG);
#pragma unroll
      for (int e = 0; e < kG; ++e) {
        const int ef = sslot[q * kG + e];
        if (ef >= 0) {
          const int o = ((ef / kE) * Nfp + N - j) * kLd + ef % kE;
          sj[o] = sup[n * kLdN + q * kG + e];
          sa[o] = snn[ef].x * a[e] + snn[ef].y * b[e];
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < kOwn; ++t) {
      const int k = tid + t * T, e = k / Np;
      if (k < kE * Np) su[(k - e * Np) * kLd + e] = own[t];
    }
    __syncthreads();
    if (mine) {  // gradient at node i: weighted by the metric, and along the normals of its faces
      float a[kG] = {}, b[kG] = {}, x[kG], y[kG];
#pragma unroll 6
      for (int m = 0; m < Np; ++m) fma_g(a, b, sDr[i * LD + m], sDs[i * LD + m], su + m * kLd + g * kG);
#pragma unroll
      for (int e = 0; e < kG; ++e) {
        const int le = g * kG + e;
        const float grr = sg[1 * kE + le], grs = sg[2 * kE + le], gss = sg[3 * kE + le];
        x[e] = grr * a[e] + grs * b[e];
        y[e] = grs * a[e] + gss * b[e];
      }
      store_vec(swr + i * kLd + g * kG, x);
      store_vec(sws + i * kLd + g * kG, y);
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        if (onf[f] < 0) continue;
#pragma unroll
        for (int e = 0; e < kG; ++e) {
          const int le = g * kG + e;
          x[e] = sg[(4 + 4 * f) * kE + le] * a[e] + sg[(5 + 4 * f) * kE + le] * b[e];
        }
        store_vec(sf + onf[f] * kLd + g * kG, x);
      }
    }
    __syncthreads();
    for (int k = tid; k < NFN * kE; k += T) {
      const int e = k % kE, r = k / kE, f = r / Nfp, o = r * kLd + e;
      const int code = scode[f * kE + e];
      const float um = su[fnode(N, f, r - f * Nfp) * kLd + e], dn = sf[o];
      float jm = 0.f, av = 0.f;
      if (code >= 0) {
        jm = sj[o] - um;
        av = 0.5f * (dn - sa[o]);  // the neighbour's normal is the opposite one
      } else if (code == -2) {     // Dirichlet: u+ = -u-, grad u+ = grad u-
        jm = -2.f * um;
        av = dn;
      }                            // Neumann: u+ = u-, grad u+ = -grad u-
      sj[o] = jm;
      sa[o] = av + cpen * sg[(7 + 4 * f) * kE + e] * jm;
    }
    __syncthreads();
    // face mass: a thread's entries are read before any is overwritten
    constexpr int kPer = (NFN * kE + T - 1) / T;
    float m1[kPer], m2[kPer];
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      const int k = tid + t * T;
      m1[t] = m2[t] = 0.f;
      if (k < NFN * kE) {
        const int e = k % kE, r = k / kE, f = r / Nfp, j = r - f * Nfp;
#pragma unroll
        for (int l = 0; l < Nfp; ++l) {
          const float mf = sMf[j * Nfp + l];
          m1[t] += mf * sa[(f * Nfp + l) * kLd + e];
          m2[t] += mf * sj[(f * Nfp + l) * kLd + e];
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      const int k = tid + t * T;
      if (k < NFN * kE) {
        const int e = k % kE, r = k / kE, f = r / Nfp;
        const float sJ = sg[(6 + 4 * f) * kE + e], f2 = 0.5f * sJ * m2[t];
        sf[r * kLd + e] = -sJ * m1[t];
        sj[r * kLd + e] = sg[(4 + 4 * f) * kE + e] * f2;
        sa[r * kLd + e] = sg[(5 + 4 * f) * kE + e] * f2;
      }
    }
    __syncthreads();
    float acc[kG] = {};
    if (mine) {  // volume term, lifted jumps, fluxes of node i: short sums apart, for their rounding and in parallel
      float vs[kG] = {}, lr[kG] = {}, ls[kG] = {};
#pragma unroll 6
      for (int m = 0; m < Np; ++m) {
        fma_g(acc, sBr[i * LD + m], swr + m * kLd + g * kG);
        fma_g(vs, sBs[i * LD + m], sws + m * kLd + g * kG);
      }
#pragma unroll
      for (int r = 0; r < NFN; ++r) {
        const int n = fnode(N, r / Nfp, r % Nfp);
        fma_g(lr, sDr[n * LD + i], sj + r * kLd + g * kG);
        fma_g(ls, sDs[n * LD + i], sa + r * kLd + g * kG);
      }
#pragma unroll
      for (int e = 0; e < kG; ++e) acc[e] = (acc[e] + vs[e]) + (lr[e] + ls[e]);
      if (HELM) {
        float mu[kG] = {};
#pragma unroll 6
        for (int m = 0; m < Np; ++m) fma_g(mu, sM[i * LD + m], su + m * kLd + g * kG);
#pragma unroll
        for (int e = 0; e < kG; ++e) acc[e] += lambda * sg[g * kG + e] * mu[e];
      }
#pragma unroll
      for (int f = 0; f < 3; ++f)
        if (onf[f] >= 0) fma_g(acc, 1.f, sf + onf[f] * kLd + g * kG);
    }
    __syncthreads();
    if (mine) store_vec(swr + i * kLd + g * kG, acc);
    __syncthreads();
    float* o = Au + e0 * Np;
    for (int k = tid; k < ne * Np; k += T) {
      const int e = k / Np;
      o[k] = swr[(k - e * Np) * kLd + e];
    }
  }
}

template <int N, bool HELM>
cudaError_t launch_n(const dg_mesh* m, int B, double lambda, const float* u, float* Au, cudaStream_t st) {
  using S = Sz<N>;
  constexpr int bytes = S::words(HELM) * 4;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 64) return cudaErrorInvalidDevice;
  static int grids[64];  // blocks that fit the device
  int grid;
  {
    std::lock_guard<std::mutex> lk(table_mutex());
    if (!grids[dev]) {
      int sms = 0, per = 0;
      e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
      if (e == cudaSuccess) e = cudaFuncSetAttribute(t32_apply<N, HELM>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
      if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, t32_apply<N, HELM>, S::threads, bytes);
      if (e != cudaSuccess) return e;
      grids[dev] = sms * std::max(1, per);
    }
    grid = grids[dev];
  }
  const int64_t nE = int64_t(B) * m->K, tiles = (nE + kE - 1) / kE;
  t32_apply<N, HELM><<<unsigned(std::min<int64_t>(tiles, grid)), S::threads, bytes, st>>>(
      m->K, nE, m->geox32, m->conn, reinterpret_cast<const float*>(m->ops32[N].buf), float(lambda), u, Au);
  note_launch();
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_apply_tile32(const dg_mesh* m, int degree, int B, double lambda, const float* u, float* Au,
                                cudaStream_t st) {
  if (B < 1) return cudaSuccess;
  if (degree == 9) return lambda != 0.0 ? launch_n<9, true>(m, B, lambda, u, Au, st) : launch_n<9, false>(m, B, lambda, u, Au, st);
  return lambda != 0.0 ? launch_n<10, true>(m, B, lambda, u, Au, st) : launch_n<10, false>(m, B, lambda, u, Au, st);
}

}  // namespace dgx
