// Host tables of the exactly sliced FP64 apply.
//
// What an apply to a smooth field yields is far smaller than the terms it is summed
// from, and what it yields when summed over an element's test functions (the field's
// flux out of the element) is smaller still. An entry's rounding error that does not
// cancel in that sum acts on every element alike, as a smooth source beta . grad u
// which the inverse operator amplifies: with the volume blocks rounded entry by entry
// to doubles, an element's sum was off by 6e-15 of its flux at degree 8 and the error of
// a solve on 512 x 512 squares 3.3e-13 to 5.8e-13 (three right-hand sides), against
// 0.2e-13 to 1.1e-13 with D^T M in two factors; with these tables 4e-17 and 0.14e-13 to
// 1.1e-13. The integer columns here therefore sum over the test functions to exactly
// zero where the basis (the constant is a sum of all test functions, and its derivative
// vanishes) says so, and the flux columns to one weight per face node for all three
// faces and both directions, so that what leaves an element is what its neighbour
// receives.
#include "tables64.h"

#include <algorithm>
#include <cmath>

#include "fix64.cuh"

namespace dgx {
namespace {

using Mat = std::vector<long double>;

// C = op(A) B, n x n, op the transpose where `t`
Mat product(int n, const Mat& A, const Mat& B, bool t) {
  Mat C(size_t(n) * n, 0.0L);
  for (int i = 0; i < n; ++i)
    for (int k = 0; k < n; ++k) {
      const long double a = t ? A[size_t(k) * n + i] : A[size_t(i) * n + k];
      for (int j = 0; j < n; ++j) C[size_t(i) * n + j] += a * B[size_t(k) * n + j];
    }
  return C;
}

// A derivative matrix whose rows sum to zero: what a row leaves is taken from all its entries.
Mat derivative(int n, const std::vector<double>& D) {
  Mat out(D.begin(), D.end());
  for (int i = 0; i < n; ++i) {
    long double s = 0.0L;
    for (int j = 0; j < n; ++j) s += out[size_t(i) * n + j];
    for (int j = 0; j < n; ++j) out[size_t(i) * n + j] -= s / n;
  }
  return out;
}

int floor_log2(long double x) {
  int e = 0;
  std::frexp(x, &e);
  return e - 1;
}

// The operator's blocks in extended precision.
struct Blocks {
  Mat S[3], F[3], M, Mf;  // volume (rr, rs + sr, ss), face (Dr^T Mf, Ds^T Mf, E Mf) [Np][3 Nfp], mass, face mass
};

Blocks blocks(const RefElem& R) {
  const int N = R.N, Np = R.Np, Nfp = R.Nfp, nface = 3 * Nfp;
  const Mat Dr = derivative(Np, R.Dr), Ds = derivative(Np, R.Ds), M(R.M.begin(), R.M.end());
  const Mat MDr = product(Np, M, Dr, false), MDs = product(Np, M, Ds, false);
  Blocks b{{product(Np, Dr, MDr, true), product(Np, Dr, MDs, true), product(Np, Ds, MDs, true)}, {}, M, {}};
  for (int i = 0; i < Np; ++i)  // S_rs + S_sr
    for (int n = i; n < Np; ++n)
      b.S[1][size_t(i) * Np + n] = b.S[1][size_t(n) * Np + i] = b.S[1][size_t(i) * Np + n] + b.S[1][size_t(n) * Np + i];
  b.Mf.resize(size_t(Nfp) * Nfp);  // the same from both ends of a face
  for (int j = 0; j < Nfp; ++j)
    for (int l = 0; l < Nfp; ++l)
      b.Mf[size_t(j) * Nfp + l] = 0.5L * ((long double)R.Mf[size_t(j) * Nfp + l] + R.Mf[size_t(N - j) * Nfp + N - l]);
  for (Mat& f : b.F) f.assign(size_t(Np) * nface, 0.0L);
  for (int i = 0; i < Np; ++i)
    for (int f = 0; f < 3; ++f)
      for (int l = 0; l < Nfp; ++l)
        for (int j = 0; j < Nfp; ++j) {
          const int k = face_node(N, f, j);
          const size_t at = size_t(i) * nface + f * Nfp + l;
          b.F[0][at] += Dr[size_t(k) * Np + i] * b.Mf[size_t(j) * Nfp + l];
          b.F[1][at] += Ds[size_t(k) * Np + i] * b.Mf[size_t(j) * Nfp + l];
          if (k == i) b.F[2][at] += b.Mf[size_t(j) * Nfp + l];
        }
  return b;
}

OutTable table(const RefElem& R, const Blocks& b, bool helm) {
  const int N = R.N, Np = R.Np, Nfp = R.Nfp, nface = 3 * Nfp;
  auto largest = [](std::initializer_list<const Mat*> ms) {
    long double m = 0.0L;
    for (const Mat* a : ms)
      for (long double v : *a) m = std::max(m, std::fabs(v));
    return m;
  };
  OutTable t;
  // powers of two that bring every block's largest entry to the volume block's
  const long double ms = largest({&b.S[0], &b.S[1], &b.S[2]});
  t.k1 = floor_log2(ms / largest({&b.F[2]}));
  t.k2 = floor_log2(ms / largest({&b.F[0], &b.F[1]}));
  t.km = floor_log2(ms / largest({&b.M}));
  t.gvol = (Np + 7) / 8;
  t.gface = t.gvol + (nface + 7) / 8;
  t.chunks = (t.gface + (helm ? (Np + 23) / 24 : 0) + 1) / 2;
  t.cols = 48 * t.chunks;
  // what column k holds: group g, item i of the group, kind c
  struct Col {
    int c, g, i;
  };
  auto col = [](int k) { return Col{(k / 16) % 3, k / 48 * 2 + k % 16 / 8, k % 8}; };
  auto entry = [&](int r, int k) -> long double {
    const Col q = col(k);
    if (q.g < t.gvol) return 8 * q.g + q.i < Np ? b.S[q.c][size_t(r) * Np + 8 * q.g + q.i] : 0.0L;
    if (q.g < t.gface) {
      const int l = 8 * (q.g - t.gvol) + q.i;
      return l < nface ? std::ldexp(b.F[q.c][size_t(r) * nface + l], q.c == 2 ? t.k1 : t.k2) : 0.0L;
    }
    const int n = 24 * (q.g - t.gface) + 3 * q.i + q.c;
    return helm && n < Np ? std::ldexp(b.M[size_t(r) * Np + n], t.km) : 0.0L;
  };
  t.ea.resize(Np);
  for (int r = 0; r < Np; ++r) {
    long double m = 0.0L, s = 0.0L;
    for (int k = 0; k < t.cols; ++k) {
      m = std::max(m, std::fabs(entry(r, k)));
      s += std::fabs(entry(r, k));
    }
    t.ea[r] = fx::row_exp(double(m), double(s));
  }
  // a unit that the flux columns' sums are multiples of on all three faces
  int eT = -(1 << 30);
  for (int f = 0; f < 3; ++f) {
    int lo = 1 << 30;
    for (int j = 0; j < Nfp; ++j) lo = std::min(lo, t.ea[face_node(N, f, j)]);
    eT = std::max(eT, lo);
  }
  std::vector<int> order(Np);  // coarsest rows first
  for (int r = 0; r < Np; ++r) order[r] = r;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return t.ea[a] > t.ea[b]; });
  t.x.assign(size_t(Np) * t.cols, 0);
  for (int k = 0; k < t.cols; ++k) {
    const Col q = col(k);
    const bool closed = q.g < t.gface;  // the column's sum is given
    long double target = 0.0L, carry = 0.0L;
    if (closed && q.g >= t.gvol && q.c == 2) {
      const int l = (8 * (q.g - t.gvol) + q.i) % Nfp;
      if (8 * (q.g - t.gvol) + q.i < nface) {
        long double w = 0.0L;  // the lower half's order of summation for both halves
        for (int j = 0; j < Nfp; ++j) w += b.Mf[size_t(j) * Nfp + std::min(l, N - l)];
        target = std::ldexp((long double)std::llround(std::ldexp(w, t.k1 + 56 - eT)), eT - 56);
      }
    }
    if (closed) {
      carry = target;
      for (int r = 0; r < Np; ++r) carry -= entry(r, k);
    }
    // each row passes on what its rounding left, so no entry is off by more than its own
    // unit, and the finest row closes the sum
    int last = -1;
    for (int r : order) {
      const long double v = entry(r, k);
      if (v == 0.0L) continue;
      const long double w = v + (closed ? carry : 0.0L);
      const long long x = std::llround(std::ldexp(w, 56 - t.ea[r]));
      carry = w - std::ldexp((long double)x, t.ea[r] - 56);
      t.x[size_t(r) * t.cols + k] = x;
      last = r;
    }
    if (!closed || last < 0) continue;
    const int unit = t.ea[last];
    __int128 sum = 0;
    for (int r = 0; r < Np; ++r) {
      const long long x = t.x[size_t(r) * t.cols + k];
      if (x != 0) sum += __int128(x) << (t.ea[r] - unit);
    }
    sum -= __int128((long long)std::ldexp(target, 56 - unit));
    t.x[size_t(last) * t.cols + k] -= (long long)sum;
  }
  return t;
}

}  // namespace

void build_out_tables(const RefElem& R, OutTable (&t)[2]) {
  const Blocks b = blocks(R);
  for (int helm = 0; helm < 2; ++helm) t[helm] = table(R, b, helm != 0);
}

}  // namespace dgx
