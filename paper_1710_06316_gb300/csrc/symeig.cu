// symeig.cu -- dense symmetric eigensolver (host code only; see symeig.h).
//
// Two textbook stages (Golub & Van Loan, Matrix Computations, Sec. 8.3):
//  1. Householder reflections H_k = I - beta v v^T reduce A to a tridiagonal T = Q^T A Q;
//  2. implicit symmetric QR steps with the Wilkinson shift chase a bulge down each
//     unreduced block of T with Givens rotations until every off-diagonal entry is
//     negligible.
// Q is kept transposed (zt = Q^T, row k = column k of Q) so that both the reflections
// and the rotations touch contiguous rows.  They act on each column of zt by itself: the
// two stages work on A and T and only record them, and they are then applied to slices of
// columns on a few threads, in the same order for every column (216 x 216: 5.9 ms with
// each applied as it arose, 2.9 ms so, on a Grace host; the rest is the chain of QR steps).
#include <algorithm>
#include <cmath>
#include <numeric>
#include <thread>
#include <vector>

#include "host_threads.h"
#include "symeig.h"

namespace afmpb {

namespace {

// What the stages do to Q: the reflections (v_k over rows k + 1 .., beta_k; 0 for none) and
// the rotations of rows (k, k + 1).
struct Rotation {
  int k;
  double c, s;
};
struct Record {
  std::vector<double> v, beta;
  std::vector<Rotation> rot;
};

constexpr int kRows = 8;

// Stage 1.  a: n x n row-major symmetric (overwritten).  d, e: diagonal and super-diagonal
// of T (e[n-1] unused).
void householder_tridiag(int n, double *a, Record &rec, double *d, double *e) {
  rec.v.assign((size_t)n * n, 0.0);
  rec.beta.assign(n, 0.0);
  std::vector<double> p(n);
  for (int k = 0; k + 2 < n; ++k) {
    const int m = n - k - 1;                       // length of x = A[k+1.., k]
    double *v = rec.v.data() + (size_t)k * n;
    double xnorm2 = 0.0;
    for (int j = 0; j < m; ++j) {
      const double x = a[(size_t)(k + 1 + j) * n + k];
      v[j] = x;
      xnorm2 += x * x;
    }
    if (xnorm2 == 0.0) continue;                   // column already reduced
    const double alpha = -std::copysign(std::sqrt(xnorm2), v[0]);   // H x = alpha e_1
    v[0] -= alpha;                                 // no cancellation: opposite signs
    double vnorm2 = 0.0;
    for (int j = 0; j < m; ++j) vnorm2 += v[j] * v[j];
    const double beta = 2.0 / vnorm2;
    rec.beta[k] = beta;
    // trailing block B = A[k+1.., k+1..] <- H B H = B - v w^T - w v^T with
    // p = beta B v, w = p - (beta/2)(v.p) v; the sums of kRows rows at a time, each in order
    // (one at a time waits for each addition of its chain)
    double vp = 0.0;
    for (int i = 0; i < m; i += kRows) {
      const int r = std::min(kRows, m - i);
      const double *row[kRows];
      double s[kRows] = {};
      for (int q = 0; q < kRows; ++q) row[q] = a + (size_t)(k + 1 + i + std::min(q, r - 1)) * n + (k + 1);
      for (int j = 0; j < m; ++j)
        for (int q = 0; q < kRows; ++q) s[q] += row[q][j] * v[j];
      for (int q = 0; q < r; ++q) {
        p[i + q] = beta * s[q];
        vp += v[i + q] * p[i + q];
      }
    }
    const double kk = 0.5 * beta * vp;
    for (int i = 0; i < m; ++i) p[i] -= kk * v[i];   // p is now w
    for (int i = 0; i < m; ++i) {
      double *row = a + (size_t)(k + 1 + i) * n + (k + 1);
      for (int j = 0; j < m; ++j) row[j] -= v[i] * p[j] + p[i] * v[j];
    }
    a[(size_t)(k + 1) * n + k] = a[(size_t)k * n + k + 1] = alpha;
    for (int j = 1; j < m; ++j) a[(size_t)(k + 1 + j) * n + k] = a[(size_t)k * n + k + 1 + j] = 0.0;
  }
  for (int i = 0; i < n; ++i) {
    d[i] = a[(size_t)i * n + i];
    e[i] = i + 1 < n ? a[(size_t)i * n + i + 1] : 0.0;
  }
}

// One implicit QR step with Wilkinson shift on the unreduced block [lo, hi] of T.
void qr_step(int lo, int hi, double *d, double *e, std::vector<Rotation> &rot) {
  const double t = 0.5 * (d[hi - 1] - d[hi]);
  const double eh = e[hi - 1];
  const double mu = d[hi] - eh * eh / (t + std::copysign(std::hypot(t, eh), t == 0.0 ? 1.0 : t));
  double x = d[lo] - mu, z = e[lo];
  for (int k = lo; k < hi; ++k) {
    // rotation G = [[c, s], [-s, c]] on (k, k+1) with s x + c z = 0
    const double r = std::hypot(x, z);
    double c = 1.0, s = 0.0;
    if (r != 0.0) { c = x / r; s = -z / r; }
    if (k > lo) e[k - 1] = r;                       // bulge at (k-1, k+1) absorbed
    const double a0 = d[k], b0 = d[k + 1], f = e[k];
    d[k] = c * c * a0 - 2.0 * c * s * f + s * s * b0;
    d[k + 1] = s * s * a0 + 2.0 * c * s * f + c * c * b0;
    e[k] = c * s * (a0 - b0) + (c * c - s * s) * f;
    if (k + 1 < hi) {                               // new bulge at (k, k+2)
      const double g = e[k + 1];
      z = -s * g;
      e[k + 1] = c * g;
      x = e[k];
    }
    rot.push_back({k, c, s});
  }
}

// Columns [c0, c1) of zt = Q^T, by the recorded reflections and rotations; work: (n + 1) x
// (c1 - c0).
void apply_columns(int n, int c0, int c1, const Record &rec, double *work, double *zt) {
  const int w = c1 - c0;
  double *z = work, *u = work + (size_t)n * w;
  std::fill(z, u, 0.0);
  for (int c = c0; c < c1; ++c) z[(size_t)c * w + (c - c0)] = 1.0;
  for (int k = 0; k + 2 < n; ++k) {
    if (rec.beta[k] == 0.0) continue;
    // Q <- Q H: rows k+1.. of zt: zt_r -= beta v_r (sum_j v_j zt_j)
    const int m = n - k - 1;
    const double *v = rec.v.data() + (size_t)k * n;
    std::fill(u, u + w, 0.0);
    for (int j = 0; j < m; ++j) {
      const double *row = z + (size_t)(k + 1 + j) * w;
      for (int c = 0; c < w; ++c) u[c] += v[j] * row[c];
    }
    for (int j = 0; j < m; ++j) {
      double *row = z + (size_t)(k + 1 + j) * w;
      const double f = rec.beta[k] * v[j];
      for (int c = 0; c < w; ++c) row[c] -= f * u[c];
    }
  }
  for (const Rotation &g : rec.rot) {
    double *qa = z + (size_t)g.k * w, *qb = z + (size_t)(g.k + 1) * w;
    for (int i = 0; i < w; ++i) {
      const double ua = qa[i], ub = qb[i];
      qa[i] = g.c * ua - g.s * ub;
      qb[i] = g.s * ua + g.c * ub;
    }
  }
  for (int r = 0; r < n; ++r) std::copy(z + (size_t)r * w, z + (size_t)(r + 1) * w, zt + (size_t)r * n + c0);
}

// zt on up to four threads (the caller's among them; a thread that is not granted or cannot be
// had leaves its columns to it).
void apply_all(int n, const Record &rec, double *zt) {
  const int parts = n >= 128 ? 4 : 1;
  std::vector<double> work((size_t)(n + 1) * n);
  const auto part = [&](int t) {
    const int c0 = n * t / parts, c1 = n * (t + 1) / parts;
    apply_columns(n, c0, c1, rec, work.data() + (size_t)(n + 1) * c0, zt);
  };
  const HostThreads extra(parts - 1);
  std::vector<std::thread> pool;
  pool.reserve(parts);
  int started = 1;
  try {
    for (; started <= extra.count(); ++started) pool.emplace_back(part, started);
  } catch (...) {
  }
  part(0);
  for (int t = started; t < parts; ++t) part(t);
  for (auto &t : pool) t.join();
}

}  // namespace

int sym_eig_desc(int n, double *A, double *w, double *zt) {
  if (n <= 0) return 0;
  std::vector<double> d(n), e(n);
  Record rec;
  householder_tridiag(n, A, rec, d.data(), e.data());
  const double eps = 0x1p-52;
  int hi = n - 1;
  long iter = 0;
  const long max_iter = 30L * n;
  while (hi > 0) {
    // deflate negligible off-diagonal entries
    for (int i = 0; i < hi; ++i)
      if (std::fabs(e[i]) <= eps * (std::fabs(d[i]) + std::fabs(d[i + 1]))) e[i] = 0.0;
    while (hi > 0 && e[hi - 1] == 0.0) --hi;       // trailing eigenvalues converged
    if (hi == 0) break;
    int lo = hi - 1;
    while (lo > 0 && e[lo - 1] != 0.0) --lo;       // start of the unreduced block
    if (++iter > max_iter) return -1;
    qr_step(lo, hi, d.data(), e.data(), rec.rot);
  }
  apply_all(n, rec, zt);
  // sort descending, permuting the eigenvector rows
  std::vector<int> idx(n);
  std::iota(idx.begin(), idx.end(), 0);
  std::stable_sort(idx.begin(), idx.end(), [&](int i, int j) { return d[i] > d[j]; });
  std::vector<double> tmp((size_t)n * n);
  for (int k = 0; k < n; ++k) {
    w[k] = d[idx[k]];
    std::copy(zt + (size_t)idx[k] * n, zt + (size_t)(idx[k] + 1) * n, tmp.begin() + (size_t)k * n);
  }
  std::copy(tmp.begin(), tmp.end(), zt);
  return 0;
}

}  // namespace afmpb
