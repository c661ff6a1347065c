// Host dense Hermitian eigensolver for the projected Lanczos matrix (m <= a few hundred).
//
// Householder reduction to tridiagonal form (Golub & Van Loan, Matrix Computations, 4th ed.,
// Alg. 8.3.1, complex Hermitian variant), a diagonal phase change that makes the
// off-diagonal real, then implicit symmetric QR steps with Wilkinson shifts and deflation
// (GvL Alg. 8.3.2 / 8.3.3), accumulating the Givens rotations.  FP64 throughout.
#include <algorithm>
#include <cmath>
#include <complex>
#include <numeric>
#include <vector>

#include "dense_eig.h"

using cd = std::complex<double>;

// Real and imaginary parts in arrays of their own, columns contiguous and every inner loop along a
// column, so that the compiler vectorises them (products of std::complex go through a library call
// that checks for NaN, one at a time).  C = false: the imaginary parts are all zero and never touched.
// n = 97 on a Grace core: 2.57 ms before, 1.11 ms (real) and 1.74 ms (complex) now; the device waits for
// this at every restart.
namespace {

template <bool C>
struct Cols {
  int n;
  std::vector<double> re, im;
  explicit Cols(int n_) : n(n_), re((size_t)n_ * n_, 0.0), im(C ? (size_t)n_ * n_ : 0, 0.0) {}
  double* r(int j) { return re.data() + (size_t)j * n; }
  double* i(int j) { return im.data() + (size_t)j * n; }
};

// y[lo..n) += x[lo..n) * (ar + i ai)
template <bool C>
inline void axpy(int lo, int n, const double* __restrict__ xr, const double* __restrict__ xi, double ar, double ai,
                 double* __restrict__ yr, double* __restrict__ yi) {
  if (C) {
    for (int t = lo; t < n; ++t) {
      yr[t] += xr[t] * ar - xi[t] * ai;
      yi[t] += xr[t] * ai + xi[t] * ar;
    }
  } else {
    for (int t = lo; t < n; ++t) yr[t] += xr[t] * ar;
  }
}

// The Givens rotations (c_k, s_k), k = lo .. hi-1, of one QR sweep applied to columns k, k+1 of Z (ld a
// multiple of kRows): kRows rows at a time, the column between two rotations kept in registers.
constexpr int kRows = 16;
inline void rotate_sweep(int ld, int lo, int hi, const double* __restrict__ c, const double* __restrict__ s, double* __restrict__ Z) {
  for (int r = 0; r < ld; r += kRows) {
    double u[kRows];
    double* z = Z + r;
    for (int t = 0; t < kRows; ++t) u[t] = z[(size_t)lo * ld + t];
    for (int k = lo; k < hi; ++k) {
      const double ck = c[k], sk = s[k];
      double* a = z + (size_t)k * ld;
      const double* b = a + ld;
      double w[kRows];
      for (int t = 0; t < kRows; ++t) w[t] = b[t];
      for (int t = 0; t < kRows; ++t) a[t] = ck * u[t] + sk * w[t];
      for (int t = 0; t < kRows; ++t) u[t] = ck * w[t] - sk * u[t];
    }
    for (int t = 0; t < kRows; ++t) z[(size_t)hi * ld + t] = u[t];
  }
}

template <bool C>
int eig(int n, const cd* A_in, double* w, cd* Z) {
  Cols<C> A(n), Q(n);                                  // Q accumulates the reflectors: A = Q T Q^H
  for (int j = 0; j < n; ++j)
    for (int i = 0; i < n; ++i) {
      A.r(j)[i] = A_in[i + (size_t)j * n].real();
      if (C) A.i(j)[i] = A_in[i + (size_t)j * n].imag();
      if (i == j) Q.r(j)[i] = 1.0;
    }
  std::vector<double> vr(n), vi(n), pr(n), pi(n), qr(n), qi(n);
  for (int k = 0; k + 2 < n; ++k) {
    const double* cr = A.r(k);
    const double* ci = C ? A.i(k) : nullptr;
    double xnorm = 0;
    for (int i = k + 1; i < n; ++i) xnorm += cr[i] * cr[i] + (C ? ci[i] * ci[i] : 0.0);
    xnorm = std::sqrt(xnorm);
    if (xnorm == 0.0) continue;
    const double x0r = cr[k + 1], x0i = C ? ci[k + 1] : 0.0, x0 = std::hypot(x0r, x0i);
    const double phr = x0 > 0 ? x0r / x0 : 1.0, phi = x0 > 0 ? x0i / x0 : 0.0;
    std::fill(vr.begin(), vr.end(), 0.0);
    std::fill(vi.begin(), vi.end(), 0.0);
    for (int i = k + 1; i < n; ++i) {
      vr[i] = cr[i];
      if (C) vi[i] = ci[i];
    }
    vr[k + 1] += phr * xnorm;                          // v = x + ph |x| e_1
    vi[k + 1] += phi * xnorm;
    double vn = 0;
    for (int i = k + 1; i < n; ++i) vn += vr[i] * vr[i] + vi[i] * vi[i];
    if (vn == 0.0) continue;
    // H = I - 2 v v^H / (v^H v);  A <- H A H:  p = tau A v, q = p - (tau/2)(v^H p) v
    const double tau = 2.0 / vn;
    std::fill(pr.begin(), pr.end(), 0.0);
    std::fill(pi.begin(), pi.end(), 0.0);
    for (int j = k + 1; j < n; ++j)
      axpy<C>(k, n, A.r(j), C ? A.i(j) : nullptr, tau * vr[j], tau * vi[j], pr.data(), pi.data());
    double Kr = 0, Ki = 0;
    for (int i = k + 1; i < n; ++i) {
      Kr += vr[i] * pr[i] + vi[i] * pi[i];
      Ki += vr[i] * pi[i] - vi[i] * pr[i];
    }
    Kr *= 0.5 * tau;
    Ki *= 0.5 * tau;
    qr = pr;
    qi = pi;
    axpy<C>(k, n, vr.data(), vi.data(), -Kr, -Ki, qr.data(), qi.data());
    // A <- A - v q^H - q v^H   (v zero at index k)
    for (int j = k; j < n; ++j) {
      axpy<C>(k, n, vr.data(), vi.data(), -qr[j], qi[j], A.r(j), C ? A.i(j) : nullptr);
      axpy<C>(k, n, qr.data(), qi.data(), -vr[j], vi[j], A.r(j), C ? A.i(j) : nullptr);
    }
    // Q <- Q H
    std::fill(pr.begin(), pr.end(), 0.0);
    std::fill(pi.begin(), pi.end(), 0.0);
    for (int j = k + 1; j < n; ++j)
      axpy<C>(0, n, Q.r(j), C ? Q.i(j) : nullptr, tau * vr[j], tau * vi[j], pr.data(), pi.data());
    for (int j = k + 1; j < n; ++j) axpy<C>(0, n, pr.data(), pi.data(), -vr[j], vi[j], Q.r(j), C ? Q.i(j) : nullptr);
  }
  // phases so that the sub-diagonal is real and non-negative: T' = D^H T D
  std::vector<double> d(n), e(n, 0.0);
  double Dr = 1.0, Di = 0.0;
  for (int i = 0; i < n; ++i) d[i] = A.r(i)[i];
  for (int j = 0; j < n; ++j) {
    if (j > 0) {
      const double tr = A.r(j - 1)[j], ti = C ? A.i(j - 1)[j] : 0.0, r = std::hypot(tr, ti);
      e[j - 1] = r;
      if (r > 0) {
        const double ur = tr / r, ui = ti / r, nr = Dr * ur - Di * ui;
        Di = Dr * ui + Di * ur;
        Dr = nr;
      }
    }
    double* xr = Q.r(j);
    if (C) {
      double* xi = Q.i(j);
      for (int i = 0; i < n; ++i) {
        const double a = xr[i], b = xi[i];
        xr[i] = a * Dr - b * Di;
        xi[i] = a * Di + b * Dr;
      }
    } else {
      for (int i = 0; i < n; ++i) xr[i] *= Dr;
    }
  }
  // implicit symmetric QR steps with a Wilkinson shift (bulge chasing by Givens rotations),
  // deflating converged off-diagonal entries from the bottom; Zr accumulates the rotations.
  const int ld = (n + kRows - 1) / kRows * kRows;
  std::vector<double> Zr((size_t)ld * n, 0.0), rc(n), rs(n);
  for (int i = 0; i < n; ++i) Zr[i + (size_t)i * ld] = 1.0;
  const double eps = 2.220446049250313e-16;
  int hi = n - 1, sweeps = 0;
  while (hi > 0) {
    if (std::fabs(e[hi - 1]) <= eps * (std::fabs(d[hi - 1]) + std::fabs(d[hi])) || e[hi - 1] == 0.0) {
      e[hi - 1] = 0.0;
      --hi;
      continue;
    }
    int lo = hi - 1;
    while (lo > 0 && std::fabs(e[lo - 1]) > eps * (std::fabs(d[lo - 1]) + std::fabs(d[lo]))) --lo;
    if (lo > 0) e[lo - 1] = 0.0;
    if (++sweeps > 60 * n) return 1;
    // Wilkinson shift from the trailing 2x2 block of the unreduced segment [lo, hi]
    const double half = 0.5 * (d[hi - 1] - d[hi]);
    const double bb = e[hi - 1];
    const double den = half + (half >= 0 ? 1.0 : -1.0) * std::hypot(half, bb);
    const double mu = (den != 0.0) ? d[hi] - bb * bb / den : d[hi] - std::fabs(bb);
    double x = d[lo] - mu, z = e[lo];
    for (int k = lo; k < hi; ++k) {
      const double r = std::hypot(x, z);
      const double c = (r == 0.0) ? 1.0 : x / r, s = (r == 0.0) ? 0.0 : z / r;
      if (k > lo) e[k - 1] = r;
      const double p = d[k], q = e[k], t = d[k + 1];
      d[k] = c * c * p + 2.0 * c * s * q + s * s * t;
      d[k + 1] = s * s * p - 2.0 * c * s * q + c * c * t;
      e[k] = c * s * (t - p) + (c * c - s * s) * q;
      if (k + 1 < hi) {
        z = s * e[k + 1];        // bulge at (k, k+2)
        e[k + 1] *= c;
        x = e[k];
      }
      rc[k] = c;
      rs[k] = s;
    }
    rotate_sweep(ld, lo, hi, rc.data(), rs.data(), Zr.data());
  }
  std::vector<int> order(n);
  std::iota(order.begin(), order.end(), 0);
  std::sort(order.begin(), order.end(), [&](int x, int y) { return d[x] < d[y]; });
  for (int jj = 0; jj < n; ++jj) {
    const int j = order[jj];
    w[jj] = d[j];
    std::fill(pr.begin(), pr.end(), 0.0);
    std::fill(pi.begin(), pi.end(), 0.0);
    for (int k = 0; k < n; ++k) {
      const double z = Zr[k + (size_t)j * ld];
      axpy<false>(0, n, Q.r(k), nullptr, z, 0.0, pr.data(), nullptr);
      if (C) axpy<false>(0, n, Q.i(k), nullptr, z, 0.0, pi.data(), nullptr);
    }
    for (int i = 0; i < n; ++i) Z[i + (size_t)jj * n] = cd(pr[i], pi[i]);
  }
  return 0;
}

}  // namespace

// A: n x n Hermitian, column-major (A[i + j*n] = A_ij); only the full matrix is read.
// On return w[0..n) ascending and Z (column-major, columns = eigenvectors).
int hermitian_eig(int n, const cd* A_in, double* w, cd* Z) {
  if (n <= 0) return 0;
  bool complex = false;
  for (size_t t = 0; t < (size_t)n * n; ++t) complex |= A_in[t].imag() != 0.0;
  return complex ? eig<true>(n, A_in, w, Z) : eig<false>(n, A_in, w, Z);
}

// Cholesky G = R^H R (R upper), column-major b x b.  Returns nonzero if not positive definite.
int cholesky_upper(int b, const cd* G, cd* R) {
  for (int i = 0; i < b * b; ++i) R[i] = 0;
  for (int j = 0; j < b; ++j) {
    cd s = G[j + (size_t)j * b];
    for (int k = 0; k < j; ++k) s -= std::conj(R[k + (size_t)j * b]) * R[k + (size_t)j * b];
    const double djj = std::real(s);
    if (!(djj > 0.0) || !std::isfinite(djj)) return 1;
    const double rjj = std::sqrt(djj);
    R[j + (size_t)j * b] = rjj;
    for (int i = j + 1; i < b; ++i) {
      cd t = G[j + (size_t)i * b];
      for (int k = 0; k < j; ++k) t -= std::conj(R[k + (size_t)j * b]) * R[k + (size_t)i * b];
      R[j + (size_t)i * b] = t / rjj;
    }
  }
  return 0;
}

// Inverse of an upper-triangular b x b matrix (column-major).
void upper_inverse(int b, const cd* R, cd* Ri) {
  for (int i = 0; i < b * b; ++i) Ri[i] = 0;
  for (int j = 0; j < b; ++j) {
    Ri[j + (size_t)j * b] = 1.0 / R[j + (size_t)j * b];
    for (int i = j - 1; i >= 0; --i) {
      cd s = 0;
      for (int k = i + 1; k <= j; ++k) s += R[i + (size_t)k * b] * Ri[k + (size_t)j * b];
      Ri[i + (size_t)j * b] = -s / R[i + (size_t)i * b];
    }
  }
}
