// Direct solve of the finite-difference Poisson equation on its box (paper Section III-A item 3:
// a finite-difference Poisson solver): the 7-point operator with periodic x and y and constant
// coefficients is diagonal in x and y under the discrete Hartley transform
// H_k = sum_j f_j (cos + sin)(2 pi j k / n), whose basis a symmetric circulant shares with the
// Fourier one, so everything stays real; what is left is one symmetric tridiagonal Toeplitz
// system along z for every (kx, ky).  A correction d = A^-1 r costs four line transforms and one
// pass of tridiagonal solves: O(n log n), where conjugate gradients take some 4 n passes over a
// grid of n points a side.  A second correction of what rounding left is applied when the first
// does not meet the tolerance; the test runs on the device, so nothing waits between the two.
//
// The transforms take two real lines as one complex line, mixed-radix Stockham stages in shared
// memory: radix 4 and 2 in registers, six fused operations for every pair a +- w b; odd primes by their
// definition, the first of them on sums and differences of mirrored inputs.  They are bound by the
// FP64 rate (13 operations a point and transform at 256 points: 0.40 ms on 256^3, 86% of the rate).
// Planes small enough for shared memory are transformed in x and y at once, two planes as one complex
// plane, with the residual formed as they are read: three launches a correction.
//
// Measured against the conjugate gradients this takes the place of (poisson.cu, one cooperative
// launch, three grid barriers an iteration): 11x11x217 grid to 1e-13 5.07 -> 0.112 ms (two corrections,
// seven launches of 6 to 14 us), 256x256x257 to 1e-10 in the mixed form 251 -> 2.53 ms (one correction
// and its check); the error against 64-bit transforms 1.2e-15 -> 1.1e-15 and 4.6e-12 -> 6.2e-14 of the
// norm.
#include <algorithm>
#include <cmath>

#include "poisson_direct.h"
#include "smem.cuh"

namespace {

constexpr int kMaxLine = 2048;       // points of a transformed line
constexpr int kMaxZ = 1024;          // unknowns of a tridiagonal system
constexpr int kPlanePoints = 3072;   // points of a plane transformed at once
constexpr int kT = 256;

struct Fft {
  int n, nf;
  int rad[12];
};

// Odd primes from the largest down (the first stage, without twiddles, then takes the dearest), then
// 4 and 2.
Fft plan_of(int n) {
  Fft p{};
  p.n = n;
  int odd[12], no = 0, m = n;
  for (int r = 3; r <= m; r += 2)
    while (m % r == 0) odd[no++] = r, m /= r;
  while (no) p.rad[p.nf++] = odd[--no];
  while (m % 4 == 0) p.rad[p.nf++] = 4, m /= 4;
  if (m == 2) p.rad[p.nf++] = 2;
  return p;
}

struct State {
  double bb, rr, stop;
  int active;          // the residual is above the stopping value
  int iterations;
  int nonzero;         // the start has a component that is not zero
  unsigned arrived;    // blocks of the running residual pass that have left their sums
};

// a + w b and a - w b in six fused operations (the difference as 2 a less the sum)
__device__ __forceinline__ void turn(double2 a, double2 w, double2 b, double2& sum, double2& dif) {
  sum.x = fma(w.x, b.x, fma(-w.y, b.y, a.x));
  sum.y = fma(w.x, b.y, fma(w.y, b.x, a.y));
  dif.x = fma(2.0, a.x, -sum.x);
  dif.y = fma(2.0, a.y, -sum.y);
}

// FFT of `count` lines of p.n points in shared memory; element e of line l at l*ls + e*es.  Ping-pong
// between a and b; returns the buffer that holds the result (all threads past a barrier).
// tw[k] = exp(-2 pi i k / n).
__device__ double2* fft_lines(double2* a, double2* b, const double2* __restrict__ tw, const Fft& p, int count, int es, int ls) {
  const int n = p.n;
  int Ns = 1;
  for (int f = 0; f < p.nf; ++f) {
    const int R = p.rad[f], q = n / R, step = q / Ns;
    const int per = R == 4 || R == 2 ? q : n;        // work items of a line
    const int items = count * per;
    const bool pairs = f == 0 && R >= 5;
    if (pairs) {
      // inputs t and R - t of a long odd stage as their sum and difference: half the products
      const int h = R / 2;
      for (int it = threadIdx.x; it < count * q * h; it += kT) {
        const int line = it / (q * h), rem = it - line * q * h, t = rem / q + 1, j = rem - (t - 1) * q;
        double2* x = a + line * ls + (j + t * q) * es;
        double2* y = a + line * ls + (j + (R - t) * q) * es;
        const double2 u = *x, w = *y;
        *x = make_double2(u.x + w.x, u.y + w.y);
        *y = make_double2(u.x - w.x, u.y - w.y);
      }
      __syncthreads();
    }
    for (int it = threadIdx.x; it < items; it += kT) {
      int line, w;
      if (es == 1) {
        line = it / per;
        w = it - line * per;
      } else {
        w = it / count;
        line = it - w * count;
      }
      const double2* src = a + line * ls;
      double2* dst = b + line * ls;
      if (R == 4) {
        // two layers of a +- w b, the twiddles 1, w, w^2, w^3 as w^2 inside both pairs and w between them
        const int jm = w % Ns, o = (w - jm) * 4 + jm;
        const double2 v0 = src[w * es], v1 = src[(w + q) * es], v2 = src[(w + 2 * q) * es], v3 = src[(w + 3 * q) * es];
        double2 s02, d02, s13, d13, y0, y1, y2, y3;
        if (Ns > 1) {   // the same for all lanes: a branch on jm would run both sides
          const double2 w1 = tw[jm * step], w2 = tw[2 * jm * step];
          turn(v0, w2, v2, s02, d02);
          turn(v1, w2, v3, s13, d13);
          turn(s02, w1, s13, y0, y2);
          turn(d02, make_double2(w1.y, -w1.x), d13, y1, y3);                  // -i w
        } else {
          s02 = make_double2(v0.x + v2.x, v0.y + v2.y), d02 = make_double2(v0.x - v2.x, v0.y - v2.y);
          s13 = make_double2(v1.x + v3.x, v1.y + v3.y), d13 = make_double2(v1.x - v3.x, v1.y - v3.y);
          y0 = make_double2(s02.x + s13.x, s02.y + s13.y), y2 = make_double2(s02.x - s13.x, s02.y - s13.y);
          y1 = make_double2(d02.x + d13.y, d02.y - d13.x), y3 = make_double2(d02.x - d13.y, d02.y + d13.x);
        }
        dst[o * es] = y0;
        dst[(o + Ns) * es] = y1;
        dst[(o + 2 * Ns) * es] = y2;
        dst[(o + 3 * Ns) * es] = y3;
      } else if (R == 2) {
        const int jm = w % Ns, o = (w - jm) * 2 + jm;
        const double2 v0 = src[w * es], v1 = src[(w + q) * es];
        double2 y0, y1;
        if (Ns > 1) turn(v0, tw[jm * step], v1, y0, y1);
        else y0 = make_double2(v0.x + v1.x, v0.y + v1.y), y1 = make_double2(v0.x - v1.x, v0.y - v1.y);
        dst[o * es] = y0;
        dst[(o + Ns) * es] = y1;
      } else if (pairs) {
        // first stage, inputs already as sums and differences of t and R - t
        const int i = w / q, j = w - i * q, e = i * q;
        double2 r = src[j * es];
        for (int t = 1, x = e; t <= R / 2; ++t) {
          const double2 a = src[(j + t * q) * es], d = src[(j + (R - t) * q) * es], c = tw[x];
          r.x = fma(-d.y, c.y, fma(a.x, c.x, r.x));
          r.y = fma(d.x, c.y, fma(a.y, c.x, r.y));
          x += e;
          if (x >= n) x -= n;
        }
        dst[(j * R + i) * es] = r;
      } else {
        // one output: sum_t src[j + t q] exp(-2 pi i t e / n)
        const int i = w / q, j = w - i * q, jm = j % Ns;
        int e = jm * step + i * q, x = e;
        double2 s = src[j * es];
        for (int t = 1; t < R; ++t) {
          const double2 v = src[(j + t * q) * es], c = tw[x];
          s.x = fma(v.x, c.x, fma(-v.y, c.y, s.x));
          s.y = fma(v.x, c.y, fma(v.y, c.x, s.y));
          x += e;
          if (x >= n) x -= n;
        }
        dst[((j - jm) * R + jm + i * Ns) * es] = s;
      }
    }
    __syncthreads();
    double2* t = a;
    a = b;
    b = t;
    Ns *= R;
  }
  return a;
}

// Twice the Hartley transforms, at k and -k, of the two real lines (planes) whose complex FFT holds z
// at k and zm at -k.
__device__ __forceinline__ void hartley2(double2 z, double2 zm, double2& at, double2& mirror) {
  const double s = z.x + zm.x, d = z.y - zm.y, t = z.y + zm.y, e = z.x - zm.x;
  at = make_double2(s - d, t + e);
  mirror = make_double2(s + d, t - e);
}

// Leaves the block's sum with the others'; the last block to arrive adds all of them in block
// order and sets the state: the squared residual, and on the first pass ||b||^2 and the stopping
// value.  All threads of the block call it.
template <bool FIRST>
__device__ void finish_residual(double lrr, double lbb, double* part, State* st, double rtol, int max_iter, int blocks) {
  __shared__ double sh[32];
  __shared__ bool last;
  const double v = block_sum(lrr, sh);
  double w = 0.0;
  if constexpr (FIRST) w = block_sum(lbb, sh);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = v;
    if constexpr (FIRST) part[blocks + blockIdx.x] = w;
    __threadfence();
    last = atomicAdd(&st->arrived, 1u) == (unsigned)blocks - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double a = 0.0, c = 0.0;
  for (int b = threadIdx.x; b < blocks; b += blockDim.x) {
    a += __ldcg(part + b);
    if constexpr (FIRST) c += __ldcg(part + blocks + b);
  }
  a = block_sum(a, sh);
  if constexpr (FIRST) c = block_sum(c, sh);
  if (threadIdx.x == 0) {
    st->arrived = 0;
    st->rr = a;
    if constexpr (FIRST) {
      st->bb = c;
      st->stop = rtol * rtol * c;
      st->iterations = 0;
    }
    st->active = c == 0.0 && FIRST ? 0 : (a > st->stop && st->iterations < max_iter);
  }
}

// How a residual is formed: b - A x, b = scale * rho; or the residual kept so far less scale * A d
enum { kFromX = 0, kFromD = 1 };

template <int HOW>
__device__ __forceinline__ double residual_at(const PGrid& g, const double* __restrict__ rho, double scale,
                                              const double* __restrict__ v, const double* r, int i, int j, int k,
                                              long long idx, double& b) {
  if constexpr (HOW == kFromX) {
    b = scale * rho[idx];
    return b - stencil_at(v, g, i, j, k, idx);
  } else {
    b = 0.0;
    return fma(-scale, stencil_at(v, g, i, j, k, idx), r[idx]);
  }
}

// Whether the start has a component that is not zero.  From the zero field, the usual start, the
// first residual is the right-hand side: 2 FP64 operations a point instead of 16, on the pipe that
// bounds it (256^3: 461 us; 80 + 28 us with this pass over
// the start).
__global__ void __launch_bounds__(kT) nonzero_kernel(const double* __restrict__ x, long long n, State* st) {
  bool any = false;
  for (long long i = (long long)blockIdx.x * kT + threadIdx.x; i < n; i += (long long)gridDim.x * kT)
    any |= (__double_as_longlong(x[i]) << 1) != 0;
  if (any) st->nonzero = 1;
}

// r = residual on the whole grid and its square sum: rows over the warps of the grid, points of a
// row over the lanes, or narrow rows' points over all lanes.
template <int HOW, bool FIRST>
__global__ void __launch_bounds__(kT) residual_kernel(PGrid g, const double* __restrict__ rho, double scale,
                                                      const double* __restrict__ v, double* r, double* part,
                                                      State* st, double rtol, int max_iter) {
  if (!FIRST && !st->active) return;
  double lrr = 0.0, lbb = 0.0;
  if (FIRST && HOW == kFromX && !st->nonzero) {
    for (long long i = (long long)blockIdx.x * kT + threadIdx.x; i < g.n; i += (long long)gridDim.x * kT) {
      const double b = scale * rho[i];
      r[i] = b;
      lrr = fma(b, b, lrr);
    }
    finish_residual<FIRST>(lrr, lrr, part, st, rtol, max_iter, (int)gridDim.x);
    return;
  }
  auto point = [&](int i, int j, int k, long long idx) {
    double b;
    const double ri = residual_at<HOW>(g, rho, scale, v, r, i, j, k, idx, b);
    r[idx] = ri;
    lrr = fma(ri, ri, lrr);
    if constexpr (FIRST) lbb = fma(b, b, lbb);
  };
  if (g.nx >= 24) {
    const int lane = threadIdx.x & 31, nw = (gridDim.x * kT) >> 5;
    const int rows = g.ny * g.nzi;
    for (int rw = (blockIdx.x * kT + threadIdx.x) >> 5; rw < rows; rw += nw) {
      const int k = rw / g.ny, j = rw - k * g.ny;
      const long long base = (long long)rw * g.nx;
      for (int i = lane; i < g.nx; i += 32) point(i, j, k, base + i);
    }
  } else {   // narrow rows: points over the lanes (n < 2^31)
    for (long long idx = (long long)blockIdx.x * kT + threadIdx.x; idx < g.n; idx += (long long)gridDim.x * kT) {
      const unsigned t = (unsigned)idx, row = t / (unsigned)g.nx;
      point((int)(t - row * g.nx), (int)(row % (unsigned)g.ny), (int)(row / (unsigned)g.ny), idx);
    }
  }
  finish_residual<FIRST>(lrr, lbb, part, st, rtol, max_iter, (int)gridDim.x);
}

// Hartley transform of every row (x lines), P pairs of rows a block.  ADD: the result is the
// correction, also added to x.
template <bool ADD>
__global__ void __launch_bounds__(kT) rows_kernel(const double* src, double* dst, double* __restrict__ x,
                                                  double scale, int nrows, int P, const __grid_constant__ Fft p,
                                                  const double2* __restrict__ tw, const State* st) {
  if (!st->active) return;
  extern __shared__ __align__(16) double2 sm[];
  const int n = p.n;
  double2 *A = sm, *B = sm + P * n, *W = sm + 2 * P * n;
  for (int i = threadIdx.x; i < n; i += kT) W[i] = tw[i];
  const int r0 = blockIdx.x * 2 * P, have = min(P, (nrows - r0 + 1) / 2);
  for (int it = threadIdx.x; it < have * n; it += kT) {
    const int l = it / n, e = it - l * n, ra = r0 + 2 * l;
    const double* s = src + (long long)ra * n + e;
    A[it] = make_double2(s[0], ra + 1 < nrows ? s[n] : 0.0);
  }
  __syncthreads();
  const double2* Z = fft_lines(A, B, W, p, have, 1, n);
  const int half = n / 2 + 1;
  for (int it = threadIdx.x; it < have * half; it += kT) {
    const int l = it / half, e = it - l * half, em = e ? n - e : 0, ra = r0 + 2 * l;
    double2 h[2];
    hartley2(Z[l * n + e], Z[l * n + em], h[0], h[1]);
    const bool both = em != e;
    for (int m = 0; m <= (both ? 1 : 0); ++m) {
      const long long at = (long long)ra * n + (m ? em : e);
      dst[at] = h[m].x;
      if constexpr (ADD) x[at] = fma(scale, h[m].x, x[at]);
      if (ra + 1 < nrows) {
        dst[at + n] = h[m].y;
        if constexpr (ADD) x[at + n] = fma(scale, h[m].y, x[at + n]);
      }
    }
  }
}

// Hartley transform of every column (y lines) in place, P pairs of neighbouring columns of one
// plane a block.
__global__ void __launch_bounds__(kT) columns_kernel(double* __restrict__ v, int nx, int P, int tiles, const __grid_constant__ Fft p,
                                                     const double2* __restrict__ tw, const State* st) {
  if (!st->active) return;
  extern __shared__ __align__(16) double2 sm[];
  const int n = p.n;
  double2 *A = sm, *B = sm + P * n, *W = sm + 2 * P * n;
  for (int i = threadIdx.x; i < n; i += kT) W[i] = tw[i];
  const int plane = blockIdx.x / tiles, c0 = (blockIdx.x - plane * tiles) * 2 * P;
  double* base = v + (long long)plane * n * nx + c0;
  const int cols = nx - c0;
  for (int it = threadIdx.x; it < P * n; it += kT) {
    const int e = it / P, l = it - e * P;
    const double* s = base + (long long)e * nx + 2 * l;
    A[it] = make_double2(2 * l < cols ? s[0] : 0.0, 2 * l + 1 < cols ? s[1] : 0.0);
  }
  __syncthreads();
  const double2* Z = fft_lines(A, B, W, p, P, P, 1);
  for (int it = threadIdx.x; it < P * (n / 2 + 1); it += kT) {
    const int e = it / P, l = it - e * P, em = e ? n - e : 0;
    double2 h[2];
    hartley2(Z[e * P + l], Z[em * P + l], h[0], h[1]);
    for (int m = 0; m <= (em != e ? 1 : 0); ++m) {
      double* s = base + (long long)(m ? em : e) * nx + 2 * l;
      if (2 * l < cols) s[0] = h[m].x;
      if (2 * l + 1 < cols) s[1] = h[m].y;
    }
  }
}

// The tridiagonal systems' pivots c_j = 1 / (delta - c_{j-1}), c_1 = 1 / delta, delta = 2 + lambda / cz,
// for the (nx/2+1)(ny/2+1) different eigenvalues lambda = 4 cx sin^2(pi kx / nx) + 4 cy sin^2(pi ky / ny):
// ctab[j-1][ky][kx].  A thread starts from the closed form (pivot_at) and runs the recurrence for
// `run` unknowns, until it stands still (most modes: after some 20 / t unknowns).
__device__ void pivots(const PGrid& g, double* __restrict__ ctab, long long t0, long long stride, int run) {
  const int hx = g.nx / 2 + 1, hy = g.ny / 2 + 1, modes = hx * hy;
  const long long total = (long long)modes * ((g.nzi + run - 1) / run);
  for (long long t = t0; t < total; t += stride) {
    const int ch = (int)(t / modes), md = (int)(t - (long long)ch * modes);
    const int ky = md / hx, kx = md - ky * hx;
    const double sx = sinpi((double)kx / g.nx), sy = sinpi((double)ky / g.ny);
    const double s = (g.cx * sx * sx + g.cy * sy * sy) / g.cz;      // lambda / (4 cz)
    const int j0 = ch * run + 1, j1 = min(j0 + run - 1, g.nzi);
    const double delta = fma(4.0, s, 2.0);
    double c = pivot_at(s, j0);
    bool still = false;
    for (int j = j0;; ++j) {
      ctab[(long long)(j - 1) * modes + md] = c;
      if (j == j1) break;
      if (!still) {
        const double next = 1.0 / (delta - c);
        still = next == c;
        c = next;
      }
    }
  }
}

// Pivots and the twiddles of both directions, for grids whose planes are not transformed at once.
__global__ void __launch_bounds__(kT) setup_kernel(PGrid g, double2* __restrict__ tw, double* __restrict__ ctab, int run) {
  const long long t0 = (long long)blockIdx.x * kT + threadIdx.x, stride = (long long)gridDim.x * kT;
  for (long long i = t0; i < g.nx + g.ny; i += stride) {
    double s, c;
    sincospi(i < g.nx ? -2.0 * i / g.nx : -2.0 * (i - g.nx) / g.ny, &s, &c);
    tw[i] = make_double2(c, s);
  }
  if (ctab) pivots(g, ctab, t0, stride, run);
}

// Twiddles of small planes, with the launch.
constexpr int kInlineTwiddles = 128;
constexpr int kPivotThreads = 64;
struct PlaneTwiddles {
  double2 w[kInlineTwiddles];
};

// Small planes: two planes a block as one complex plane, x and y lines transformed together (the
// Hartley transform over the plane, cas of the summed phase, which the operator's eigenvectors
// share as well).  FORWARD: the residual is formed as the planes are read (and kept in r), its
// transform written to `hat`; else `hat` is transformed back into the correction d (still to be
// multiplied by `inv`), added to x.  The first launch forms the pivots as well, in blocks of its own.
template <bool FORWARD, bool FIRST>
__global__ void __launch_bounds__(kT) planes_kernel(PGrid g, const double* __restrict__ rho, double scale, double* __restrict__ x,
                                                    double* r, double* __restrict__ d, double* __restrict__ hat,
                                                    double* part, State* st, double rtol, int max_iter, double inv,
                                                    const __grid_constant__ Fft px, const __grid_constant__ Fft py,
                                                    const __grid_constant__ PlaneTwiddles tw, const double2* __restrict__ twd,
                                                    double* __restrict__ ctab, int nplanes) {
  if (!FIRST && !st->active) return;
  if (FIRST && (int)blockIdx.x >= nplanes) {           // the blocks past the planes form the pivots,
    if (threadIdx.x < kPivotThreads)                   // in few warps each: some 200 FP64 operations deep
      pivots(g, ctab, ((long long)blockIdx.x - nplanes) * kPivotThreads + threadIdx.x,
             (long long)(gridDim.x - nplanes) * kPivotThreads, 1);
    return;
  }
  extern __shared__ __align__(16) double2 sm[];
  const int nx = g.nx, ny = g.ny, np = nx * ny;
  double2 *A = sm, *B = sm + np, *WX = sm + 2 * np, *WY = WX + nx;
  for (int i = threadIdx.x; i < nx + ny; i += kT) WX[i] = twd ? twd[i] : tw.w[i];
  const int k0 = blockIdx.x * 2;
  const bool two = k0 + 1 < g.nzi;
  const long long base = (long long)k0 * np;
  double lrr = 0.0, lbb = 0.0;
  for (int it = threadIdx.x; it < np; it += kT) {
    const int j = it / nx, i = it - j * nx;
    if constexpr (FORWARD) {
      double b0, b1 = 0.0, q1 = 0.0;
      const double q0 = residual_at<kFromX>(g, rho, scale, x, r, i, j, k0, base + it, b0);
      r[base + it] = q0;
      if (two) {
        q1 = residual_at<kFromX>(g, rho, scale, x, r, i, j, k0 + 1, base + np + it, b1);
        r[base + np + it] = q1;
      }
      lrr = fma(q0, q0, fma(q1, q1, lrr));
      if constexpr (FIRST) lbb = fma(b0, b0, fma(b1, b1, lbb));
      A[it] = make_double2(q0, q1);
    } else {
      A[it] = make_double2(hat[base + it], two ? hat[base + np + it] : 0.0);
    }
  }
  __syncthreads();
  double2* X = fft_lines(A, B, WX, px, ny, 1, nx);
  const double2* Z = fft_lines(X, X == A ? B : A, WY, py, nx, nx, 1);
  for (int it = threadIdx.x; it < np; it += kT) {
    const int j = it / nx, i = it - j * nx;
    const int im = (j ? ny - j : 0) * nx + (i ? nx - i : 0);
    if (im < it) continue;                             // the lower of k and -k does both
    double2 h[2];
    hartley2(Z[it], Z[im], h[0], h[1]);
    for (int m = 0; m <= (im != it ? 1 : 0); ++m) {
      const long long at = base + (m ? im : it);
      if constexpr (FORWARD) {
        hat[at] = h[m].x;
        if (two) hat[at + np] = h[m].y;
      } else {
        d[at] = h[m].x;
        x[at] = fma(inv, h[m].x, x[at]);
        if (two) {
          d[at + np] = h[m].y;
          x[at + np] = fma(inv, h[m].y, x[at + np]);
        }
      }
    }
  }
  if constexpr (FORWARD) finish_residual<FIRST>(lrr, lbb, part, st, rtol, max_iter, nplanes);
}

// The tridiagonal systems of blockDim.x modes (kx, ky), in place: thread row s of the block takes
// unknowns [s L, (s+1) L) of each.  Forward g_j = c_j (f_j + g_{j-1}) and backward u_j = g_j + c_j u_{j+1}
// are linear in what enters a segment, so each warp first finds what its segment returns for
// nothing entering, the segments' chain is followed by one warp, and the sweeps run with it.
// The segment's f and c stay in registers between the sweeps: v is read and written once.
// (L = 32 with 1024 threads, for more than 256 unknowns, spills part of them to L1.)
template <int L, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) tridiag_kernel(PGrid g, double* __restrict__ v, const double* __restrict__ ctab,
                                                                 State* st) {
  if (!st->active) return;
  __shared__ double out[32][33], prod[32][33];       // [segment][lane]
  const int lane = threadIdx.x, s = threadIdx.y, S = blockDim.y;
  const int np = g.nx * g.ny;
  const int mode = blockIdx.x * blockDim.x + lane;
  const bool live = mode < np;
  const int ky = live ? mode / g.nx : 0, kx = live ? mode - ky * g.nx : 0;
  const int hx = g.nx / 2 + 1, modes = hx * (g.ny / 2 + 1);
  const int md = min(ky, g.ny - ky) * hx + min(kx, g.nx - kx);
  const int j0 = s * L;
  double h[L], c[L];
#pragma unroll
  for (int j = 0; j < L; ++j) {
    const bool in = live && j0 + j < g.nzi;
    h[j] = in ? v[(long long)(j0 + j) * np + mode] : 0.0;
    c[j] = in ? ctab[(long long)(j0 + j) * modes + md] : 0.0;
  }
  double e = 0.0, pr = 1.0;
#pragma unroll
  for (int j = 0; j < L; ++j) {
    h[j] *= c[j];
    e = fma(c[j], e, h[j]);
    pr *= c[j];
  }
  out[s][lane] = e;
  prod[s][lane] = pr;
  __syncthreads();
  if (s == 0) {                                      // what enters segment i, left in out[i]
    double in = 0.0;
    for (int i = 0; i < S; ++i) {
      const double nxt = fma(prod[i][lane], in, out[i][lane]);
      out[i][lane] = in;
      in = nxt;
    }
  }
  __syncthreads();
  e = out[s][lane];
#pragma unroll
  for (int j = 0; j < L; ++j) {
    e = fma(c[j], e, h[j]);
    h[j] = e;
  }
  __syncthreads();
  e = 0.0;
#pragma unroll
  for (int j = L - 1; j >= 0; --j) e = fma(c[j], e, h[j]);
  out[s][lane] = e;
  __syncthreads();
  if (s == 0) {
    double in = 0.0;
    for (int i = S - 1; i >= 0; --i) {
      const double nxt = fma(prod[i][lane], in, out[i][lane]);
      out[i][lane] = in;
      in = nxt;
    }
  }
  __syncthreads();
  e = out[s][lane];
#pragma unroll
  for (int j = L - 1; j >= 0; --j) {
    e = fma(c[j], e, h[j]);
    if (live && j0 + j < g.nzi) v[(long long)(j0 + j) * np + mode] = e;
  }
  if (blockIdx.x == 0 && lane == 0 && s == 0) st->iterations += 1;
}

}  // namespace

// Work items of the transforms' launches for grids that are transformed line by line.
struct LineShape {
  int PX, PY;              // pairs of lines a block: rows, columns
};
static LineShape line_shape(const PGrid& g, int sms) {
  // up to 2048 complex points a block, and enough blocks for every SM
  auto pairs_of = [&](int len, long long pairs) {
    const long long most = std::max(1, kMaxLine / len);
    return (int)std::max<long long>(1, std::min(most, (pairs + 4 * sms - 1) / (4 * sms)));
  };
  LineShape L;
  L.PX = pairs_of(g.nx, ((long long)g.ny * g.nzi + 1) / 2);
  L.PY = std::min((g.nx + 1) / 2, std::max(pairs_of(g.ny, (long long)((g.nx + 1) / 2) * g.nzi), std::min(8, std::max(1, kMaxLine / g.ny))));
  return L;
}

// FP64 operations of the transform of a pair of lines: six for a pair a +- w b, 2 R an output for the
// first stage of a long prime R, 4 (R - 1) for other odd ones.
static double line_ops(int n) {
  const Fft p = plan_of(n);
  double s = 0.0;
  for (int f = 0; f < p.nf; ++f) {
    const int R = p.rad[f];
    s += (double)n * (R == 4 ? 6 : R == 2 ? 3 : f == 0 && R >= 5 ? 2 * R : 4 * (R - 1));
  }
  return s;
}

// Whether direct corrections are the faster way.  A line with a large prime costs operations in
// proportion to it, while a grid of few planes, or a loose tolerance, needs few CG iterations; so
// both are estimated, in us, from the FP64 rate (4,130 operations a us and SM) and the times of a
// launch and of an iteration's grid barriers.  The lines lie where these estimates cross, 15% on the
// direct side.  Measured, direct / CG (FP64, to 1e-13): 2039x2039x2 59.2 / 5.7 ms, 1021x1021x5 29.3 /
// 13.6, 2039x16x3 4.3 / 1.4 go to CG; 1021x1021x17 111 / 168, 509x509x33 29 / 155, 1024x1024x2 0.8 / 1.8
// and every grid of factors 2, 3 and 5 stay.  max_iter keeps twice the estimated iterations in hand,
// and the mixed form, whose test is b - A x, a tolerance that its iterations reach.
static bool direct_pays(const PGrid& g, double rtol, int max_iter, bool mixed, int sms) {
  if (mixed && rtol < 1e-12) return true;
  constexpr double kOpsPerUs = 4130.0;
  auto waves = [&](double blocks) { return std::max(1.0, blocks / sms); };
  const double ox = line_ops(g.nx), oy = line_ops(g.ny);
  double transform;                                   // x and y once
  if ((long long)g.nx * g.ny <= kPlanePoints) {
    transform = 1.5 * (g.ny * ox + g.nx * oy) / kOpsPerUs * waves(0.5 * g.nzi);
  } else {
    const LineShape L = line_shape(g, sms);
    transform = (ox * L.PX * waves(0.5 * g.ny * g.nzi / L.PX) + oy * L.PY * waves(0.5 * g.nx * g.nzi / L.PY)) / kOpsPerUs;
  }
  const double direct = 80.0 + 2.0 * transform + 60.0 * g.n / (kOpsPerUs * sms);
  // CG: error falls by (k - 1) / (k + 1) an iteration, k^2 the condition number
  const double t = M_PI / (2.0 * (g.nzi + 1)), sn = std::sin(t), cs = std::cos(t);
  const double k = std::sqrt((4.0 * g.cx + 4.0 * g.cy + 4.0 * g.cz * cs * cs) / (4.0 * g.cz * sn * sn));
  const double its = k > 1.0 + 1e-6 ? std::min((double)g.n, std::log(2.0 / rtol) / std::log((k + 1.0) / (k - 1.0))) : 1.0;
  const double cg = 200.0 + (mixed ? 1.2 : 1.0) * its * ((mixed ? 55.0 : 15.0) + (mixed ? 8.0 : 23.0) * g.n / (kOpsPerUs * sms));
  return !(cg < 0.85 * direct && 2.0 * its < max_iter);
}

// Whether n has no prime factor above 31: such lines always pay.
static bool smooth(int n) {
  for (int p : {2, 3, 5, 7, 11, 13, 17, 19, 23, 29, 31})
    while (n % p == 0) n /= p;
  return n == 1;
}

bool poisson_direct_fits(const omen_ctx* ctx, const PGrid& g, double rtol, int max_iter, bool mixed) {
  if (g.nx > kMaxLine || g.ny > kMaxLine || g.nzi > kMaxZ) return false;
  if (smooth(g.nx) && smooth(g.ny)) return true;
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device) != cudaSuccess) return true;
  return direct_pays(g, rtol, max_iter, mixed, sms);
}

omen_status poisson_direct(omen_ctx* ctx, const PGrid& g, const double* rho, double scale, double* x, double rtol,
                           int max_iter, bool true_residual, DirectResult* res) {
  cudaStream_t st = ctx->stream;
  const long long n = g.n;
  const int np = g.nx * g.ny;
  const bool planes = np <= kPlanePoints;
  int sms = 0;
  OMEN_CUDA(ctx, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device));
  const long long modes = (long long)(g.nx / 2 + 1) * (g.ny / 2 + 1);
  const int rblocks = (int)std::min<long long>(((long long)g.ny * g.nzi + 7) / 8, (long long)sms * 8);
  const int pblocks = (g.nzi + 1) / 2;
  const int nblocks = std::max(rblocks, pblocks);
  auto pad = [](size_t b) { return (b + 255) / 256 * 256; };
  const size_t bv = pad(sizeof(double) * (size_t)n), bc = pad(sizeof(double) * (size_t)(modes * g.nzi));
  const size_t bt = pad(sizeof(double2) * ((size_t)g.nx + g.ny));
  const size_t bytes = (planes ? 3 : 2) * bv + bc + bt + pad(sizeof(double) * 2 * (size_t)nblocks) + pad(sizeof(State));
  char* buf = nullptr;
  if (ctx_alloc(ctx, &buf, bytes) != cudaSuccess) {
    cudaGetLastError();
    return set_err(ctx, OMEN_ENOMEM, "Poisson work vectors");
  }
  char* at = buf;
  auto take = [&](size_t b) { char* p = at; at += pad(b); return p; };
  double* r = reinterpret_cast<double*>(take(bv));
  double* d = reinterpret_cast<double*>(take(bv));
  double* hat = planes ? reinterpret_cast<double*>(take(bv)) : d;
  double* ctab = reinterpret_cast<double*>(take(bc));
  double2* tw = reinterpret_cast<double2*>(take(bt));
  double* part = reinterpret_cast<double*>(take(sizeof(double) * 2 * nblocks));
  State* state = reinterpret_cast<State*>(take(sizeof(State)));
  const Fft px = plan_of(g.nx), py = plan_of(g.ny);
  cudaError_t e = cudaMemsetAsync(state, 0, sizeof(State), st);
  auto ok = [&](cudaError_t c) { if (e == cudaSuccess) e = c; };

  // planes at once take their twiddles with the launch (else from a table) and form the pivots, one a
  // thread, beside their first transform; line by line, longer runs of the recurrence cost less
  PlaneTwiddles inl{};
  const bool with_launch = planes && g.nx + g.ny <= kInlineTwiddles;
  if (with_launch) {
    for (int i = 0; i < g.nx + g.ny; ++i) {
      const double a = i < g.nx ? -2.0 * M_PI * i / g.nx : -2.0 * M_PI * (i - g.nx) / g.ny;
      inl.w[i] = make_double2(std::cos(a), std::sin(a));
    }
  } else {
    const int run = 64;
    const long long work = planes ? g.nx + g.ny : std::max<long long>(g.nx + g.ny, modes * ((g.nzi + run - 1) / run));
    setup_kernel<<<(unsigned)std::min<long long>((work + kT - 1) / kT, (long long)sms * 8), kT, 0, st>>>(g, tw, planes ? nullptr : ctab, run);
    ok(cudaGetLastError());
  }
  const double2* twd = with_launch ? nullptr : tw;
  const double2 *twx = tw, *twy = tw + g.nx;

  // each transform doubles (hartley2) and the inverse leaves nx ny; the factor goes in where the
  // correction is added to x and where A d is taken from the residual
  const double inv = 1.0 / ((planes ? 4.0 : 16.0) * np * g.cz);
  // modes a block: 32, or fewer where those blocks leave SMs idle; unknowns per thread: long segments
  // (fewer operations) once the modes alone give every SM a block
  auto tridiag = [&]() {
    const int per = np >= 32 * sms ? 32 : np >= 8 * sms ? 8 : 4;
    const unsigned blocks = (unsigned)((np + per - 1) / per);
    const int L = g.nzi > 256 || np >= 64 * sms ? 32 : np >= 32 * sms ? 16 : 8;
    const dim3 thr(per, (g.nzi + L - 1) / L);
    if (g.nzi > 256) tridiag_kernel<32, 1024><<<blocks, thr, 0, st>>>(g, hat, ctab, state);
    else if (L == 32) tridiag_kernel<32, 256><<<blocks, thr, 0, st>>>(g, hat, ctab, state);
    else if (L == 16) tridiag_kernel<16, 512><<<blocks, thr, 0, st>>>(g, hat, ctab, state);
    else tridiag_kernel<8, 1024><<<blocks, thr, 0, st>>>(g, hat, ctab, state);
    ok(cudaGetLastError());
  };
  const int rounds = std::min(2, max_iter);
  if (planes) {
    const size_t smem = sizeof(double2) * (2 * (size_t)np + g.nx + g.ny);
    ok(smem_limit(planes_kernel<true, true>, smem));
    ok(smem_limit(planes_kernel<true, false>, smem));
    ok(smem_limit(planes_kernel<false, false>, smem));
    const int pivot_blocks = (int)std::min<long long>((modes * g.nzi + kPivotThreads - 1) / kPivotThreads, (long long)sms * 8);
    auto plane_pass = [&](auto kernel, int blocks, double factor) {
      kernel<<<blocks, kT, smem, st>>>(g, rho, factor, x, r, d, hat, part, state, rtol, max_iter, inv, px, py, inl, twd, ctab, pblocks);
      ok(cudaGetLastError());
    };
    for (int i = 0; i < rounds && e == cudaSuccess; ++i) {
      if (i == 0) plane_pass(planes_kernel<true, true>, pblocks + pivot_blocks, scale);
      else plane_pass(planes_kernel<true, false>, pblocks, scale);
      tridiag();
      plane_pass(planes_kernel<false, false>, pblocks, scale);
    }
  } else {
    const LineShape L = line_shape(g, sms);
    const int PX = L.PX, PY = L.PY, nrows = g.ny * g.nzi;
    const unsigned bx = (unsigned)((nrows + 2 * PX - 1) / (2 * PX));
    const int tiles = (g.nx + 2 * PY - 1) / (2 * PY);
    const unsigned by = (unsigned)tiles * g.nzi;
    const size_t smx = sizeof(double2) * (2 * (size_t)PX + 1) * g.nx, smy = sizeof(double2) * (2 * (size_t)PY + 1) * g.ny;
    ok(smem_limit(rows_kernel<false>, smx));
    ok(smem_limit(rows_kernel<true>, smx));
    ok(smem_limit(columns_kernel, smy));
    nonzero_kernel<<<(unsigned)(sms * 8), kT, 0, st>>>(x, n, state);
    residual_kernel<kFromX, true><<<rblocks, kT, 0, st>>>(g, rho, scale, x, r, part, state, rtol, max_iter);
    ok(cudaGetLastError());
    for (int i = 0; i < rounds && e == cudaSuccess; ++i) {
      rows_kernel<false><<<bx, kT, smx, st>>>(r, d, x, inv, nrows, PX, px, twx, state);
      columns_kernel<<<by, kT, smy, st>>>(d, g.nx, PY, tiles, py, twy, state);
      ok(cudaGetLastError());
      tridiag();
      columns_kernel<<<by, kT, smy, st>>>(d, g.nx, PY, tiles, py, twy, state);
      rows_kernel<true><<<bx, kT, smx, st>>>(d, d, x, inv, nrows, PX, px, twx, state);
      ok(cudaGetLastError());
      if (i + 1 < rounds) {
        residual_kernel<kFromX, false><<<rblocks, kT, 0, st>>>(g, rho, scale, x, r, part, state, rtol, max_iter);
        ok(cudaGetLastError());
      }
    }
  }
  if (e == cudaSuccess) {   // what the last correction leaves (skipped once one has passed the test)
    if (true_residual) residual_kernel<kFromX, false><<<rblocks, kT, 0, st>>>(g, rho, scale, x, r, part, state, rtol, max_iter);
    else residual_kernel<kFromD, false><<<rblocks, kT, 0, st>>>(g, rho, inv, d, r, part, state, rtol, max_iter);
    ok(cudaGetLastError());
  }
  State h{};
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, state, sizeof(State), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e == cudaSuccess && h.bb == 0.0) {   // b = 0: the solution is x = 0 whatever the initial guess
    e = cudaMemsetAsync(x, 0, sizeof(double) * (size_t)n, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  }
  cudaFreeAsync(buf, st);
  if (e != cudaSuccess) return set_err(ctx, OMEN_ECUDA, "Poisson solve: %s", cudaGetErrorString(e));
  res->iterations = h.iterations;
  res->converged = h.bb == 0.0 || h.rr <= h.stop;
  res->rel = h.bb > 0.0 ? std::sqrt(h.rr / h.bb) : 0.0;
  return OMEN_OK;
}
