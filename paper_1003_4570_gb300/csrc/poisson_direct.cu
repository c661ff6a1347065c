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
// memory (radix 4 and 2 in registers, other primes by their definition), and are bound by the FP64
// rate (some 85 operations a point for four transforms of 256 points).  Planes small enough for
// shared memory are transformed in x and y at once, two planes as one complex plane, with the
// residual formed as they are read: three launches a correction.
//
// Measured against the conjugate gradients this takes the place of (poisson.cu, one cooperative
// launch, three grid barriers an iteration): 11x11x217 grid to 1e-13 4.95 -> 0.157 ms (two
// corrections; launches), 256x256x257 to 1e-10 in the mixed form 250 -> 3.41 ms (one correction
// and its check; the FP64 rate), the error against 64-bit transforms 1.1e-15 -> 0.7e-15 and
// 9.6e-12 -> 1.1e-14 of the norm.
#include <algorithm>
#include <cmath>

#include "poisson_direct.h"

namespace {

constexpr int kMaxLine = 2048;       // points of a transformed line
constexpr int kMaxZ = 1024;          // unknowns of a tridiagonal system
constexpr int kPlanePoints = 3072;   // points of a plane transformed at once
constexpr int kT = 256;

struct Fft {
  int n, nf;
  int rad[12];
};

Fft plan_of(int n) {
  Fft p{};
  p.n = n;
  int m = n;
  while (m % 4 == 0) p.rad[p.nf++] = 4, m /= 4;
  for (int r = 2; m > 1; ++r)
    while (m % r == 0) p.rad[p.nf++] = r, m /= r;
  return p;
}

struct State {
  double bb, rr, stop;
  int active;          // the residual is above the stopping value
  int iterations;
  unsigned arrived;    // blocks of the running residual pass that have left their sums
};

__device__ __forceinline__ double2 cx_mul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
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
        const int jm = w % Ns;
        double2 v0 = src[w * es], v1 = src[(w + q) * es], v2 = src[(w + 2 * q) * es], v3 = src[(w + 3 * q) * es];
        if (jm) {
          const int t = jm * step;
          v1 = cx_mul(v1, tw[t]);
          v2 = cx_mul(v2, tw[2 * t]);
          v3 = cx_mul(v3, tw[3 * t]);
        }
        const double2 s02 = make_double2(v0.x + v2.x, v0.y + v2.y), d02 = make_double2(v0.x - v2.x, v0.y - v2.y);
        const double2 s13 = make_double2(v1.x + v3.x, v1.y + v3.y), d13 = make_double2(v1.x - v3.x, v1.y - v3.y);
        const int o = (w - jm) * 4 + jm;
        dst[o * es] = make_double2(s02.x + s13.x, s02.y + s13.y);
        dst[(o + Ns) * es] = make_double2(d02.x + d13.y, d02.y - d13.x);       // d02 - i d13
        dst[(o + 2 * Ns) * es] = make_double2(s02.x - s13.x, s02.y - s13.y);
        dst[(o + 3 * Ns) * es] = make_double2(d02.x - d13.y, d02.y + d13.x);
      } else if (R == 2) {
        const int jm = w % Ns;
        const double2 v0 = src[w * es];
        double2 v1 = src[(w + q) * es];
        if (jm) v1 = cx_mul(v1, tw[jm * step]);
        const int o = (w - jm) * 2 + jm;
        dst[o * es] = make_double2(v0.x + v1.x, v0.y + v1.y);
        dst[(o + Ns) * es] = make_double2(v0.x - v1.x, v0.y - v1.y);
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

// Twice the Hartley transforms of the two real lines (planes) whose complex FFT holds z at k and
// zm at -k.
__device__ __forceinline__ double2 hartley2(double2 z, double2 zm) {
  return make_double2((z.x + zm.x) - (z.y - zm.y), (z.y + zm.y) + (z.x - zm.x));
}

// Leaves the block's sum with the others'; the last block to arrive adds all of them in block
// order and sets the state: the squared residual, and on the first pass ||b||^2 and the stopping
// value.  All threads of the block call it.
template <bool FIRST>
__device__ void finish_residual(double lrr, double lbb, double* part, State* st, double rtol, int max_iter) {
  __shared__ double sh[32];
  __shared__ bool last;
  const double v = block_sum(lrr, sh);
  double w = 0.0;
  if constexpr (FIRST) w = block_sum(lbb, sh);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = v;
    if constexpr (FIRST) part[gridDim.x + blockIdx.x] = w;
    __threadfence();
    last = atomicAdd(&st->arrived, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double a = 0.0, c = 0.0;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) {
    a += __ldcg(part + b);
    if constexpr (FIRST) c += __ldcg(part + gridDim.x + b);
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

// How a residual is formed
enum { kFromX = 0, kFromD = 1 };     // b - A x; or the residual kept so far less A d

template <int HOW>
__device__ __forceinline__ double residual_at(const PGrid& g, const double* __restrict__ rho, double scale,
                                              const double* __restrict__ v, const double* r, int i, int j, int k,
                                              long long idx, double& b) {
  if constexpr (HOW == kFromX) {
    b = scale * rho[idx];
    return b - stencil_at(v, g, i, j, k, idx);
  } else {
    b = 0.0;
    return r[idx] - stencil_at(v, g, i, j, k, idx);
  }
}

// r = residual on the whole grid and its square sum: rows over the warps of the grid, points of a
// row over the lanes.
template <int HOW, bool FIRST>
__global__ void __launch_bounds__(kT) residual_kernel(PGrid g, const double* __restrict__ rho, double scale,
                                                      const double* __restrict__ v, double* r, double* part,
                                                      State* st, double rtol, int max_iter) {
  if (!FIRST && !st->active) return;
  const int lane = threadIdx.x & 31, nw = (gridDim.x * kT) >> 5;
  const int rows = g.ny * g.nzi;
  double lrr = 0.0, lbb = 0.0;
  for (int rw = (blockIdx.x * kT + threadIdx.x) >> 5; rw < rows; rw += nw) {
    const int k = rw / g.ny, j = rw - k * g.ny;
    const long long base = (long long)rw * g.nx;
    for (int i = lane; i < g.nx; i += 32) {
      double b;
      const double ri = residual_at<HOW>(g, rho, scale, v, r, i, j, k, base + i, b);
      r[base + i] = ri;
      lrr = fma(ri, ri, lrr);
      if constexpr (FIRST) lbb = fma(b, b, lbb);
    }
  }
  finish_residual<FIRST>(lrr, lbb, part, st, rtol, max_iter);
}

// Hartley transform of every row (x lines), P pairs of rows a block.  ADD: the result is the
// correction, also added to x.
template <bool ADD>
__global__ void __launch_bounds__(kT) rows_kernel(const double* src, double* dst, double* __restrict__ x,
                                                  int nrows, int P, const __grid_constant__ Fft p,
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
  for (int it = threadIdx.x; it < have * n; it += kT) {
    const int l = it / n, e = it - l * n, ra = r0 + 2 * l;
    const double2 h = hartley2(Z[it], Z[l * n + (e ? n - e : 0)]);
    const long long at = (long long)ra * n + e;
    dst[at] = h.x;
    if constexpr (ADD) x[at] += h.x;
    if (ra + 1 < nrows) {
      dst[at + n] = h.y;
      if constexpr (ADD) x[at + n] += h.y;
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
  for (int it = threadIdx.x; it < P * n; it += kT) {
    const int e = it / P, l = it - e * P;
    const double2 h = hartley2(Z[it], Z[(e ? n - e : 0) * P + l]);
    double* s = base + (long long)e * nx + 2 * l;
    if (2 * l < cols) s[0] = h.x;
    if (2 * l + 1 < cols) s[1] = h.y;
  }
}

// Small planes: two planes a block as one complex plane, x and y lines transformed together (the
// Hartley transform over the plane, cas of the summed phase, which the operator's eigenvectors
// share as well).  FORWARD: the residual is formed as the planes are read (and kept in r), its
// transform written to `hat`; else `hat` is transformed back into the correction d, added to x.
template <bool FORWARD, int HOW, bool FIRST>
__global__ void __launch_bounds__(kT) planes_kernel(PGrid g, const double* __restrict__ rho, double scale, double* __restrict__ x,
                                                    double* r, double* __restrict__ d, double* __restrict__ hat,
                                                    double* part, State* st, double rtol, int max_iter,
                                                    const __grid_constant__ Fft px, const __grid_constant__ Fft py,
                                                    const double2* __restrict__ twx, const double2* __restrict__ twy) {
  if (!FIRST && !st->active) return;
  extern __shared__ __align__(16) double2 sm[];
  const int nx = g.nx, ny = g.ny, np = nx * ny;
  double2 *A = sm, *B = sm + np, *WX = sm + 2 * np, *WY = WX + nx;
  for (int i = threadIdx.x; i < nx; i += kT) WX[i] = twx[i];
  for (int i = threadIdx.x; i < ny; i += kT) WY[i] = twy[i];
  const int k0 = blockIdx.x * 2;
  const bool two = k0 + 1 < g.nzi;
  const long long base = (long long)k0 * np;
  double lrr = 0.0, lbb = 0.0;
  for (int it = threadIdx.x; it < np; it += kT) {
    const int j = it / nx, i = it - j * nx;
    if constexpr (FORWARD) {
      const double* v = HOW == kFromX ? x : d;
      double b0, b1 = 0.0, q1 = 0.0;
      const double q0 = residual_at<HOW>(g, rho, scale, v, r, i, j, k0, base + it, b0);
      r[base + it] = q0;
      if (two) {
        q1 = residual_at<HOW>(g, rho, scale, v, r, i, j, k0 + 1, base + np + it, b1);
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
    const double2 h = hartley2(Z[it], Z[(j ? ny - j : 0) * nx + (i ? nx - i : 0)]);
    if constexpr (FORWARD) {
      hat[base + it] = h.x;
      if (two) hat[base + np + it] = h.y;
    } else {
      d[base + it] = h.x;
      x[base + it] += h.x;
      if (two) {
        d[base + np + it] = h.y;
        x[base + np + it] += h.y;
      }
    }
  }
  if constexpr (FORWARD) finish_residual<FIRST>(lrr, lbb, part, st, rtol, max_iter);
}

// Twiddles of both directions, and the tridiagonal systems' pivots c_j = 1 / (delta - c_{j-1}),
// c_1 = 1 / delta, delta = 2 + lambda / cz, for the (nx/2+1)(ny/2+1) different eigenvalues
// lambda = 4 cx sin^2(pi kx / nx) + 4 cy sin^2(pi ky / ny): ctab[j-1][ky][kx].  In closed form
// c_j = e^-t expm1(-2 j t) / expm1(-2 (j+1) t), sinh^2(t/2) = lambda / (4 cz) (j / (j+1) for
// lambda = 0); a thread starts from it and runs the recurrence for kPivots unknowns.
constexpr int kPivots = 16;

__global__ void __launch_bounds__(kT) setup_kernel(PGrid g, double2* __restrict__ twx, double2* __restrict__ twy,
                                                   double* __restrict__ ctab, State* st) {
  const long long t0 = (long long)blockIdx.x * kT + threadIdx.x, stride = (long long)gridDim.x * kT;
  if (t0 == 0) st->arrived = 0;
  const int hx = g.nx / 2 + 1, hy = g.ny / 2 + 1, modes = hx * hy;
  const int chunks = (g.nzi + kPivots - 1) / kPivots;
  const long long total = (long long)modes * chunks;
  for (long long t = t0; t < total + g.nx + g.ny; t += stride) {
    if (t >= total) {
      const int i = (int)(t - total);
      double s, c;
      if (i < g.nx) {
        sincospi(-2.0 * i / g.nx, &s, &c);
        twx[i] = make_double2(c, s);
      } else {
        sincospi(-2.0 * (i - g.nx) / g.ny, &s, &c);
        twy[i - g.nx] = make_double2(c, s);
      }
      continue;
    }
    const int ch = (int)(t / modes), md = (int)(t - (long long)ch * modes);
    const int ky = md / hx, kx = md - ky * hx;
    const double sx = sinpi((double)kx / g.nx), sy = sinpi((double)ky / g.ny);
    const double s = (g.cx * sx * sx + g.cy * sy * sy) / g.cz;      // lambda / (4 cz)
    const int j0 = ch * kPivots + 1, j1 = min(j0 + kPivots - 1, g.nzi);
    const double delta = fma(4.0, s, 2.0);
    double c;
    if (s == 0.0) {
      c = (double)j0 / (j0 + 1);
    } else {
      const double th = 2.0 * asinh(sqrt(s));
      c = exp(-th) * (expm1(-2.0 * j0 * th) / expm1(-2.0 * (j0 + 1) * th));
    }
    ctab[(long long)(j0 - 1) * modes + md] = c;
    for (int j = j0 + 1; j <= j1; ++j) {
      c = 1.0 / (delta - c);
      ctab[(long long)(j - 1) * modes + md] = c;
    }
  }
}

// The tridiagonal systems of 32 modes (kx, ky), in place: warp s of the block takes unknowns
// [s L, (s+1) L) of each.  Forward g_j = c_j (f_j + g_{j-1}) and backward u_j = g_j + c_j u_{j+1}
// are linear in what enters a segment, so each warp first finds what its segment returns for
// nothing entering, the segments' chain is followed by one warp, and the sweeps run with it.
// The segment's f and c stay in registers between the sweeps: v is read and written once.
// (L = 32 with 1024 threads, for more than 256 unknowns, spills part of them to L1.)
template <int L, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) tridiag_kernel(PGrid g, double* __restrict__ v, const double* __restrict__ ctab,
                                                                 double scale, State* st) {
  if (!st->active) return;
  __shared__ double out[32][33], prod[32][33];       // [segment][lane]
  const int lane = threadIdx.x, s = threadIdx.y, S = blockDim.y;
  const int np = g.nx * g.ny;
  const int mode = blockIdx.x * 32 + lane;
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
    h[j] = h[j] * scale * c[j];
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

template <typename K>
cudaError_t allow_smem(K kernel, size_t bytes) {
  return bytes > 48 * 1024 ? cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) : cudaSuccess;
}

}  // namespace

bool poisson_direct_fits(const PGrid& g) { return g.nx <= kMaxLine && g.ny <= kMaxLine && g.nzi <= kMaxZ; }

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
  const size_t bt = pad(sizeof(double2) * (size_t)g.nx) + pad(sizeof(double2) * (size_t)g.ny);
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
  double2* twx = reinterpret_cast<double2*>(take(sizeof(double2) * g.nx));
  double2* twy = reinterpret_cast<double2*>(take(sizeof(double2) * g.ny));
  double* part = reinterpret_cast<double*>(take(sizeof(double) * 2 * nblocks));
  State* state = reinterpret_cast<State*>(take(sizeof(State)));
  const Fft px = plan_of(g.nx), py = plan_of(g.ny);
  cudaError_t e = cudaSuccess;
  auto ok = [&](cudaError_t c) { if (e == cudaSuccess) e = c; };

  const long long work = modes * ((g.nzi + kPivots - 1) / kPivots) + g.nx + g.ny;
  setup_kernel<<<(unsigned)std::min<long long>((work + kT - 1) / kT, (long long)sms * 8), kT, 0, st>>>(g, twx, twy, ctab, state);
  ok(cudaGetLastError());

  // each transform doubles (hartley2) and the inverse leaves nx ny
  const double inv = 1.0 / ((planes ? 4.0 : 16.0) * np * g.cz);
  // unknowns per thread of the tridiagonal solves: long segments (fewer operations) once the modes
  // alone give every SM a block
  auto tridiag = [&]() {
    const unsigned blocks = (unsigned)((np + 31) / 32);
    const int L = g.nzi > 256 || blocks >= 2u * sms ? 32 : blocks >= (unsigned)sms ? 16 : 8;
    const dim3 thr(32, (g.nzi + L - 1) / L);
    if (g.nzi > 256) tridiag_kernel<32, 1024><<<blocks, thr, 0, st>>>(g, hat, ctab, inv, state);
    else if (L == 32) tridiag_kernel<32, 256><<<blocks, thr, 0, st>>>(g, hat, ctab, inv, state);
    else if (L == 16) tridiag_kernel<16, 512><<<blocks, thr, 0, st>>>(g, hat, ctab, inv, state);
    else tridiag_kernel<8, 1024><<<blocks, thr, 0, st>>>(g, hat, ctab, inv, state);
    ok(cudaGetLastError());
  };
  const int rounds = std::min(2, max_iter);
  if (planes) {
    const size_t smem = sizeof(double2) * (2 * (size_t)np + g.nx + g.ny);
    ok(allow_smem(planes_kernel<true, kFromX, true>, smem));
    ok(allow_smem(planes_kernel<true, kFromX, false>, smem));
    ok(allow_smem(planes_kernel<true, kFromD, false>, smem));
    ok(allow_smem(planes_kernel<false, kFromX, false>, smem));
    for (int i = 0; i < rounds && e == cudaSuccess; ++i) {
      if (i == 0)
        planes_kernel<true, kFromX, true><<<pblocks, kT, smem, st>>>(g, rho, scale, x, r, d, hat, part, state, rtol, max_iter, px, py, twx, twy);
      else if (true_residual)
        planes_kernel<true, kFromX, false><<<pblocks, kT, smem, st>>>(g, rho, scale, x, r, d, hat, part, state, rtol, max_iter, px, py, twx, twy);
      else
        planes_kernel<true, kFromD, false><<<pblocks, kT, smem, st>>>(g, rho, scale, x, r, d, hat, part, state, rtol, max_iter, px, py, twx, twy);
      ok(cudaGetLastError());
      tridiag();
      planes_kernel<false, kFromX, false><<<pblocks, kT, smem, st>>>(g, rho, scale, x, r, d, hat, part, state, rtol, max_iter, px, py, twx, twy);
      ok(cudaGetLastError());
    }
  } else {
    // pairs of lines a block: up to 2048 complex points, and enough blocks for every SM
    auto pairs_of = [&](int len, long long pairs) {
      const long long most = std::max(1, kMaxLine / len);
      return (int)std::max<long long>(1, std::min(most, (pairs + 4 * sms - 1) / (4 * sms)));
    };
    const int nrows = g.ny * g.nzi;
    const int PX = pairs_of(g.nx, (nrows + 1) / 2);
    const int PY = std::min((g.nx + 1) / 2, std::max(pairs_of(g.ny, (long long)((g.nx + 1) / 2) * g.nzi), std::min(8, std::max(1, kMaxLine / g.ny))));
    const unsigned bx = (unsigned)((nrows + 2 * PX - 1) / (2 * PX));
    const int tiles = (g.nx + 2 * PY - 1) / (2 * PY);
    const unsigned by = (unsigned)tiles * g.nzi;
    const size_t smx = sizeof(double2) * (2 * (size_t)PX + 1) * g.nx, smy = sizeof(double2) * (2 * (size_t)PY + 1) * g.ny;
    ok(allow_smem(rows_kernel<false>, smx));
    ok(allow_smem(rows_kernel<true>, smx));
    ok(allow_smem(columns_kernel, smy));
    residual_kernel<kFromX, true><<<rblocks, kT, 0, st>>>(g, rho, scale, x, r, part, state, rtol, max_iter);
    ok(cudaGetLastError());
    for (int i = 0; i < rounds && e == cudaSuccess; ++i) {
      rows_kernel<false><<<bx, kT, smx, st>>>(r, d, x, nrows, PX, px, twx, state);
      columns_kernel<<<by, kT, smy, st>>>(d, g.nx, PY, tiles, py, twy, state);
      ok(cudaGetLastError());
      tridiag();
      columns_kernel<<<by, kT, smy, st>>>(d, g.nx, PY, tiles, py, twy, state);
      rows_kernel<true><<<bx, kT, smx, st>>>(d, d, x, nrows, PX, px, twx, state);
      ok(cudaGetLastError());
      if (i + 1 < rounds) {
        if (true_residual) residual_kernel<kFromX, false><<<rblocks, kT, 0, st>>>(g, rho, scale, x, r, part, state, rtol, max_iter);
        else residual_kernel<kFromD, false><<<rblocks, kT, 0, st>>>(g, rho, scale, d, r, part, state, rtol, max_iter);
        ok(cudaGetLastError());
      }
    }
  }
  if (e == cudaSuccess) {   // the residual the last correction leaves (skipped once one has passed the test)
    if (true_residual) residual_kernel<kFromX, false><<<rblocks, kT, 0, st>>>(g, rho, scale, x, r, part, state, rtol, max_iter);
    else residual_kernel<kFromD, false><<<rblocks, kT, 0, st>>>(g, rho, scale, d, r, part, state, rtol, max_iter);
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
  res->zero = h.bb == 0.0;
  res->converged = res->zero || h.rr <= h.stop;
  res->rel = h.bb > 0.0 ? std::sqrt(h.rr / h.bb) : 0.0;
  return OMEN_OK;
}
