// Direct corrections for the finite-difference Poisson solver (poisson_direct.cu).
#pragma once

#include <cmath>

#include "omen_internal.h"
#include "fd.cuh"

struct DirectResult {
  int iterations;      // corrections applied
  bool converged;
  double rel;          // ||r|| / ||b||
};

// Whether the grid's lines fit the transforms and these are the faster way (else the caller iterates).
bool poisson_direct_fits(const omen_ctx* ctx, const PGrid& g, double rtol, int max_iter, bool mixed);

// Up to two corrections x += A^-1 r of the solution x of A x = scale * rho, r = b - A x.  The residual
// of the second correction, tested against rtol ||b||, is r - A d, carried like the recurrence residual
// of conjugate gradients (b - A x itself ends at the rounding of x), or with `true_residual` b - A x.
// Waits for the context's stream.  ENOMEM leaves x as it was.
omen_status poisson_direct(omen_ctx* ctx, const PGrid& g, const double* rho, double scale, double* x, double rtol,
                           int max_iter, bool true_residual, DirectResult* out);

// The j-th pivot of a mode's tridiagonal system, c_j = 1 / (2 + 4 s - c_{j-1}), c_0 = 0, in closed form:
// c_j = e^-t expm1(-2 j t) / expm1(-2 (j+1) t) with sinh^2(t/2) = s (j / (j+1) for s = 0).  With a =
// sqrt(s) and u = 1 / (a + sqrt(1 + s)), e^-t = u^2 and expm1(-t) = -2 a u, so nothing cancels for any
// s: e^-t as expm1(-t) + 1 would lose e^t of its digits (1e-10 where the spacing in z is a thousand
// times the lateral one).
__host__ __device__ inline double pivot_at(double s, int j) {
  if (s == 0.0) return (double)j / (j + 1);
  const double a = sqrt(s), b = sqrt(1.0 + s), u = 1.0 / (a + b), q = u * u;
  const double ej = expm1(-4.0 * j * log1p(a + s / (1.0 + b)));    // asinh(a) from the root at hand
  return q * (ej / fma(ej, q * q, -2.0 * a * u * (q + 1.0)));
}
