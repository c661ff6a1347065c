// Direct corrections for the finite-difference Poisson solver (poisson_direct.cu).
#pragma once

#include "omen_internal.h"
#include "fd.cuh"

struct DirectResult {
  int iterations;      // corrections applied
  bool converged;
  bool zero;           // the right-hand side is zero
  double rel;          // ||r|| / ||b||
};

// Whether the grid's lines fit the transforms (else the caller iterates).
bool poisson_direct_fits(const PGrid& g);

// Up to two corrections x += A^-1 r of the solution x of A x = scale * rho, r = b - A x.  The residual
// of the second correction, tested against rtol ||b||, is r - A d, carried like the recurrence residual
// of conjugate gradients (b - A x itself ends at the rounding of x), or with `true_residual` b - A x.  Waits for the
// context's stream.  ENOMEM leaves x as it was.
omen_status poisson_direct(omen_ctx* ctx, const PGrid& g, const double* rho, double scale, double* x, double rtol,
                           int max_iter, bool true_residual, DirectResult* out);
