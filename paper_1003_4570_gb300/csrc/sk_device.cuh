// Slater–Koster two-centre blocks in reduced form and the zincblende neighbour geometry shared
// by the assembly and H·X kernels.
#pragma once

#include <cuda_runtime.h>

#include "omen_internal.h"

// Integral indices
enum { P_SS = 0, P_SSSS, P_SSS, P_SP, P_SSP, P_SD, P_SSD, P_PPS, P_PPP, P_PDS, P_PDP, P_DDS, P_DDP, P_DDD };

// Numbers of a reduced block, padded so that every block starts on a 16-byte boundary.
__host__ __device__ constexpr int coef_stride(int norb) { return norb == 10 ? 28 : 12; }

// The reduced block (see hx.cu) of a bond along (1,1,1): Slater & Koster, Phys. Rev. 94, 1498
// (1954), Table I at direction cosines 1/sqrt(3), written in the sums and multiples of the
// identity that the rotations about the bond leave.  V12: integrals with the first-named orbital
// on atom 1, V21 with it on atom 2; a pair out of the table's order takes (-1)^(l1+l2) and V21.
// Rows are those of atom 1, or of atom 2 (`transposed`).
//   sp3d5s*: s: ss, sP, sT, ss*;  s*: s*s, s*P, s*T, s*s*;
//            p: ps, ps*, P (all-ones part), T (all-ones part), p (identity part), t (identity part), q;
//            t: ts, ts*, P, T, p, t, q;  e: p, t, e;  p and t of the first e row (times sqrt(3)/2).
//   sp3s*:   s: ss, sP, ss*;  s*: s*s, s*P, s*s*;  p: ps, ps*, P, p.
__host__ __device__ inline void reduced_block(const double* V12, const double* V21, int norb, bool transposed, double* c) {
  const double i3 = 0.57735026918962576;   // 1/sqrt(3)
  const double ss = V12[P_SS], SS = V12[P_SSSS], sS = V12[P_SSS], Ss = V21[P_SSS];
  const double sp = i3 * V12[P_SP], Sp = i3 * V12[P_SSP], ps = -i3 * V21[P_SP], pS = -i3 * V21[P_SSP];
  const double ppi = V12[P_PPP], pps = (V12[P_PPS] - V12[P_PPP]) / 3.0;
  if (norb == 5) {
    const double a[10] = {ss, sp, sS, Ss, Sp, SS, ps, pS, pps, ppi};
    const double t[10] = {ss, ps, Ss, sS, pS, SS, sp, Sp, pps, ppi};
    for (int i = 0; i < 12; ++i) c[i] = i < 10 ? (transposed ? t[i] : a[i]) : 0.0;
    return;
  }
  const double sd = i3 * V12[P_SD], Sd = i3 * V12[P_SSD], ds = i3 * V21[P_SD], dS = i3 * V21[P_SSD];
  // p-d: all-ones, identity and e parts; d-p the same of V21, negated
  const double pdb = V12[P_PDS] / 3.0 + V12[P_PDP] * i3 / 3.0, pda = -i3 * V12[P_PDP], pde = 2.0 / 3.0 * V12[P_PDP];
  const double dpb = -(V21[P_PDS] / 3.0 + V21[P_PDP] * i3 / 3.0), dpa = i3 * V21[P_PDP], dpe = -2.0 / 3.0 * V21[P_PDP];
  const double ddb = V12[P_DDS] / 3.0 - V12[P_DDP] / 9.0 - 2.0 / 9.0 * V12[P_DDD];
  const double dda = V12[P_DDP] / 3.0 + 2.0 / 3.0 * V12[P_DDD];
  const double dde = 2.0 / 3.0 * i3 * (V12[P_DDD] - V12[P_DDP]);   // t2g-e
  const double ee = 2.0 / 3.0 * V12[P_DDP] + V12[P_DDD] / 3.0;
  const double r = 0.86602540378443865;
  const double a[27] = {ss, sp, sd, sS, Ss, Sp, Sd, SS, ps, pS, pps, pdb, ppi, pda, pde,
                        ds, dS, dpb, ddb, dpa, dda, dde, dpe, dde, ee, r * dpe, r * dde};
  const double t[27] = {ss, ps, ds, Ss, sS, pS, dS, SS, sp, Sp, pps, dpb, ppi, dpa, dpe,
                        sd, Sd, pdb, ddb, pda, dda, dde, pde, dde, ee, r * pde, r * dde};
  for (int i = 0; i < 28; ++i) c[i] = i < 27 ? (transposed ? t[i] : a[i]) : 0.0;
}

// Geometry helpers ---------------------------------------------------------------------------
struct Geo {
  int nx, ny, nz, ncells, natoms;
  int periodic[3];
};
