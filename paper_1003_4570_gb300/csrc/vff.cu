// Valence-force-field strain relaxation on the device (paper Section II-B: the atom positions of
// a structure are relaxed by minimising an atomistic VFF strain energy before the electronic
// structure is computed; Fig. 4 benchmarks that step).  The paper prints no form; this is
// Keating's (Phys. Rev. 145, 637 (1966)), per bond and per bond angle:
//
//   E = sum_bonds 3 alpha_b / (8 d_b^2) (r_b.r_b - d_b^2)^2
//     + sum_atoms sum_{bond pairs p<q at the atom} 3 beta_pq / (8 d_p d_q) (r_p.r_q + d_p d_q / 3)^2
//
// r_p leaves the vertex atom along bond p; d_b is the natural bond length of the pair (mean of
// sqrt(3)/4 a of the two species), alpha_b the mean stretching constant, beta_b the mean bending
// constant of the bond's species and beta_pq the mean over the two bonds.  Positions are
// x = F x0 + u with F a fixed homogeneous deformation of the box and u the displacements; the
// ideal A->B bond vector of direction k is dir_k a/4, so r = +-F dir_k a/4 + u_n - u_i needs no
// stored positions and no neighbour list (neighbours come from the cell index, as in H·X).
//
// Kernels.  Every term belongs to a vertex: the angles between the four bonds r_p of an atom, and
// half of each bond's stretch, so with G_pq = r_p.r_q
//   E_i = sum_p k_p (G_pp - d_p^2)^2 + sum_{p<q} k_pq (G_pq + d_p d_q / 3)^2,
//   f_p = dE_i/dr_p = sum_q M_pq r_q,  M_pp = 4 k_p (G_pp - d_p^2),  M_pq = 2 k_pq (G_pq + d_p d_q / 3),
// and the gradient of atom j along its bonds k to atoms n_k is -sum_k (f_k(j) - f_k(n_k)).  One kernel
// writes the 12 numbers f of every atom, a second gathers them (no atomics, a bit-reproducible
// result): 140 FP64 operations an atom, where gathering every term that touches an atom took some
// 900, 40 divisions by natural lengths among them; the constants of every species triple now come
// from a table in shared memory.  All of it is bound by the FP64 rate.  1M atoms, one iteration: gradient
// 1.46 ms before, 0.20 + 0.08 ms now; line coefficients 0.73 -> 0.42 ms (218 operations an atom); step 0.104 -> 0.008 ms (every
// block bisected the quartic); direction 0.032 -> 0.015 ms; 100 iterations 237 -> 75 ms.
// For the line search of the nonlinear conjugate-gradient relaxation, a kernel accumulates the
// coefficients of the energy along a search direction.  Every term is
// the square of a quadratic polynomial in the step t (r is affine in t), so E(u + t p) is a
// quartic whose derivative c1 + 2 c2 t + 3 c3 t^2 + 4 c4 t^3 is minimised exactly; c1 = g.p is
// accumulated term by term, so no energy difference (and no cancellation) enters the step.
#include <algorithm>
#include <chrono>
#include <cmath>

#include "neighbours.cuh"
#include "omen_internal.h"
#include "sk_device.cuh"

namespace {

constexpr int kThreads = 256;

// Constants of a vertex of species v: bond to species p {k_p, d_p^2}, angle between bonds to p and
// q {k_pq, d_p d_q / 3}.
struct VffTable {
  double2 bond[4][4];
  double2 angle[4][4][4];
};

struct VffArgs {
  Geo g;
  const uint8_t* species;
  double fd[4][3];            // F dir_k a/4: deformed ideal A->B vector of direction k (nm)
  double dnat[4];             // natural bond length sqrt(3)/4 a per species (nm)
  VffTable t;
};

// One atom's site, species and bonds (neighbour atoms; -1 where a bond leaves a hard wall).
struct Vertex {
  int sp;
  int nb[4];
  int sn[4];
  double sg;                  // A atoms sit at the tail of dir_k, B atoms at its head
};

__device__ __forceinline__ Vertex vertex_of(const VffArgs& a, int atom) {
  const Geo& g = a.g;
  const int b = atom / g.ncells, cell = atom - b * g.ncells;
  const int nxy = g.nx * g.ny;
  const int iz = cell / nxy, rem = cell - iz * nxy, iy = rem / g.nx, ix = rem - iy * g.nx;
  const Steps steps = steps_of(g, b, ix, iy, iz);
  Vertex v;
  v.sp = a.species[atom];
  v.sg = b < 4 ? 1.0 : -1.0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const Neighbour n = neighbour_of(g, steps, b, k, cell);
    v.nb[k] = n.ok ? n.atom : -1;
    v.sn[k] = n.ok ? a.species[n.atom] : 0;
  }
  return v;
}

__device__ __forceinline__ void load3(const double* __restrict__ v, long long n, int i, double out[3]) {
  out[0] = v[i];
  out[1] = v[n + i];
  out[2] = v[2 * n + i];
}

__device__ __forceinline__ double dot3(const double x[3], const double y[3]) {
  return fma(x[2], y[2], fma(x[1], y[1], x[0] * y[0]));
}
// c + x.y
__device__ __forceinline__ double dot3(double c, const double x[3], const double y[3]) {
  return fma(x[2], y[2], fma(x[1], y[1], fma(x[0], y[0], c)));
}

// Bond vectors of a vertex at displacements u ([3][natoms]); zero for absent bonds.
__device__ __forceinline__ void bond_vectors(const VffArgs& a, const Vertex& v, const double* __restrict__ u, int atom,
                                             double (&r)[4][3]) {
  const long long N = a.g.natoms;
  double ui[3];
  load3(u, N, atom, ui);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    double un[3] = {0.0, 0.0, 0.0};
    if (v.nb[k] >= 0) load3(u, N, v.nb[k], un);
#pragma unroll
    for (int c = 0; c < 3; ++c) r[k][c] = v.nb[k] >= 0 ? (v.sg * a.fd[k][c] - ui[c]) + un[c] : 0.0;
  }
}

// Constants of the pair of bonds (p, q) of a vertex; k = 0 where one of them is absent.
__device__ __forceinline__ double2 pair_of(const VffTable& t, const Vertex& v, int p, int q) {
  double2 k = p == q ? t.bond[v.sp][v.sn[p]] : t.angle[v.sp][v.sn[p]][v.sn[q]];
  if (v.nb[p] < 0 || v.nb[q] < 0) k.x = 0.0;
  return k;
}

// The table to shared memory, k of the bonds and of the angles times a factor.
__device__ __forceinline__ void stage_table(const VffTable& t, VffTable& sm, double bond = 1.0, double angle = 1.0) {
  const double2* src = reinterpret_cast<const double2*>(&t);
  double2* dst = reinterpret_cast<double2*>(&sm);
  for (int i = threadIdx.x; i < (int)(sizeof(VffTable) / sizeof(double2)); i += blockDim.x)
    dst[i] = make_double2((i < 16 ? bond : angle) * src[i].x, src[i].y);
  __syncthreads();
}

// Relaxation state on the device (one small record).
struct VffState {
  double t;          // last step length
  double gg;         // g.g of the current gradient
  double beta;       // of the next direction
  double gmax;       // max |g_c| of the current gradient
  int restart;       // the last direction was not a descent direction: next direction is -g
  unsigned arrived;  // blocks of the running reduction that have left their sums
};

// Deterministic block sums of NV values per thread into partial[v * nblocks + block]; with
// MAX_LAST the last value is reduced by max instead of sum.
template <int NV, bool MAX_LAST>
__device__ __forceinline__ void block_reduce(double (&v)[NV], double* __restrict__ partial) {
  __shared__ double sm[NV][kThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    double x = v[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double y = __shfl_down_sync(0xffffffffu, x, o);
      x = (MAX_LAST && q == NV - 1) ? fmax(x, y) : x + y;
    }
    if (lane == 0) sm[q][w] = x;
  }
  __syncthreads();
  if (threadIdx.x < NV) {
    const int q = threadIdx.x;
    double x = sm[q][0];
    for (int i = 1; i < kThreads / 32; ++i) x = (MAX_LAST && q == NV - 1) ? fmax(x, sm[q][i]) : x + sm[q][i];
    partial[(size_t)q * gridDim.x + blockIdx.x] = x;
  }
}

// The last block to leave its partials reduces all of them in block order: v valid in thread 0 of
// that block, which alone gets true.
template <int NV, bool MAX_LAST>
__device__ __forceinline__ bool grid_reduce(double (&v)[NV], double* partial, VffState* st) {
  __shared__ bool last;
  block_reduce<NV, MAX_LAST>(v, partial);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&st->arrived, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return false;
  __threadfence();
  __shared__ double sm[NV][kThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    const bool mx = MAX_LAST && q == NV - 1;
    double x = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += kThreads) {
      const double y = __ldcg(partial + (size_t)q * gridDim.x + i);
      x = mx ? fmax(x, y) : x + y;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double y = __shfl_down_sync(0xffffffffu, x, o);
      x = mx ? fmax(x, y) : x + y;
    }
    if (lane == 0) sm[q][w] = x;
  }
  __syncthreads();
  if (threadIdx.x != 0) return false;
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    v[q] = sm[q][0];
    for (int i = 1; i < kThreads / 32; ++i) v[q] = (MAX_LAST && q == NV - 1) ? fmax(v[q], sm[q][i]) : v[q] + sm[q][i];
  }
  st->arrived = 0;
  return true;
}

// f_k = dE_i/dr_k of every atom: f[(3 k + c) natoms + atom].
__global__ void __launch_bounds__(kThreads) vff_vertex_kernel(const __grid_constant__ VffArgs a, const double* __restrict__ u,
                                                              double* __restrict__ f) {
  __shared__ VffTable t;
  stage_table(a.t, t, 4.0, 2.0);
  const long long N = a.g.natoms;
  const int atom = blockIdx.x * blockDim.x + threadIdx.x;
  if (atom >= N) return;
  const Vertex v = vertex_of(a, atom);
  double r[4][3], fk[4][3];
  bond_vectors(a, v, u, atom, r);
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const double2 k = pair_of(t, v, p, p);
    const double m = k.x * dot3(-k.y, r[p], r[p]);
#pragma unroll
    for (int c = 0; c < 3; ++c) fk[p][c] = m * r[p][c];
  }
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = p + 1; q < 4; ++q) {
      const double2 k = pair_of(t, v, p, q);
      const double m = k.x * dot3(k.y, r[p], r[q]);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        fk[p][c] = fma(m, r[q][c], fk[p][c]);
        fk[q][c] = fma(m, r[p][c], fk[q][c]);
      }
    }
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int c = 0; c < 3; ++c) f[(3 * k + c) * N + atom] = fk[k][c];
}

// Gradient (times `sign`) from the vertices' f.  With a state: g.g, g.g_prev (0 if g_prev is null)
// and max |g_c| over the structure, and from them beta of the next direction p = -g + beta p
// (Polak–Ribière, clipped at 0; 0 on the first iteration or after a restart).
__global__ void __launch_bounds__(kThreads) vff_gather_kernel(const __grid_constant__ VffArgs a, const double* __restrict__ f,
                                                              double* __restrict__ g, const double* __restrict__ g_prev,
                                                              double sign, double* partial, VffState* st) {
  const long long N = a.g.natoms;
  double acc[3] = {0.0, 0.0, 0.0};
  const int flip = sign < 0.0 ? 0x80000000 : 0;
  long long gmax = 0;
  for (int atom = blockIdx.x * blockDim.x + threadIdx.x; atom < N; atom += gridDim.x * blockDim.x) {
    const Vertex v = vertex_of(a, atom);
    double gi[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (v.nb[k] < 0) continue;                     // f_k of an absent bond is zero
      double own[3], back[3];
      load3(f + 3 * k * N, N, atom, own);
      load3(f + 3 * k * N, N, v.nb[k], back);
#pragma unroll
      for (int c = 0; c < 3; ++c) gi[c] += back[c] - own[c];
    }
    double gp[3] = {0.0, 0.0, 0.0};
    if (g_prev) load3(g_prev, N, atom, gp);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      // the sign and the largest |g_c| on the integer pipe (a NaN compares as the largest)
      g[c * N + atom] = __hiloint2double(__double2hiint(gi[c]) ^ flip, __double2loint(gi[c]));
      acc[0] = fma(gi[c], gi[c], acc[0]);
      acc[1] = fma(gi[c], gp[c], acc[1]);
      gmax = max(gmax, __double_as_longlong(gi[c]) & 0x7fffffffffffffffll);
    }
  }
  if (!st) return;
  acc[2] = __longlong_as_double(gmax);
  if (grid_reduce<3, true>(acc, partial, st)) {
    double beta = 0.0;
    if (g_prev && !st->restart && st->gg > 0.0) beta = fmax(0.0, (acc[0] - acc[1]) / st->gg);
    st->beta = beta;
    st->gg = acc[0];
    // fmax drops a NaN: the sum of squares carries it
    st->gmax = acc[0] == acc[0] ? acc[2] : acc[0];
  }
}

// Energy of every vertex.
__global__ void __launch_bounds__(kThreads) vff_energy_kernel(const __grid_constant__ VffArgs a, const double* __restrict__ u,
                                                              double* __restrict__ partial) {
  __shared__ VffTable t;
  stage_table(a.t, t);
  const long long N = a.g.natoms;
  double acc[1] = {0.0};
  for (int atom = blockIdx.x * blockDim.x + threadIdx.x; atom < N; atom += gridDim.x * blockDim.x) {
    const Vertex v = vertex_of(a, atom);
    double r[4][3];
    bond_vectors(a, v, u, atom, r);
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = p; q < 4; ++q) {
        const double2 k = pair_of(t, v, p, q);
        const double x = dot3(p == q ? -k.y : k.y, r[p], r[q]);
        acc[0] = fma(k.x * x, x, acc[0]);
      }
  }
  block_reduce<1, false>(acc, partial);
}

// Step length minimising the quartic along the line: the first sign change of its derivative
// c1 + 2 c2 t + 3 c3 t^2 + 4 c4 t^3 (c1 < 0) bracketed by doubling, then Newton's method kept
// inside the bracket (bisection where it leaves it), to rounding.
__device__ double quartic_step(double c1, double c2, double c3, double c4) {
  if (!(c1 < 0.0)) return 0.0;
  auto dE = [&](double t) { return c1 + t * (2.0 * c2 + t * (3.0 * c3 + t * 4.0 * c4)); };
  double hi = c2 > 0.0 ? -c1 / (2.0 * c2) : 1e-6;
  int n = 0;
  while (!(dE(hi) > 0.0) && n < 400) {
    hi *= 2.0;
    ++n;
  }
  if (!(dE(hi) > 0.0)) return 0.0;                 // no minimum along the line: restart
  double lo = 0.0, t = n ? 0.5 * hi : hi;
  for (int i = 0; i < 200 && hi - lo > 1e-16 * hi; ++i) {
    const double d = dE(t);
    if (d > 0.0) hi = t; else lo = t;
    const double slope = 2.0 * c2 + t * (6.0 * c3 + t * 12.0 * c4);
    double next = t - d / slope;
    if (!(next > lo && next < hi)) next = 0.5 * (lo + hi);
    if (fabs(next - t) <= 1e-16 * t) break;
    t = next;
  }
  return t;
}

// Coefficients c1..c4 of E(u + t p) - E(u) = c1 t + c2 t^2 + c3 t^3 + c4 t^4, and the step they
// give.  A term K (q0 + q1 t + q2 t^2)^2 contributes 2K q0 q1, K (q1^2 + 2 q0 q2), 2K q1 q2, K q2^2.
__global__ void __launch_bounds__(kThreads) vff_line_kernel(const __grid_constant__ VffArgs a, const double* __restrict__ u,
                                                            const double* __restrict__ p, double* partial, VffState* st) {
  __shared__ VffTable t;
  stage_table(a.t, t);
  const long long N = a.g.natoms;
  // sums of K q0 q1, K q1^2, K q0 q2, K q1 q2, K q2^2
  double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  for (int atom = blockIdx.x * blockDim.x + threadIdx.x; atom < N; atom += gridDim.x * blockDim.x) {
    const Vertex v = vertex_of(a, atom);
    double r[4][3], s[4][3], pi[3];                  // bond vectors and their change per unit step
    bond_vectors(a, v, u, atom, r);
    load3(p, N, atom, pi);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      double pn[3] = {pi[0], pi[1], pi[2]};
      if (v.nb[k] >= 0) load3(p, N, v.nb[k], pn);
#pragma unroll
      for (int c = 0; c < 3; ++c) s[k][c] = pn[c] - pi[c];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int q = i; q < 4; ++q) {
        const double2 k = pair_of(t, v, i, q);
        const double q0 = dot3(i == q ? -k.y : k.y, r[i], r[q]);
        const double q1 = i == q ? 2.0 * dot3(r[i], s[i]) : dot3(dot3(r[i], s[q]), s[i], r[q]);
        const double q2 = dot3(s[i], s[q]);
        const double k1 = k.x * q1, k2 = k.x * q2;
        acc[0] = fma(k1, q0, acc[0]);
        acc[1] = fma(k1, q1, acc[1]);
        acc[2] = fma(k2, q0, acc[2]);
        acc[3] = fma(k2, q1, acc[3]);
        acc[4] = fma(k2, q2, acc[4]);
      }
  }
  double c[4] = {acc[0], fma(2.0, acc[2], acc[1]), acc[3], acc[4]};   // c1 / 2, c2, c3 / 2, c4
  if (grid_reduce<4, false>(c, partial, st)) {
    const double c1 = 2.0 * c[0];
    const double step = quartic_step(c1, c[1], 2.0 * c[2], c[3]);
    st->t = step;
    st->restart = step > 0.0 ? 0 : 1;
  }
}

// u += t p with the step of the line kernel.
__global__ void __launch_bounds__(kThreads) vff_step_kernel(double* __restrict__ u, const double* __restrict__ p,
                                                            long long n3, const VffState* __restrict__ st) {
  const double t = st->t;
  if (t == 0.0) return;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n3; i += (long long)gridDim.x * blockDim.x)
    u[i] = fma(t, p[i], u[i]);
}

// New direction p = -g + beta p.
__global__ void __launch_bounds__(kThreads) vff_dir_kernel(const double* __restrict__ g, double* __restrict__ p,
                                                           long long n3, const VffState* __restrict__ st, int first) {
  const double beta = st->beta;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n3; i += (long long)gridDim.x * blockDim.x)
    p[i] = first ? -g[i] : fma(beta, p[i], -g[i]);
}

__global__ void vff_strain_kernel(VffArgs a, const double* __restrict__ u, double* __restrict__ strain) {
  const long long nslots = 16ll * a.g.ncells;
  const long long N = a.g.natoms;
  for (long long sl = blockIdx.x * (long long)blockDim.x + threadIdx.x; sl < nslots; sl += (long long)gridDim.x * blockDim.x) {
    const int ks = (int)(sl / a.g.ncells);
    const int cell = (int)(sl - (long long)ks * a.g.ncells);
    const int k = ks >> 2, s = ks & 3;
    const int atom = s * a.g.ncells + cell;
    const int nxy = a.g.nx * a.g.ny;
    const int iz = cell / nxy, rem = cell - iz * nxy, iy = rem / a.g.nx, ix = rem - iy * a.g.nx;
    const Neighbour to = neighbour_of(a.g, steps_of(a.g, s, ix, iy, iz), s, k, cell);
    const int n = to.atom;
    if (!to.ok) {
      strain[sl] = 0.0;
      continue;
    }
    double ui[3], un[3], r[3];
    load3(u, N, atom, ui);
    load3(u, N, n, un);
#pragma unroll
    for (int c = 0; c < 3; ++c) r[c] = a.fd[k][c] + un[c] - ui[c];
    const double d = 0.5 * (a.dnat[a.species[atom]] + a.dnat[a.species[n]]);
    strain[sl] = sqrt(dot3(r, r)) / d - 1.0;
  }
}

omen_status make_args(omen_ctx* ctx, const omen_lattice* L, const omen_vff_params* vp, const double* F, VffArgs& a) {
  if (!vp) return set_err(ctx, OMEN_EINVAL, "null VFF parameters");
  if (vp->nspecies < 1 || vp->nspecies > 4) return set_err(ctx, OMEN_EINVAL, "nspecies must be 1..4");
  for (int s = 0; s < vp->nspecies; ++s)
    if (!(vp->a_nm[s] > 0) || !(vp->alpha[s] >= 0) || !(vp->beta[s] >= 0))
      return set_err(ctx, OMEN_EINVAL, "species %d: a_nm must be > 0 and alpha, beta >= 0", s);
  // the kernels look the constants up in a table of four species
  if (L->max_species > 3) return set_err(ctx, OMEN_EINVAL, "species index %d: at most 4 species", L->max_species);
  a.g.nx = L->nx; a.g.ny = L->ny; a.g.nz = L->nz;
  a.g.ncells = L->ncells; a.g.natoms = L->natoms;
  for (int d = 0; d < 3; ++d) a.g.periodic[d] = L->periodic[d];
  a.species = L->d_species;
  static const int dir[4][3] = {{1, 1, 1}, {1, -1, -1}, {-1, 1, -1}, {-1, -1, 1}};
  const double q4 = 0.25 * L->a_nm;
  for (int k = 0; k < 4; ++k)
    for (int r = 0; r < 3; ++r) {
      double x = 0.0;
      for (int c = 0; c < 3; ++c) x += (F ? F[r * 3 + c] : (r == c ? 1.0 : 0.0)) * dir[k][c];
      a.fd[k][r] = x * q4;
    }
  double alpha[4], beta[4];
  for (int s = 0; s < 4; ++s) {
    const int t = s < vp->nspecies ? s : 0;
    a.dnat[s] = 0.25 * std::sqrt(3.0) * vp->a_nm[t];
    alpha[s] = vp->alpha[t];
    beta[s] = vp->beta[t];
  }
  for (int v = 0; v < 4; ++v)
    for (int p = 0; p < 4; ++p) {
      const double dp = 0.5 * (a.dnat[v] + a.dnat[p]), bp = 0.5 * (beta[v] + beta[p]);
      a.t.bond[v][p] = make_double2(0.5 * 0.375 * 0.5 * (alpha[v] + alpha[p]) / (dp * dp), dp * dp);
      for (int q = 0; q < 4; ++q) {
        const double dd = dp * 0.5 * (a.dnat[v] + a.dnat[q]), bq = 0.5 * (beta[v] + beta[q]);
        a.t.angle[v][p][q] = make_double2(0.375 * 0.5 * (bp + bq) / dd, dd / 3.0);
      }
    }
  return OMEN_OK;
}

int reduce_blocks(omen_ctx* ctx, long long n) {
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
  const long long want = (n + kThreads - 1) / kThreads;
  return (int)std::max<long long>(1, std::min<long long>(want, 4ll * std::max(1, sms)));
}

unsigned blocks_of(long long n) { return (unsigned)((n + kThreads - 1) / kThreads); }

// Host sum of the partials of one row, in block order.
double host_sum(const std::vector<double>& h, int q, int nb, bool take_max = false) {
  double s = 0.0;
  for (int i = 0; i < nb; ++i) s = take_max ? std::max(s, h[(size_t)q * nb + i]) : s + h[(size_t)q * nb + i];
  return s;
}

}  // namespace

extern "C" omen_status omen_vff_energy_forces(omen_ctx* ctx, const omen_lattice* L, const omen_vff_params* vp,
                                              const double* F_host, const double* u_dev, double* E_host,
                                              double* force_dev) {
  if (!ctx || !L || !u_dev) return set_err(ctx, OMEN_EINVAL, "null argument");
  VffArgs a;
  omen_status s = make_args(ctx, L, vp, F_host, a);
  if (s != OMEN_OK) return s;
  const long long N = L->natoms;
  const int nb = reduce_blocks(ctx, N);
  if ((size_t)4 * nb * sizeof(double) > ctx->work_bytes) return set_err(ctx, OMEN_EINVAL, "work area too small");
  double* part = ctx->d_work;
  std::vector<double> h((size_t)3 * nb);
  if (force_dev) {
    double* f = nullptr;
    if (ctx_alloc(ctx, &f, sizeof(double) * 12 * (size_t)N) != cudaSuccess) {
      cudaGetLastError();
      return set_err(ctx, OMEN_ENOMEM, "VFF work vectors");
    }
    vff_vertex_kernel<<<blocks_of(N), kThreads, 0, ctx->stream>>>(a, u_dev, f);
    // force = -dE/du
    vff_gather_kernel<<<nb, kThreads, 0, ctx->stream>>>(a, f, force_dev, nullptr, -1.0, nullptr, nullptr);
    const cudaError_t e = cudaGetLastError();
    cudaFreeAsync(f, ctx->stream);
    if (e != cudaSuccess) return set_err(ctx, OMEN_ECUDA, "VFF forces: %s", cudaGetErrorString(e));
  }
  if (E_host) {
    vff_energy_kernel<<<nb, kThreads, 0, ctx->stream>>>(a, u_dev, part);
    OMEN_CHECK_LAUNCH(ctx);
    OMEN_CUDA(ctx, cudaMemcpyAsync(h.data(), part, sizeof(double) * nb, cudaMemcpyDeviceToHost, ctx->stream));
  }
  OMEN_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  if (E_host) *E_host = host_sum(h, 0, nb);
  return OMEN_OK;
}

extern "C" omen_status omen_relax_vff(omen_ctx* ctx, const omen_lattice* L, const omen_vff_params* vp,
                                      const double* F_host, const omen_vff_opts* o, double* u_dev, double* strain_dev,
                                      omen_vff_info* info) {
  if (!ctx || !L || !o || !u_dev) return set_err(ctx, OMEN_EINVAL, "null argument");
  if (!(o->gtol > 0) || o->max_iter < 0) return set_err(ctx, OMEN_EINVAL, "gtol must be > 0 and max_iter >= 0");
  const auto t0 = std::chrono::steady_clock::now();
  VffArgs a;
  omen_status s = make_args(ctx, L, vp, F_host, a);
  if (s != OMEN_OK) return s;
  const long long N = L->natoms, n3 = 3 * N;
  const int nb = reduce_blocks(ctx, N);
  const int check = 10;                                 // iterations between host convergence checks
  // work: two gradients (ping-pong), the direction, the vertices' f, partials of the gradient (3
  // rows) and of the line coefficients (4 rows), and the state record
  const size_t bytes = sizeof(double) * (7 * (size_t)n3 + 7 * (size_t)nb) + sizeof(VffState);
  char* buf = nullptr;
  if (ctx_alloc(ctx, &buf, bytes) != cudaSuccess) {
    cudaGetLastError();
    return set_err(ctx, OMEN_ENOMEM, "VFF work vectors (%zu bytes)", bytes);
  }
  double* g[2] = {reinterpret_cast<double*>(buf), reinterpret_cast<double*>(buf) + n3};
  double* p = g[1] + n3;
  double* f = p + n3;
  double* gpart = f + 4 * n3;
  double* lpart = gpart + 3 * (size_t)nb;
  VffState* st = reinterpret_cast<VffState*>(lpart + 4 * (size_t)nb);
  std::vector<double> h((size_t)nb);
  VffState hs{};
  cudaError_t e = cudaMemsetAsync(st, 0, sizeof(VffState), ctx->stream);
  double E0 = 0.0;
  if (e == cudaSuccess) {
    vff_energy_kernel<<<nb, kThreads, 0, ctx->stream>>>(a, u_dev, gpart);
    e = cudaMemcpyAsync(h.data(), gpart, sizeof(double) * nb, cudaMemcpyDeviceToHost, ctx->stream);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  if (e == cudaSuccess) E0 = host_sum(h, 0, nb);
  int cur = 0, it = 0;
  bool converged = false;
  if (e == cudaSuccess) {
    vff_vertex_kernel<<<blocks_of(N), kThreads, 0, ctx->stream>>>(a, u_dev, f);
    vff_gather_kernel<<<nb, kThreads, 0, ctx->stream>>>(a, f, g[cur], nullptr, 1.0, gpart, st);
    vff_dir_kernel<<<nb, kThreads, 0, ctx->stream>>>(g[cur], p, n3, st, 1);
    e = cudaGetLastError();
  }
  while (e == cudaSuccess) {
    if (it % check == 0 || it == o->max_iter) {
      e = cudaMemcpyAsync(&hs, st, sizeof(VffState), cudaMemcpyDeviceToHost, ctx->stream);
      if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
      if (e != cudaSuccess) break;
      if (!std::isfinite(hs.gmax)) break;
      if (hs.gmax < o->gtol) {
        converged = true;
        break;
      }
      if (it == o->max_iter) break;
    }
    vff_line_kernel<<<nb, kThreads, 0, ctx->stream>>>(a, u_dev, p, lpart, st);
    vff_step_kernel<<<nb, kThreads, 0, ctx->stream>>>(u_dev, p, n3, st);
    vff_vertex_kernel<<<blocks_of(N), kThreads, 0, ctx->stream>>>(a, u_dev, f);
    vff_gather_kernel<<<nb, kThreads, 0, ctx->stream>>>(a, f, g[cur ^ 1], g[cur], 1.0, gpart, st);
    cur ^= 1;
    ++it;
    vff_dir_kernel<<<nb, kThreads, 0, ctx->stream>>>(g[cur], p, n3, st, 0);
    e = cudaGetLastError();
  }
  double E1 = 0.0;
  if (e == cudaSuccess) {
    vff_energy_kernel<<<nb, kThreads, 0, ctx->stream>>>(a, u_dev, gpart);
    e = cudaMemcpyAsync(h.data(), gpart, sizeof(double) * nb, cudaMemcpyDeviceToHost, ctx->stream);
  }
  if (e == cudaSuccess && strain_dev) {
    const long long nslots = 16ll * L->ncells;
    const int sb = (int)std::min<long long>((nslots + kThreads - 1) / kThreads, 65535);
    vff_strain_kernel<<<sb, kThreads, 0, ctx->stream>>>(a, u_dev, strain_dev);
    e = cudaGetLastError();
  }
  cudaFreeAsync(buf, ctx->stream);
  const cudaError_t e2 = cudaStreamSynchronize(ctx->stream);
  if (e != cudaSuccess || e2 != cudaSuccess)
    return set_err(ctx, OMEN_ECUDA, "VFF relaxation: %s", cudaGetErrorString(e != cudaSuccess ? e : e2));
  E1 = host_sum(h, 0, nb);
  if (info) {
    info->iterations = it;
    info->converged = converged ? 1 : 0;
    info->energy_start = E0;
    info->energy = E1;
    info->max_force = hs.gmax;
    info->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  }
  if (!std::isfinite(hs.gmax) || !std::isfinite(E1))
    return set_err(ctx, OMEN_ENUMERIC, "VFF relaxation produced a non-finite force or energy");
  if (!converged)
    return set_err(ctx, OMEN_ENOCONV, "VFF relaxation stopped at %d iterations, max force %.3e eV/nm", it, hs.gmax);
  return OMEN_OK;
}
