// Charge from eigenstates, grid deposit and gather, Fermi level (paper Section III-A item 2:
// the charge profile from filling the states at a given Fermi level, or charge and Fermi level
// together under charge neutrality).
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "omen_internal.h"
#include "sk_device.cuh"
#include "vec.cuh"
#include "cic.cuh"
#include "param_copy.cuh"
#include "df.cuh"

// n_atom[i] += w * sum_n occ[n] * sum_o |psi_n[o*N + i]|^2
//
// The squares are summed on the FP32 pipe in double-float arithmetic (GB300's FP64 rate would
// otherwise bound the kernel, one FP64 FMA per 8-byte amplitude).  Each FP64 amplitude v is
// split, scaled by 2^32 (exact), into FP32 parts with integer operations only: hi keeps the
// sign, the exponent and the leading 24 significant bits, lo is the rest rounded to FP32 (48
// significant bits in all).  v^2 2^64 is then hi^2 (the FP32 product plus its exact FMA error)
// + 2 hi lo + lo^2, the terms added with TwoSum into an FP32 pair (about 1e-14 relative).  The
// scaling keeps amplitudes in [2^-83, 2^32) clear of FP32 underflow and overflow; smaller ones
// (contributing below 2^-166) count as zero, and so do occupations below 2^-126.  Infinite or
// NaN amplitudes (and finite ones of 2^96 or more) give NaN.
__device__ __forceinline__ void df_add_square(float& S, float& Cc, double v) {
  const float2 h = split_fp64<32>(v);
  const float p = __fmul_rn(h.x, h.x);
  float e = __fmaf_rn(h.x, h.x, -p);
  e = __fmaf_rn(__fmul_rn(2.f, h.x), h.y, e);
  e = __fmaf_rn(h.y, h.y, e);
  const float s = __fadd_rn(S, p);
  const float bb = __fsub_rn(s, S);
  const float t = __fadd_rn(__fsub_rn(S, __fsub_rn(s, bb)), __fsub_rn(p, bb));
  Cc = __fadd_rn(Cc, __fadd_rn(t, e));
  S = s;
}

// Occupations of a few states travel with the launch, more of them in device memory.
constexpr int kInlineStates = 64;
struct OccInline {
  double f[kInlineStates];
};

template <bool C, int NB>
__global__ void __launch_bounds__(256) density_kernel(const void* __restrict__ psiv, long long nrows, int natoms,
                                                      int nb_rt, int nstates, const __grid_constant__ OccInline few,
                                                      const double* __restrict__ many, double w,
                                                      double* __restrict__ n_atom) {
  using E = Elem<double, C>;
  const typename E::V* psi = static_cast<const typename E::V*>(psiv);
  const int nb = NB > 0 ? NB : nb_rt;
  const double* occ = many ? many : few.f;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < natoms; i += gridDim.x * blockDim.x) {
    float AS = 0.f, AC = 0.f;   // sum over states of occ * (state's sum of squares)
    for (int s = 0; s < nstates; ++s) {
      const double f = occ[s];
      if (f == 0.0) continue;
      const typename E::V* ps = psi + (size_t)s * nrows + i;
      float S = 0.f, Cc = 0.f;
      if constexpr (NB > 0) {
        typename E::V v[NB];
#pragma unroll
        for (int o = 0; o < NB; ++o) v[o] = ps[(size_t)o * natoms];
#pragma unroll
        for (int o = 0; o < NB; ++o) {
          df_add_square(S, Cc, E::re(v[o]));
          if constexpr (C) df_add_square(S, Cc, E::im(v[o]));
        }
      } else {
        for (int o = 0; o < nb; ++o) {
          const typename E::V v = ps[(size_t)o * natoms];
          df_add_square(S, Cc, E::re(v));
          if constexpr (C) df_add_square(S, Cc, E::im(v));
        }
      }
      df_mac(AS, AC, df_norm(S, Cc), split_fp64<0>(f));
    }
    // the squares carry the factor 2^64 of the split
    n_atom[i] += w * (((double)AS + (double)AC) * 0x1p-64);
  }
}

// The atoms' coordinates along one axis are the quarter cells Q a/4, Q = 0 .. 4 n - 1, so the
// cloud-in-cell position of every atom is a look-up: node below, and weight of the node above.
struct AxisTable {
  double* f;      // [nq] weight of the node above
  int* node;      // [nq] node below, wrapped on the periodic axes
  double h;       // grid spacing (nm)
  int nq, wrap;   // wrap: nodes of a periodic axis, 0 for z
};

__global__ void axis_tables_kernel(AxisTable ax, AxisTable ay, AxisTable az, double quarter) {
  const AxisTable& A = blockIdx.y == 0 ? ax : blockIdx.y == 1 ? ay : az;
  const int Q = blockIdx.x * blockDim.x + threadIdx.x;
  if (Q >= A.nq) return;
  const double t = (Q * quarter) / A.h;
  const int node = (int)floor(t);
  A.f[Q] = t - node;
  A.node[Q] = A.wrap ? node % A.wrap : node;
}

// Cloud-in-cell place of one atom from the axis tables.
struct Place {
  int i0, i1, j0, j1, k0;
  double fx, fy, fz;
};

__device__ __forceinline__ Place place_of(const Geo& g, const AxisTable& X, const AxisTable& Y, const AxisTable& Z, int atom) {
  const int b = atom / g.ncells, cell = atom - b * g.ncells;
  const int nxy = g.nx * g.ny;
  const int iz = cell / nxy, rem = cell - iz * nxy, iy = rem / g.nx, ix = rem - iy * g.nx;
  const int s = b & 3, o = b >> 2;                       // sites (000) (022) (202) (220), B those plus (111)
  const int Qx = 4 * ix + (s & 2) + o, Qy = 4 * iy + 2 * (s & 1) + o, Qz = 4 * iz + 2 * ((s ^ (s >> 1)) & 1) + o;
  Place p;
  p.fx = X.f[Qx];
  p.fy = Y.f[Qy];
  p.fz = Z.f[Qz];
  p.i0 = X.node[Qx];
  p.j0 = Y.node[Qy];
  p.k0 = Z.node[Qz];
  p.i1 = p.i0 + 1 == X.wrap ? 0 : p.i0 + 1;
  p.j1 = p.j0 + 1 == Y.wrap ? 0 : p.j0 + 1;
  return p;
}

// Deposit straight into the (cleared) density, already divided by the cell volume; nodes on the
// grounded planes take nothing.  Both kernels were bound by the FP64 rate: three divisions, three
// floors and the weights of 8 nodes an atom, on a pipe of 1/64 the FP32 rate; the tables leave 15
// (gather 14) FP64 operations.  1M atoms on 256^3: deposit 128 us of atomics + 22 us clearing +
// 41 us copying out of a padded node array before, 53 + 21 us now (a kernel by node without atomics
// took 292 us: most lanes of its FP64 instructions idle).
__global__ void __launch_bounds__(256) deposit_kernel(Geo g, AxisTable X, AxisTable Y, AxisTable Z, int nz,
                                                      const double* __restrict__ q, double inv_vol, double* __restrict__ rho) {
  const int atom = blockIdx.x * blockDim.x + threadIdx.x;
  if (atom >= g.natoms) return;
  const double qi = q[atom] * inv_vol;
  if (qi == 0.0) return;
  const Place p = place_of(g, X, Y, Z, atom);
  const double qz1 = qi * p.fz, qz0 = qi - qz1;
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    const int k = p.k0 + d;
    if (k < 1 || k > nz - 1) continue;
    const double qz = d ? qz1 : qz0, qy1 = qz * p.fy, qy0 = qz - qy1;
    const double a = qy0 * p.fx, c = qy1 * p.fx;
    double* r0 = rho + ((long long)(k - 1) * Y.wrap + p.j0) * X.wrap;
    double* r1 = rho + ((long long)(k - 1) * Y.wrap + p.j1) * X.wrap;
    atomicAdd(r0 + p.i0, qy0 - a);
    atomicAdd(r0 + p.i1, a);
    atomicAdd(r1 + p.i0, qy1 - c);
    atomicAdd(r1 + p.i1, c);
  }
}

// Trilinear interpolation at every atom.  1M atoms on 256^3: 124 us before, 32 us now.
__global__ void __launch_bounds__(256) gather_kernel(Geo g, AxisTable X, AxisTable Y, AxisTable Z, int nz,
                                                     const double* __restrict__ phi, double* __restrict__ out) {
  const int atom = blockIdx.x * blockDim.x + threadIdx.x;
  if (atom >= g.natoms) return;
  const Place p = place_of(g, X, Y, Z, atom);
  double v[2];
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    const int k = p.k0 + d;
    double p00 = 0.0, p01 = 0.0, p10 = 0.0, p11 = 0.0;
    if (k >= 1 && k <= nz - 1) {
      const double* __restrict__ r0 = phi + ((long long)(k - 1) * Y.wrap + p.j0) * X.wrap;
      const double* __restrict__ r1 = phi + ((long long)(k - 1) * Y.wrap + p.j1) * X.wrap;
      p00 = r0[p.i0];
      p01 = r0[p.i1];
      p10 = r1[p.i0];
      p11 = r1[p.i1];
    }
    const double a = fma(p.fx, p01 - p00, p00), c = fma(p.fx, p11 - p10, p10);
    v[d] = fma(p.fy, c - a, a);
  }
  out[atom] = fma(p.fz, v[1] - v[0], v[0]);
}

// The three axis tables of a structure on a grid, in one buffer on the context's stream.
static omen_status make_tables(omen_ctx* ctx, const omen_lattice* L, const GridGeo& G, AxisTable (&t)[3], char** buf) {
  const int nc[3] = {L->nx, L->ny, L->nz}, wrap[3] = {G.nx, G.ny, 0};
  const double h[3] = {G.hx, G.hy, G.hz};
  size_t n = 0;
  for (int c : nc) n += 4 * (size_t)c;
  if (ctx_alloc(ctx, buf, n * (sizeof(double) + sizeof(int))) != cudaSuccess) {
    cudaGetLastError();
    return set_err(ctx, OMEN_ENOMEM, "interpolation tables");
  }
  double* f = reinterpret_cast<double*>(*buf);
  int* node = reinterpret_cast<int*>(f + n);
  int most = 0;
  for (int d = 0; d < 3; ++d) {
    t[d] = AxisTable{f, node, h[d], 4 * nc[d], wrap[d]};
    f += 4 * nc[d];
    node += 4 * nc[d];
    most = std::max(most, 4 * nc[d]);
  }
  axis_tables_kernel<<<dim3((most + 127) / 128, 3), 128, 0, ctx->stream>>>(t[0], t[1], t[2], 0.25 * L->a_nm);
  return OMEN_OK;
}

extern "C" omen_status omen_density_accum(omen_ctx* ctx, const omen_ham* h, const void* psi, int nstates,
                                          const double* occ_host, double w, double* n_atom) {
  if (!ctx || !h || !psi || !occ_host || !n_atom || nstates < 0) return set_err(ctx, OMEN_EINVAL, "null argument");
  if (nstates == 0) return OMEN_OK;
  double* d_occ = nullptr;
  OccInline few{};
  if (nstates <= kInlineStates) {
    std::copy(occ_host, occ_host + nstates, few.f);
  } else {
    if (ctx_alloc(ctx, &d_occ, sizeof(double) * nstates) != cudaSuccess) {
      cudaGetLastError();
      return set_err(ctx, OMEN_ENOMEM, "occupations");
    }
    const cudaError_t e = copy_as_params(ctx->stream, d_occ, occ_host, sizeof(double) * nstates);
    if (e != cudaSuccess) {
      cudaFreeAsync(d_occ, ctx->stream);
      return set_err(ctx, OMEN_ECUDA, "occupations: %s", cudaGetErrorString(e));
    }
  }
  const int N = (int)(h->nrows / h->nb);   // atoms, or grid points of an effective-mass Hamiltonian
  // one atom a thread: a grid cut to whole waves left its last round a fifth full at 1M atoms
  // (0.259 ms for 16 states, 0.228 ms now: 83% of the HBM copy rate)
  const unsigned grid = (unsigned)std::max(1, (N + 255) / 256);
  auto launch = [&](auto cplx, auto nbc) {
    constexpr bool Cx = decltype(cplx)::value;
    constexpr int NB = decltype(nbc)::value;
    density_kernel<Cx, NB><<<grid, 256, 0, ctx->stream>>>(psi, h->nrows, N, h->nb, nstates, few, d_occ, w, n_atom);
  };
  using T_ = std::true_type;
  using F_ = std::false_type;
  using I1 = std::integral_constant<int, 1>;
  using I5 = std::integral_constant<int, 5>;
  using I10 = std::integral_constant<int, 10>;
  using I20 = std::integral_constant<int, 20>;
  using I0 = std::integral_constant<int, 0>;
  if (h->is_complex) {
    if (h->nb == 1) launch(T_{}, I1{});
    else if (h->nb == 5) launch(T_{}, I5{});
    else if (h->nb == 10) launch(T_{}, I10{});
    else if (h->nb == 20) launch(T_{}, I20{});
    else launch(T_{}, I0{});
  } else {
    if (h->nb == 1) launch(F_{}, I1{});
    else if (h->nb == 5) launch(F_{}, I5{});
    else if (h->nb == 10) launch(F_{}, I10{});
    else if (h->nb == 20) launch(F_{}, I20{});
    else launch(F_{}, I0{});
  }
  cudaError_t e = cudaGetLastError();
  if (d_occ) cudaFreeAsync(d_occ, ctx->stream);
  if (e != cudaSuccess) return set_err(ctx, OMEN_ECUDA, "density: %s", cudaGetErrorString(e));
  return OMEN_OK;
}

static omen_status check_grid(omen_ctx* ctx, const omen_grid* gr) {
  if (!gr || gr->nx < 1 || gr->ny < 1 || gr->nz < 2 || !(gr->Lx_nm > 0) || !(gr->Ly_nm > 0) || !(gr->Lz_nm > 0))
    return set_err(ctx, OMEN_EINVAL, "invalid grid");
  return OMEN_OK;
}

extern "C" omen_status omen_deposit(omen_ctx* ctx, const omen_lattice* L, const omen_grid* gr, const double* q,
                                    double* rho) {
  if (!ctx || !L || !q || !rho) return set_err(ctx, OMEN_EINVAL, "null argument");
  omen_status s = check_grid(ctx, gr);
  if (s != OMEN_OK) return s;
  const GridGeo G = grid_geo(gr);
  AxisTable t[3];
  char* buf = nullptr;
  s = make_tables(ctx, L, G, t, &buf);
  if (s != OMEN_OK) return s;
  const cudaError_t ec = cudaMemsetAsync(rho, 0, sizeof(double) * (size_t)G.nx * G.ny * (G.nz - 1), ctx->stream);
  deposit_kernel<<<(unsigned)((L->natoms + 255) / 256), 256, 0, ctx->stream>>>(lat_geo(L), t[0], t[1], t[2], G.nz, q,
                                                                               1.0 / G.vol_m3, rho);
  if (ec != cudaSuccess) {
    cudaFreeAsync(buf, ctx->stream);
    return set_err(ctx, OMEN_ECUDA, "deposit: %s", cudaGetErrorString(ec));
  }
  cudaError_t e = cudaGetLastError();
  cudaFreeAsync(buf, ctx->stream);
  if (e != cudaSuccess) return set_err(ctx, OMEN_ECUDA, "deposit: %s", cudaGetErrorString(e));
  return OMEN_OK;
}

extern "C" omen_status omen_gather(omen_ctx* ctx, const omen_lattice* L, const omen_grid* gr, const double* phi,
                                   double* out) {
  if (!ctx || !L || !phi || !out) return set_err(ctx, OMEN_EINVAL, "null argument");
  omen_status s = check_grid(ctx, gr);
  if (s != OMEN_OK) return s;
  const GridGeo G = grid_geo(gr);
  AxisTable t[3];
  char* buf = nullptr;
  s = make_tables(ctx, L, G, t, &buf);
  if (s != OMEN_OK) return s;
  gather_kernel<<<(unsigned)((L->natoms + 255) / 256), 256, 0, ctx->stream>>>(lat_geo(L), t[0], t[1], t[2], G.nz, phi, out);
  cudaError_t e = cudaGetLastError();
  cudaFreeAsync(buf, ctx->stream);
  if (e != cudaSuccess) return set_err(ctx, OMEN_ECUDA, "gather: %s", cudaGetErrorString(e));
  return OMEN_OK;
}

static double fermi_fn(double x) {  // 1 / (1 + exp(x)), overflow-safe
  if (x > 0) {
    const double e = exp(-x);
    return e / (1.0 + e);
  }
  return 1.0 / (1.0 + exp(x));
}

extern "C" omen_status omen_fermi_level(const double* E, const double* wgt, int n, double n_target, double kT, double* EF) {
  if (!E || !wgt || !EF || n < 1 || !(kT > 0)) return OMEN_EINVAL;
  double total = 0.0, lo = E[0], hi = E[0];
  for (int i = 0; i < n; ++i) {
    total += wgt[i];
    lo = std::min(lo, E[i]);
    hi = std::max(hi, E[i]);
  }
  if (!(n_target >= 0) || n_target > total) return OMEN_EINVAL;
  lo -= 50 * kT;
  hi += 50 * kT;
  auto count = [&](double ef) {
    double c = 0.0;
    for (int i = 0; i < n; ++i) c += wgt[i] * fermi_fn((E[i] - ef) / kT);
    return c;
  };
  for (int it = 0; it < 200 && hi - lo > 1e-13; ++it) {
    const double mid = 0.5 * (lo + hi);
    if (count(mid) < n_target) lo = mid; else hi = mid;
  }
  *EF = 0.5 * (lo + hi);
  return OMEN_OK;
}
