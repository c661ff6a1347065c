// Device-side Hamiltonian assembly (paper Section I: sp3s*/sp3d5s* tight binding with strain).
//
// 1. the Slater–Koster block of every species pair at d0, in the reduced form the product
//    applies (sk_device.cuh), for both ends of the bond;
// 2. the factor (d0/d)^eta of every bond slot, d = d0 (1 + strain): a bond's block is its
//    factor times its pair's reduced block, with the signs of its direction.
// Stored and matrix-free Hamiltonians hold the same data, in the precisions their products use.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "omen_internal.h"
#include "sk_device.cuh"

// coef[end][pair][coef_stride(norb)]: end 0 the rows of the A atom, end 1 those of the B atom
__global__ void coef_table_kernel(const double* __restrict__ V, int ns, int norb, double* __restrict__ c64,
                                  float* __restrict__ c32, float2* __restrict__ cdf) {
  const int cs = coef_stride(norb);
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 2 * ns * ns) return;
  const int end = t / (ns * ns), pair = t - end * ns * ns;
  const int sa = pair / ns, sb = pair - sa * ns;
  double c[28];
  reduced_block(V + (sa * ns + sb) * 14, V + (sb * ns + sa) * 14, norb, end != 0, c);
  for (int i = 0; i < cs; ++i) {
    const size_t at = (size_t)t * cs + i;
    const float hi = __double2float_rn(c[i]);
    if (c64) c64[at] = c[i];
    if (c32) c32[at] = hi;
    if (cdf) cdf[at] = make_float2(hi, __double2float_rn(c[i] - (double)hi));
  }
}

__global__ void bond_scale_kernel(const double* __restrict__ strain, long long nslots, double eta,
                                  double* __restrict__ s64, float* __restrict__ s32, float2* __restrict__ sdf) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nslots; i += (long long)gridDim.x * blockDim.x) {
    const double f = pow(1.0 + strain[i], -eta);
    const float hi = __double2float_rn(f);
    if (s64) s64[i] = f;
    if (s32) s32[i] = hi;
    if (sdf) sdf[i] = make_float2(hi, __double2float_rn(f - (double)hi));
  }
}

__global__ void max_species_kernel(const uint8_t* __restrict__ sp, int n, int* __restrict__ out) {
  int m = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) m = max(m, (int)sp[i]);
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

static void free_ham_buffers(omen_ham* h) {
  cudaFree(h->d_coef64);
  cudaFree(h->d_coef32);
  cudaFree(h->d_coefdf);
  cudaFree(h->d_scale64);
  cudaFree(h->d_scale32);
  cudaFree(h->d_scaledf);
  cudaFree(h->d_onsite);
  cudaFree(h->d_onsite32);
  cudaFree(h->d_onsite_df);
  cudaFree(h->d_U);
  cudaFree(h->d_U32);
  cudaFree(h->d_lambda);
}

extern "C" void omen_free_ham(omen_ham* h) {
  if (!h) return;
  free_ham_buffers(h);
  delete h;
}

#define ALLOC_OR_FAIL(ptr, bytes)                                                          \
  do {                                                                                     \
    if (cudaMalloc(&(ptr), (bytes)) != cudaSuccess) {                                      \
      cudaGetLastError();                                                                  \
      omen_free_ham(h);                                                                    \
      return set_err(ctx, OMEN_ENOMEM, "device allocation of %zu bytes failed", (size_t)(bytes)); \
    }                                                                                      \
  } while (0)

extern "C" omen_status omen_assemble_H(omen_ctx* ctx, const omen_lattice* lat, const omen_tb_params* p,
                                       const omen_ham_opts* opts, omen_ham** out) {
  if (!ctx || !lat || !p || !opts || !out) return set_err(ctx, OMEN_EINVAL, "null argument");
  *out = nullptr;
  if (p->basis != OMEN_SP3S && p->basis != OMEN_SP3D5S) return set_err(ctx, OMEN_EINVAL, "basis must be 5 or 10");
  if (p->nspecies < 1 || p->nspecies > 4) return set_err(ctx, OMEN_EINVAL, "nspecies must be 1..4");
  if (opts->precision < OMEN_F64 || opts->precision > OMEN_F64_DF)
    return set_err(ctx, OMEN_EINVAL, "unknown precision %d", opts->precision);
  if (opts->precision == OMEN_F64_DF && (opts->spin_orbit || opts->matrix_free || (opts->k && (lat->periodic[0] == OMEN_BLOCH || lat->periodic[1] == OMEN_BLOCH || lat->periodic[2] == OMEN_BLOCH))))
    return set_err(ctx, OMEN_EUNSUPPORTED, "double-float precision supports real stored Hamiltonians only");
  OMEN_CUDA(ctx, cudaSetDevice(ctx->device));
  {  // species indices must be < nspecies
    int* d_m = (int*)ctx->d_status;
    OMEN_CUDA(ctx, cudaMemsetAsync(d_m, 0, sizeof(int), ctx->stream));
    max_species_kernel<<<64, 256, 0, ctx->stream>>>(lat->d_species, lat->natoms, d_m);
    OMEN_CHECK_LAUNCH(ctx);
    int hm = 0;
    OMEN_CUDA(ctx, cudaMemcpyAsync(&hm, d_m, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    OMEN_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    if (hm >= p->nspecies) return set_err(ctx, OMEN_EINVAL, "species index %d >= nspecies %d", hm, p->nspecies);
  }
  auto* h = new omen_ham();
  h->lat = lat;
  h->norb = p->basis;
  h->spin_orbit = opts->spin_orbit ? 1 : 0;
  h->nspin = h->spin_orbit ? 2 : 1;
  h->nb = h->norb * h->nspin;
  h->precision = opts->precision;
  h->matrix_free = opts->matrix_free ? 1 : 0;
  h->nspecies = p->nspecies;
  h->eta = p->eta;
  h->nrows = (long long)h->nb * lat->natoms;
  h->bloch = 0;
  if (opts->k) {
    for (int d = 0; d < 3; ++d) h->kvec[d] = opts->k[d];
    for (int d = 0; d < 3; ++d)
      if (lat->periodic[d] == OMEN_BLOCH) h->bloch = 1;
  }
  const int ncell_d[3] = {lat->nx, lat->ny, lat->nz};
  for (int d = 0; d < 3; ++d) {
    double ph = 0.0;
    if (lat->periodic[d] == OMEN_BLOCH) ph = h->kvec[d] * ncell_d[d] * lat->a_nm;
    h->phase[d] = make_double2(cos(ph), sin(ph));
  }
  h->is_complex = (h->spin_orbit || h->bloch) ? 1 : 0;
  for (int s = 0; s < 4; ++s) h->lambda_so[s] = p->lambda_so[s];

  const int ns = p->nspecies, norb = p->basis;
  const size_t nslots = 16 * (size_t)lat->ncells;
  const size_t ncoef = 2 * (size_t)ns * ns * coef_stride(norb);
  ALLOC_OR_FAIL(h->d_onsite, sizeof(double) * ns * norb);
  ALLOC_OR_FAIL(h->d_onsite32, sizeof(float) * ns * norb);
  ALLOC_OR_FAIL(h->d_U, sizeof(double) * lat->natoms);
  ALLOC_OR_FAIL(h->d_lambda, sizeof(double) * 4);
  // the precisions the products of this Hamiltonian use (matrix-free: FP64 and FP32)
  const bool need64 = h->matrix_free || h->precision == OMEN_F64 || h->precision == OMEN_F32_REFINE64;
  const bool need32 = h->matrix_free || h->precision == OMEN_F32 || h->precision == OMEN_F32_REFINE64;
  const bool needdf = h->precision == OMEN_F64_DF;
  if (need64) {
    ALLOC_OR_FAIL(h->d_coef64, ncoef * sizeof(double));
    ALLOC_OR_FAIL(h->d_scale64, nslots * sizeof(double));
  }
  if (need32) {
    ALLOC_OR_FAIL(h->d_coef32, ncoef * sizeof(float));
    ALLOC_OR_FAIL(h->d_scale32, nslots * sizeof(float));
  }
  if (needdf) {
    ALLOC_OR_FAIL(h->d_coefdf, ncoef * sizeof(float2));
    ALLOC_OR_FAIL(h->d_scaledf, nslots * sizeof(float2));
  }

  // parameter tables
  std::vector<double> V(ns * ns * 14), on(ns * norb);
  for (int a = 0; a < ns; ++a)
    for (int b = 0; b < ns; ++b)
      for (int q = 0; q < 14; ++q) V[(a * ns + b) * 14 + q] = p->V[a][b][q];
  for (int a = 0; a < ns; ++a) {
    int o = 0;
    on[a * norb + o++] = p->onsite[a][0];
    for (int i = 0; i < 3; ++i) on[a * norb + o++] = p->onsite[a][1];
    if (norb == 10)
      for (int i = 0; i < 5; ++i) on[a * norb + o++] = p->onsite[a][2];
    on[a * norb + o++] = p->onsite[a][3];
  }
  double* d_V = nullptr;
  if (cudaMalloc(&d_V, sizeof(double) * V.size()) != cudaSuccess) {
    omen_free_ham(h);
    return set_err(ctx, OMEN_ENOMEM, "device allocation failed");
  }
  cudaError_t e = cudaMemcpyAsync(d_V, V.data(), sizeof(double) * V.size(), cudaMemcpyHostToDevice, ctx->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(h->d_onsite, on.data(), sizeof(double) * on.size(), cudaMemcpyHostToDevice, ctx->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(h->d_lambda, p->lambda_so, sizeof(double) * 4, cudaMemcpyHostToDevice, ctx->stream);
  std::vector<float> on32(on.begin(), on.end());
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(h->d_onsite32, on32.data(), sizeof(float) * on32.size(), cudaMemcpyHostToDevice, ctx->stream);
  std::vector<float2> ondf(on.size());
  if (e == cudaSuccess && needdf) {
    for (size_t i = 0; i < on.size(); ++i) {
      const float hi = (float)on[i];
      ondf[i] = make_float2(hi, (float)(on[i] - (double)hi));
    }
    if (cudaMalloc(&h->d_onsite_df, sizeof(float2) * ondf.size()) != cudaSuccess) {
      cudaGetLastError();
      cudaFree(d_V);
      omen_free_ham(h);
      return set_err(ctx, OMEN_ENOMEM, "device allocation failed");
    }
    e = cudaMemcpyAsync(h->d_onsite_df, ondf.data(), sizeof(float2) * ondf.size(), cudaMemcpyHostToDevice, ctx->stream);
  }
  if (e == cudaSuccess) {
    if (opts->U_atom_dev)
      e = cudaMemcpyAsync(h->d_U, opts->U_atom_dev, sizeof(double) * lat->natoms, cudaMemcpyDeviceToDevice, ctx->stream);
    else
      e = cudaMemsetAsync(h->d_U, 0, sizeof(double) * lat->natoms, ctx->stream);
  }
  if (e == cudaSuccess) {
    coef_table_kernel<<<1, 64, 0, ctx->stream>>>(d_V, ns, norb, h->d_coef64, h->d_coef32, h->d_coefdf);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) {
    bond_scale_kernel<<<(unsigned)std::min<size_t>((nslots + 255) / 256, 65535), 256, 0, ctx->stream>>>(
        lat->d_strain, (long long)nslots, p->eta, h->d_scale64, h->d_scale32, h->d_scaledf);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  cudaFree(d_V);
  if (e != cudaSuccess) {
    omen_free_ham(h);
    return set_err(ctx, OMEN_ECUDA, "assembly failed: %s", cudaGetErrorString(e));
  }
  *out = h;
  return OMEN_OK;
}

extern "C" omen_status omen_ham_shape(const omen_ham* h, long long* nrows, int* is_complex, int* elem_bytes) {
  if (!h) return OMEN_EINVAL;
  if (nrows) *nrows = h->nrows;
  if (is_complex) *is_complex = h->is_complex;
  if (elem_bytes) *elem_bytes = (int)vec_elem_bytes(h, h->precision);
  return OMEN_OK;
}

extern "C" omen_status omen_ham_set_potential(omen_ctx* ctx, omen_ham* h, const double* U) {
  if (!ctx || !h) return set_err(ctx, OMEN_EINVAL, "null argument");
  if (h->effmass) return effmass_set_potential(ctx, h, U);
  if (U)
    OMEN_CUDA(ctx, cudaMemcpyAsync(h->d_U, U, sizeof(double) * h->lat->natoms, cudaMemcpyDeviceToDevice, ctx->stream));
  else
    OMEN_CUDA(ctx, cudaMemsetAsync(h->d_U, 0, sizeof(double) * h->lat->natoms, ctx->stream));
  return OMEN_OK;
}
