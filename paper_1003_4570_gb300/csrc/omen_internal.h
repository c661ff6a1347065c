// Internal definitions shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>
#include <cstdint>
#include <cstdio>
#include <string>
#include <vector>

#include "../../include/omen.h"

struct omen_ctx {
  int device = 0;
  cudaStream_t stream = nullptr;
  std::string err;
  // small device work area: reduction partials and a status word
  double* d_work = nullptr;
  size_t work_bytes = 0;
  int* d_status = nullptr;
  // Lanczos step sequences between host checks are captured once as CUDA graphs and replayed
  bool use_graphs = true;
  int reorth = OMEN_REORTH_FULL;        // full Gram–Schmidt pass policy of the Lanczos steps
  bool lock_check = true;               // single-vector lowest solves check for missed copies
  cudaStream_t cap_stream = nullptr;   // private stream the captures are recorded on
  cudaStream_t copy_stream[2] = {nullptr, nullptr};  // host<->device copies overlapped with H·X
  // device buffers of the host-buffer product, kept between calls (grown, never shrunk): a fresh
  // allocation per call costs more than the copies it serves
  void* host_scratch = nullptr;
  size_t host_scratch_bytes = 0;
  std::vector<cudaEvent_t> host_events;  // the pipeline's events, created once
  // pinned host memory that small coefficient tables are copied from, and the event after the last
  // such copy (made on first use)
  void* stage = nullptr;
  cudaEvent_t stage_done = nullptr;
  // work areas of the calls come from a pool of the context's own, which keeps up to kPoolKeep
  // bytes mapped between calls (the default pool gives everything back at the next
  // synchronisation, and a call then spends 0.1 to 0.4 ms mapping it again); gone with the context
  cudaMemPool_t pool = nullptr;
};
constexpr unsigned long long kPoolKeep = 512ull << 20;
constexpr size_t kStageBytes = 512 << 10;

// `bytes` of host memory that the caller may drop on return, to dst on the context's stream: through
// the pinned stage, else waited for (the runtime may read pageable memory until the stream is next
// synchronised).
omen_status copy_to_device(omen_ctx* ctx, void* dst, const void* src, size_t bytes);

// Stream-ordered device memory for one call on the context's stream (free with cudaFreeAsync).
template <typename T>
inline cudaError_t ctx_alloc(omen_ctx* ctx, T** p, size_t bytes) {
  return ctx->pool ? cudaMallocFromPoolAsync(reinterpret_cast<void**>(p), bytes, ctx->pool, ctx->stream)
                   : cudaMallocAsync(reinterpret_cast<void**>(p), bytes, ctx->stream);
}

struct omen_lattice {
  int nx, ny, nz, ncells, natoms;
  int periodic[3];
  double a_nm;
  uint8_t* d_species = nullptr;  // [natoms]
  int max_species = 0;           // the largest of them
  double* d_strain = nullptr;    // [16*ncells]
  long long nbonds = 0;
};

// Launch shape of an H·X kernel: CTA width and rows per register batch (k batch: wave vectors
// per thread); zeros select the built-in defaults.
struct HxTile {
  int threads = 0, rb = 0;
};

struct omen_ham {
  const omen_lattice* lat = nullptr;
  int norb = 0, nspin = 1, nb = 0;        // nb = norb * nspin
  int spin_orbit = 0, precision = OMEN_F64, matrix_free = 0, bloch = 0, is_complex = 0;
  int nspecies = 1;
  long long nrows = 0;
  double eta = 2.0;
  double kvec[3] = {0, 0, 0};
  double2 phase[3];                       // exp(i k.L_d e_d) for a +1 supercell wrap along d
  // reduced bond blocks of every species pair, both ends ([2][ns*ns][coef_stride(norb)], see
  // sk_device.cuh), and the bond-length factor (d0/d)^eta of every slot from the structure's
  // strain at assembly ([16*ncells], slot layout): FP64, FP32 and double-float copies as the
  // products of this Hamiltonian need them, else null
  double* d_coef64 = nullptr;
  float* d_coef32 = nullptr;
  float2* d_coefdf = nullptr;
  double* d_scale64 = nullptr;
  float* d_scale32 = nullptr;
  float2* d_scaledf = nullptr;
  // onsite energies per species and orbital [ns][norb], potential per atom
  double* d_onsite = nullptr;
  float* d_onsite32 = nullptr;            // the same in FP32
  float2* d_onsite_df = nullptr;          // the same as double-float pairs (OMEN_F64_DF)
  double* d_U = nullptr;                  // [natoms]
  double lambda_so[4] = {0, 0, 0, 0};
  double* d_lambda = nullptr;             // [ns]
  HxTile tile[2];                         // H·X launch shape for FP64 [0] and FP32 [1] vectors
  HxTile ktile[2];                        // the same for the k-batched product
  // single-band effective-mass Hamiltonian on a uniform grid (lat is null; nb = 1, d_U holds
  // one potential per grid point, d_U32 its FP32 copy for FP32 vectors)
  int effmass = 0;
  int gdim[3] = {0, 0, 0};
  int gper[3] = {0, 0, 0};
  double t_hop[3] = {0, 0, 0};            // hbar^2 / (2 m0 m_d h_d^2) (eV)
  double ec = 0.0;
  float* d_U32 = nullptr;
};

// effective-mass product y = (H - sigma) x (effmass.cu)
omen_status launch_hx_effmass(omen_ctx* ctx, const omen_ham* h, const void* x, void* y, int nvec, double sigma,
                              int vec_precision, cudaStream_t st);
// U per grid point (device, eV) or null for zero; refreshes the FP32 copy
omen_status effmass_set_potential(omen_ctx* ctx, omen_ham* h, const double* U);

// status / error helpers ---------------------------------------------------------------------
omen_status set_err(omen_ctx* ctx, omen_status s, const char* fmt, ...);
#define OMEN_CUDA(ctx, call)                                                            \
  do {                                                                                  \
    cudaError_t e_ = (call);                                                            \
    if (e_ != cudaSuccess)                                                              \
      return set_err(ctx, OMEN_ECUDA, "%s failed: %s", #call, cudaGetErrorString(e_));  \
  } while (0)
#define OMEN_CHECK_LAUNCH(ctx) OMEN_CUDA(ctx, cudaGetLastError())

// kernels launched from the C-ABI layer ------------------------------------------------------
omen_status launch_assemble(omen_ctx* ctx, omen_ham* ham, const omen_tb_params* p);
omen_status launch_hx(omen_ctx* ctx, const omen_ham* ham, const void* x, void* y, int nvec,
                      double sigma, int vec_precision);
omen_status launch_hx_kbatch(omen_ctx* ctx, const omen_ham* h, int nk, const double2* phases_dev, const void* x, void* y,
                             double sigma, int vec_precision);
// One structure of a multi-structure k batch: its nk wave vectors' phase table (device) and the
// element offset of its first vector in the batch's vector buffers ([nk][nrows] from there).
struct KItem {
  const omen_ham* ham;
  int nk;
  const double2* phases;
  long long x_off;
  const double2* phases_host = nullptr;   // where `phases` is null: [nk][3], passed with the launch
};
constexpr int kInlinePhases = 128;        // wave vectors of a batch whose phases fit the launch
omen_status launch_hx_kmulti(omen_ctx* ctx, const KItem* items, int nitems, const void* x, void* y, double sigma,
                             int vec_precision);
omen_status make_phases(omen_ctx* ctx, const omen_ham* h, int nk, const double* k_host, double2** out);
std::vector<double2> phase_table(const omen_ham* h, int nk, const double* k_host);

// Krylov helpers (lanczos.cu)
size_t vec_elem_bytes(const omen_ham* ham, int precision);
omen_status krylov_start_from(omen_ctx* ctx, const omen_ham* ham, int prec, const void* X, int k, void* out, int nout,
                              unsigned long long seed);
