// y = (H - sigma) x: the block-sparse tight-binding product repeated by the Lanczos
// recurrence (paper Section II-B benchmarks "500 Lanczos iterations"; Section III-A item 1).
//
// Bond blocks are applied in reduced form.  A two-centre block is invariant under rotations
// about its bond, so along (1,1,1), with the p and t2g amplitudes written (x, y, z) and
// (yz, zx, xy), it holds 25 numbers (10 for sp3s*) instead of 100 (25): the s, s* rows see
// only the sums P = px+py+pz and T = dyz+dzx+dxy; p-p, p-t2g, t2g-t2g parts are a multiple of
// the identity plus a multiple of the all-ones matrix; the e pair couples to p and t2g through
// the zero-sum triple q = (-e2/2 + r e1, -e2/2 - r e1, e2), r = sqrt(3)/2.  The other three
// directions differ by the signs of (px, py, pz) and (dyz, dzx, dxy), the same three signs for
// both; the bond's length multiplies the whole block by (d0/d)^eta.  A bond end costs 61
// operations (FP64: the bound) instead of 100, and reads one factor instead of a block, so no
// block is stored: the reduced numbers of every species pair (a few KB, both ends of the bond)
// sit in shared memory.
//
// Measured on the sp3d5s* alloy of 1M atoms, full blocks before and this form after: FP64 0.706 ->
// 0.451 ms (88% of the FP64 rate in the operations needed, FP64 pipe 93% busy; bound by it), FP32
// stored 0.169 -> 0.040 ms, FP32 matrix-free 0.061 -> 0.040 ms (bound by the shared-memory reads of the reduced blocks, 27 words a bond end
// and lane, and the latency of the neighbours' amplitudes: 54% of the LSU data rate, 57% of the
// issue slots).  The rounding error against 64 bits falls with the number of terms: FP32 1.3e-7
// -> 0.7e-7 of the result's norm.
//
// One thread per atom; a warp takes 32 consecutive cells of one site, the eight warps of a CTA
// the eight sites of the same cells, so that of the sixteen bonds of a cell nine find their
// neighbour's amplitudes in the lines the CTA has just read.  Vectors are orbital-major,
// atom-minor: the per-orbital loads of x and stores of y are coalesced.
// Bloch phase: a neighbour reached across the high (low) face of a Bloch-periodic direction d
// is its periodic image shifted by +L_d (-L_d); its amplitude is multiplied by
// exp(+i k_d L_d) (resp. the conjugate).
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "omen_internal.h"
#include "sk_device.cuh"
#include "df.cuh"
#include "neighbours.cuh"
#include "param_copy.cuh"
#include "pdl.cuh"

template <typename T> struct Cx;
template <> struct Cx<double> { using t = double2; };
template <> struct Cx<float> { using t = float2; };

template <typename T, bool CPLX> struct VecT { using t = T; };
template <typename T> struct VecT<T, true> { using t = typename Cx<T>::t; };

// Amplitudes (real, or complex as a pair) times real numbers.  FP32 pairs use the packed
// FP32x2 instructions: each lane an ordinary fma, add or multiply.
__device__ __forceinline__ double v_fma(double c, double x, double a) { return fma(c, x, a); }
__device__ __forceinline__ float v_fma(float c, float x, float a) { return fmaf(c, x, a); }
__device__ __forceinline__ double2 v_fma(double c, double2 x, double2 a) { return make_double2(fma(c, x.x, a.x), fma(c, x.y, a.y)); }
__device__ __forceinline__ float2 v_fma(float c, float2 x, float2 a) { return __ffma2_rn(make_float2(c, c), x, a); }
__device__ __forceinline__ double v_mul(double c, double x) { return c * x; }
__device__ __forceinline__ float v_mul(float c, float x) { return c * x; }
__device__ __forceinline__ double2 v_mul(double c, double2 x) { return make_double2(c * x.x, c * x.y); }
__device__ __forceinline__ float2 v_mul(float c, float2 x) { return __fmul2_rn(make_float2(c, c), x); }
__device__ __forceinline__ double v_add(double a, double b) { return a + b; }
__device__ __forceinline__ float v_add(float a, float b) { return a + b; }
__device__ __forceinline__ double2 v_add(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 v_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ double v_neg(double a) { return -a; }
__device__ __forceinline__ float v_neg(float a) { return -a; }
__device__ __forceinline__ double2 v_neg(double2 a) { return make_double2(-a.x, -a.y); }
__device__ __forceinline__ float2 v_neg(float2 a) { return make_float2(-a.x, -a.y); }
template <typename V> __device__ __forceinline__ V v_zero();
template <> __device__ __forceinline__ double v_zero<double>() { return 0.0; }
template <> __device__ __forceinline__ float v_zero<float>() { return 0.f; }
template <> __device__ __forceinline__ double2 v_zero<double2>() { return make_double2(0.0, 0.0); }
template <> __device__ __forceinline__ float2 v_zero<float2>() { return make_float2(0.f, 0.f); }

template <typename C>
__device__ __forceinline__ C cmul(C a, C b) {
  C r;
  r.x = a.x * b.x - a.y * b.y;
  r.y = a.x * b.y + a.y * b.x;
  return r;
}

// The reduced numbers of one bond end, shared memory to registers in 16-byte loads.
template <typename T, int NORB>
__device__ __forceinline__ void load_coef(const T* __restrict__ s, T (&c)[coef_stride(NORB)]) {
  constexpr int N = coef_stride(NORB);
  if constexpr (sizeof(T) == 4) {
    const float4* s4 = reinterpret_cast<const float4*>(s);
#pragma unroll
    for (int i = 0; i < N / 4; ++i) {
      const float4 v = s4[i];
      c[4 * i] = v.x; c[4 * i + 1] = v.y; c[4 * i + 2] = v.z; c[4 * i + 3] = v.w;
    }
  } else {
    const double2* s2 = reinterpret_cast<const double2*>(s);
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
      const double2 v = s2[i];
      c[2 * i] = v.x; c[2 * i + 1] = v.y;
    }
  }
}

// r = B x for the bond along (1,1,1), from its reduced numbers (the order of coef_table).
template <typename T, int NORB, typename V>
__device__ __forceinline__ void bond_product(const T (&c)[coef_stride(NORB)], const V (&x)[NORB], V (&r)[NORB]) {
  if constexpr (NORB == 5) {
    const V P = v_add(v_add(x[1], x[2]), x[3]);
    r[0] = v_fma(c[2], x[4], v_fma(c[1], P, v_mul(c[0], x[0])));
    r[4] = v_fma(c[5], x[4], v_fma(c[4], P, v_mul(c[3], x[0])));
    const V C = v_fma(c[8], P, v_fma(c[7], x[4], v_mul(c[6], x[0])));
#pragma unroll
    for (int i = 0; i < 3; ++i) r[1 + i] = v_fma(c[9], x[1 + i], C);
  } else {
    constexpr T kHalf = (T)0.5, kR = (T)0.86602540378443865;   // sqrt(3)/2
    const V p12 = v_add(x[1], x[2]), t12 = v_add(x[4], x[5]);
    const V P = v_add(p12, x[3]), Q = v_add(t12, x[6]);
    r[0] = v_fma(c[3], x[9], v_fma(c[2], Q, v_fma(c[1], P, v_mul(c[0], x[0]))));
    r[9] = v_fma(c[7], x[9], v_fma(c[6], Q, v_fma(c[5], P, v_mul(c[4], x[0]))));
    const V Cp = v_fma(c[11], Q, v_fma(c[10], P, v_fma(c[9], x[9], v_mul(c[8], x[0]))));
    const V Ct = v_fma(c[18], Q, v_fma(c[17], P, v_fma(c[16], x[9], v_mul(c[15], x[0]))));
    const V h = v_mul(-kHalf, x[8]);
    const V q[3] = {v_fma(kR, x[7], h), v_fma(-kR, x[7], h), x[8]};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      r[1 + i] = v_fma(c[13], x[4 + i], v_fma(c[12], x[1 + i], v_fma(c[14], q[i], Cp)));
      r[4 + i] = v_fma(c[20], x[4 + i], v_fma(c[19], x[1 + i], v_fma(c[21], q[i], Ct)));
    }
    const V pe1 = v_add(x[1], v_neg(x[2])), te1 = v_add(x[4], v_neg(x[5]));
    const V pe2 = v_fma(-kHalf, p12, x[3]), te2 = v_fma(-kHalf, t12, x[6]);
    r[7] = v_fma(c[24], x[7], v_fma(c[26], te1, v_mul(c[25], pe1)));
    r[8] = v_fma(c[24], x[8], v_fma(c[23], te2, v_mul(c[22], pe2)));
  }
}

// One structure of a product.  Real and complex vectors, FP64 and FP32.
template <typename T>
struct HxInst {
  Geo g;
  const T* __restrict__ coef;         // [2 ends][ns*ns][coef_stride] reduced blocks
  const T* __restrict__ scale;        // [16*ncells] (d0/d)^eta per bond slot
  const uint8_t* __restrict__ species;
  const T* __restrict__ onsite;       // [ns][norb]
  const double* U;                    // [natoms]; kernels of the stream may write it (see pdl.cuh)
  const double* __restrict__ lambda;  // [ns]
  const double2* __restrict__ phases; // k batch: [nk][3] exp(i k_d L_d); null: with the launch,
  int ph_at;                          // from this entry
  long long nrows;
  long long x_off;                    // first element of this structure's vectors
  double2 phase[3];                   // the same for the one wave vector of a plain product
  int ns;
  int nvec;                           // vectors (k batch: wave vectors)
  int cta0, tiles;                    // k batch: first CTA, CTAs per group of wave vectors
};

// exp(i k.T) of a wrapped bond
template <typename T>
__device__ __forceinline__ typename Cx<T>::t wrap_phase(unsigned wrap, bool is_a, const double2* __restrict__ ph) {
  typename Cx<T>::t f;
  f.x = (T)1;
  f.y = (T)0;
#pragma unroll
  for (int d = 0; d < 3; ++d)
    if (wrap >> d & 1u) {
      typename Cx<T>::t p;
      p.x = (T)ph[d].x;
      p.y = (T)(is_a ? -ph[d].y : ph[d].y);
      f = cmul(f, p);
    }
  return f;
}

// Onsite rows: (E_o + U - sigma) x, and lambda L.sigma on the p amplitudes with spin-orbit
// (basis (spin, orbital), spin up first; spin `q` of this thread, xo the other spin's vector).
template <typename T, int NORB, bool CPLX, bool SO>
__device__ __forceinline__ void onsite_rows(const HxInst<T>& I, int atom, int sp, double sigma, int q,
                                            const typename VecT<T, CPLX>::t* __restrict__ x,
                                            typename VecT<T, CPLX>::t (&acc)[NORB]) {
  using V = typename VecT<T, CPLX>::t;
  const size_t N = I.g.natoms;
  const T u = (T)(I.U[atom] - sigma);
  const V* __restrict__ xp = x + (size_t)(SO ? q * NORB : 0) * N + atom;
  V xv[NORB];
#pragma unroll
  for (int o = 0; o < NORB; ++o) xv[o] = xp[o * N];
  // one energy for each of s, p, d, s*
  const T* __restrict__ e = I.onsite + sp * NORB;
  const T es = e[0] + u, ep = e[1] + u, ed = e[NORB == 10 ? 4 : 1] + u, eS = e[NORB - 1] + u;
#pragma unroll
  for (int o = 0; o < NORB; ++o) acc[o] = v_mul(o == 0 ? es : o < 4 ? ep : o == NORB - 1 ? eS : ed, xv[o]);
  if constexpr (SO) {
    const T lam = (T)I.lambda[sp];
    const V* __restrict__ xo = x + (size_t)((1 - q) * NORB) * N + atom;
    const V o0 = xo[N], o1 = xo[2 * N], o2 = xo[3 * N];   // the other spin's px, py, pz
    const V m0 = xv[1], m1 = xv[2], m2 = xv[3];
    // i*z = (-z.y, z.x)
    if (q == 0) {   // up x: -i xu_y + xd_z ; up y: i xu_x - i xd_z ; up z: i xd_y - xd_x
      acc[1].x += lam * (m1.y + o2.x);
      acc[1].y += lam * (-m1.x + o2.y);
      acc[2].x += lam * (-m0.y + o2.y);
      acc[2].y += lam * (m0.x - o2.x);
      acc[3].x += lam * (-o1.y - o0.x);
      acc[3].y += lam * (o1.x - o0.y);
    } else {        // dn x: i xd_y - xu_z ; dn y: -i xd_x - i xu_z ; dn z: i xu_y + xu_x
      acc[1].x += lam * (-m1.y - o2.x);
      acc[1].y += lam * (m1.x - o2.y);
      acc[2].x += lam * (m0.y + o2.y);
      acc[2].y += lam * (-m0.x - o2.x);
      acc[3].x += lam * (-o1.y + o0.x);
      acc[3].y += lam * (o1.x + o0.y);
    }
  }
}

// Rows of one atom for NV vectors v0.. (nv of them present).  LB bonds' amplitudes are loaded
// before their arithmetic; every accumulator sums its terms in the same order for any LB, NV
// and CTA width: the result does not depend on them.
template <typename T, int NORB, bool CPLX, bool SO, bool KPH, int NV, int LB>
__device__ __forceinline__ void hx_rows(const HxInst<T>& I, const T* __restrict__ tab, double sigma, int b, int cell, int q, int v0, int nv, const void* xv, void* yv,
                                        const double2* __restrict__ phases = nullptr) {
  using V = typename VecT<T, CPLX>::t;
  constexpr int CS = coef_stride(NORB);
  const Geo& g = I.g;
  const size_t N = g.natoms;
  const int atom = b * g.ncells + cell;
  const int nxy = g.nx * g.ny;
  const int iz = cell / nxy, rem = cell - iz * nxy, iy = rem / g.nx, ix = rem - iy * g.nx;
  const Steps steps = steps_of(g, b, ix, iy, iz);
  const V* __restrict__ x = static_cast<const V*>(xv) + I.x_off + (size_t)v0 * I.nrows;
  V* __restrict__ y = static_cast<V*>(yv) + I.x_off + (size_t)v0 * I.nrows;
  const int sp = I.species[atom];
  const bool is_a = b < 4;
  const T* __restrict__ tb = tab + (is_a ? 0 : I.ns * I.ns * CS);
  V acc[NV][NORB];
#pragma unroll
  for (int w = 0; w < NV; ++w) {
    if (w < nv) {
      onsite_rows<T, NORB, CPLX, SO>(I, atom, sp, sigma, q, x + (size_t)w * I.nrows, acc[w]);
    } else {
#pragma unroll
      for (int o = 0; o < NORB; ++o) acc[w][o] = v_zero<V>();
    }
  }
  const size_t spin = SO ? (size_t)(q * NORB) * N : 0;
  T c[CS];
  if (I.ns == 1) load_coef<T, NORB>(tb, c);   // one species: the same block for every bond
#pragma unroll
  for (int k0 = 0; k0 < 4; k0 += LB) {
    Neighbour n[LB];
    V xn[LB][NV][NORB];
    T sc[LB];
    int sp2[LB];
#pragma unroll
    for (int j = 0; j < LB; ++j) {
      n[j] = neighbour_of(g, steps, b, k0 + j, cell);
      sc[j] = (T)0;
      sp2[j] = 0;
      if (n[j].ok) {
        sc[j] = I.scale[n[j].slot];
        sp2[j] = I.species[n[j].atom];
      }
#pragma unroll
      for (int w = 0; w < NV; ++w) {
        const V* __restrict__ xp = x + (size_t)w * I.nrows + spin + n[j].atom;
#pragma unroll
        for (int o = 0; o < NORB; ++o) xn[j][w][o] = (n[j].ok && w < nv) ? xp[o * N] : v_zero<V>();
      }
    }
#pragma unroll
    for (int j = 0; j < LB; ++j) {
      const int k = k0 + j;
      if (I.ns > 1) load_coef<T, NORB>(tb + (is_a ? sp * I.ns + sp2[j] : sp2[j] * I.ns + sp) * CS, c);
#pragma unroll
      for (int w = 0; w < NV; ++w) {
        V(&xw)[NORB] = xn[j][w];
        if constexpr (CPLX) {
          if (n[j].wrap) {
            const V f = wrap_phase<T>(n[j].wrap, is_a, KPH ? phases + (size_t)min(v0 + w, I.nvec - 1) * 3 : I.phase);
#pragma unroll
            for (int o = 0; o < NORB; ++o) xw[o] = cmul(xw[o], f);
          }
        }
#pragma unroll
        for (int i = 0; i < 3; ++i)
          if (dir_minus(k, i)) {
            xw[1 + i] = v_neg(xw[1 + i]);
            if constexpr (NORB == 10) xw[4 + i] = v_neg(xw[4 + i]);
          }
        V r[NORB];
        bond_product<T, NORB>(c, xw, r);
#pragma unroll
        for (int o = 0; o < NORB; ++o) {
          const bool odd = o >= 1 && o <= (NORB == 10 ? 6 : 3);
          acc[w][o] = v_fma(odd && dir_minus(k, (o - 1) % 3) ? -sc[j] : sc[j], r[o], acc[w][o]);
        }
      }
    }
  }
#pragma unroll
  for (int w = 0; w < NV; ++w)
    if (w < nv) {
      V* __restrict__ yp = y + (size_t)w * I.nrows + spin + atom;
#pragma unroll
      for (int o = 0; o < NORB; ++o) yp[o * N] = acc[w][o];
    }
}

// The reduced blocks of every species pair, both ends, into shared memory.
template <typename T, int NORB>
__device__ __forceinline__ void stage_coef(const T* __restrict__ coef, int ns, T* tab) {
  const int n = 2 * ns * ns * coef_stride(NORB);
  for (int i = threadIdx.x; i < n; i += blockDim.x) tab[i] = coef[i];
  __syncthreads();
}

// y = (H - sigma) x.  grid.x: work items (site fastest, then tiles of 32 cells) over the warps;
// grid.y: the two spins with spin-orbit (the bonds are spin diagonal); grid.z: vectors.
template <typename T, int NORB, bool CPLX, bool SO, int LB>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 5 : CPLX ? 2 : 4) hx_kernel(const __grid_constant__ HxInst<T> I,
                                                 double sigma, int cell0, int cell1, const void* x, void* y) {
  __shared__ __align__(16) T tab[2 * 16 * coef_stride(NORB)];
  stage_coef<T, NORB>(I.coef, I.ns, tab);
  const int item = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int b = item & 7;
  const int cell = cell0 + (item >> 3) * 32 + (threadIdx.x & 31);
  if (cell >= cell1) return;
  const int q = SO ? blockIdx.y : 0, v = blockIdx.z;
  hx_rows<T, NORB, CPLX, SO, false, 1, LB>(I, tab, sigma, b, cell, q, v, 1, x, y);
}

// lambda (L.sigma x) of p orbital i (0..2) at spin q: `first` and `second` are the amplitudes it
// needs (see onsite_rows): its spin's p_1 (i = 0) or p_0 (i = 1), or the other spin's p_1 (i = 2);
// and the other spin's p_2 (i = 0, 1) or p_0 (i = 2).
template <typename V>
__device__ __forceinline__ V so_term(int q, int i, V first, V second) {
  const bool p1 = q == 0 ? i == 0 : i == 1;                        // sign of first.y in the real part
  const bool p2 = q == 0 ? i != 2 : i != 0;                        // sign of second in the real part
  const auto a = i == 1 ? second.y : second.x, b = i == 1 ? second.x : second.y;
  const bool p3 = i == 1 ? false : q == 0 ? i == 0 : i == 2;       // sign of second in the imaginary part
  V r;
  r.x = (p1 ? first.y : -first.y) + (p2 ? a : -a);
  r.y = (p1 ? -first.x : first.x) + (p3 ? b : -b);
  return r;
}

// One lane's bond end in the products below: 8 atoms x 4 bonds a warp (complex vectors: 4 x 4 x 2
// components).  Nothing here is written by an earlier kernel of the stream.
template <typename T, int NORB, bool CPLX>
struct BondLane {
  static constexpr int kCells = CPLX ? 4 : 8;
  int k, b, cell, atom, sp;
  bool im, live, is_a;      // im: the lane's component
  Neighbour n;
  T sc;                     // (d0/d)^eta; 0 for an absent bond
  const T* coef;            // its reduced block
  typename Cx<T>::t f;      // Bloch phase, the imaginary part with the sign the component takes

  __device__ __forceinline__ BondLane(const HxInst<T>& I, const T* tab, int item, int cell0, int cell1) {
    const Geo& g = I.g;
    const int lane = threadIdx.x & 31;
    k = (lane / kCells) & 3;
    im = CPLX && lane >= 16;
    b = item & 7;
    is_a = b < 4;
    const int cell_raw = cell0 + (item >> 3) * kCells + lane % kCells;
    live = cell_raw < cell1;
    cell = live ? cell_raw : cell1 - 1;              // idle lanes repeat the last cell, and store nothing
    atom = b * g.ncells + cell;
    const int nxy = g.nx * g.ny;
    const int iz = cell / nxy, rem = cell - iz * nxy, iy = rem / g.nx, ix = rem - iy * g.nx;
    n = neighbour_of(g, steps_of(g, b, ix, iy, iz), b, k, cell);
    sp = I.species[atom];
    sc = (T)0;
    int sp2 = 0;
    if (n.ok) {
      sc = I.scale[n.slot];
      sp2 = I.species[n.atom];
    }
    coef = tab + ((is_a ? 0 : I.ns * I.ns) + (is_a ? sp * I.ns + sp2 : sp2 * I.ns + sp)) * coef_stride(NORB);
    f.x = (T)1;
    f.y = (T)0;
    if (CPLX && n.wrap) f = wrap_phase<T>(n.wrap, is_a, I.phase);
    if (!im) f.y = -f.y;
  }

  // the lane's component of a neighbour's amplitude, times the phase
  __device__ __forceinline__ T component(typename VecT<T, CPLX>::t x) const {
    if constexpr (CPLX) {
      const T mine = im ? x.y : x.x, other = im ? x.x : x.y;
      return n.wrap ? fma(mine, f.x, other * f.y) : mine;
    } else {
      return x;
    }
  }
};

// The same product with one lane per bond, and for complex vectors one per bond and component: a
// warp takes 8 atoms x 4 bonds (4 x 4 x 2 complex), the bonds' rows are summed by shuffles that leave
// each lane the orbitals o = bond mod 4, and those lanes add the onsite rows and store.  For
// products too small to fill the chip: FP64 issues one warp instruction in 64 cycles on a
// sub-partition, so the product of a small block costs the FP64 instructions of one thread.
// The dependents are released after the wait, not before it: released at the start, kernel after kernel
// of a run of products comes to sit on the SMs, and blocks go where one has just left instead of
// spreading (8^3 cells, FP64, back to back: 8.1 against 5.2 us; 3x3x16, complex128: 9.9 against 5.6).
template <typename T, int NORB, bool CPLX, bool SO>
__global__ void __launch_bounds__(32) hx_split_kernel(const __grid_constant__ HxInst<T> I, double sigma, int cell0, int cell1,
                                                      const void* xv, void* yv) {
  using V = typename VecT<T, CPLX>::t;
  constexpr int CS = coef_stride(NORB), CELLS = CPLX ? 4 : 8, G = (NORB + 3) / 4;
  __shared__ __align__(16) T tab[2 * 16 * coef_stride(NORB)];
  stage_coef<T, NORB>(I.coef, I.ns, tab);
  const BondLane<T, NORB, CPLX> B(I, tab, blockIdx.x, cell0, cell1);
  const size_t N = I.g.natoms;
  const int k = B.k, atom = B.atom, sp = B.sp;
  const bool im = B.im;
  const T sc = B.sc;
  const int q = SO ? blockIdx.y : 0, v = blockIdx.z;
  const V* x = static_cast<const V*>(xv) + I.x_off + (size_t)v * I.nrows;
  const size_t spin = SO ? (size_t)(q * NORB) * N : 0;
  T c[CS];
  load_coef<T, NORB>(B.coef, c);
  pdl_wait();      // the vectors and the potential; structure and blocks do not change
  pdl_trigger();
  const V* xp = x + spin + B.n.atom;
  V xn[NORB], own[G];
#pragma unroll
  for (int o = 0; o < NORB; ++o) xn[o] = B.n.ok ? xp[o * N] : v_zero<V>();
#pragma unroll
  for (int j = 0; j < G; ++j) {
    const int o = 4 * j + k;
    own[j] = o < NORB ? x[spin + o * N + atom] : v_zero<V>();
  }
  T xs[NORB];
#pragma unroll
  for (int o = 0; o < NORB; ++o) xs[o] = B.component(xn[o]);
  T sg[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const bool minus = dir_minus(k, i);
    sg[i] = minus ? -sc : sc;
    if (minus) {
      xs[1 + i] = -xs[1 + i];
      if constexpr (NORB == 10) xs[4 + i] = -xs[4 + i];
    }
  }
  T r[4 * G];
  {
    T r0[NORB];
    bond_product<T, NORB>(c, xs, r0);
#pragma unroll
    for (int o = 0; o < 4 * G; ++o) {
      const bool odd = o >= 1 && o <= (NORB == 10 ? 6 : 3);
      r[o] = o < NORB ? (odd ? sg[(o - 1) % 3] : sc) * r0[o < NORB ? o : 0] : (T)0;
    }
  }
  const T u = (T)(I.U[atom] - sigma);
#pragma unroll
  for (int j = 0; j < G; ++j) {
    // bonds k and k^2, then k and k^1: of orbitals 4j..4j+3 the lane keeps 4j + k
    const bool h = k & 2, l = k & 1;
    const T a0 = (h ? r[4 * j + 2] : r[4 * j]) + __shfl_xor_sync(0xffffffffu, h ? r[4 * j] : r[4 * j + 2], 2 * CELLS);
    const T a1 = (h ? r[4 * j + 3] : r[4 * j + 1]) + __shfl_xor_sync(0xffffffffu, h ? r[4 * j + 1] : r[4 * j + 3], 2 * CELLS);
    const T sum = (l ? a1 : a0) + __shfl_xor_sync(0xffffffffu, l ? a0 : a1, CELLS);
    const int o = 4 * j + k;
    if (B.live && o < NORB) {
      T mine;
      if constexpr (CPLX) mine = im ? own[j].y : own[j].x; else mine = own[j];
      T out = fma(I.onsite[sp * NORB + o] + u, mine, sum);
      if constexpr (SO) {
        if (o >= 1 && o <= 3) {
          const int i = o - 1;
          const V* xo = x + (size_t)((1 - q) * NORB) * N + atom;
          const V first = i == 2 ? xo[2 * N] : x[spin + (i == 0 ? 2 : 1) * N + atom];
          const V t = so_term(q, i, first, i == 2 ? xo[N] : xo[3 * N]);
          out = fma((T)I.lambda[sp], im ? t.y : t.x, out);
        }
      }
      V* y = static_cast<V*>(yv) + I.x_off + (size_t)v * I.nrows + spin + o * N + atom;
      if constexpr (CPLX) (im ? y->y : y->x) = out; else *y = out;
    }
  }
}

template <typename T>
__device__ __forceinline__ T flip(T v, bool minus) {
  if constexpr (sizeof(T) == 8) return __hiloint2double(__double2hiint(v) ^ (minus ? 0x80000000 : 0), __double2loint(v));
  else return __int_as_float(__float_as_int(v) ^ (minus ? 0x80000000 : 0));
}

// And with one warp per kind of row besides, s and s*, p, t2g, e, for the smallest products: each
// warp reads the amplitudes of its kind, gives them the Bloch phase and the bond's signs and leaves
// them with their sums in shared memory for the others; then it forms its rows of the bond, sums
// them over the bonds by shuffles that leave lane k the k-th row, adds the onsite part and stores.
// Some 30 FP64 instructions of a warp between the vectors' arrival and the result, where a lane
// with all rows takes 100.  1x1x16 cells, complex128: 41.0 us with one thread per atom and full
// blocks, 26.7 us with one thread per atom and reduced blocks, 5.8 us with one lane per bond, 2.5 us
// here (back to back).
template <typename T, int NORB, bool CPLX, bool SO>
__global__ void __launch_bounds__(NORB == 10 ? 128 : 64) hx_kinds_kernel(const __grid_constant__ HxInst<T> I, double sigma, int cell0,
                                                                         int cell1, const void* xv, void* yv) {
  using V = typename VecT<T, CPLX>::t;
  constexpr int CELLS = CPLX ? 4 : 8;
  // what a kind leaves for the others: its amplitudes, their sum, and the zero-sum parts the e rows see
  enum { S = 0, SS, P0, PSUM = P0 + 3, PE1, PE2, T0, TSUM = T0 + 3, TE1, TE2, Q0, kShared = Q0 + 3 };
  __shared__ __align__(16) T tab[2 * 16 * coef_stride(NORB)];
  __shared__ T ex[kShared][32];
  stage_coef<T, NORB>(I.coef, I.ns, tab);
  const BondLane<T, NORB, CPLX> B(I, tab, blockIdx.x, cell0, cell1);
  const size_t N = I.g.natoms;
  // the kinds' warps in a turning order: the p and t2g ones, the longer, spread over an SM's sub-partitions
  const int lane = threadIdx.x & 31, kind = ((threadIdx.x >> 5) + blockIdx.x) & (NORB == 10 ? 3 : 1);
  const int k = B.k;
  const int q = SO ? blockIdx.y : 0, v = blockIdx.z;
  const V* x = static_cast<const V*>(xv) + I.x_off + (size_t)v * I.nrows;
  const size_t spin = SO ? (size_t)(q * NORB) * N : 0;
  // this kind's numbers of the reduced block, and its rows: orbitals o0 + j od
  constexpr int kS = NORB == 10 ? 8 : 6, kP = NORB == 10 ? 7 : 4;
  const int nc = kind == 0 ? kS : kind == 3 ? 5 : kP, c0 = kind == 0 ? 0 : kind == 1 ? kS : kind == 2 ? kS + kP : kS + 2 * kP;
  T c[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) c[i] = i < nc ? B.coef[c0 + i] : (T)0;
  const int rows = kind == 0 || kind == 3 ? 2 : 3;
  const int o0 = kind == 0 ? 0 : kind == 1 ? 1 : kind == 2 ? 4 : 7, od = kind == 0 ? NORB - 1 : 1;
  bool minus[3];
  T sg[3];                                         // the bond's factor with the row's sign
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    minus[i] = (kind == 1 || kind == 2) && dir_minus(k, i);
    sg[i] = flip(B.sc, minus[i]);
  }
  const int o = o0 + min(k, rows - 1) * od;        // the row this lane stores
  const T e0 = I.onsite[B.sp * NORB + o];
  pdl_wait();      // the vectors and the potential; structure and blocks do not change
  pdl_trigger();
  const V* xp = x + spin + B.n.atom;
  V xn[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) xn[j] = B.n.ok && j < rows ? xp[(o0 + j * od) * N] : v_zero<V>();
  const V own = x[spin + o * N + B.atom];
  const T u = (T)(I.U[B.atom] - sigma);
  T a[3];                                          // this lane's component, times phase and sign
#pragma unroll
  for (int j = 0; j < 3; ++j) a[j] = flip(B.component(xn[j]), minus[j]);
  constexpr T kHalf = (T)0.5, kR = (T)0.86602540378443865;   // sqrt(3)/2
  if (kind == 0) {
    ex[S][lane] = a[0];
    ex[SS][lane] = a[1];
  } else if (NORB == 5 || kind < 3) {
    const int at = kind == 1 ? P0 : T0;
    const T s = a[0] + a[1];
#pragma unroll
    for (int j = 0; j < 3; ++j) ex[at + j][lane] = a[j];
    ex[at + 3][lane] = s + a[2];
    if constexpr (NORB == 10) {
      ex[at + 4][lane] = a[0] - a[1];
      ex[at + 5][lane] = fma(-kHalf, s, a[2]);
    }
  } else {
    const T h = -kHalf * a[1];
    ex[Q0][lane] = fma(kR, a[0], h);
    ex[Q0 + 1][lane] = fma(-kR, a[0], h);
    ex[Q0 + 2][lane] = a[1];
  }
  __syncthreads();
  T r[3];
  if (kind == 0) {
    const T P = ex[PSUM][lane];
    if constexpr (NORB == 10) {
      const T Q = ex[TSUM][lane];
      r[0] = fma(c[3], a[1], fma(c[2], Q, fma(c[1], P, c[0] * a[0])));
      r[1] = fma(c[7], a[1], fma(c[6], Q, fma(c[5], P, c[4] * a[0])));
    } else {
      r[0] = fma(c[2], a[1], fma(c[1], P, c[0] * a[0]));
      r[1] = fma(c[5], a[1], fma(c[4], P, c[3] * a[0]));
    }
    r[2] = (T)0;
  } else if (NORB == 5) {
    const T C = fma(c[2], ex[PSUM][lane], fma(c[1], ex[SS][lane], c[0] * ex[S][lane]));
#pragma unroll
    for (int i = 0; i < 3; ++i) r[i] = fma(c[3], a[i], C);
  } else if (kind < 3) {
    // c: s, s*, P, T, p, t, q
    const T C = fma(c[3], ex[TSUM][lane], fma(c[2], ex[PSUM][lane], fma(c[1], ex[SS][lane], c[0] * ex[S][lane])));
#pragma unroll
    for (int i = 0; i < 3; ++i)
      r[i] = fma(c[5], ex[T0 + i][lane], fma(c[4], ex[P0 + i][lane], fma(c[6], ex[Q0 + i][lane], C)));
  } else {
    // c: p and t of the second row, t, e, p and t of the first
    r[0] = fma(c[2], a[0], fma(c[4], ex[TE1][lane], c[3] * ex[PE1][lane]));
    r[1] = fma(c[2], a[1], fma(c[1], ex[TE2][lane], c[0] * ex[PE2][lane]));
    r[2] = (T)0;
  }
#pragma unroll
  for (int j = 0; j < 3; ++j) r[j] *= sg[j];
  // bonds k and k^2, then k and k^1: of its kind's rows the lane keeps row k
  const bool h = k & 2, l = k & 1;
  const T a0 = (h ? r[2] : r[0]) + __shfl_xor_sync(0xffffffffu, h ? r[0] : r[2], 2 * CELLS);
  const T a1 = (h ? (T)0 : r[1]) + __shfl_xor_sync(0xffffffffu, h ? r[1] : (T)0, 2 * CELLS);
  const T sum = (l ? a1 : a0) + __shfl_xor_sync(0xffffffffu, l ? a0 : a1, CELLS);
  if (B.live && k < rows) {
    T mine;
    if constexpr (CPLX) mine = B.im ? own.y : own.x; else mine = own;
    T out = fma(e0 + u, mine, sum);
    if constexpr (SO) {
      if (kind == 1) {
        const V* xo = x + (size_t)((1 - q) * NORB) * N + B.atom;
        const V first = k == 2 ? xo[2 * N] : x[spin + (k == 0 ? 2 : 1) * N + B.atom];
        const V t = so_term(q, k, first, k == 2 ? xo[N] : xo[3 * N]);
        out = fma((T)I.lambda[B.sp], B.im ? t.y : t.x, out);
      }
    }
    V* y = static_cast<V*>(yv) + I.x_off + (size_t)v * I.nrows + spin + o * N + B.atom;
    if constexpr (CPLX) (B.im ? y->y : y->x) = out; else *y = out;
  }
}

// ---------------------------------------------------------------------------------------
// Double-float product (precision OMEN_F64_DF): every value is an FP32 pair (hi, lo) with
// value = hi + lo, products and sums by the error-free transformations of df.cuh, all on the
// FP32 pipe (57x GB300's FP64 rate), on reduced blocks like the rest: 1M atoms 0.325 ms with full
// blocks (79% of the HBM rate), 0.131 ms here (bound by the FP32 pipe, some 750 instructions a
// bond end).
struct HxDfArgs {
  Geo g;
  const float2* __restrict__ coef;     // as HxInst::coef, double-float
  const float2* __restrict__ scale;
  const uint8_t* __restrict__ species;
  const float2* __restrict__ onsite;   // [ns][norb] double-float
  const double* __restrict__ U;
  const float2* x;
  float2* y;
  long long nrows;
  double sigma;
  int ns;
  int cell0, cell1;                    // cells [cell0, cell1) of this launch
};

// Running double-float sum (S, C)
struct DfSum {
  float S, C;
  __device__ __forceinline__ float2 value() const { return df_norm(S, C); }
};
__device__ __forceinline__ DfSum ds_mul(float2 a, float2 b) {
  DfSum r;
  r.S = __fmul_rn(a.x, b.x);
  r.C = __fmaf_rn(a.y, b.x, __fmaf_rn(a.x, b.y, __fmaf_rn(a.x, b.x, -r.S)));
  return r;
}
__device__ __forceinline__ DfSum ds_mac(float2 a, float2 b, DfSum s) {
  df_mac(s.S, s.C, a, b);
  return s;
}
__device__ __forceinline__ float2 df_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 df_half(float2 a) { return make_float2(0.5f * a.x, 0.5f * a.y); }   // exact

// bond_product in double-float arithmetic
template <int NORB>
__device__ __forceinline__ void bond_product_df(const float2* __restrict__ c, const float2 (&x)[NORB], float2 (&r)[NORB]) {
  if constexpr (NORB == 5) {
    const float2 P = df_add(df_add(x[1], x[2]), x[3]);
    r[0] = ds_mac(c[2], x[4], ds_mac(c[1], P, ds_mul(c[0], x[0]))).value();
    r[4] = ds_mac(c[5], x[4], ds_mac(c[4], P, ds_mul(c[3], x[0]))).value();
    const DfSum C = ds_mac(c[8], P, ds_mac(c[7], x[4], ds_mul(c[6], x[0])));
#pragma unroll
    for (int i = 0; i < 3; ++i) r[1 + i] = ds_mac(c[9], x[1 + i], C).value();
  } else {
    const float2 kR = make_float2(0.866025388f, 1.55436253e-8f);   // sqrt(3)/2 as hi + lo
    const float2 p12 = df_add(x[1], x[2]), t12 = df_add(x[4], x[5]);
    const float2 P = df_add(p12, x[3]), Q = df_add(t12, x[6]);
    r[0] = ds_mac(c[3], x[9], ds_mac(c[2], Q, ds_mac(c[1], P, ds_mul(c[0], x[0])))).value();
    r[9] = ds_mac(c[7], x[9], ds_mac(c[6], Q, ds_mac(c[5], P, ds_mul(c[4], x[0])))).value();
    const DfSum Cp = ds_mac(c[11], Q, ds_mac(c[10], P, ds_mac(c[9], x[9], ds_mul(c[8], x[0]))));
    const DfSum Ct = ds_mac(c[18], Q, ds_mac(c[17], P, ds_mac(c[16], x[9], ds_mul(c[15], x[0]))));
    const float2 h = df_neg(df_half(x[8])), re = ds_mul(kR, x[7]).value();
    const float2 q[3] = {df_add(h, re), df_add(h, df_neg(re)), x[8]};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      r[1 + i] = ds_mac(c[13], x[4 + i], ds_mac(c[12], x[1 + i], ds_mac(c[14], q[i], Cp))).value();
      r[4 + i] = ds_mac(c[20], x[4 + i], ds_mac(c[19], x[1 + i], ds_mac(c[21], q[i], Ct))).value();
    }
    const float2 pe1 = df_add(x[1], df_neg(x[2])), te1 = df_add(x[4], df_neg(x[5]));
    const float2 pe2 = df_add(x[3], df_neg(df_half(p12))), te2 = df_add(x[6], df_neg(df_half(t12)));
    r[7] = ds_mac(c[24], x[7], ds_mac(c[26], te1, ds_mul(c[25], pe1))).value();
    r[8] = ds_mac(c[24], x[8], ds_mac(c[23], te2, ds_mul(c[22], pe2))).value();
  }
}

template <int NORB>
__global__ void __launch_bounds__(256) hx_df_kernel(const __grid_constant__ HxDfArgs a) {
  constexpr int CS = coef_stride(NORB);
  __shared__ __align__(16) float2 tab[2 * 16 * CS];
  stage_coef<float2, NORB>(a.coef, a.ns, tab);
  const Geo& g = a.g;
  const int item = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int b = item & 7;
  const int cell = a.cell0 + (item >> 3) * 32 + (threadIdx.x & 31);
  if (cell >= a.cell1) return;
  const size_t N = g.natoms;
  const int atom = b * g.ncells + cell;
  const int nxy = g.nx * g.ny;
  const int iz = cell / nxy, rem = cell - iz * nxy, iy = rem / g.nx, ix = rem - iy * g.nx;
  const Steps steps = steps_of(g, b, ix, iy, iz);
  const float2* __restrict__ x = a.x + (size_t)blockIdx.z * a.nrows;
  float2* __restrict__ y = a.y + (size_t)blockIdx.z * a.nrows;
  const int sp = a.species[atom];
  const bool is_a = b < 4;
  const float2* __restrict__ tb = tab + (is_a ? 0 : a.ns * a.ns * CS);
  DfSum acc[NORB];
  {
    const float2 u = df_from_double(a.U[atom] - a.sigma);
#pragma unroll
    for (int o = 0; o < NORB; ++o) acc[o] = ds_mul(df_add(a.onsite[sp * NORB + o], u), x[o * N + atom]);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const Neighbour n = neighbour_of(g, steps, b, k, cell);
    if (!n.ok) continue;
    const float2 sc = a.scale[n.slot];
    const int sp2 = a.species[n.atom];
    float2 xn[NORB], r[NORB];
#pragma unroll
    for (int o = 0; o < NORB; ++o) xn[o] = x[o * N + n.atom];
#pragma unroll
    for (int i = 0; i < 3; ++i)
      if (dir_minus(k, i)) {
        xn[1 + i] = df_neg(xn[1 + i]);
        if constexpr (NORB == 10) xn[4 + i] = df_neg(xn[4 + i]);
      }
    bond_product_df<NORB>(tb + (is_a ? sp * a.ns + sp2 : sp2 * a.ns + sp) * CS, xn, r);
#pragma unroll
    for (int o = 0; o < NORB; ++o) {
      const bool odd = o >= 1 && o <= (NORB == 10 ? 6 : 3);
      acc[o] = ds_mac(odd && dir_minus(k, (o - 1) % 3) ? df_neg(sc) : sc, r[o], acc[o]);
    }
  }
#pragma unroll
  for (int o = 0; o < NORB; ++o) y[o * N + atom] = acc[o].value();
}

__global__ void f64_to_df_kernel(const double* __restrict__ src, float2* __restrict__ dst, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    dst[i] = df_from_double(src[i]);
}
__global__ void df_to_f64_kernel(const float2* __restrict__ src, double* __restrict__ dst, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    dst[i] = (double)src[i].x + (double)src[i].y;
}

static cudaError_t launch_df(const omen_ham* h, const void* x, void* y, int nvec, double sigma, cudaStream_t st,
                             int cell0, int cell1) {
  const omen_lattice* L = h->lat;
  HxDfArgs a;
  a.g = Geo{L->nx, L->ny, L->nz, L->ncells, L->natoms, {L->periodic[0], L->periodic[1], L->periodic[2]}};
  a.coef = h->d_coefdf;
  a.scale = h->d_scaledf;
  a.species = L->d_species;
  a.onsite = h->d_onsite_df;
  a.U = h->d_U;
  a.x = static_cast<const float2*>(x);
  a.y = static_cast<float2*>(y);
  a.nrows = h->nrows;
  a.sigma = sigma;
  a.ns = h->nspecies;
  a.cell0 = cell0;
  a.cell1 = cell1;
  dim3 grid((cell1 - cell0 + 31) / 32, 1, nvec);   // a CTA's eight warps: the eight sites of 32 cells
  if (h->norb == 10) hx_df_kernel<10><<<grid, 256, 0, st>>>(a);
  else hx_df_kernel<5><<<grid, 256, 0, st>>>(a);
  return cudaGetLastError();
}

extern "C" omen_status omen_convert_vectors(omen_ctx* ctx, const void* src, int sp, void* dst, int dp, long long n) {
  if (!ctx || !src || !dst || n < 0) return set_err(ctx, OMEN_EINVAL, "null argument");
  const unsigned grid = (unsigned)std::max<long long>(1, std::min<long long>((n + 255) / 256, 152 * 16));
  if (sp == OMEN_F64 && dp == OMEN_F64_DF)
    f64_to_df_kernel<<<grid, 256, 0, ctx->stream>>>(static_cast<const double*>(src), static_cast<float2*>(dst), n);
  else if (sp == OMEN_F64_DF && dp == OMEN_F64)
    df_to_f64_kernel<<<grid, 256, 0, ctx->stream>>>(static_cast<const float2*>(src), static_cast<double*>(dst), n);
  else
    return set_err(ctx, OMEN_EINVAL, "conversion supports F64 <-> F64_DF");
  OMEN_CHECK_LAUNCH(ctx);
  return OMEN_OK;
}

// ---------------------------------------------------------------------------------------
// k-batched product over several structures: y = (H_i(k) - sigma) x for every wave vector k of
// every structure i, all in one launch (the (structure, k) work list).  Within a structure only
// the phase on bonds that wrap a Bloch face depends on k, so each thread finds its neighbours and
// reads their factors and reduced blocks once for KB wave vectors.  The CTAs of structure i are
// [cta0_i, cta0_i + tiles_i * ceil(nk_i / KB)); within them the tile index runs fastest.
// phases_i[k*3 + d] = exp(i k_d L_d).  Structure i's vectors are [nk_i][nrows_i] starting at
// element x_off_i of x and y.
// 4x4x80 cells, 32 wave vectors, complex64: 56 us per launch with full blocks, 28 us here (one wave
// vector a thread at 100 registers: 25 us; two at 160: 27 us; latency, 27 MB read and written in L2).
// Up to 128 wave vectors' phases travel as kernel parameters: allocating, copying and freeing a table
// held a call to 42 us among others and 285 us alone; 24 and 60 us without.
static constexpr int kMaxKInst = 16;

template <typename T>
struct KMulti {
  HxInst<T> in[kMaxKInst];
  int n;
  const void* x;
  void* y;
  double sigma;
  double2 ph[3 * kInlinePhases];      // phases of the structures whose table is null, in order
};

template <typename T, int NORB, int KB>
__global__ void __launch_bounds__(128, sizeof(T) == 8 ? 2 : KB == 1 ? 5 : KB == 2 ? 3 : 2) hx_kbatch_kernel(const __grid_constant__ KMulti<T> m) {
  __shared__ __align__(16) T tab[2 * 16 * coef_stride(NORB)];
  int inst = 0;
  while (inst + 1 < m.n && (int)blockIdx.x >= m.in[inst + 1].cta0) ++inst;
  const HxInst<T>& I = m.in[inst];
  stage_coef<T, NORB>(I.coef, I.ns, tab);
  const int local = (int)blockIdx.x - I.cta0;
  const int item = (local % I.tiles) * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int cell = (item >> 3) * 32 + (threadIdx.x & 31);
  if (cell >= I.g.ncells) return;
  const int k0 = (local / I.tiles) * KB;
  hx_rows<T, NORB, true, false, true, KB, 1>(I, tab, m.sigma, item & 7, cell, 0, k0, min(KB, I.nvec - k0), m.x, m.y,
                                              I.phases ? I.phases : m.ph + I.ph_at);
}

size_t vec_elem_bytes(const omen_ham* h, int precision) {
  const size_t r = (precision == OMEN_F64 || precision == OMEN_F64_DF) ? 8 : 4;
  return h->is_complex ? 2 * r : r;
}

// Up to this many CTAs (8 cells of a site, complex 4, a vector, a spin) take a warp per kind of row,
// and products of fewer warps (32 cells of a site, a vector, a spin) than split_below one lane per
// bond.  Back to back, us, row per lane / lane per bond / kinds (warps, CTAs), either side of the lines:
//   FP64    8^3 cells (128, 512) 14.4 / 4.6 / 4.4    9^3 (184, 736) 14.4 / 5.1 / 8.2
//           15^3 (848) 22.6 / 20.4                   16^3 (1024) 22.6 / 23.3
//   complex128  4x4x16 (64, 512) 26.7 / 5.8 / 5.9    5x5x16 (104, 800) 26.7 / 7.2 / 10.9
//           10x10x16 (400) 26.7 / 23.4
//   FP32    11^3 (336, 1336) 4.2 / 3.5 / 3.4         12^3 (432, 1728) 4.1 / 3.8 / 4.1
//           14^3 (688) 6.2 / 4.8                     16^3 (1024) 6.2 / 6.2
//   complex64   10x10x16 (400) 6.2 / 4.5             12x12x16 (576) 6.2 / 6.2
// sp3s*: FP64 12^3 (432) 6.2 / 4.9, 14^3 (688) 10.3 / 10.6; complex128 256 warps 12.4 / 6.9, 400
// 12.4 / 13.8.  Past 512 CTAs a sub-partition gets more than three and a half warps of the kinds, and
// FP64 instructions of one warp after the other bind; the lane per bond spends fewer in all.
static constexpr long long kinds_upto(bool f64, bool cplx) { return f64 || cplx ? 512 : 1336; }
static constexpr long long split_below(bool f64, bool cplx, int norb) {
  return norb == 5 ? (cplx ? 350 : 600) : !cplx ? 900 : f64 ? 450 : 560;
}

template <typename T, int NORB, bool CPLX, bool SO, int LB>
static cudaError_t launch_t(const HxInst<T>& I, int nvec, int threads, double sigma, int cell0, int cell1, const void* x,
                            void* y, cudaStream_t st) {
  const int warps = threads / 32;
  const long long items = (long long)((cell1 - cell0 + 31) / 32) * 8;
  const dim3 grid((unsigned)((items + warps - 1) / warps), SO ? 2 : 1, nvec);
  hx_kernel<T, NORB, CPLX, SO, LB><<<grid, threads, 0, st>>>(I, sigma, cell0, cell1, x, y);
  return cudaGetLastError();
}

// Whether `rb` is one of the load batches accepted for this kind of product (0 = the built-in
// rule): FP32 1, 2, 5, or the orbital count without spin-orbit; FP64 and matrix-free 1, 2; each must
// divide the orbital count.  (The values of an earlier kernel's register batches, accepted as before;
// loads_of says what they select.)
static bool rb_valid(int norb, bool f64, bool so, bool mf, int rb) {
  if (rb == 0) return true;
  if (rb < 0 || norb % rb != 0) return false;
  if (mf || f64) return rb == 1 || rb == 2;
  return rb == 1 || rb == 2 || rb == 5 || (rb == norb && !so);
}

// The kernel of a product, from the whole structure (so that a product computed in pieces has the same
// bits).
enum class HxRoute { kKinds, kSplit, kRows };
static HxRoute hx_route(int ncells, bool f64, bool cplx, bool so, int norb, int nvec) {
  const int cells = cplx ? 4 : 8;
  const long long each = 8ll * (so ? 2 : 1) * nvec;
  if ((ncells + cells - 1) / cells * each <= kinds_upto(f64, cplx)) return HxRoute::kKinds;
  return (ncells + 31) / 32 * each < split_below(f64, cplx, norb) ? HxRoute::kSplit : HxRoute::kRows;
}

// Bonds whose amplitudes are loaded together: rb 1 -> 1, 2 -> 2, 5 or 10 -> 4.
static int loads_of(bool f64, bool cplx, int rb) { return rb == 0 ? (!f64 && !cplx ? 2 : 1) : rb == 1 ? 1 : rb == 2 ? 2 : 4; }

template <typename T, int NORB, bool CPLX, bool SO>
static cudaError_t launch_rows(const HxInst<T>& I, int nvec, HxTile t, double sigma, int cell0, int cell1, const void* x,
                               void* y, cudaStream_t st) {
  constexpr int cells = CPLX ? 4 : 8;
  // a warp (kinds: a CTA) each; small CTAs spread over the SMs
  const dim3 grid((unsigned)((cell1 - cell0 + cells - 1) / cells) * 8, SO ? 2 : 1, nvec);
  const HxRoute route = hx_route(I.g.ncells, sizeof(T) == 8, CPLX, SO, NORB, nvec);
  if (route == HxRoute::kKinds)
    return launch_dependent(hx_kinds_kernel<T, NORB, CPLX, SO>, grid, dim3(NORB == 10 ? 128 : 64), 0, st, I, sigma, cell0, cell1, x, y);
  if (route == HxRoute::kSplit)
    return launch_dependent(hx_split_kernel<T, NORB, CPLX, SO>, grid, dim3(32), 0, st, I, sigma, cell0, cell1, x, y);
  const int thr = t.threads ? t.threads : 128;
  const int lb = loads_of(sizeof(T) == 8, CPLX, t.rb);
  if constexpr (sizeof(T) == 4) if (lb == 4) return launch_t<T, NORB, CPLX, SO, 4>(I, nvec, thr, sigma, cell0, cell1, x, y, st);
  if (lb == 2) return launch_t<T, NORB, CPLX, SO, 2>(I, nvec, thr, sigma, cell0, cell1, x, y, st);
  return launch_t<T, NORB, CPLX, SO, 1>(I, nvec, thr, sigma, cell0, cell1, x, y, st);
}

// Whether (threads, rb) is an accepted launch shape for this Hamiltonian and vector precision.
bool hx_tile_valid(const omen_ham* h, int vec_precision, int threads, int rb) {
  if (threads != 0 && (threads < 32 || threads > 128 || threads % 32 != 0)) return false;
  return rb_valid(h->norb, vec_precision == OMEN_F64, h->spin_orbit, h->matrix_free, rb);
}

// Whether products of nvec vectors look at the launch shape (small ones take one kernel whatever is set),
// and what distinguishes the shapes (threads, rb) there.
bool hx_takes_tile(const omen_ham* h, int vec_precision, int nvec) {
  return hx_route(h->lat->ncells, vec_precision == OMEN_F64, h->is_complex, h->spin_orbit, h->norb, nvec) == HxRoute::kRows;
}
int hx_tile_loads(const omen_ham* h, int vec_precision, int rb) { return loads_of(vec_precision == OMEN_F64, h->is_complex, rb); }

// The structure, reduced blocks and potential of a Hamiltonian for FP64 or FP32 products.
template <typename T>
static HxInst<T> make_inst(const omen_ham* h) {
  const omen_lattice* L = h->lat;
  HxInst<T> I{};
  I.g = Geo{L->nx, L->ny, L->nz, L->ncells, L->natoms, {L->periodic[0], L->periodic[1], L->periodic[2]}};
  if constexpr (sizeof(T) == 8) {
    I.coef = h->d_coef64;
    I.scale = h->d_scale64;
    I.onsite = h->d_onsite;
  } else {
    I.coef = h->d_coef32;
    I.scale = h->d_scale32;
    I.onsite = h->d_onsite32;
  }
  I.species = L->d_species;
  I.U = h->d_U;
  I.lambda = h->d_lambda;
  I.nrows = h->nrows;
  for (int d = 0; d < 3; ++d) I.phase[d] = h->phase[d];
  I.ns = h->nspecies;
  return I;
}

template <typename T>
static cudaError_t launch_prec(const omen_ham* h, const void* x, void* y, int nvec, double sigma, cudaStream_t st,
                               int cell0, int cell1) {
  const HxInst<T> I = make_inst<T>(h);
  const HxTile t = h->tile[sizeof(T) == 8 ? 0 : 1];
  auto go = [&](auto norb) {
    constexpr int NORB = decltype(norb)::value;
    if (!h->is_complex) return launch_rows<T, NORB, false, false>(I, nvec, t, sigma, cell0, cell1, x, y, st);
    if (!h->spin_orbit) return launch_rows<T, NORB, true, false>(I, nvec, t, sigma, cell0, cell1, x, y, st);
    return launch_rows<T, NORB, true, true>(I, nvec, t, sigma, cell0, cell1, x, y, st);
  };
  return h->norb == 10 ? go(std::integral_constant<int, 10>{}) : go(std::integral_constant<int, 5>{});
}

// y rows of the cells [cell0, cell1) (all orbitals, sites, vectors); the rest of y is untouched
static omen_status launch_hx_cells(omen_ctx* ctx, const omen_ham* h, const void* x, void* y, int nvec, double sigma,
                                   int vec_precision, int cell0, int cell1, cudaStream_t st) {
  if (nvec < 1 || nvec > 65535) return set_err(ctx, OMEN_EINVAL, "nvec must be 1..65535");
  if (cell1 <= cell0) return OMEN_OK;
  cudaError_t e;
  if (vec_precision == OMEN_F64_DF) {
    if (!h->d_scaledf) return set_err(ctx, OMEN_EINVAL, "Hamiltonian has no double-float blocks");
    e = launch_df(h, x, y, nvec, sigma, st, cell0, cell1);
  } else if (vec_precision == OMEN_F64) {
    if (!h->d_scale64) return set_err(ctx, OMEN_EINVAL, "Hamiltonian has no FP64 blocks");
    e = launch_prec<double>(h, x, y, nvec, sigma, st, cell0, cell1);
  } else {
    if (!h->d_scale32) return set_err(ctx, OMEN_EINVAL, "Hamiltonian has no FP32 blocks");
    e = launch_prec<float>(h, x, y, nvec, sigma, st, cell0, cell1);
  }
  if (e != cudaSuccess) return set_err(ctx, OMEN_ECUDA, "H·X launch failed: %s", cudaGetErrorString(e));
  return OMEN_OK;
}

omen_status launch_hx(omen_ctx* ctx, const omen_ham* h, const void* x, void* y, int nvec, double sigma, int vec_precision) {
  if (h->effmass) return launch_hx_effmass(ctx, h, x, y, nvec, sigma, vec_precision, ctx->stream);
  return launch_hx_cells(ctx, h, x, y, nvec, sigma, vec_precision, 0, h->lat->ncells, ctx->stream);
}

// The vector type of the Hamiltonian's products: FP32 for OMEN_F32 and OMEN_F32_REFINE64 (the
// refinement is internal to omen_eigs), double-float pairs for OMEN_F64_DF, else FP64.
static int native_precision(const omen_ham* h) {
  if (h->precision == OMEN_F64_DF) return OMEN_F64_DF;
  return (h->precision == OMEN_F32 || h->precision == OMEN_F32_REFINE64) ? OMEN_F32 : OMEN_F64;
}

extern "C" omen_status omen_hx(omen_ctx* ctx, const omen_ham* h, const void* x, void* y, int nvec, double sigma) {
  if (!ctx || !h || !x || !y) return set_err(ctx, OMEN_EINVAL, "null argument");
  return launch_hx(ctx, h, x, y, nvec, sigma, native_precision(h));
}

// Host-buffer product with the copies overlapped: the structure is cut into slabs of whole
// z-planes; slab i of x goes up on one copy stream, its rows of y are computed on the context's
// stream as soon as the planes they touch (the slab and one plane on each side) are on the
// device, and go down on the other copy stream while later slabs compute.  A slab of every
// vector is one strided copy: rows (vector, orbital, site) are ncells apart and a slab's cells
// are contiguous within each.  With a periodic z axis the first slab also needs the last
// plane, so it is computed last.
static omen_status hx_host_pipelined(omen_ctx* ctx, const omen_ham* h, const void* xh, void* yh, void* dx, void* dy,
                                     int nvec, double sigma) {
  const omen_lattice* L = h->lat;
  const int prec = native_precision(h);
  const size_t el = vec_elem_bytes(h, prec);
  const int plane = L->nx * L->ny;
  const int S = std::max(1, std::min(8, L->nz / 2));
  const size_t pitch = (size_t)L->ncells * el;
  const size_t rows = (size_t)nvec * (size_t)(h->nrows / L->ncells);   // (vector, orbital, site) runs
  for (int k = 0; k < 2; ++k)
    if (!ctx->copy_stream[k] && cudaStreamCreateWithFlags(&ctx->copy_stream[k], cudaStreamNonBlocking) != cudaSuccess) {
      ctx->copy_stream[k] = nullptr;
      return set_err(ctx, OMEN_ECUDA, "could not create a copy stream");
    }
  cudaStream_t sin = ctx->copy_stream[0], sout = ctx->copy_stream[1];
  omen_status st = OMEN_OK;
  while (st == OMEN_OK && ctx->host_events.size() < (size_t)(2 * S + 2)) {
    cudaEvent_t e = nullptr;
    if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) st = set_err(ctx, OMEN_ECUDA, "event creation failed");
    else ctx->host_events.push_back(e);
  }
  if (st != OMEN_OK) return st;
  std::vector<cudaEvent_t>& ev = ctx->host_events;
  auto z0 = [&](int i) { return (int)((long long)L->nz * i / S); };
  cudaEvent_t* ein = ev.data();
  cudaEvent_t* ecomp = ev.data() + S;
  cudaEvent_t start = ev[2 * S], done = ev[2 * S + 1];
  cudaError_t e = cudaSuccess;
  if (st == OMEN_OK) {
    // order the copy streams after the context's stream (earlier work on the buffers)
    e = cudaEventRecord(start, ctx->stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(sin, start, 0);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(sout, start, 0);
  }
  for (int i = 0; i < S && st == OMEN_OK && e == cudaSuccess; ++i) {
    const size_t c0 = (size_t)z0(i) * plane, c1 = (size_t)z0(i + 1) * plane;
    e = cudaMemcpy2DAsync(static_cast<char*>(dx) + c0 * el, pitch, static_cast<const char*>(xh) + c0 * el, pitch,
                          (c1 - c0) * el, rows, cudaMemcpyHostToDevice, sin);
    if (e == cudaSuccess) e = cudaEventRecord(ein[i], sin);
  }
  const bool zper = L->periodic[2] != OMEN_HARD_WALL;
  for (int t = 0; t < S && st == OMEN_OK && e == cudaSuccess; ++t) {
    const int i = zper ? (t + 1) % S : t;     // periodic z: slab 0 last
    const int need = zper && i == 0 ? S - 1 : std::min(i + 1, S - 1);
    e = cudaStreamWaitEvent(ctx->stream, ein[need], 0);
    if (e != cudaSuccess) break;
    st = launch_hx_cells(ctx, h, dx, dy, nvec, sigma, prec, z0(i) * plane, z0(i + 1) * plane, ctx->stream);
    if (st != OMEN_OK) break;
    e = cudaEventRecord(ecomp[i], ctx->stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(sout, ecomp[i], 0);
    const size_t c0 = (size_t)z0(i) * plane, c1 = (size_t)z0(i + 1) * plane;
    if (e == cudaSuccess)
      e = cudaMemcpy2DAsync(static_cast<char*>(yh) + c0 * el, pitch, static_cast<const char*>(dy) + c0 * el, pitch,
                            (c1 - c0) * el, rows, cudaMemcpyDeviceToHost, sout);
  }
  // the context's stream (and the caller's frees on it) wait for the last copy down
  if (st == OMEN_OK && e == cudaSuccess) e = cudaEventRecord(done, sout);
  if (st == OMEN_OK && e == cudaSuccess) e = cudaStreamWaitEvent(ctx->stream, done, 0);
  if (st == OMEN_OK && e != cudaSuccess) st = set_err(ctx, OMEN_ECUDA, "host H·X copies: %s", cudaGetErrorString(e));
  if (st != OMEN_OK) {
    // leave nothing in flight on the copy streams before the buffers go back
    cudaStreamSynchronize(sin);
    cudaStreamSynchronize(sout);
  }
  return st;
}

extern "C" omen_status omen_hx_host(omen_ctx* ctx, const omen_ham* h, const void* xh, void* yh, int nvec, double sigma) {
  if (!ctx || !h || !xh || !yh) return set_err(ctx, OMEN_EINVAL, "null argument");
  if (nvec < 1) return set_err(ctx, OMEN_EINVAL, "nvec must be >= 1");
  const size_t bytes = vec_elem_bytes(h, native_precision(h)) * (size_t)h->nrows * nvec;
  if (h->precision == OMEN_F64_DF) {
    // FP64 host arrays; double-float conversion on the device
    const long long n = h->nrows * nvec;
    void *dx = nullptr, *dy = nullptr, *fx = nullptr;
    if (ctx_alloc(ctx, &dx, bytes) != cudaSuccess || ctx_alloc(ctx, &dy, bytes) != cudaSuccess ||
        ctx_alloc(ctx, &fx, 8 * (size_t)n) != cudaSuccess) {
      cudaGetLastError();
      if (dx) cudaFreeAsync(dx, ctx->stream);
      if (dy) cudaFreeAsync(dy, ctx->stream);
      return set_err(ctx, OMEN_ENOMEM, "device allocation of %zu bytes failed", bytes);
    }
    omen_status st = OMEN_OK;
    cudaError_t e = cudaMemcpyAsync(fx, xh, 8 * (size_t)n, cudaMemcpyHostToDevice, ctx->stream);
    if (e == cudaSuccess) st = omen_convert_vectors(ctx, fx, OMEN_F64, dx, OMEN_F64_DF, n);
    if (e == cudaSuccess && st == OMEN_OK) st = launch_hx(ctx, h, dx, dy, nvec, sigma, OMEN_F64_DF);
    if (e == cudaSuccess && st == OMEN_OK) st = omen_convert_vectors(ctx, dy, OMEN_F64_DF, fx, OMEN_F64, n);
    if (e == cudaSuccess && st == OMEN_OK) e = cudaMemcpyAsync(yh, fx, 8 * (size_t)n, cudaMemcpyDeviceToHost, ctx->stream);
    cudaFreeAsync(dx, ctx->stream);
    cudaFreeAsync(dy, ctx->stream);
    cudaFreeAsync(fx, ctx->stream);
    cudaError_t e2 = cudaStreamSynchronize(ctx->stream);
    if (st != OMEN_OK) return st;
    if (e != cudaSuccess || e2 != cudaSuccess)
      return set_err(ctx, OMEN_ECUDA, "host H·X failed: %s", cudaGetErrorString(e != cudaSuccess ? e : e2));
    return OMEN_OK;
  }
  const size_t half = (bytes + 255) / 256 * 256;
  if (ctx->host_scratch_bytes < 2 * half) {
    // grow the context's scratch (synchronises the device once; later calls reuse it)
    OMEN_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    if (ctx->host_scratch) cudaFree(ctx->host_scratch);
    ctx->host_scratch = nullptr;
    ctx->host_scratch_bytes = 0;
    if (cudaMalloc(&ctx->host_scratch, 2 * half) != cudaSuccess) {
      cudaGetLastError();
      ctx->host_scratch = nullptr;
      return set_err(ctx, OMEN_ENOMEM, "device allocation of %zu bytes failed", 2 * half);
    }
    ctx->host_scratch_bytes = 2 * half;
  }
  void* dx = ctx->host_scratch;
  void* dy = static_cast<char*>(ctx->host_scratch) + half;
  omen_status st = OMEN_OK;
  if (h->effmass) {
    // one copy up, the product, one copy down
    cudaError_t e = cudaMemcpyAsync(dx, xh, bytes, cudaMemcpyHostToDevice, ctx->stream);
    if (e == cudaSuccess) st = launch_hx(ctx, h, dx, dy, nvec, sigma, native_precision(h));
    if (e == cudaSuccess && st == OMEN_OK) e = cudaMemcpyAsync(yh, dy, bytes, cudaMemcpyDeviceToHost, ctx->stream);
    if (e != cudaSuccess && st == OMEN_OK) st = set_err(ctx, OMEN_ECUDA, "host H·X copies: %s", cudaGetErrorString(e));
  } else {
    st = hx_host_pipelined(ctx, h, xh, yh, dx, dy, nvec, sigma);
  }
  cudaError_t e2 = cudaStreamSynchronize(ctx->stream);
  if (st != OMEN_OK) return st;
  if (e2 != cudaSuccess) return set_err(ctx, OMEN_ECUDA, "host H·X failed: %s", cudaGetErrorString(e2));
  return OMEN_OK;
}

// Wave vectors per thread KB: 1 by default (registers: two FP64 ones spill, two FP32 ones leave 12
// warps an SM); 1, 2, 4 compiled for FP32 and 1, 2 for FP64.
static bool kb_compiled(bool f64, int kb) { return kb == 0 || kb == 1 || kb == 2 || (!f64 && kb == 4); }

bool hx_kbatch_tile_valid(int vec_precision, int threads, int kb) {
  if (threads != 0 && (threads < 32 || threads > 128 || threads % 32 != 0)) return false;
  return kb_compiled(vec_precision == OMEN_F64, kb);
}

template <typename T, int KB>
static cudaError_t launch_kb(KMulti<T>& m, int norb, int threads, cudaStream_t st) {
  const int warps = threads / 32;
  long long total = 0;
  for (int i = 0; i < m.n; ++i) {
    const int items = ((m.in[i].g.ncells + 31) / 32) * 8;
    m.in[i].tiles = (items + warps - 1) / warps;
    m.in[i].cta0 = (int)total;
    total += (long long)m.in[i].tiles * ((m.in[i].nvec + KB - 1) / KB);
  }
  if (total > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  if (norb == 10) hx_kbatch_kernel<T, 10, KB><<<(unsigned)total, threads, 0, st>>>(m);
  else hx_kbatch_kernel<T, 5, KB><<<(unsigned)total, threads, 0, st>>>(m);
  return cudaGetLastError();
}

template <typename T>
static cudaError_t launch_kmulti_prec(const KItem* items, int nitems, const void* x, void* y, double sigma,
                                      cudaStream_t st) {
  KMulti<T> m;
  m.n = nitems;
  m.x = x;
  m.y = y;
  m.sigma = sigma;
  int ph = 0;
  for (int i = 0; i < nitems; ++i) {
    m.in[i] = make_inst<T>(items[i].ham);
    if (!items[i].phases) {
      m.in[i].ph_at = ph;
      std::copy(items[i].phases_host, items[i].phases_host + 3 * items[i].nk, m.ph + ph);
      ph += 3 * items[i].nk;
    }
    m.in[i].phases = items[i].phases;
    m.in[i].x_off = items[i].x_off;
    m.in[i].nvec = items[i].nk;
  }
  const HxTile t = items[0].ham->ktile[sizeof(T) == 8 ? 0 : 1];
  const int thr = t.threads ? t.threads : 128;
  if (t.rb == 1) return launch_kb<T, 1>(m, items[0].ham->norb, thr, st);
  if constexpr (sizeof(T) == 4) if (t.rb == 4) return launch_kb<T, 4>(m, items[0].ham->norb, thr, st);
  if (t.rb == 2) return launch_kb<T, 2>(m, items[0].ham->norb, thr, st);
  return launch_kb<T, 1>(m, items[0].ham->norb, thr, st);
}

omen_status launch_hx_kmulti(omen_ctx* ctx, const KItem* items, int nitems, const void* x, void* y, double sigma,
                             int vec_precision) {
  if (nitems < 1 || nitems > kMaxKInst) return set_err(ctx, OMEN_EINVAL, "1..%d structures per k batch", kMaxKInst);
  const bool f64 = vec_precision == OMEN_F64;
  for (int i = 0; i < nitems; ++i) {
    const omen_ham* h = items[i].ham;
    if (!h || items[i].nk < 1 || items[i].nk > 65535) return set_err(ctx, OMEN_EINVAL, "structure %d: null or nk out of range", i);
    if (!h->bloch || h->matrix_free || h->spin_orbit)
      return set_err(ctx, OMEN_EUNSUPPORTED, "k batch needs Bloch structures with stored blocks and no spin-orbit");
    if (h->norb != items[0].ham->norb) return set_err(ctx, OMEN_EINVAL, "structures of one k batch share the basis");
    if (f64 ? !h->d_scale64 : !h->d_scale32) return set_err(ctx, OMEN_EINVAL, "structure %d has no blocks of this precision", i);
  }
  const cudaError_t e = f64 ? launch_kmulti_prec<double>(items, nitems, x, y, sigma, ctx->stream)
                            : launch_kmulti_prec<float>(items, nitems, x, y, sigma, ctx->stream);
  if (e != cudaSuccess) return set_err(ctx, OMEN_ECUDA, "k-batched H·X launch: %s", cudaGetErrorString(e));
  return OMEN_OK;
}

omen_status launch_hx_kbatch(omen_ctx* ctx, const omen_ham* h, int nk, const double2* phases_dev, const void* x, void* y,
                             double sigma, int vec_precision) {
  const KItem item{h, nk, phases_dev, 0};
  return launch_hx_kmulti(ctx, &item, 1, x, y, sigma, vec_precision);
}

std::vector<double2> phase_table(const omen_ham* h, int nk, const double* k_host) {
  const omen_lattice* L = h->lat;
  std::vector<double2> ph((size_t)nk * 3);
  const int nc[3] = {L->nx, L->ny, L->nz};
  for (int q = 0; q < nk; ++q)
    for (int d = 0; d < 3; ++d) {
      const double t = (L->periodic[d] == OMEN_BLOCH) ? k_host[q * 3 + d] * nc[d] * L->a_nm : 0.0;
      ph[(size_t)q * 3 + d] = make_double2(cos(t), sin(t));
    }
  return ph;
}

omen_status make_phases(omen_ctx* ctx, const omen_ham* h, int nk, const double* k_host, double2** out) {
  const std::vector<double2> ph = phase_table(h, nk, k_host);
  if (ctx_alloc(ctx, out, sizeof(double2) * ph.size()) != cudaSuccess) {
    cudaGetLastError();
    return set_err(ctx, OMEN_ENOMEM, "phase table");
  }
  OMEN_CUDA(ctx, copy_as_params(ctx->stream, *out, ph.data(), sizeof(double2) * ph.size()));   // ph goes on return
  return OMEN_OK;
}

extern "C" omen_status omen_hx_kbatch_multi(omen_ctx* ctx, int nitems, const omen_kbatch_item* it, const void* x, void* y,
                                            double sigma) {
  if (!ctx || !it || !x || !y || nitems < 1 || nitems > kMaxKInst) return set_err(ctx, OMEN_EINVAL, "null argument or 1..%d structures", kMaxKInst);
  std::vector<KItem> items(nitems);
  std::vector<double2*> ph(nitems, nullptr);
  std::vector<std::vector<double2>> inl(nitems);
  long long off = 0, total = 0;
  for (int i = 0; i < nitems; ++i) total += std::max(0, it[i].nk);
  // a few wave vectors travel with the launch: no table to allocate, copy and free
  const bool with_launch = total <= kInlinePhases;
  omen_status s = OMEN_OK;
  for (int i = 0; i < nitems && s == OMEN_OK; ++i) {
    if (!it[i].ham || !it[i].k_host || it[i].nk < 1) { s = set_err(ctx, OMEN_EINVAL, "structure %d: null argument or nk < 1", i); break; }
    if (it[i].ham->effmass) { s = set_err(ctx, OMEN_EUNSUPPORTED, "k batch runs on tight-binding Hamiltonians"); break; }
    if (!it[i].ham->bloch) { s = set_err(ctx, OMEN_EINVAL, "structure %d has no Bloch-periodic direction", i); break; }
    if (with_launch) inl[i] = phase_table(it[i].ham, it[i].nk, it[i].k_host);
    else s = make_phases(ctx, it[i].ham, it[i].nk, it[i].k_host, &ph[i]);
    items[i] = KItem{it[i].ham, it[i].nk, ph[i], off, inl[i].data()};
    off += (long long)it[i].nk * it[i].ham->nrows;
  }
  if (s == OMEN_OK) {
    const omen_ham* h0 = it[0].ham;
    for (int i = 1; i < nitems && s == OMEN_OK; ++i)
      if (it[i].ham->precision != h0->precision) s = set_err(ctx, OMEN_EINVAL, "structures of one k batch share the precision");
    if (s == OMEN_OK) s = launch_hx_kmulti(ctx, items.data(), nitems, x, y, sigma, native_precision(h0));
  }
  for (double2* q : ph)
    if (q) cudaFreeAsync(q, ctx->stream);
  return s;
}

extern "C" omen_status omen_hx_kbatch(omen_ctx* ctx, const omen_ham* h, int nk, const double* k_host, const void* x,
                                      void* y, double sigma) {
  if (!ctx || !h || !k_host || !x || !y || nk < 1) return set_err(ctx, OMEN_EINVAL, "null argument or nk < 1");
  if (h->effmass) return set_err(ctx, OMEN_EUNSUPPORTED, "k batch runs on tight-binding Hamiltonians");
  if (!h->bloch) return set_err(ctx, OMEN_EINVAL, "k batch needs a structure with Bloch-periodic directions");
  const omen_kbatch_item item{h, nk, k_host};
  return omen_hx_kbatch_multi(ctx, 1, &item, x, y, sigma);
}
