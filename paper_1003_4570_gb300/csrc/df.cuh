// Double-float arithmetic: a value is an FP32 pair (hi, lo) with value = hi + lo (about 48
// significant bits).  A product a*b is formed exactly in its leading part (p = fl(a.hi b.hi),
// e = fma(a.hi, b.hi, -p); Dekker 1971) plus the cross terms; it is added to a running (S, C)
// pair with Knuth's TwoSum, the rounding error of the sum going into C.  The _rn intrinsics keep
// the compiler from contracting the additions into FMAs, which would break the error-free
// transformations.
#pragma once
#include <cuda_runtime.h>

__device__ __forceinline__ void df_mac(float& S, float& C, float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  float e = __fmaf_rn(a.x, b.x, -p);
  e = __fmaf_rn(a.x, b.y, e);
  e = __fmaf_rn(a.y, b.x, e);
  const float s = __fadd_rn(S, p);
  const float bb = __fsub_rn(s, S);
  const float t = __fadd_rn(__fsub_rn(S, __fsub_rn(s, bb)), __fsub_rn(p, bb));
  C = __fadd_rn(C, __fadd_rn(t, e));
  S = s;
}
__device__ __forceinline__ float2 df_norm(float S, float C) {
  const float h = __fadd_rn(S, C);
  return make_float2(h, __fsub_rn(C, __fsub_rn(h, S)));
}
__device__ __forceinline__ float2 df_add(float2 a, float2 b) {
  const float s = __fadd_rn(a.x, b.x);
  const float bb = __fsub_rn(s, a.x);
  const float t = __fadd_rn(__fsub_rn(a.x, __fsub_rn(s, bb)), __fsub_rn(b.x, bb));
  return df_norm(s, __fadd_rn(t, __fadd_rn(a.y, b.y)));
}
__device__ __forceinline__ float2 df_from_double(double v) {
  const float hi = __double2float_rn(v);
  return make_float2(hi, __double2float_rn(v - (double)hi));
}

// v 2^kSplitShift as an FP32 pair (hi, lo), by integer operations only (the FP64 pipe, which
// df_from_double uses, has 1/64 of the FP32 rate).  kRound: hi is v rounded to 24 significant bits and
// lo the signed rest rounded to 24, so the pair is within 2^-49 of v relatively, as df_from_double's
// is.  Else hi is the leading 24 bits: within 2^-48, twice the error on average, in fewer
// instructions (electrons per atom of 16 states of 1M atoms: 229 us, 260 us with rounding).
// Magnitudes too small for FP32 give zero, too large or non-finite ones NaN.
struct SplitBits {
  unsigned hi, scale;                  // hi, and the unit of the rest with v's sign, as FP32 bits
  int rest;
};
template <int kSplitShift, bool kRound>
__host__ __device__ __forceinline__ SplitBits split_bits(unsigned long long b) {
  const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
  const int e = (int)((unsigned)(b >> 52) & 0x7FFu);                       // biased FP64 exponent
  // half of hi's last place, which may carry up to the exponent, leaves the bits of hi on top
  const unsigned long long top = kRound ? b + 0x10000000u : b;
  const int eh = (kRound ? (int)((unsigned)(top >> 52) & 0x7FFu) : e) - 896 + kSplitShift;   // FP32 exponent of hi
  if (eh <= 0) return SplitBits{0, 0, 0};                                  // |v| < 2^-158 (shift 32), or zero
  if (eh >= 255) return SplitBits{0x7fc00000u, 0, 0};                      // beyond FP32, inf or NaN: NaN
  // the rest in units of 2^(e - 1075 + shift)
  const int el = e - 948 + kSplitShift;
  return SplitBits{sign | ((unsigned)eh << 23) | ((unsigned)(top >> 29) & 0x7FFFFFu), el > 0 ? sign | ((unsigned)el << 23) : 0u,
                   (int)((unsigned)top & 0x1FFFFFFFu) - (kRound ? 0x10000000 : 0)};
}
template <int kSplitShift, bool kRound>
__device__ __forceinline__ float2 split_fp64(double v) {
  const SplitBits s = split_bits<kSplitShift, kRound>((unsigned long long)__double_as_longlong(v));
  return make_float2(__uint_as_float(s.hi), __fmul_rn(__int2float_rn(s.rest), __uint_as_float(s.scale)));
}
