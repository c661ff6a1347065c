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
// df_from_double uses, has 1/64 of the FP32 rate): hi keeps the sign, the exponent and the leading
// 24 significant bits, lo is the rest rounded to FP32 (48 significant bits in all: the pair is within
// 2^-48 of v relatively).  Magnitudes too small for FP32 give zero, too large or non-finite ones NaN.
template <int kSplitShift>
__device__ __forceinline__ float2 split_fp64(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const unsigned hi32 = (unsigned)(b >> 32), lo32 = (unsigned)b;
  const int e = (int)((hi32 >> 20) & 0x7FFu);   // biased FP64 exponent
  // FP32 exponent of hi: e - 1023 + 127 + shift
  const int eh = e - 896 + kSplitShift;
  if (eh <= 0) return make_float2(0.f, 0.f);     // |v| < 2^-158, or zero
  if (eh >= 255) return make_float2(__int_as_float(0x7fc00000), 0.f);   // beyond FP32, inf or NaN: NaN
  const unsigned sign = hi32 & 0x80000000u;
  const unsigned top23 = ((hi32 & 0xFFFFFu) << 3) | (lo32 >> 29);
  const float hi = __uint_as_float(sign | ((unsigned)eh << 23) | top23);
  // the remaining 29 bits: rem * 2^(e - 1075 + shift)
  const unsigned rem = lo32 & 0x1FFFFFFFu;
  const int el = e - 948 + kSplitShift;
  const float scale = el > 0 ? __uint_as_float((unsigned)el << 23) : 0.f;
  const float lo = __fmul_rn(__uint2float_rn(rem), scale);
  return make_float2(hi, sign ? -lo : lo);
}

// The same with hi rounded to 24 significant bits and lo the signed rest: within 2^-49 of v, as
// df_from_double is, with half the error on average, for some more instructions (electrons per atom
// of 16 states of 1M atoms would take 260 us with it, 229 us with the leading bits).
struct SplitBits {
  unsigned hi, scale;                  // hi, and the unit of the rest with v's sign, as FP32 bits
  int rest;
};
template <int kSplitShift>
__host__ __device__ __forceinline__ SplitBits split_rounded_bits(unsigned long long b) {
  const unsigned long long up = b + 0x10000000u;    // half of hi's last place, which may carry up to the exponent
  const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
  const int e = (int)((unsigned)(b >> 52) & 0x7FFu), eu = (int)((unsigned)(up >> 52) & 0x7FFu);   // biased FP64 exponents
  const int eh = eu - 896 + kSplitShift;            // FP32 exponent of hi
  if (eh <= 0) return SplitBits{0, 0, 0};
  if (eh >= 255) return SplitBits{0x7fc00000u, 0, 0};
  // the rest in units of 2^(e - 1075 + shift)
  const int el = e - 948 + kSplitShift;
  return SplitBits{sign | ((unsigned)eh << 23) | ((unsigned)(up >> 29) & 0x7FFFFFu), el > 0 ? sign | ((unsigned)el << 23) : 0u,
                   (int)((unsigned)up & 0x1FFFFFFFu) - 0x10000000};
}
template <int kSplitShift>
__device__ __forceinline__ float2 split_fp64_rounded(double v) {
  const SplitBits s = split_rounded_bits<kSplitShift>((unsigned long long)__double_as_longlong(v));
  return make_float2(__uint_as_float(s.hi), __fmul_rn(__int2float_rn(s.rest), __uint_as_float(s.scale)));
}
