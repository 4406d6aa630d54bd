// Double-float ("ff") arithmetic for the float64-accuracy kernels of the
// mixed-precision path.  A value is hi + lo in two float32s (about 47
// significant bits), evaluated on the float32 pipes, which GB300 runs at 64x
// its float64 rate.  Products use the exact float32 product error of an FMA,
// sums Knuth's two-sum; every rounding-sensitive operation uses the _rn
// intrinsics so that the compiler cannot contract or reorder it.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

// float64 -> hi + lo from the bit fields, with no float64 instruction: hi = x
// truncated to 24 significant bits, lo = the next 23 bits (truncated), both
// with the sign of x; |x - hi - lo| < 2^-46 |x|.  |x| < 2^-126 gives 0, lo is
// dropped below |x| = 2^-80, and NaN, Inf or |x| >= 2^128 give NaN.
__device__ __forceinline__ void ff_split(double x, float& hi, float& lo) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  const uint32_t w1 = (uint32_t)(b >> 32), w0 = (uint32_t)b;
  const uint32_t sign = w1 & 0x80000000u;
  const int e = (int)((w1 >> 20) & 0x7FFu);
  const int ef = e - 896;  // float exponent field of x
  const uint32_t hb = sign | ((uint32_t)ef << 23) | ((w1 & 0xFFFFFu) << 3) | (w0 >> 29);
  hi = ef > 0 ? __uint_as_float(hb) : __uint_as_float(sign);
  if (ef >= 255) hi = __uint_as_float(0x7FC00000u);
  // the next 23 significand bits as an exact float integer, times 2^(e - 1069)
  const float m = __fsub_rn(__uint_as_float(0x4B000000u | ((w0 & 0x1FFFFFFFu) >> 6)), 8388608.0f);
  const int es = e - 942;
  const float s = __uint_as_float((uint32_t)(es > 0 ? (es < 255 ? es : 0) : 0) << 23);
  lo = __uint_as_float(__float_as_uint(__fmul_rn(m, s)) | sign);
}

// float32 -> float64 from the bit fields (float subnormals flush to 0).
__device__ __forceinline__ double ff_f2d(float f) {
  const uint32_t u = __float_as_uint(f);
  const uint32_t ef = (u >> 23) & 0xFFu;
  if (ef == 0) return __longlong_as_double((long long)((uint64_t)(u & 0x80000000u) << 32));
  const uint64_t ed = ef == 255 ? 2047ull : (uint64_t)(ef + 896);
  return __longlong_as_double(
      (long long)(((uint64_t)(u & 0x80000000u) << 32) | (ed << 52) | ((uint64_t)(u & 0x7FFFFFu) << 29)));
}

// hi + lo rounded to float64 (one float64 addition).
__device__ __forceinline__ double ff_to_double(float hi, float lo) { return __dadd_rn(ff_f2d(hi), ff_f2d(lo)); }

// ----------------------------------------------------------------------------------------------
// The arithmetic, on two values at once: the packed float32 instructions of sm_100 and later (f32x2)
// take one issue slot for two lanes' worth of work.  The float32 pipe's rate is the same and so are the
// results.  It takes the bordering kernel from 266 to 174 thread instructions an entry and its issue slots
// from 65 to 46 % busy (h = 1/512, k = 64; 182 -> 172 us): what is left is the latency of the gathers at
// half occupancy, beside a float32 pipe that is 53 % busy.  A block vector "in pairs" stores two columns as
// one 16-byte chunk (hi0, hi1, lo0, lo1), so that a 16-byte load gives both packed operands.
typedef unsigned long long ff2;  // two float32

__device__ __forceinline__ ff2 ff2_pack(float a, float b) {
  ff2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void ff2_unpack(ff2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ ff2 ff2_addrn(ff2 a, ff2 b) {
  ff2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ ff2 ff2_subrn(ff2 a, ff2 b) {
  ff2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ ff2 ff2_mulrn(ff2 a, ff2 b) {
  ff2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ ff2 ff2_fmarn(ff2 a, ff2 b, ff2 c) {
  ff2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ ff2 ff2_neg(ff2 a) { return a ^ 0x8000000080000000ull; }

// (hi, lo) += -n + e for the product -n with exact error e (two-sum of hi and -n)
__device__ __forceinline__ void ff2_accumulate(ff2& hi, ff2& lo, ff2 n, ff2 e) {
  const ff2 s = ff2_subrn(hi, n);
  const ff2 bb = ff2_subrn(s, hi);
  const ff2 t = ff2_subrn(ff2_subrn(hi, ff2_subrn(s, bb)), ff2_addrn(n, bb));
  hi = s;
  lo = ff2_addrn(lo, ff2_addrn(t, e));
}
// (hi, lo) += (ah + al) * (xh + xl); na = -ah
__device__ __forceinline__ void ff2_mac(ff2& hi, ff2& lo, ff2 ah, ff2 na, ff2 al, ff2 xh, ff2 xl) {
  const ff2 n = ff2_mulrn(na, xh);
  ff2 e = ff2_fmarn(ah, xh, n);
  e = ff2_fmarn(ah, xl, e);
  e = ff2_fmarn(al, xh, e);
  ff2_accumulate(hi, lo, n, e);
}
// ff2_mac for a float32 coefficient a (no low part)
__device__ __forceinline__ void ff2_mac_exact(ff2& hi, ff2& lo, ff2 a, ff2 na, ff2 xh, ff2 xl) {
  const ff2 n = ff2_mulrn(na, xh);
  ff2 e = ff2_fmarn(a, xh, n);
  e = ff2_fmarn(a, xl, e);
  ff2_accumulate(hi, lo, n, e);
}
// (hi, lo) += v
__device__ __forceinline__ void ff2_add(ff2& hi, ff2& lo, ff2 v) {
  const ff2 s = ff2_addrn(hi, v);
  const ff2 bb = ff2_subrn(s, hi);
  const ff2 t = ff2_addrn(ff2_subrn(hi, ff2_subrn(s, bb)), ff2_subrn(v, bb));
  hi = s;
  lo = ff2_addrn(lo, t);
}
__device__ __forceinline__ void ff2_norm(ff2& hi, ff2& lo) {
  const ff2 s = ff2_addrn(hi, lo);
  lo = ff2_subrn(lo, ff2_subrn(s, hi));
  hi = s;
}
// (hi, lo) = (ah + al) * (bh + bl), renormalised
__device__ __forceinline__ void ff2_mul(ff2 ah, ff2 al, ff2 bh, ff2 bl, ff2& hi, ff2& lo) {
  hi = ff2_mulrn(ah, bh);
  ff2 e = ff2_fmarn(ah, bh, ff2_neg(hi));
  e = ff2_fmarn(ah, bl, e);
  lo = ff2_fmarn(al, bh, e);
  ff2_norm(hi, lo);
}
