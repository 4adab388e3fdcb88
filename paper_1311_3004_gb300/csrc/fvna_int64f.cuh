// fvna_int64f.cuh -- binary64 reciprocal, quotient, square root and product
// computed in integer arithmetic and correctly rounded (to nearest even), so
// that each returns the bits the binary64 unit returns.
//
// Why: a GB300 SM takes a binary64 instruction of one warp every 16 cycles
// (two lanes a cycle), while its integer pipes take two to four instructions
// a cycle.  Measured on a full SM, cycles per warp instruction or function
// (16 warps, four independent chains each):
//     binary64 fma 16.1, add or multiply 19.1,
//     1/x 86,  x/y 137,  sqrt 143   (the compiler's sequences on the unit)
//     rcp 29,  div 35,   sqrt 35    (below)
//     mulz 15.5, and 16.6 for a mulz and a binary64 add together: the two
//     pipes work side by side.
// The reciprocal is Newton's iteration from the binary32 approximation, in
// fixed point; the quotient multiplies by it, the square root refines
// m rsqrt(m) by its residual.  The approximation is within a few units of
// 2^-63 (bounds beside each function), so its rounding to 53 bits is the
// correct one unless it lies within that many units of a rounding boundary;
// then the exact remainder of the candidate decides (Markstein's method of
// rounding by the remainder, IBM J. Res. Dev. 34 (1990), in integers).
#pragma once

#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define INT64F_FN __host__ __device__ __forceinline__
#else
#define INT64F_FN static inline
#endif

namespace fvna {
namespace int64f {

typedef uint32_t u32;
typedef uint64_t u64;
typedef int32_t i32;
typedef int64_t i64;

#ifdef __CUDA_ARCH__
__device__ __forceinline__ u64 bits_of(double x) { return (u64)__double_as_longlong(x); }
__device__ __forceinline__ double of_bits(u64 b) { return __longlong_as_double((long long)b); }
__device__ __forceinline__ u64 mul_hi(u64 a, u64 b) { return __umul64hi(a, b); }
__device__ __forceinline__ u32 shift_left(u32 lo, u32 hi, u32 s) { return __funnelshift_l(lo, hi, s); }
// approximations of 1/f and 1/sqrt(f) as binary32 bit patterns
__device__ __forceinline__ u32 rcp_seed(u32 f) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(f)));
  return __float_as_uint(r);
}
__device__ __forceinline__ u32 rsqrt_seed(u32 f) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(f)));
  return __float_as_uint(r);
}
#else
// the same on the host (for checks); INT64F_SEED_OFF displaces the seeds by
// that many units in the last place
#ifndef INT64F_SEED_OFF
#define INT64F_SEED_OFF 0
#endif
INT64F_FN u64 bits_of(double x) { u64 b; memcpy(&b, &x, 8); return b; }
INT64F_FN double of_bits(u64 b) { double x; memcpy(&x, &b, 8); return x; }
INT64F_FN u64 mul_hi(u64 a, u64 b) { return (u64)(((unsigned __int128)a * b) >> 64); }
INT64F_FN u32 shift_left(u32 lo, u32 hi, u32 s) { return s ? (hi << s) | (lo >> (32 - s)) : hi; }
INT64F_FN u32 rcp_seed(u32 f) {
  float x;
  memcpy(&x, &f, 4);
  x = 1.0f / x;
  memcpy(&f, &x, 4);
  return f + (u32)(INT64F_SEED_OFF);
}
INT64F_FN u32 rsqrt_seed(u32 f) {
  float x;
  memcpy(&x, &f, 4);
  x = (float)(1.0 / __builtin_sqrt((double)x));
  memcpy(&f, &x, 4);
  return f + (u32)(INT64F_SEED_OFF);
}
#endif

INT64F_FN u64 wide(u32 a, u32 b) { return (u64)a * b; }
INT64F_FN u32 hi_of(double x) { return (u32)(bits_of(x) >> 32); }
INT64F_FN u64 significand(u64 b) { return (b & 0xfffffffffffffull) | 0x10000000000000ull; }

// exponent field in [512, 1535], i.e. 2^-511 <= |x| < 2^513: the two top bits
// of the field differ
INT64F_FN bool mid(u32 hi) { return ((hi ^ (hi << 1)) & 0x40000000u) != 0; }

// a seed kept in [1/2, 1), where the fixed-point forms below expect it
INT64F_FN u32 clamp_seed(u32 s) {
  s = s < 0x3f7fffffu ? s : 0x3f7fffffu;
  return s > 0x3f000000u ? s : 0x3f000000u;
}

// 1/m with 63 fractional bits for m = A 2^-63 in [1, 2).  The seed's relative
// error is below 2^-21 (its own few units, the truncation of m to 24 bits),
// the first iteration's below 2^-42; the second adds floor((f X1) 2^-62) with
// f in [0, 1) the truncation of m x1, and truncates once more: the result
// minus the exact value lies in (-1.01, 2) units of 2^-63.
INT64F_FN u64 recip63(u64 A) {
  const u32 ah = (u32)(A >> 32), al = (u32)A;
  const u32 s = clamp_seed(rcp_seed(0x3f800000u | ((ah >> 8) & 0x7fffffu)));
  const u32 x0 = (s << 8) | 0x80000000u;                        // 32 fractional bits
  const u64 p = wide(ah, x0) + (u32)(wide(al, x0) >> 32);       // m x0, 63 fractional bits
  const i32 e = (i32)((i64)(0x8000000000000000ull - p) >> 12);  // 1 - m x0, 51 fractional bits
  const u64 x1 = ((u64)x0 << 31) + (u64)(((i64)e * (i64)(u64)x0) >> 20);
  const i32 e1 = -(i32)(u32)mul_hi(A, x1);                      // 1 - m x1, 62 fractional bits
  return x1 + (u64)(((i64)e1 * (i64)(x1 >> 32)) >> 30);
}

// is t (the approximation plus half a unit of the rounded place, ten bits
// below it) within w units of a rounding boundary?
INT64F_FN bool close_call(u64 t, u32 w) { return (((u32)t + w) & 1023u) <= 2 * w; }

// 1/a for mid(a).  No tie exists: a quotient of 53-bit numbers is never
// half-way between two of them.
INT64F_FN double rcp_mid(double a) {
  const u64 b = bits_of(a);
  const u32 hi = (u32)(b >> 32);
  const u64 M = significand(b);
  const u64 t = recip63(M << 11) + 512;
  u64 Q = t >> 10;                                // 53 fractional bits, in [2^52, 2^53]
  if (close_call(t, 2)) {
    const i64 r = (i64)(0ull - M * Q);            // 2^105 - M Q, small: exact in 64 bits
    if (2 * r > (i64)M) Q++;
    else if (2 * r < -(i64)M) Q--;
  }
  // the sign, and the exponent field less one (Q's leading bit adds one)
  const u32 e = (hi & 0x80000000u) + 0x7fc00000u - (hi & 0x7ff00000u);
  return of_bits(Q + ((u64)e << 32));
}

// n/d for normal n and d whose exponents differ by less than 1000 (so that the
// quotient is normal).  The approximation is (-4.1, 4.1) units off after the normalising shift.
INT64F_FN double div_normal(u64 nb, u64 db) {
  const u64 M = significand(db), N = significand(nb);
  const u64 q = mul_hi(N << 11, recip63(M << 11));  // 62 fractional bits, in (1/2, 2)
  const u32 lt = 1u - (u32)(q >> 62);               // 1: the quotient is below 1
  const u64 t = (q << lt) + 512;
  u64 Q = t >> 10;
  if (close_call(t, 5)) {
    const i64 r = (i64)((N << (52 + lt)) - M * Q);
    if (2 * r > (i64)M) Q++;
    else if (2 * r < -(i64)M) Q--;
  }
  const u32 nh = (u32)(nb >> 32), dh = (u32)(db >> 32);
  const u32 e = (nh & 0xfff00000u) - (dh & 0xfff00000u) + 0x3fe00000u - (lt << 20);
  return of_bits(Q + ((u64)e << 32));
}

// sqrt(a) for mid(a), a > 0.  y0 ~ 1/sqrt(m), s0 = m y0, then twice
// s += (m - s^2) y0 / 2; the result is within (-1.8, 1.3) units of 2^-62.
INT64F_FN double sqrt_mid(double a) {
  const u64 b = bits_of(a);
  const u32 hi = (u32)(b >> 32);
  const u32 odd = ((hi >> 20) & 1u) ^ 1u;          // a = m 4^k with m in [1, 2) or [2, 4)
  const u64 M = significand(b);
  const u64 A = M << (10 + odd);                   // m, 62 fractional bits
  const u32 f = (0x3f800000u + (odd << 23)) | ((u32)(M >> 29) & 0x7fffffu);
  const u32 y0 = (clamp_seed(rsqrt_seed(f)) << 8) | 0x80000000u;             // 32 fractional bits
  const u64 s0 = wide((u32)(A >> 32), y0) + (u32)(wide((u32)A, y0) >> 32);   // m y0, 62
  const u32 sh = (i64)s0 < 0 ? 0xffffffffu : (u32)(s0 >> 31);                // 31, below 2
  const i32 e0 = (i32)((i64)(A - wide(sh, sh)) >> 15);                       // m - sh^2, 47
  u64 s1 = ((u64)sh << 31) + (u64)(((i64)e0 * (i64)(u64)y0) >> 18);          // 62
  const i32 e1 = (i32)(u32)(A - mul_hi(s1 << 1, s1 << 1));                   // m - s1^2, 62
  s1 += (u64)(((i64)e1 * (i64)(u64)y0) >> 33);
  const u64 t = s1 + 512;
  u64 Q = t >> 10;                                 // 52 fractional bits
  if (close_call(t, 3)) {
    const i64 r = (i64)((A << 42) - Q * Q);        // against (Q + 1/2)^2 and (Q - 1/2)^2
    if (r > (i64)Q) Q++;
    else if (r <= -(i64)Q) Q--;
  }
  const u32 e = (((hi >> 20) - 1023u - odd) >> 1) + 1022u;   // exponent field less one
  return of_bits(Q + ((u64)(e & 0x7ffu) << 52));
}

// x y, for factors that are zero or normal with exponent fields that add up
// to at least 1034 (product >= 2^-1012) and to less than 3069: callers bound
// their factors.  The product of the significands has 53 or 54 bits above
// 2^52 2^64 (top) and 64 below; a left shift by s brings the first case to
// the second, so that the top's last bit is the rounding bit.
INT64F_FN double mulz(double x, double y) {
  const u64 xb = bits_of(x), yb = bits_of(y);
  const u32 xh = (u32)(xb >> 32), xl = (u32)xb, yh = (u32)(yb >> 32), yl = (u32)yb;
  const u32 fl = xl << 12, fh = shift_left(xl, xh, 12);    // fraction of x, 64 bits
  const u32 mh = (yh & 0xfffffu) | 0x100000u;              // significand of y, 53 bits
  const u64 p0 = wide(fl, yl);
  const u64 p1 = wide(fh, yl) + (p0 >> 32);
  const u64 p2 = wide(fl, mh) + (u32)p1;
  const u64 top = wide(fh, mh) + (((u64)mh << 32) | yl) + (p1 >> 32) + (p2 >> 32);
  const u32 c = (u32)(top >> 53), s = c ^ 1u;              // c: the product is 2 or more
  const u32 th = shift_left((u32)top, (u32)(top >> 32), s), tl = shift_left((u32)p2, (u32)top, s);
  const u32 rest = ((u32)p2 << s) | (u32)p0;
  const u64 T = ((u64)th << 32) | tl;
  const u64 R = (T + (rest ? 1u : (tl >> 1) & 1u)) >> 1;   // to nearest even
  const u32 es = (xh & 0x7ff00000u) + (yh & 0x7ff00000u);
  const bool zero = es < (1034u << 20);                    // a factor is zero
  const u32 rh = zero ? 0u : (u32)(R >> 32) + es + (c << 20) - 0x40000000u;
  const u32 rl = zero ? 0u : (u32)R;
  return of_bits(((u64)(rh | ((xh ^ yh) & 0x80000000u)) << 32) | rl);
}

// x/2 and 2x of a number that stays normal
INT64F_FN double half_of(double x) { return of_bits(bits_of(x) - 0x10000000000000ull); }
INT64F_FN double twice(double x) { return of_bits(bits_of(x) + 0x10000000000000ull); }

}  // namespace int64f
}  // namespace fvna
