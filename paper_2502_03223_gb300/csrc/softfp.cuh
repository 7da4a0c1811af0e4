// FP64 arithmetic on the integer and FP32 units.
//
// On this part a warp's FP64 instruction takes 16 cycles of the SM's FP64
// pipe, a division or square root 97 to 151 (measured, all lanes busy), while
// a 32 x 32 + 64-bit integer multiply-add (mad.wide) takes 0.6 and a 32-bit
// integer operation about 0.5.  The kernels of this library were bound by the
// FP64 pipe with the integer and FP32 units idle.  sdiv, srcp, ssqrt and
// srsqrt form the quotient, reciprocal, square root and its reciprocal of
// doubles there: an FP32 seed (24 bits) and one third-order (Householder) step
// on the exact residual, all in integers, give 60 bits; the result is then
// rounded once.  Quotient, reciprocal and square root are corrected by their
// exact remainder, so they are the correctly rounded ones, bit for bit those
// of the FP64 instructions (decisions such as rho < rho_atm compare values
// formed by them); srsqrt is off by less than 0.52 ulp.  Operands outside the
// normal range (zeros, infinities, NaN, subnormals) and results near its ends
// take the FP64 instruction sequence.  36 (srcp) to 57 (ssqrt) SM cycles per
// warp on the integer pipe.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define SF_HD __host__ __device__ __forceinline__
#else
#define SF_HD inline
#endif

namespace sacra {
namespace sf {

typedef long long i64;
typedef unsigned long long u64;

SF_HD i64 bits(double v) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(v);
#else
  i64 b; memcpy(&b, &v, 8); return b;
#endif
}
SF_HD double of_bits(i64 b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(b);
#else
  double v; memcpy(&v, &b, 8); return v;
#endif
}
SF_HD float f_of_bits(unsigned u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float f; memcpy(&f, &u, 4); return f;
#endif
}
SF_HD unsigned f_bits(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(f);
#else
  unsigned u; memcpy(&u, &f, 4); return u;
#endif
}
SF_HD unsigned hiw(i64 b) { return (unsigned)((u64)b >> 32); }
SF_HD unsigned low(i64 b) { return (unsigned)b; }
SF_HD unsigned umulhi32(unsigned a, unsigned b) { return (unsigned)(((u64)a * b) >> 32); }
SF_HD i64 wide(int a, int b) { return (i64)a * b; }
// FP32 seeds: the hardware approximations (the host form, for tests, may be nudged)
#ifndef SF_SEED
#define SF_SEED(f) (f)
#endif
SF_HD float seed_rcp(float f) {
#ifdef __CUDA_ARCH__
  float r; asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(f)); return r;
#else
  return SF_SEED(1.0f / f);
#endif
}
SF_HD float seed_rsqrt(float f) {
#ifdef __CUDA_ARCH__
  float r; asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(f)); return r;
#else
  return SF_SEED(1.0f / sqrtf(f));
#endif
}

// ---------------------------------------------------------------- quotients and roots

// 1 / m for m = M 2^-52 in [1, 2) as an integer multiple of 2^-62 (error
// below 2^-60): r0 an FP32 seed, e = 1 - m r0 exactly (|e| < 2^-21), then
// r0 (1 + e + e^2); the next term is e^3 < 2^-63.
SF_HD i64 rcp62(unsigned mh, unsigned ml) {
  const float f = f_of_bits(0x3f800000u | ((mh & 0xFFFFFu) << 3) | (ml >> 29));
  const float r = fminf(fmaxf(seed_rcp(f), 0.5f), 0.99999994f);
  const int R = (int)((f_bits(r) & 0x7FFFFFu) | 0x800000u);             // r0 2^24
  const i64 E = -(i64)((u64)ml * (unsigned)R + ((u64)(mh * (unsigned)R) << 32));   // e 2^76
  const i64 T = wide(R, (int)(E >> 32)) + (i64)umulhi32((unsigned)R, low(E));      // r0 e 2^68
  const int e2 = (int)(E >> 24);                                         // e 2^52
  const int sq = (int)(wide(e2, e2) >> 32);                              // e^2 2^72
  return ((i64)R << 38) + (T >> 6) + (wide(R, sq) >> 34);
}

// 1 / sqrt(m) for m = M 2^-52 in [1, 4) (M < 2^54) as a multiple of 2^-62:
// e = 1 - m y0^2 (|e| < 2^-20) to 2^-64, then y0 (1 + e/2 + 3/8 e^2); the
// next term is 5/16 e^3 < 2^-61.
SF_HD i64 rsqrt62(i64 M, float f) {
  const float y = fminf(fmaxf(seed_rsqrt(f), 0.5f), 0.99999994f);
  const unsigned Y = (f_bits(y) & 0x7FFFFFu) | 0x800000u;                // y0 2^24
  const u64 Z = (u64)Y * Y;                                              // y0^2 2^48
  const unsigned zh = (unsigned)(Z >> 24), zl = (unsigned)Z & 0xFFFFFFu;
  const unsigned mh = hiw(M), ml = low(M);
  // m y0^2 2^64 mod 2^64 (the integer part cancels the 1)
  const u64 S = (((u64)ml * zh) >> 12) + (((u64)mh * zh) << 20) + (((u64)mh * zl) >> 4) + (((u64)ml * zl) >> 36);
  const i64 e = -(i64)S;                                                 // e 2^64
  const i64 es = e << 18;                                                // e 2^82
  const i64 T = wide((int)Y, (int)(es >> 32)) + (i64)umulhi32(Y, low(es));   // y0 e 2^74
  const int e2 = (int)(e >> 14);                                         // e 2^50
  const int sq = 3 * (int)(wide(e2, e2) >> 32);                          // 3 e^2 2^68
  return ((i64)Y << 38) + (T >> 13) + (wide((int)Y, sq) >> 33);
}

// A B 2^-62 for 0 <= A, B < 2^62 (error below 2 units)
SF_HD i64 mulhi62(i64 A, i64 B) {
  const int ah = (int)(A >> 31), al = (int)(low(A) & 0x7FFFFFFFu);
  const int bh = (int)(B >> 31), bl = (int)(low(B) & 0x7FFFFFFFu);
  return wide(ah, bh) + ((wide(ah, bl) + wide(al, bh)) >> 31);
}

// Q 2^-61 for Q in [2^60, 2^62), times 2^(ex - 1023), rounded to nearest
SF_HD double pack61(u64 Q, int ex, unsigned sign) {
  const int up = (int)(Q >> 61);                     // 1: in [1, 2)
  const int s = 8 + up;
  const u64 m = (Q + (1ull << (s - 1))) >> s;        // 53 bits with the leading one (or the next power of two)
  return of_bits((i64)(m + ((u64)(unsigned)(ex - 2 + up) << 52)) | ((i64)(int)sign << 32));
}

#ifdef __CUDACC__
__device__ __noinline__ inline double div_fp64(double a, double b) { return a / b; }
__device__ __noinline__ inline double sqrt_fp64(double a) { return sqrt(a); }
__device__ __noinline__ inline double rsqrt_fp64(double a) { return rsqrt(a); }
#endif
SF_HD double slow_div(double a, double b) {
#ifdef __CUDA_ARCH__
  return div_fp64(a, b);
#else
  return a / b;
#endif
}
SF_HD double slow_sqrt(double a) {
#ifdef __CUDA_ARCH__
  return sqrt_fp64(a);
#else
  return sqrt(a);
#endif
}
SF_HD double slow_rsqrt(double a) {
#ifdef __CUDA_ARCH__
  return rsqrt_fp64(a);
#else
  return 1.0 / sqrt(a);
#endif
}

// The correctly rounded quotient ma 2^k / mb (53-bit significands, k = 52 or
// 53) from its neighbour q (mq its significand, off by less than one unit):
// q one unit up or down where the remainder exceeds half a divisor.  The
// remainder is below 2^54, so its low 64 bits hold it; a tie cannot occur.
SF_HD double round_quotient(double q, u64 ma, u64 mb, int k) {
  const i64 bq = bits(q);
  const u64 mq = ((u64)bq & ((1ull << 52) - 1)) | (1ull << 52);
  const i64 r2 = (i64)((ma << k) - mq * mb) * 2;
  return of_bits(bq + (r2 > (i64)mb) - (r2 < -(i64)mb));
}

// a / b
SF_HD double sdiv(double a, double b) {
  const i64 ba = bits(a), bb = bits(b);
  const int ea = (int)(hiw(ba) >> 20) & 0x7FF, eb = (int)(hiw(bb) >> 20) & 0x7FF;
  const int ex = ea - eb + 1023;
  if ((unsigned)(ea - 1) >= 2046u || (unsigned)(eb - 1) >= 2046u || (unsigned)(ex - 3) >= 2040u) {
    if ((ba << 1) == 0 && (unsigned)(eb - 1) < 2046u)       // zero over a normal number
      return of_bits((i64)(((u64)ba ^ (u64)bb) & (1ull << 63)));
    return slow_div(a, b);
  }
  const u64 ma = ((u64)ba & ((1ull << 52) - 1)) | (1ull << 52), mb = ((u64)bb & ((1ull << 52) - 1)) | (1ull << 52);
  const i64 A = (i64)(ma << 9);                                                    // [2^61, 2^62)
  const i64 r = rcp62((unsigned)(mb >> 32), low(bb));                              // (2^61, 2^62]
  // A r 2^-62 lies in [2^60, 2^62); r may reach 2^62 only for b a power of two
  const i64 Q = mulhi62(A, r - (r >> 62));
  const double q = pack61((u64)Q, ex, (hiw(ba) ^ hiw(bb)) & 0x80000000u);
  const int eq = (int)(hiw(bits(q)) >> 20) & 0x7FF;
  return round_quotient(q, ma, mb, ex - eq + 52);
}

// 1 / b
SF_HD double srcp(double b) {
  const i64 bb = bits(b);
  const int eb = (int)(hiw(bb) >> 20) & 0x7FF;
  if ((unsigned)(eb - 3) >= 2040u) return slow_div(1.0, b);
  const u64 mb = ((u64)bb & ((1ull << 52) - 1)) | (1ull << 52);
  const i64 r = rcp62((unsigned)(mb >> 32), low(bb));
  const double q = pack61((u64)(r >> 1), 2046 - eb, hiw(bb) & 0x80000000u);
  const int eq = (int)(hiw(bits(q)) >> 20) & 0x7FF;
  return round_quotient(q, 1ull << 52, mb, 2046 - eb - eq + 52);
}

// the pieces of a positive normal a = m 4^k: M = m 2^52 (m in [1, 4)), m in FP32, k
SF_HD void root_parts(i64 b, i64 &M, float &f, int &k) {
  const int ea = (int)(hiw(b) >> 20) - 1023;
  const int odd = ea & 1;
  k = (ea - odd) >> 1;
  M = (i64)((((u64)b & ((1ull << 52) - 1)) | (1ull << 52)) << odd);
  f = f_of_bits((0x3f800000u + ((unsigned)odd << 23)) | ((hiw(b) & 0xFFFFFu) << 3) | (low(b) >> 29));
}

// sqrt(a)
SF_HD double ssqrt(double a) {
  const i64 b = bits(a);
  if ((unsigned)((int)hiw(b) - 0x00300000) >= 0x7FC00000u) return slow_sqrt(a);    // not positive, normal and finite
  i64 M; float f; int k;
  root_parts(b, M, f, k);
  const i64 y = rsqrt62(M, f);                             // (2^61, 2^62]
  // m y in [1, 2): (M 2^8) y 2^-62 = sqrt(m) 2^60
  const i64 Q = mulhi62(M << 8, y - (y >> 62));
  const i64 bq = bits(pack61((u64)(Q << 1), 1023 + k, 0u));
  // q on the grid of [1, 2) (2 itself may come out of the rounding), off by less than one
  // unit: corrected by the remainder M 2^52 - q^2, which the low 64 bits hold
  const i64 q = (i64)((((u64)bq & ((1ull << 52) - 1)) | (1ull << 52)) << ((int)(hiw(bq) >> 20) - 1023 - k));
  const i64 rem = (i64)(((u64)M << 52) - (u64)q * (u64)q);
  return of_bits(bq + (rem > q) - (rem <= -q));
}

// 1 / sqrt(a)
SF_HD double srsqrt(double a) {
  const i64 b = bits(a);
  if ((unsigned)((int)hiw(b) - 0x00300000) >= 0x7FC00000u) return slow_rsqrt(a);
  i64 M; float f; int k;
  root_parts(b, M, f, k);
  return pack61((u64)(rsqrt62(M, f) >> 1), 1023 - k, 0u);
}

}  // namespace sf
}  // namespace sacra
