// FP64 building blocks for a part whose FP64 pipe takes about two operations
// per SM and clock (1/64 of its FP32 rate): quotients, square roots,
// comparisons and scalings by two done in the integer and FP32 pipes, which
// the FP64 kernels leave idle.  Every function returns exactly the value of
// the IEEE operation it replaces (round to nearest even), so results do not
// change; operands or results outside the normal range take the native
// operation.
//
// Measured on a GB300 (1024 x 1024 radial dam break, 32 x 32 patches, 36 %
// wet): a wet cell took about 1770 FP64-pipe operations, of which the scheme
// needs 468; the division and square-root sequences (some eight to ten
// FP64 operations each, about 50 of them per cell) were most of the rest.
//
// The header also compiles for the host, where a program provides the seeds:
// a test draws their relative errors from the whole range that the device's
// approximations may have (reciprocals and roots up to 2^-22, about twice the
// documented bounds; cube roots 2^-20).
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define GF_HD __device__ __forceinline__
// out of line: a quotient or root is some sixty instructions, and the FP64
// kernels hold dozens of them
#define GF_HD_CALL static __device__ __noinline__
#else
#define GF_HD inline
#define GF_HD_CALL inline
#endif

namespace gfk {

#ifdef __CUDACC__
GF_HD long long dbits(double x) { return __double_as_longlong(x); }
GF_HD double bitsd(long long b) { return __longlong_as_double(b); }
GF_HD float bitsf(unsigned b) { return __uint_as_float(b); }
GF_HD int f2i_magic(float x) { return __float_as_int(__fadd_rn(x, 12582912.0f)) - 0x4b400000; }
GF_HD float i2f(int i) { return __int2float_rn(i); }
GF_HD float fmul(float a, float b) { return __fmul_rn(a, b); }
GF_HD float seed_rcp(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
GF_HD float seed_rsqrt(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
GF_HD float seed_cbrt(float x) { return exp2f(log2f(x) * (1.0f / 3.0f)); }
GF_HD double native_sqrt(double x) { return sqrt(x); }
GF_HD double native_cbrt(double x) { return cbrt(x); }
GF_HD double ffma(double a, double b, double c) { return __fma_rn(a, b, c); }
GF_HD unsigned fbits(float x) { return __float_as_uint(x); }
#else
inline long long dbits(double x) { long long b; std::memcpy(&b, &x, 8); return b; }
inline double bitsd(long long b) { double x; std::memcpy(&x, &b, 8); return x; }
inline float bitsf(unsigned b) { float x; std::memcpy(&x, &b, 4); return x; }
inline int f2i_magic(float x) {
  volatile float s = x + 12582912.0f;
  const float t = s;
  int b;
  std::memcpy(&b, &t, 4);
  return b - 0x4b400000;
}
inline float i2f(int i) { return (float)i; }
inline float fmul(float a, float b) { volatile float r = a * b; return r; }
float seed_rcp(float x);
float seed_rsqrt(float x);
float seed_cbrt(float x);
double native_sqrt(double x);
double native_cbrt(double x);
inline double ffma(double a, double b, double c) { return std::fma(a, b, c); }
inline unsigned fbits(float x) { unsigned b; std::memcpy(&b, &x, 4); return b; }
#endif

// Remainders below are exact modulo 2^64 although the products they come from
// are longer: formed unsigned, read signed.
typedef unsigned long long u64;

constexpr long long D_MANT = (1ll << 52) - 1;
constexpr long long D_HID = 1ll << 52;
constexpr long long D_INF = 0x7ffll << 52;

// a / b.  Digit recurrence on the 53-bit significands ma, mb: three quotient
// digits of 20, 20 and 15 bits, each the remainder's leading bits times an
// FP32 reciprocal of mb rounded to an integer, with the remainder updated
// exactly modulo 2^64.  The reciprocal is within 2^-21.4 of 1 / mb (2^-23
// from the truncation of mb to 23 bits, 2^-22 allowed to the approximation),
// so a digit is off by less than 2 units, the
// remainder stays below 2^55 and the last digit (15 bits) is within 0.6 of
// the exact one: the sign of the last remainder says whether the 56-bit
// quotient is one too large, and whether it is zero is the sticky bit.
GF_HD_CALL double div_rn(double a, double b) {
  const long long ab = dbits(a), bb = dbits(b);
  const int ea = (int)(ab >> 52) & 0x7ff, eb = (int)(bb >> 52) & 0x7ff;
  const int e = ea - eb;
  // both operands and the quotient well inside the normal range
  if ((unsigned)(ea - 1) < 2046u && (unsigned)(eb - 1) < 2046u && (unsigned)(e + 1021) < 2043u) {
    const u64 ma = (u64)((ab & D_MANT) | D_HID), mb = (u64)((bb & D_MANT) | D_HID);
    const float fa = bitsf(0x3f800000u | (unsigned)((ab & D_MANT) >> 29));
    const float fb = bitsf(0x3f800000u | (unsigned)((bb & D_MANT) >> 29));
    const float y = seed_rcp(fb);
    const int q1 = f2i_magic(fmul(fa, fmul(y, 1048576.0f)));
    const long long r1 = (long long)((ma << 20) - (u64)(long long)q1 * mb);
    const int q2 = f2i_magic(fmul(i2f((int)(r1 >> 24)), fmul(y, 0x1p-8f)));
    const long long r2 = (long long)(((u64)r1 << 20) - (u64)(long long)q2 * mb);
    const int q3 = f2i_magic(fmul(i2f((int)(r2 >> 24)), fmul(y, 0x1p-13f)));
    const long long r3 = (long long)(((u64)r2 << 15) - (u64)(long long)q3 * mb);
    // quotient ma 2^55 / mb in (2^54, 2^56): floor, then the sticky bit
    long long Q = (long long)((u64)q1 << 35) + (long long)q2 * 32768 + q3;
    Q += r3 >> 63;
    Q |= r3 != 0 ? 1 : 0;
    const bool small = Q < (1ll << 55);
    Q = small ? Q + Q : Q;
    const long long m = (Q + 3 + ((Q >> 3) & 1)) >> 3;
    const long long r = ((long long)(e + (small ? 1021 : 1022)) << 52) + m;
    return bitsd(r | ((ab ^ bb) & (long long)0x8000000000000000ull));
  }
  if ((u64)ab << 1 == 0 && (unsigned)(eb - 1) < 2046u)  // signed zero
    return bitsd((ab ^ bb) & (long long)0x8000000000000000ull);
  return a / b;
}

// sqrt(x).  The same recurrence for the root: m in [2^52, 2^54) (the exponent
// made even), digits of the root at 2^20, 2^40 and 2^53, each the exact
// residual times half an FP32 reciprocal square root.  The last digit is
// within 0.6 of the exact one, so the residual's sign gives the floor of the
// 54-bit root; a root is never halfway between two results.
GF_HD_CALL double sqrt_rn(double x) {
  const long long xb = dbits(x);
  const int ex = (int)(xb >> 52);  // sign included: negative values fall out
  if ((unsigned)(ex - 1) < 2046u) {
    const int odd = (ex + 1) & 1;  // ex - 1023 odd
    const u64 m = (u64)((xb & D_MANT) | D_HID) << odd;
    const float f0 = bitsf(0x3f800000u | (unsigned)((xb & D_MANT) >> 29));
    const float f = odd ? f0 + f0 : f0;
    const float y = seed_rsqrt(f);
    const int s1 = f2i_magic(fmul(fmul(f, y), 1048576.0f));
    const long long r1 = (long long)(m - ((u64)((long long)s1 * s1) << 12));
    const int s2 = f2i_magic(fmul(i2f((int)(r1 >> 8)), fmul(y, 0x1p-5f)));
    const long long r2 = (long long)(((u64)r1 << 28) - ((u64)((long long)s1 * s2) << 21) -
                                     (u64)((long long)s2 * s2));
    const long long S2 = ((long long)s1 << 20) + s2;
    const int s3 = f2i_magic(fmul(i2f((int)(r2 >> 16)), fmul(y, 0x1p-12f)));
    const long long r3 = (long long)(((u64)r2 << 26) - ((u64)(S2 * s3) << 14) -
                                     (u64)((long long)s3 * s3));
    long long S = (S2 << 13) + s3;
    S += r3 >> 63;
    const long long mr = (S + 1) >> 1;  // [2^52, 2^53]
    const int er = (ex - 1023 - odd) / 2 + 1022;
    return bitsd(((long long)er << 52) + mr);
  }
  if ((u64)xb << 1 == 0) return x;
  return native_sqrt(x);
}

// x rounded towards zero to FP32, without the FP64 pipe's conversion: zero
// below 2^-126, NaN from 2^127 on.
GF_HD float trunc_f32(double x) {
  const u64 b = (u64)dbits(x);
  const int t = (int)((b >> 32) & 0x7fffffffu) - 0x38000000;
  // the exponent's bias off, the significand's first 23 bits up to its place
  const float f = bitsf(((unsigned)t << 3 | (unsigned)b >> 29) | ((unsigned)(b >> 32) & 0x80000000u));
  return t < 0x00100000 ? 0.0f : (t >= 0x0fe00000 ? bitsf(0x7fffffffu) : f);
}

// Cube root of a positive number, within an ulp: the FP32 estimate (2^-20)
// corrected by two terms of the binomial series of the exact residual ratio
// d = x / y^3 - 1, y (1 + d/3 - d^2/9), whose third term is below 2^-59 of y.
// (At the ends of the range, and for anything else, the native function.)
GF_HD double cbrt_pos(double x) {
  const int e = (int)(dbits(x) >> 52);  // biased exponent
  if ((unsigned)(e - 4) >= 2040u) return native_cbrt(x);
  const int k = (e - 1023 + 1533) / 3 - 511;          // floor((e - 1023) / 3)
  const double m = bitsd(dbits(x) - 3 * k * D_HID);   // [1, 8)
  const unsigned fb = fbits(seed_cbrt(trunc_f32(m)));
  // the estimate to FP64 by its bits
  const double y = bitsd(((long long)((fb >> 23) + 896u) << 52) | ((long long)(fb & 0x7fffffu) << 29));
  const double y2 = y * y;  // exact: 48 bits
  const double y3 = y2 * y;
  const double r = ffma(-y2, y, m);
  const double d = div_rn(r, y3);
  const double c = d * ffma(d, -1.0 / 9.0, 1.0 / 3.0);
  const double t = ffma(y, c, y);
  return bitsd(dbits(t) + k * D_HID);
}

// a < b and a <= 0 style tests on the bit patterns (no NaN operands: a NaN
// orders beyond infinity here, and the step reports it as a non-finite value
// whichever branch it takes).
GF_HD long long okey(double x) {  // order-preserving; -0 and +0 alike
  const long long b = dbits(x);
  return b < 0 ? (long long)(0x8000000000000000ull - (unsigned long long)b) : b;
}
GF_HD bool dlt(double a, double b) { return okey(a) < okey(b); }
GF_HD bool neg(double x) { return dbits(x) < 0 && (u64)dbits(x) << 1 != 0; }
GF_HD bool pos(double x) { return dbits(x) > 0; }
GF_HD bool iszero(double x) { return (u64)dbits(x) << 1 == 0; }
GF_HD double dabs(double x) { return bitsd(dbits(x) & 0x7fffffffffffffffll); }
GF_HD double dneg(double x) { return bitsd(dbits(x) ^ (long long)0x8000000000000000ull); }
GF_HD double dmin(double a, double b) { return dlt(a, b) ? a : b; }
GF_HD double dmax(double a, double b) { return dlt(b, a) ? a : b; }
// h > d for a positive threshold d; false for NaN
GF_HD bool above(double h, double d) {
  return (u64)dbits(h) - (u64)dbits(d) - 1u < (u64)D_INF - (u64)dbits(d);
}
// x / 2 and 2 x by the exponent, at the ends of the range too (a product
// there, however rare, would take a slot of the FP64 pipe each time: the
// compiler predicates it)
GF_HD double half(double x) {
  const long long b = dbits(x), m = b & 0x7fffffffffffffffll;
  // below twice the smallest normal number: the significand halved, to even
  const long long lo = (m >> 1) + ((m & 3) == 3 ? 1 : 0);
  const long long hi = m >= D_INF ? m : m - D_HID;
  return bitsd((m < 2 * D_HID ? lo : hi) | (b & (long long)0x8000000000000000ull));
}
GF_HD double twice(double x) {
  const long long b = dbits(x), m = b & 0x7fffffffffffffffll;
  const long long hi = m >= D_INF - D_HID ? (m > D_INF ? m : D_INF) : m + D_HID;
  return bitsd((m < D_HID ? 2 * m : hi) | (b & (long long)0x8000000000000000ull));
}
// Marks a rare branch: keeps the compiler from executing its FP64 operations
// under a predicate (each would take its slot of the FP64 pipe all the same).
GF_HD void rare() {
#ifdef __CUDACC__
  asm volatile("");
#endif
}

}  // namespace gfk
