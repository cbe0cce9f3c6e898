// intdiv.cuh -- correctly rounded FP64 reciprocal and quotient from integer arithmetic.
//
// The FP64 pipe of this GPU takes one warp instruction per 64 cycles, so the hardware's division sequence costs
// 344 cycles for 1/x and 562 for x/y of the pipe that bounds every kernel here, while the integer units stand
// idle (a 64-bit high product takes 19 cycles).  Both functions below use no FP64 instruction: a reciprocal of
// the 53-bit mantissa by Newton's iteration in 64-bit fixed point, a quotient rounded to nearest from it, and
// the exact remainder, which corrects the last place.  A quotient of two doubles never lies half-way between
// two doubles in the normal range, so the nearest one is unique and the result is the IEEE one, bit for bit.
// Zero (as a divisor), subnormal, infinite and NaN operands and results outside the normal range take the
// hardware division.  With them, with decisions taken from the bits of doubles (fmax costs 152 cycles) and with
// sums that share a butterfly, the source term of 65,536 cells of 53 species / 325 reactions went from 2667 to
// 2456 us and the Jacobian of 8,191 cells from 1071 to 1033 us.
#pragma once

#ifdef __CUDACC__
#define CHEM_DEV __device__ __forceinline__
#else   // host build of the same source, for checks without a GPU
#include <cmath>
#include <cstdint>
#include <cstring>
#define CHEM_DEV inline
#endif

namespace chemgb {

#ifdef __CUDACC__
// the hardware's sequence, out of line: the usual case does not reach it
static __device__ __noinline__ double slow_div(double a, double b) { return a / b; }
CHEM_DEV unsigned long long dbits(double x) { return (unsigned long long)__double_as_longlong(x); }
CHEM_DEV double bitsd(unsigned long long x) { return __longlong_as_double((long long)x); }
CHEM_DEV float f_of_bits(unsigned x) { return __uint_as_float(x); }
CHEM_DEV unsigned bits_of_f(float x) { return __float_as_uint(x); }
CHEM_DEV unsigned long long mul_hi64(unsigned long long a, unsigned long long b) { return __umul64hi(a, b); }
CHEM_DEV float rcp_seed(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
#else
inline double slow_div(double a, double b) { return a / b; }
CHEM_DEV unsigned long long dbits(double x) { unsigned long long u; std::memcpy(&u, &x, 8); return u; }
CHEM_DEV double bitsd(unsigned long long u) { double x; std::memcpy(&x, &u, 8); return x; }
CHEM_DEV float f_of_bits(unsigned u) { float x; std::memcpy(&x, &u, 4); return x; }
CHEM_DEV unsigned bits_of_f(float x) { unsigned u; std::memcpy(&u, &x, 4); return u; }
CHEM_DEV unsigned long long mul_hi64(unsigned long long a, unsigned long long b) {
  return (unsigned long long)(((unsigned __int128)a * b) >> 64);
}
static int seed_ulps = 0;   // the check moves the seed by up to +-2 units in the last place
CHEM_DEV float rcp_seed(float x) { return f_of_bits(bits_of_f(1.0f / x) + (unsigned)seed_ulps); }
#endif

// y 2^63 with y = 1/x for the normalised x = X / 2^63 in [1, 2), relative error below 2^-58.  From a 23-bit seed
// (kept below 1 so that its bits are a fixed-point fraction): e = 1 - x y0, y = y0 (1 + e + e^2).
CHEM_DEV unsigned long long recip63(unsigned long long X) {
  const unsigned xh = (unsigned)(X >> 32), xl = (unsigned)X;
  const float f0 = rcp_seed(f_of_bits(0x3f800000u | ((xh >> 8) & 0x7fffffu)));
#ifdef __CUDACC__
  const float f1 = __fmaf_rn(f0, 0.999999f, 1.0f);
#else
  const float f1 = std::fma(f0, 0.999999f, 1.0f);
#endif
  const unsigned y0 = (bits_of_f(f1) & 0x7fffffu) << 9;   // y0 2^32
  const unsigned long long P = (unsigned long long)xh * y0 + (((unsigned long long)xl * y0) >> 32);
  const long long e = (long long)(0x8000000000000000ull - P);   // e 2^63, |e| < 2^-19
  const int e1 = (int)(e >> 14);                                // e 2^49
  const long long s = e + (((long long)e1 * e1) >> 35);         // e + e^2
  const long long t = (long long)(int)(s >> 32) * (long long)(unsigned long long)y0 +
                      (long long)(((unsigned long long)(unsigned)s * y0) >> 32);   // y0 (e + e^2) 2^63
  return ((unsigned long long)y0 << 31) + (unsigned long long)t;
}

// 1/d, rounded to nearest.
CHEM_DEV double rcp_rn(double d) {
  const unsigned long long b = dbits(d);
  const unsigned ed = (unsigned)(b >> 52) & 0x7ffu;
  if (ed - 1u >= 2044u) return slow_div(1.0, d);
  const unsigned long long m = (b & 0xfffffffffffffull) | 0x10000000000000ull;
  unsigned long long q = (recip63(m << 11) + 512u) >> 10;   // 2^105 / m within one
  const long long r = -(long long)(q * m);                  // 2^105 - q m, exact modulo 2^64
  if (2 * r > (long long)m) ++q;
  else if (2 * r < -(long long)m) --q;
  return bitsd((b & 0x8000000000000000ull) | (((unsigned long long)(2044u - ed) << 52) + q));
}

// a/d, rounded to nearest.
CHEM_DEV double div_rn(double a, double d) {
  const unsigned long long ba = dbits(a), bd = dbits(d);
  const int ea = (int)(ba >> 52) & 0x7ff, ed = (int)(bd >> 52) & 0x7ff;
  const unsigned long long ma = (ba & 0xfffffffffffffull) | 0x10000000000000ull;
  const unsigned long long md = (bd & 0xfffffffffffffull) | 0x10000000000000ull;
  const bool less = ma < md;
  const int B = 1023 + ea - ed - (less ? 1 : 0);   // biased exponent of the quotient
  const bool zero = (ba << 1) == 0;
  if (ed - 1u >= 2046u || (!zero && (ea - 1u >= 2046u || B - 1u >= 2045u))) return slow_div(a, d);
  const unsigned long long h = mul_hi64(ma << 11, recip63(md << 11));   // ma/md 2^62
  unsigned long long q = (h + (less ? 256u : 512u)) >> (less ? 9 : 10);
  const long long r = (long long)((ma << (less ? 53 : 52)) - q * md);
  if (2 * r > (long long)md) ++q;
  else if (2 * r < -(long long)md) --q;
  const unsigned long long sign = (ba ^ bd) & 0x8000000000000000ull;
  return bitsd(sign | (zero ? 0ull : ((unsigned long long)(B - 1) << 52) + q));
}

}  // namespace chemgb
