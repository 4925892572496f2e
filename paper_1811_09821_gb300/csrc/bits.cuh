// Arithmetic on the bits of doubles, the same on the device and on the host (where a plain C++ compiler takes
// this file, so that it can be tested without a GPU).
#ifndef MTO_BITS_CUH
#define MTO_BITS_CUH

#include <cmath>
#include <cstring>

#ifdef __CUDACC__
#define MTO_BITS __host__ __device__ __forceinline__
#else
#define MTO_BITS inline
#endif

namespace mto {

// floor(|v| 2^(56 - ex)) of a finite double v, |v| < 2^ex, by its bits
MTO_BITS unsigned long long fixed56(unsigned long long bits, int ex) {
  const int be = (int)(bits >> 52) & 0x7ff;
  bits &= 0x7fffffffffffffffull;
  const unsigned long long m = be ? (bits & 0xfffffffffffffull) | (1ull << 52) : bits;
  const int sh = (be ? be : 1) - 1075 + 56 - ex;
  return sh >= 0 ? m << (sh & 63) : (sh > -64 ? m >> (-sh & 63) : 0ull);
}

// The exact sum of the level integers, X 2^(ex - 70) with X = H 2^28 + Lw, rounded once to FP64 (to
// nearest even), as its bits.  |H| < 2^52.
MTO_BITS unsigned long long levels_to_double(long long H, long long Lw, int ex) {
  long long h = H + (Lw >> 28);
  unsigned lo = (unsigned)Lw & 0xfffffffu;   // X = h 2^28 + lo, 0 <= lo < 2^28
  const bool neg = h < 0;
  if (neg) {
    lo = (0u - lo) & 0xfffffffu;
    h = ~h + (lo == 0u);
  }
  unsigned long long W = ((unsigned long long)h << 12) | (lo >> 16);   // the upper 64 of 80 bits
  unsigned long long R = (unsigned long long)(lo & 0xffffu) << 48;     // the rest, left-aligned
  if (W == 0ull) {
    if (R == 0ull) return 0ull;
    W = R;
    R = 0ull;
    ex -= 64;
  }
#ifdef __CUDA_ARCH__
  const int z = __clzll((long long)W);
#else
  const int z = __builtin_clzll(W);
#endif
  const unsigned long long A = z ? (W << z) | (R >> (64 - z)) : W;   // leading one at bit 63
  const unsigned long long sticky = (R << z) != 0ull;
  const unsigned rem = (unsigned)(A & 0x7ffu) * 2u + (unsigned)sticky;
  unsigned long long m = A >> 11;
  m += rem + (unsigned)(m & 1u) > 0x800u;
  const int be = 9 - z + ex + 1023;   // X = A 2^(16 - z)
  unsigned long long bits;
  if (be >= 1 && be <= 2046) {
    bits = ((unsigned long long)(be - 1) << 52) + m;
  } else {
    const double v = ldexp((double)m, be - 1075);
    memcpy(&bits, &v, 8);
  }
  return neg ? bits | (1ull << 63) : bits;
}

// The split pair of an FP64 value: hi = fl32(v), lo = fl32(v - hi), by integer instructions where the
// exponents allow it (from 2^-98 on a lo below the normal range has at most 24 bits, so that the
// conversion and the scaling below round once between them).
MTO_BITS void split_pair(unsigned long long bits, float& hi, float& lo) {
  const int be = (int)(bits >> 52) & 0x7ff;
  const int e = be - 1023;
  if (e < -98 || e > 110) {
    double v;
    memcpy(&v, &bits, 8);
    hi = (float)v;
    lo = (float)(v - (double)hi);
    return;
  }
  const unsigned long long m = (bits & 0xfffffffffffffull) | (1ull << 52);
  const unsigned h24 = (unsigned)(m >> 29), rem = (unsigned)m & 0x1fffffffu;
  const unsigned up = rem + (h24 & 1u) > 0x10000000u;
  const unsigned sgn = (unsigned)(bits >> 32) & 0x80000000u;
  const unsigned hb = (sgn | ((unsigned)(e + 126) << 23)) + h24 + up;
  const int D = (int)rem - (int)(up << 29);   // v - hi = D 2^(e - 52)
  const unsigned sb = (unsigned)(e + 8 + 127) << 23;   // 2^(e + 8); the product rounds once (exact before)
  float s;
  memcpy(&hi, &hb, 4);
  memcpy(&s, &sb, 4);
  const float d = (float)(sgn ? -D : D);
  lo = (d * 8.673617379884035e-19f) * s;   // 2^-60 2^(e + 8)
}

// 1 / d, correctly rounded: Newton's iteration x <- x + x (1 - d x) on the mantissa from its FP32 reciprocal
// (2^-23, squared twice, then once more from a value within one unit in the last place, which rounds
// correctly but for a mantissa of ones only: Markstein, IBM J. Res. Dev. 34, 1990); plain division for that
// mantissa, at the ends of the exponent range, for negative values, infinities and NaN.  A branch-free chain of
// FMAs where the division's subroutine call cost the elimination kernels their overlap.
MTO_BITS double newton_rcp(double d) {
  unsigned long long b;
  memcpy(&b, &d, 8);
  const int be = (int)(b >> 52);   // sign and exponent
  const unsigned long long man = b & 0xfffffffffffffull;
  if (be < 8 || be > 2038 || man == 0xfffffffffffffull) return 1.0 / d;
  const unsigned long long mb = man | (1023ull << 52);
  const unsigned fb = 0x3f800000u | (unsigned)(man >> 29);
  double m;
  float f;
  memcpy(&m, &mb, 8);
  memcpy(&f, &fb, 4);
  double r = (double)(1.0f / f);
  r = fma(r, fma(-m, r, 1.0), r);
  r = fma(r, fma(-m, r, 1.0), r);
  r = fma(r, fma(-m, r, 1.0), r);
  unsigned long long rb;
  memcpy(&rb, &r, 8);
  rb -= (unsigned long long)(long long)(be - 1023) << 52;
  memcpy(&r, &rb, 8);
  return r;
}

}  // namespace mto

#endif
