// fxmath.cuh -- 64-bit fixed-point arithmetic on the integer pipes: upper products, conversion to double,
// the inverse square root, and the Stumpff functions of the Kepler drift.
#pragma once
#include "fxpair.cuh"

namespace genga {
namespace fx {

// upper half of the product of two 64-bit numbers, to one unit; the cross products must not carry
// out of 64 bits together (one factor below 2^63 suffices when the other is, too, and one high word
// is below 2^31)
FX_HD u64 mulhi(u64 a, u64 b) {
  const u64 c = madu(hi32(a), lo32(b), mulu(lo32(a), hi32(b)));
  return madu(hi32(a), hi32(b), pair64(hi32(c), 0u));
}
FX_HD u64 mul32(u64 a, u32 b) {  // (a b) >> 32
  return madu(hi32(a), b, pair64(hi32(mulu(lo32(a), b)), 0u));
}
FX_HD u64 sqrhi(u64 a) {  // (a^2) >> 64, a <= 2^63
  const u64 c = mulu(hi32(a), lo32(a));
  return madu(hi32(a), hi32(a), c >> 31);
}
FX_HD int clz64(u64 a) {
#ifdef __CUDA_ARCH__
  return __clzll((i64)a);
#else
  return a ? __builtin_clzll(a) : 64;
#endif
}

// z 2^ex as a double (round to nearest; z > 0 or 0).
FX_HD double to_double(u64 z, int ex) {
  if (z == 0ULL) return 0.0;
  const int lz = clz64(z);
  z <<= lz;
  const u64 m = (z + 0x400ULL) >> 11;                           // 53 bits (2^53 carries into the exponent)
  const int be = 1023 + 63 - lz + ex;
  if (be <= 0 || be >= 0x7fe || z + 0x400ULL < z) return be <= 0 ? 0.0 : scalbn((double)(z >> 1), ex - lz + 1);
  return u2d(m + ((u64)(be - 1) << 52));
}

// r^-1 and r from r2 > 0 (normal), each rounded once from 2^-59 of itself.
FX_HD void inverse_root(double r2, double &ir, double &r) {
  const u64 b = d2u(r2);
  const int q = (int)(b >> 52) - 1022, odd = q & 1, k = (q - odd) >> 1;  // r2 = R 4^k, R in [0.5, 2)
  const u64 R = (((b & 0xfffffffffffffULL) | 0x10000000000000ULL) << 9) << odd;  // 2^-62
  const float rho2 = i2f(((126 + odd) << 23) | (int)((u32)(b >> 29) & 0x7fffffu));
  const u32 U = (u32)f2i(frsqrt(rho2) + 2.0f) << 9;             // 2^-31
  const u64 e = (1ULL << 60) - mulhi(R, mulu(U, U));            // 2^-60, signed
  const int e1 = (int)((i64)e >> 11);                           // 2^-49
  const u32 ee = hi32((u64)muls(e1, e1));                       // 2^-66
  const u64 Y = mul32((1ULL << 63) + 4ULL * e + (ee * 3u >> 6), U);  // rho^-1, 2^-62
  ir = to_double(Y, -62 - k);
  r = to_double(mulhi(R, Y), -60 + k);
}

// a w + b for w in units of 2^-64, |w| < 2^63; a, b and the result in one unit, |a| < 2^62.
FX_HD i64 step64(i64 a, int wh, int wl, i64 b) {
  const int ah = hi_s((u64)a), al = (int)lo32((u64)a);
  return mads(ah, wh, mads(al, wh, muls(ah, wl)) >> 32) + b;
}

// The Stumpff functions c_k(z) = sum_m (-z)^m / (2m + k)!, k = 0..3, for |z| <= 0.4 (Taylor series to
// m = 8 of c2, c3; c0 = 1 - z c2, c1 = 1 - z c3), to 2^-60. An FP64 step of the series takes 76 cycles of
// a busy sub-partition, a fixed-point one about 26 on pipes the drift leaves idle.
FX_HD void stumpff(double z, double &c0, double &c1, double &c2, double &c3) {
  const u64 w = (u64)fixed(-z, -2);                             // 2^-64
  const int wh = hi_s(w), wl = (int)lo32(w);
  // 2^62 / (2m + 2)!, 2^62 / (2m + 3)! rounded
  constexpr i64 C2[9] = {2305843009213693952LL, 192153584101141163LL, 6405119470038039LL, 114377133393536LL, 1270857037706LL,
                         9627704831LL, 52899477LL, 220414LL, 720LL};
  constexpr i64 C3[9] = {768614336404564651LL, 38430716820228233LL, 915017067148291LL, 12708570377060LL, 115532457973LL,
                         740592679LL, 3526632LL, 12966LL, 38LL};
  i64 a = C2[8], b = C3[8];
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int m = 7; m >= 0; --m) { a = step64(a, wh, wl, C2[m]); b = step64(b, wh, wl, C3[m]); }
  c2 = to_double((u64)a, -62);
  c3 = to_double((u64)b, -62);
  c0 = to_double((u64)step64(a, wh, wl, 1LL << 62), -62);
  c1 = to_double((u64)step64(b, wh, wl, 1LL << 62), -62);
}

}  // namespace fx
}  // namespace genga
