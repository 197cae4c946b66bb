// fxforce.cuh -- the scalar factor of a Bulirsch-Stoer pull, G m W_A(r) / r^3 from r^2, in 64-bit
// fixed point.
//
// A force evaluation of the Bulirsch-Stoer kernels is one chain of FP64 instructions, 64-76 cycles
// each whatever the warp's active lanes, and it sets their time. Of the 33 instructions of a term 20
// turn r^2 into the factor (the refined inverse square root, the changeover weight with its
// reciprocal, the products). Here that part runs on the integer pipes: a 64 x 64 bit product's upper
// half takes three wide multiply-adds and about 15 cycles of latency. Every quantity carries 57 or
// more significant bits (the weight: 57 bits after the point), so the factor is the correctly rounded
// one to about 0.6 ulp, the FP64 form to about 2. Measured: 8192 systems x 4 steps 8.69 -> 7.23 ms, 300
// systems 2.98 -> 2.55 ms, 10^5 test particles x 4 steps 2.17 -> 1.90 ms.
//
//   r^2 = R 4^k, R in [0.5, 2); u = 2^-23-accurate R^(-1/2); e = 1 - R u^2 (exact to 2^-59)
//   r^-3 = 8^-k u^3 (1 + 3/2 e + 15/8 e^2), r = 2^k R u (1 + e/2 + 3/8 e^2)
//   y = r A - 1/9 clamped to [0, 1], W_A = (1 - y)^2 / (y^2 + (1 - y)^2) with the reciprocal from its
//   single-precision seed s: s (1 + e' + e'^2), e' = 1 - s (y^2 + (1 - y)^2)
#pragma once
#include "fxmath.cuh"
#ifdef __CUDACC__
#include "genga_dev.cuh"
#endif

namespace genga {
namespace fx {

// A positive double's mantissa in [2^62, 2^63) and exponent: x = M 2^(me - 63); zero: M = 0.
struct Num {
  u64 M;
  int me;
};
FX_HD Num num(double x) {
  Num n;
  set_mass(x, n.M, n.me);
  return n;
}

// pref w rho^-3 in 2^-59 (times 2^pref.me) from rho^2 = R 2^-62 in [0.5, 2) and its single-precision
// value; r = rho 2^k. w = 1 (full), W_A of the changeover zone with A = 1/(0.9 rc) (zone), or 0.
FX_HD u64 factor(u64 R, float rho2, int k, const Num &pref, const Num &A, bool full, bool zone) {
  const u32 U = (u32)f2i(frsqrt(rho2) + 2.0f) << 9;             // 2^-31
  const u64 W = mulu(U, U);                                     // 2^-62
  const u64 e = (1ULL << 60) - mulhi(R, W);                     // 2^-60, signed
  const int e1 = (int)((i64)e >> 11);                           // 2^-49
  const u32 ee = hi32((u64)muls(e1, e1));                       // 2^-66
  const u64 F = (1ULL << 63) + 12ULL * e + (ee * 15u >> 6);
  const u64 Y3 = mulhi(mul32(W, U), F);                         // rho^-3, 2^-60
  u64 w = full ? (1ULL << 63) : 0ULL;                           // 2^-63
  if (zone && !full) {
    const u64 rho = mulhi(mul32(R, U), (1ULL << 63) + 4ULL * e + (ee * 3u >> 6));  // 2^-60
    const int n = k + A.me;                                     // r A = rho M_A 2^n
    i64 y = (i64)((mulhi(rho, A.M) << ((n + 3) & 63)) >> 1);    // r A in 2^-61 for -3 <= n <= 1
    y -= 256204778801521550LL;                                  // 2^61 / 9
    if (n < -3) y = 0;
    if (n > 1) y = 1LL << 61;
    y = y < 0 ? 0 : (y > (1LL << 61) ? (1LL << 61) : y);
    const u64 yy = sqrhi((u64)y << 2), oo = sqrhi((1ULL << 63) - ((u64)y << 2));  // 2^-62
    const u64 D = yy + oo;                                      // in [0.5, 1]
    const float s = frcp((float)(int)hi32(D) * 9.313225746154785e-10f);  // 1 .. 2
    const u32 S = (u32)f2i(s + 4.0f) << 9;                      // 2^-30
    const u64 d = (1ULL << 60) - mul32(D, S);                   // 2^-60, signed
    const int d1 = (int)((i64)d >> 11);
    const u64 H = (1ULL << 63) + 8ULL * d + (hi32((u64)muls(d1, d1)) >> 3);
    w = mulhi(mul32(oo, S), H) << 4;
  }
  return mulhi(mulhi(Y3 << 1, w), pref.M);
}

// pref w / r^3 for r2 > 0 (normal); full, zone as in factor.
FX_HD double pull_factor(double r2, const Num &pref, const Num &A, bool full, bool zone) {
  const u64 b = d2u(r2);
  const int q = (int)(b >> 52) - 1022, odd = q & 1, k = (q - odd) >> 1;  // r2 = R 4^k, R in [0.5, 2)
  const u64 R = (((b & 0xfffffffffffffULL) | 0x10000000000000ULL) << 9) << odd;  // 2^-62
  const float rho2 = i2f(((126 + odd) << 23) | (int)((u32)(b >> 29) & 0x7fffffu));
  return to_double(factor(R, rho2, k, pref, A, full, zone), pref.me - 59 - 3 * k);
}

// r^-3 and r^-5 for r2 > 0 (normal).
FX_HD void inverse_powers(double r2, double &y3, double &y5) {
  const u64 b = d2u(r2);
  const int q = (int)(b >> 52) - 1022, odd = q & 1, k = (q - odd) >> 1;  // r2 = R 4^k, R in [0.5, 2)
  const u64 R = (((b & 0xfffffffffffffULL) | 0x10000000000000ULL) << 9) << odd;  // 2^-62
  const float rho2 = i2f(((126 + odd) << 23) | (int)((u32)(b >> 29) & 0x7fffffu));
  const u32 U = (u32)f2i(frsqrt(rho2) + 2.0f) << 9;             // 2^-31
  const u64 W = mulu(U, U);                                     // 2^-62
  const u64 e = (1ULL << 60) - mulhi(R, W);                     // 2^-60, signed
  const int e1 = (int)((i64)e >> 11);                           // 2^-49
  const u32 ee = hi32((u64)muls(e1, e1));                       // 2^-66
  const u64 Y3 = mulhi(mul32(W, U), (1ULL << 63) + 12ULL * e + (ee * 15u >> 6));  // rho^-3, 2^-60
  const u64 Y2 = mulhi(W, (1ULL << 63) + 8ULL * e + (ee >> 3)); // rho^-2, 2^-61
  y3 = to_double(Y3, -60 - 3 * k);
  y5 = to_double(mulhi(Y3 << 1, Y2 << 1), -59 - 5 * k);
}

}  // namespace fx

#ifdef __CUDACC__
// The factor of one Bulirsch-Stoer term from its r^2: the whole pull (central mass), the pull weighted
// by W_A (inside the pair's critical radius), else 0 without evaluating anything. kmode 1 (the exact
// gradient of H_B) keeps the FP64 form, and so does an r^2 that has no normalised mantissa: for members
// at one position it gives a finite factor, which their separation of zero then annuls.
__device__ __forceinline__ bool bs_factor_is_fixed(double r2, int kmode) {
  return kmode == 0 && (unsigned)__double2hiint(r2) >= 0x00100000u;
}
static __device__ __noinline__ double bs_factor_fp64(double r2, double pref, double A, bool full, int kmode) {
  const double yr = rsqrt_refined(r2);
  const double w = full ? 1.0 : changeover_wA_clamped(r2 * yr, A, kmode);
  return pref * w * (yr * yr * yr);
}
__device__ __forceinline__ double bs_factor(double r2, double pref, double A, bool full, bool inside, int kmode) {
  if (!full && !inside) return 0.0;
  if (bs_factor_is_fixed(r2, kmode)) {
    const double f = fx::pull_factor(r2, fx::num(pref), fx::num(A), full, inside);
    return __longlong_as_double(__double_as_longlong(f) | (__double_as_longlong(pref) & (long long)0x8000000000000000ULL));
  }
  return bs_factor_fp64(r2, pref, A, full, kmode);
}
#endif
}  // namespace genga
