// fxpair.cuh -- the Newtonian pull G m_j d / r^3 of a pair in 64-bit fixed point on the integer and
// FP32 pipes.
//
// FP64 is issued at two lanes per clock per SM (64-76 cycles a warp instruction and sub-partition);
// a 32 x 32 + 64 bit multiply-add takes 4 cycles, a 32-bit integer operation 2, an FP32 one 1
// (measured). A pull costs about 17 FP64 instructions (1200 cycles a warp of ordered pairs); here it
// takes about 20 wide multiply-adds, 50 other integer and 35 FP32 operations, and it is the more
// accurate of the two: every quantity carries 55 or more significant bits, and the sums are exact.
//
//   positions   X = x 2^(62 - E) rounded to an integer, |x| < 2^E (2-norm) for the bodies of one
//               call: a component is exact from 2^(E - 10) on (a double has 53 bits), else within
//               2^(E - 63); d = X_j - X_i exact
//   unit vector rho = r scaled by a power of two into [0.70, 1.42), U = 2^29/rho to 2^-21 from the
//               single-precision inverse square root, v = d U: |v| = 2^61 (1 - delta)
//   residual    e = 1 - |v|^2 / 2^122 to 2^-57, |e| < 2^-19.9
//   pull        G m_j / r^2 . (d / r) = (G m_j U^2)(1 + 3/2 e + 15/8 e^2) v (Taylor series of
//               (1 - e)^(-3/2); the next term is below 2^-58)
//   sum         the scalar factor as a 61-bit integer in units of 2^A, A chosen per body so that the
//               factors of one chunk of partners add up to less than 2^61 (a first pass over the
//               chunk bounds the sum in single precision); the products are summed exactly
//
// A pair closer than FX_RMIN2 (r < 2^(E - 9)) is left to the FP64 code: there the rounding of X
// could exceed the rounding of the FP64 formula.
#pragma once
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define FX_HD __host__ __device__ __forceinline__
#else
#define FX_HD inline
#endif

namespace genga {
namespace fx {

typedef long long i64;
typedef unsigned long long u64;
typedef unsigned int u32;

constexpr float FX_RMIN2 = 4398046511104.0f;  // 2^42: smallest r^2 in units of 2^(2E - 60)
constexpr int FX_CHUNK = 64;                  // most partners summed in one set of accumulators
constexpr int FX_FLUSH = 4;                   // partners between two carries of the low sums (6 fit)

FX_HD int f2i(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_int(f);
#else
  int i; memcpy(&i, &f, 4); return i;
#endif
}
FX_HD float i2f(int i) {
#ifdef __CUDA_ARCH__
  return __int_as_float(i);
#else
  float f; memcpy(&f, &i, 4); return f;
#endif
}
FX_HD u64 d2u(double d) {
#ifdef __CUDA_ARCH__
  return (u64)__double_as_longlong(d);
#else
  u64 u; memcpy(&u, &d, 8); return u;
#endif
}
FX_HD double u2d(u64 u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((i64)u);
#else
  double d; memcpy(&d, &u, 8); return d;
#endif
}
#ifndef __CUDACC__
float fx_host_rsqrt(float x);  // the host test supplies an approximation with the device's error
float fx_host_rcp(float x);
#endif
FX_HD float frsqrt(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#elif defined(__CUDACC__)
  return x;  // device code only
#else
  return fx_host_rsqrt(x);
#endif
}
FX_HD float frcp(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#elif defined(__CUDACC__)
  return x;
#else
  return fx_host_rcp(x);
#endif
}
FX_HD float ffma(float a, float b, float c) {
#ifdef __CUDA_ARCH__
  return __fmaf_rn(a, b, c);
#else
  return __builtin_fmaf(a, b, c);
#endif
}
// Wide multiply-adds as PTX: the compiler's own expansion of the C expressions moves operands about
// (measured: 85 against 52 instructions on the multiply-add pipe a pull).
FX_HD i64 mads(int a, int b, i64 c) {  // signed 32 x 32 + 64
#ifdef __CUDA_ARCH__
  i64 r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (i64)a * b + c;
#endif
}
FX_HD i64 muls(int a, int b) {
#ifdef __CUDA_ARCH__
  i64 r;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
#else
  return (i64)a * b;
#endif
}
FX_HD u64 madu(u32 a, u32 b, u64 c) {  // unsigned
#ifdef __CUDA_ARCH__
  u64 r;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (u64)a * b + c;
#endif
}
FX_HD u64 mulu(u32 a, u32 b) {
#ifdef __CUDA_ARCH__
  u64 r;
  asm("mul.wide.u32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
#else
  return (u64)a * b;
#endif
}
FX_HD u32 lo32(u64 a) {
#ifdef __CUDA_ARCH__
  u32 l, h;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(l), "=r"(h) : "l"(a));
  return l;
#else
  return (u32)a;
#endif
}
FX_HD u32 hi32(u64 a) {
#ifdef __CUDA_ARCH__
  u32 l, h;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(l), "=r"(h) : "l"(a));
  return h;
#else
  return (u32)(a >> 32);
#endif
}
FX_HD u64 pair64(u32 lo, u32 hi) {
#ifdef __CUDA_ARCH__
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
  return r;
#else
  return (u64)hi << 32 | lo;
#endif
}
FX_HD u64 shr_clamp(u64 a, int s) {                                   // a >> s, 0 from 64 on
#ifdef __CUDA_ARCH__
  u64 r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(s));
  return r;
#else
  return s > 63 ? 0 : a >> s;
#endif
}
// The high word of a 64-bit number whose low word is read as signed: a = hi_s(a) 2^32 + (int)lo(a).
FX_HD int hi_s(u64 a) { return (int)(hi32(a) + (lo32(a) >> 31)); }

// Biased exponent field of a double (0x7ff: not finite).
FX_HD int expo(double x) { return (int)((d2u(x) >> 52) & 0x7ffu); }

// x 2^(62 - E) to the nearest integer; |x| < 2^E and finite.
FX_HD i64 fixed(double x, int E) {
  const u64 b = d2u(x);
  const int ex = (int)((b >> 52) & 0x7ffu), sh = ex - 1013 - E;  // value = mant 2^sh
  const u64 mant = ex ? ((b & 0xfffffffffffffULL) | 0x10000000000000ULL) : 0ULL;
  u64 r;
  if (sh >= 0) r = mant << (sh & 63);
  else r = sh < -60 ? 0ULL : ((mant >> (-sh - 1)) + 1ULL) >> 1;
  return (b >> 63) ? -(i64)r : (i64)r;
}

// A body as a partner: position, the position in single precision (h + m, units of 2^32), G m as
// M 2^(me - 63) with M in [2^62, 2^63) (0: massless).
struct Pos {
  i64 X, Y, Z;
  float hx, hy, hz, mx, my, mz;
};

FX_HD void split(i64 X, float &h, float &m) {
  const int hi = (int)(X >> 32);
  h = (float)hi;
  m = ffma((float)(u32)X, 2.3283064365386963e-10f, (float)(hi - (int)h));
}
FX_HD void set_pos(Pos &p, double x, double y, double z, int E) {
  p.X = fixed(x, E); p.Y = fixed(y, E); p.Z = fixed(z, E);
  split(p.X, p.hx, p.mx); split(p.Y, p.hy, p.my); split(p.Z, p.hz, p.mz);
}
FX_HD void set_mass(double gm, u64 &M, int &me) {  // gm >= 0, finite (denormals count as zero)
  const u64 b = d2u(gm);
  const int ex = (int)((b >> 52) & 0x7ffu);
  M = ex ? (((b & 0xfffffffffffffULL) | 0x10000000000000ULL) << 10) : 0ULL;
  me = ex - 1022;
}
// G m in single precision times 2^(60 - me_max), for the bound pass.
FX_HD float mass_f(u64 M, int me, int me_max) {
  const int ex = 127 + 60 + me - me_max - 1;
  return (M == 0ULL || ex <= 0) ? 0.0f : i2f((ex << 23) | (int)((M >> 39) & 0x7fffffu));
}

// The units exponent A of a body's sums, from the single-precision bound B of its chunk (sum of
// mass_f / r^2 with the rough r^2, within 2^-12, so rounded up by 2^-10); the sum of the factors is then
// below 2^61.
FX_HD int units(float B, int me_max) {
  int ex = ((f2i(B * 1.001f) >> 23) & 0xff) - 127;  // the bound in [2^ex, 2^(ex+1))
  if (ex < -120) ex = -120;
  return ex + 1 + me_max - 120;
}

struct Acc {
  i64 h[3], l[3];  // sums of the products' 2^64 and 2^32 parts
};

FX_HD void clear(Acc &a) {
  for (int c = 0; c < 3; ++c) { a.h[c] = 0; a.l[c] = 0; }
}
FX_HD void flush(Acc &a) {  // carries the low sums
  for (int c = 0; c < 3; ++c) {
    a.h[c] += (int)hi32((u64)a.l[c]);
    a.l[c] = (i64)pair64(lo32((u64)a.l[c]), 0u);
  }
}
// The sum (after flush) in the caller's units (positions scaled by 2^(62 - E)); |h| < 2^58.
FX_HD double value(i64 h, i64 l, int A, int E) {
  const i64 s = (i64)((u64)h << 4 | (u64)l >> 28);
  if (s == 0) return 0.0;
  const double d = (double)s;
  const int k = A + 59 - 2 * E, ex = expo(d) + k;
  if (ex > 0 && ex < 0x7ff) return u2d(d2u(d) + ((u64)(i64)k << 52));  // exact
  return scalbn(d, k);
}

// (d U) >> s as 64 bits, 0 < s < 32.
FX_HD u64 unit(i64 d, u32 U, int s) {
  const u64 lo = mulu(lo32((u64)d), U);
  const u64 hi = (u64)mads((int)hi32((u64)d), (int)U, (i64)pair64(hi32(lo), 0u));
#ifdef __CUDA_ARCH__
  return pair64(__funnelshift_r(lo32(lo), lo32(hi), s), __funnelshift_r(lo32(hi), hi32(hi), s));
#else
  return (u64)(((__int128)(i64)hi << 32 | lo32(lo)) >> (s & 31));
#endif
}

// One partner: adds the pull of M_j to the sums, from the separation (dX, dY, dZ) and the same in single
// precision (fx, fy, fz; units of 2^32). use: false leaves the partner out.
FX_HD void pull(float fx, float fy, float fz, i64 dX, i64 dY, i64 dZ, u64 M, int me, int A, bool use, Acc &acc) {
  // single precision: r^2 in units of 2^64, its exponent, the inverse square root
  const float r2 = ffma(fz, fz, ffma(fy, fy, fx * fx));
  const int eb = f2i(r2), kk = eb >> 24;                      // r = rho 2^(kk - 63)
  const float rho2 = i2f(eb - (kk << 24) + (126 << 23));      // in [0.5, 2)
  const float u2 = frsqrt(rho2) + 2.0f;
  const u32 U2 = (u32)f2i(u2) << 9, U = U2 >> 2;              // 2^31 / rho, 2^29 / rho: 23 bits
  // unit vector, |v| = 2^61: the 96-bit products d U, shifted down by their exponent (21 .. 31)
  const u64 vx = unit(dX, U, kk - 63), vy = unit(dY, U, kk - 63), vz = unit(dZ, U, kk - 63);
  const int ax = hi_s(vx), ay = hi_s(vy), az = hi_s(vz);
  const int bx = (int)lo32(vx), by = (int)lo32(vy), bz = (int)lo32(vz);
  // e = 1 - |v|^2, in 2^-58
  const i64 cr = mads(az, bz, mads(ay, by, muls(ax, bx))) >> 31;
  const u64 S = (u64)mads(az, az, mads(ay, ay, mads(ax, ax, cr)));
  const u64 e = (1ULL << 58) - S;
#ifdef __CUDA_ARCH__
  const int e1 = (int)__funnelshift_r(lo32(e), hi32(e), 9);   // 2^-49
#else
  const int e1 = (int)(e >> 9);
#endif
  const u32 q = hi32((u64)muls(e1, e1));                      // e^2 in 2^-66
  // F = 2^63 (1 + 3/2 e + 15/8 e^2)
  u64 F = madu(lo32(e), 48u, pair64(q * 15u >> 6, 0x80000000u));
  F = pair64(lo32(F), hi32(F) + hi32(e) * 48u);
  // G m_j / r^2: (M W >> 64) F >> 64, W = U2^2
  const u64 W = mulu(U2, U2);
  const u64 cq = madu(hi32(M), lo32(W), mulu(lo32(M), hi32(W)));
  const u64 Q = madu(hi32(M), hi32(W), pair64(hi32(cq), 0u));
  const u64 cf = madu(hi32(Q), lo32(F), mulu(lo32(Q), hi32(F)));
  const u64 C = madu(hi32(Q), hi32(F), pair64(hi32(cf), 0u));
  // C = M / (8 rho^2), in [2^58, 2^61] up to the error of U: the largest M at rho^2 = 0.5 passes 2^61, so
  // the product keeps a spare bit on top; the smallest C with a factor below 2^61 leaves the shift at 0
  const int sh = use ? A - me - 64 + 2 * kk : 64;
  const u64 g = shr_clamp(C << 2, sh);
  const int gh = hi_s(g), gl = (int)lo32(g);
  acc.h[0] = mads(ax, gh, acc.h[0]); acc.h[1] = mads(ay, gh, acc.h[1]); acc.h[2] = mads(az, gh, acc.h[2]);
  acc.l[0] = mads(ax, gl, mads(bx, gh, acc.l[0]));
  acc.l[1] = mads(ay, gl, mads(by, gh, acc.l[1]));
  acc.l[2] = mads(az, gl, mads(bz, gh, acc.l[2]));
}

FX_HD void pull(const Pos &i, const Pos &j, u64 M, int me, int A, bool use, Acc &acc) {
  pull((j.hx - i.hx) + (j.mx - i.mx), (j.hy - i.hy) + (j.my - i.my), (j.hz - i.hz) + (j.mz - i.mz), j.X - i.X, j.Y - i.Y,
       j.Z - i.Z, M, me, A, use, acc);
}

// Rough r^2 (units of 2^64) of the first pass.
FX_HD float rough_r2(const Pos &i, float hx, float hy, float hz) {
  const float fx = hx - i.hx, fy = hy - i.hy, fz = hz - i.hz;
  return ffma(fz, fz, ffma(fy, fy, fx * fx));
}

}  // namespace fx
}  // namespace genga
