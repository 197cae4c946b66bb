// Host run of the fixed-point pair pull (fxpair.cuh) against extended precision, on pairs at the ends of its
// ranges: G m at the top and the bottom of a binade, r^2 around even and odd powers of two (the ends of
// the normalised rho^2), the inverse root exact, low and high by the device's error. Prints the largest
// error of a sum relative to the sum of its terms' magnitudes, in units of 2^-53, and what it was met at.
#include <cmath>
#include <cstdio>
#include <random>
#include "fxpair.cuh"

static double seed_error = 0.0;
namespace genga {
namespace fx {
float fx_host_rsqrt(float x) { return (float)(1.0 / std::sqrt((double)x) * (1.0 + seed_error)); }
float fx_host_rcp(float x) { return (float)(1.0 / (double)x * (1.0 + seed_error)); }
}  // namespace fx
}  // namespace genga
using namespace genga::fx;

int main() {
  std::mt19937_64 rng(3);
  std::uniform_real_distribution<double> u01(0.0, 1.0);
  std::normal_distribution<double> normal;
  const double mantissas[] = {1.0 - 0x1p-53, 1.0 - 1e-12, 1.0 - 1e-8, 1.0 - 1e-7, 1.0 - 3e-7, 0.5, 0.5 * (1.0 + 0x1p-52), 0.5 * (1.0 + 1e-7)};
  const double seeds[] = {0.0, -1.2e-7, 1.2e-7};
  double worst = 0.0;
  long pairs = 0;
  for (int E = 1; E <= 3; ++E)
    for (double se : seeds)
      for (double mant : mantissas)
        for (int p = -6; p <= 2; ++p)        // r^2 around 2^p
          for (int trial = 0; trial < 150; ++trial) {
            seed_error = se;
            const int n = trial % 3 == 0 ? 1 : (trial % 3 == 1 ? 8 : 64);  // partners of a chunk
            const double gm = std::ldexp(mant, -10);
            double xi[3], xj[64][3];
            for (int c = 0; c < 3; ++c) xi[c] = 0.1 * (2.0 * u01(rng) - 1.0);
            for (int j = 0; j < n; ++j) {
              double d[3], s = 0.0;
              for (int c = 0; c < 3; ++c) { d[c] = normal(rng); s += d[c] * d[c]; }
              const double r = std::sqrt(std::ldexp(1.0, p)) * (1.0 + 3e-7 * (2.0 * u01(rng) - 1.0));
              double m = 0.0;
              for (int c = 0; c < 3; ++c) { xj[j][c] = xi[c] + d[c] * r / std::sqrt(s); m += xj[j][c] * xj[j][c]; }
              if (m >= std::ldexp(1.0, 2 * E)) --j;  // outside this grid: draw again
              if (p > 2 * E - 2) break;
            }
            if (p > 2 * E - 2) break;
            Pos pi;
            set_pos(pi, xi[0], xi[1], xi[2], E);
            u64 M;
            int me;
            set_mass(gm, M, me);
            Pos pj[64];
            float B = 0.0f;
            for (int j = 0; j < n; ++j) {
              set_pos(pj[j], xj[j][0], xj[j][1], xj[j][2], E);
              B = ffma(mass_f(M, me, me), fx_host_rcp(rough_r2(pi, pj[j].hx, pj[j].hy, pj[j].hz)), B);
            }
            const int A = units(B, me);
            Acc acc;
            clear(acc);
            long double want[3] = {0, 0, 0}, mag = 0;
            for (int j = 0; j < n; ++j) {
              pull(pi, pj[j], M, me, A, true, acc);
              if (j % FX_FLUSH == FX_FLUSH - 1) flush(acc);
              const long double dx = (long double)xj[j][0] - xi[0], dy = (long double)xj[j][1] - xi[1], dz = (long double)xj[j][2] - xi[2];
              const long double r2 = dx * dx + dy * dy + dz * dz, f = (long double)gm / (r2 * std::sqrt(r2));
              want[0] += f * dx; want[1] += f * dy; want[2] += f * dz;
              mag += (long double)gm / r2;
            }
            flush(acc);
            long double err = 0;
            for (int c = 0; c < 3; ++c) {
              const long double e = (long double)value(acc.h[c], acc.l[c], A, E) - want[c];
              err += e * e;
            }
            const double rel = (double)(std::sqrt(err) / mag * 0x1p53L);
            pairs += n;
            if (!(rel <= worst)) {
              worst = rel;
              std::fprintf(stderr, "E %d seed %g mantissa 1 - %g r^2 ~ 2^%d partners %d: %g\n", E, se, 1.0 - mant, p, n, rel);
            }
          }
  std::printf("%ld %.6g\n", pairs, worst);
  return 0;
}
