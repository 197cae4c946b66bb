// kick_fx.cuh -- the fixed-point sum of the pulls on tiles of bodies, shared by the main mode's pair
// kernel (kick.cu) and the differentiable engine's (adjoint.cu).
//
// A CTA holds TW tiles of 32 bodies, a warp each, one body a lane, and CW chunks of at most 64
// partners in shared memory (TW CW = 8 warps); a warp sums one tile's pulls from one chunk.
//
// Pass 1 separates the near partners -- inside the caller's limit radius, or closer than the
// fixed-point grid resolves, or the body itself -- into a bit mask and bounds the sum of the others.
// Pass 2 sums the far pulls (fxpair.cuh). The near pairs of the warp are then listed and handed to
// the caller one a lane, in FP64 with its exact decisions. A CTA with a number the fixed-point form
// cannot hold (not finite, a negative mass) takes every pair as near.
//
// Radii over many octaves: one grid for all would be that of the largest radius, and every pair closer than
// 2^-9 of it near. A CTA with more than a few bodies at less than 1/32 of its largest radius gives each body
// the grid of its own radius instead and evaluates a pair on the coarser grid of the two (kx_far<true>).
// Measured with 2048 bodies at 0.5-4 AU (33.9 us a kick; the FP64 tile ring took 87 whatever the
// positions): 1, 8 or 64 of them moved to 3000 AU 143-144 us on one grid, 42 so; a tenth, half or all of
// them spread over 4-4000 AU 140, 109, 53 us on one grid, 42-43 so.
//
// What bounds it at N = 2048 (32.6 us, 33.6 with its event nodes; the FP64 tile ring it replaced 87):
// the wide multiply-adds' pipe, 62 % busy, 30 of them a pull at 4 cycles; pass 1 about 6 us, set-up and
// launch 8 us, the near pairs 3 us. Two CTAs per SM measured the same as three.
//
// No Newton's third law: the sums of the j side would rotate through the lanes with 24 more
// shuffled words a pair (4 cycles each), as much as evaluating the pair once more.
#pragma once
#include "fxpair.cuh"
#include "genga_launch.h"

namespace genga {

constexpr int KX_WARPS = 8;
constexpr int KX_CTAS = 3;  // CTAs per SM (80 registers; measured at N = 2048: two 33.9 us, three 33.7 us a kick)
constexpr int KX_LIST = 96;  // near pairs of a warp taken together
constexpr int KX_INNER = 8;  // threads with a body far inside the others that one grid for all may have
constexpr int KX_FINEST = 40;  // octaves between the finest grid and the coarsest
constexpr int KX_SMALL = 8;  // partners a chunk for fewer than 8 tiles
template <int CAP>
struct KxShared {
  float4 h[CAP], m[CAP];  // position in single precision (h + m); .w: mass, its exponent
  longlong2 xy[CAP], zM[CAP];
  float lim[CAP];
};
struct KxList {  // near pairs: body lane << 8 | partner, and their pulls
  int e[KX_LIST];
  double f[3][KX_LIST];
};

// max(T, grid limit) as the first pass's limit on rough r^2 (units of 2^(2E - 60)), rounded up by
// 2^-10 (rough r^2 is within 2^-12).
__device__ __forceinline__ float kx_limit(u64 T, int E, float grid = fx::FX_RMIN2) {
  const float t = scalbnf(d2f_safe(__longlong_as_double((long long)T)), 60 - 2 * E);
  return fmaxf(t, grid) * 1.001f;
}
__device__ __forceinline__ float kx_norm2(double x, double y, double z) {  // |x|^2, rounded up
  const float a = d2f_safe(x), b = d2f_safe(y), c = d2f_safe(z);
  return fmaf(c, c, fmaf(b, b, a * a)) * 1.000002f;
}
__device__ __forceinline__ bool kx_odd(double x) { return fx::expo(x) == 0x7ff; }
__device__ __forceinline__ int kx_exponent(float n2) { return ((__float_as_int(n2) >> 23) - 127 + 2) >> 1; }  // |x| < 2^E

// Both passes of one warp over a chunk's cnt partners: the near partners as bit masks, the sum of the far
// pulls. WIDE: body and partners are on grids of their own, di and the upper half of the partner's
// mass exponent word octaves finer than the grid of exponent E. A position moves to the pair's coarser
// grid by a shift that truncates, so that pairs are near up to twice the distance. The sums' units stay
// those of the grid E: a factor formed dl octaves finer counts 4^dl times.
template <bool WIDE, int CAP>
__device__ __forceinline__ void kx_far(const KxShared<CAP> &sm, int cnt, const fx::Pos &pi, int di, float limi, int me_max,
                                       int E, unsigned (&near)[2], double &ax, double &ay, double &az) {
  auto octaves = [&](int word, int &a, int &b) {  // from the body's and the partner's grid to the pair's; returns dl
    const int dj = (word + 0x8000) >> 16, dl = min(di, dj);
    a = di - dl; b = dj - dl;
    return dl;
  };
  auto pow2 = [](int k) { return __int_as_float((127 + k) << 23); };
  float B = 0.0f;
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    const int n = min(cnt - 32 * w, 32);
#pragma unroll 4
    for (int k = 0; k < n; ++k) {
      const float4 h = sm.h[32 * w + k];
      const float lim = fmaxf(limi, sm.lim[32 * w + k]);
      if (!WIDE) {
        const float r2 = fx::rough_r2(pi, h.x, h.y, h.z);
        if (r2 >= lim) B = fmaf(h.w, fx::frcp(r2), B);
        else near[w] |= 1u << k;
      } else {
        int a, b;
        const int dl = octaves(__float_as_int(sm.m[32 * w + k].w), a, b);
        const float sa = pow2(-a), sb = pow2(-b);
        const float dx = h.x * sb - pi.hx * sa, dy = h.y * sb - pi.hy * sa, dz = h.z * sb - pi.hz * sa;
        const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
        if (r2 >= 4.004f * fx::FX_RMIN2 && r2 * pow2(-2 * dl) >= lim) B = fmaf(h.w, fx::frcp(r2) * pow2(2 * dl), B);
        else near[w] |= 1u << k;
      }
    }
  }
  const int A = fx::units(B, me_max);
  fx::Acc acc;
  fx::clear(acc);
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    const int n = min(cnt - 32 * w, 32);
    for (int k0 = 0; k0 < n; k0 += fx::FX_FLUSH) {
      const int k1 = min(n, k0 + fx::FX_FLUSH);
#pragma unroll 2
      for (int k = k0; k < k1; ++k) {
        const float4 h = sm.h[32 * w + k], m = sm.m[32 * w + k];
        const longlong2 p = sm.xy[32 * w + k], q = sm.zM[32 * w + k];
        const bool use = !((near[w] >> k) & 1u);
        if (!WIDE) {
          const fx::Pos pj = {p.x, p.y, q.x, h.x, h.y, h.z, m.x, m.y, m.z};
          fx::pull(pi, pj, (u64)q.y, __float_as_int(m.w), A, use, acc);
        } else {
          const int word = __float_as_int(m.w);
          int a, b;
          const int dl = octaves(word, a, b);
          const float sa = pow2(-a), sb = pow2(-b);
          fx::pull((h.x * sb - pi.hx * sa) + (m.x * sb - pi.mx * sa), (h.y * sb - pi.hy * sa) + (m.y * sb - pi.my * sa),
                   (h.z * sb - pi.hz * sa) + (m.z * sb - pi.mz * sa), (p.x >> b) - (pi.X >> a), (p.y >> b) - (pi.Y >> a),
                   (q.x >> b) - (pi.Z >> a), (u64)q.y, word - ((dl + b) << 16), A - 2 * dl, use, acc);
        }
      }
      fx::flush(acc);
    }
  }
  ax = fx::value(acc.h[0], acc.l[0], A, E);
  ay = fx::value(acc.h[1], acc.l[1], A, E);
  az = fx::value(acc.h[2], acc.l[2], A, E);
}

template <int CAP>
__device__ __noinline__ void kx_far_wide(const KxShared<CAP> &sm, int cnt, const fx::Pos &pi, int di, float limi, int me_max, int E,
                                         unsigned (&near)[2], double (&f)[3]) {
  kx_far<true>(sm, cnt, pi, di, limi, me_max, E, near, f[0], f[1], f[2]);
}

// The pulls on body (base + I 32 + lane), I = tg TW + wid % TW, from the partners of chunk c0 = cg CW +
// wid / TW (kchunk partners each, np bodies, nt tiles, C chunks) into (ax, ay, az); x: component-major
// with leading dimension ld. lim: squared limit radii (bits); a pair inside max(lim_i, lim_j), or
// closer than the grid resolves, is near(i, j, dx, dy, dz)'s, which returns the pull's factor.
// Returns false for a warp without a tile and chunk. All threads of the CTA call it.
// OUT: the rare kx_far<true> as a call, otherwise in line. In line the kernel's code is longer, which short
// launches pay for: 10 steps of 500 bodies +1.2%, gradients of systems of up to seven tiles +1.6%; as a
// call the gradient of 64 systems of eight tiles +0.3%.
template <int TW, bool OUT, class Near>
__device__ __forceinline__ bool kx_block(const double *__restrict__ X, int ld, const double *__restrict__ gm,
                                         const int *__restrict__ alive, const u64 *__restrict__ lim, int base, int np,
                                         int nt, int C, int kchunk, int tg, int cg, Near near_pair, int &I, int &c0,
                                         bool &ali, double &ax, double &ay, double &az) {
  constexpr int CW = KX_WARPS / TW, CAP = TW == 8 ? fx::FX_CHUNK : KX_SMALL;
  __shared__ KxShared<CAP> smem[CW];
  __shared__ KxList slist[KX_WARPS];
  __shared__ int s_n2, s_lo, s_me[CW];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int cw = wid / TW;
  I = tg * TW + wid % TW;
  c0 = cg * CW + cw;
  const bool on = I < nt && c0 < C;
  if (tid == 0) { s_n2 = 0; s_lo = 0x7f800000; }
  if (tid < CW) s_me[tid] = -2000;
  // own body; partners (one a thread, twice over when the CTA holds more than four chunks)
  const int i = base + min(I, nt - 1) * 32 + lane;
  ali = on && alive[i] != 0;
  const double xi = ali ? X[i] : 0.0, yi = ali ? X[ld + i] : 0.0, zi = ali ? X[2 * ld + i] : 0.0;
  const u64 Ti = ali ? lim[i] : 0ULL;
  constexpr int NB = CW * CAP, PB = (NB + 32 * KX_WARPS - 1) / (32 * KX_WARPS);
  double bx[PB], by[PB], bz[PB], bg[PB];
  u64 bT[PB];
  const float ni = kx_norm2(xi, yi, zi);
  float nb[PB], n2 = ni, lo = ni > 0.0f ? ni : __int_as_float(0x7f800000);  // of the thread: largest, smallest
  bool odd = kx_odd(xi) || kx_odd(yi) || kx_odd(zi);
#pragma unroll
  for (int k = 0; k < PB; ++k) {
    const int q = tid + 32 * KX_WARPS * k, ch = cg * CW + q / CAP, u = q % CAP;
    const int jl = ch * kchunk + u, j = base + jl;
    const bool al = q < NB && ch < C && u < kchunk && jl < np && alive[j] != 0;
    bx[k] = al ? X[j] : 0.0; by[k] = al ? X[ld + j] : 0.0; bz[k] = al ? X[2 * ld + j] : 0.0;
    bg[k] = al ? gm[j] : 0.0;
    bT[k] = al ? lim[j] : 0ULL;
    nb[k] = kx_norm2(bx[k], by[k], bz[k]);
    n2 = fmaxf(n2, nb[k]);
    if (nb[k] > 0.0f) lo = fminf(lo, nb[k]);
    odd |= kx_odd(bx[k]) || kx_odd(by[k]) || kx_odd(bz[k]) || kx_odd(bg[k]) || (long long)dbits(bg[k]) < 0;
  }
  __syncthreads();
  // common scale: |x| < 2^E; per chunk the largest mass exponent
  const int wn2 = __reduce_max_sync(0xffffffffu, odd ? 0x7f800000 : __float_as_int(n2));
  const int wlo = __reduce_min_sync(0xffffffffu, __float_as_int(lo));
  if (lane == 0) { atomicMax(&s_n2, wn2); atomicMin(&s_lo, wlo); }
#pragma unroll
  for (int k = 0; k < PB; ++k) {
    const int q = tid + 32 * KX_WARPS * k;
    if (q >= NB) continue;
    u64 M;
    int me;
    fx::set_mass(bg[k], M, me);
    if (M) atomicMax(&s_me[q / CAP], me);
  }
  __syncthreads();
  odd = s_n2 >= 0x7f000000;
  const int E = odd ? 0 : kx_exponent(__int_as_float(s_n2)), inner = s_n2 - (10 << 23);
  bool wide = !odd && s_lo < inner;
  if (wide) wide = __syncthreads_count(__float_as_int(lo) < inner) > KX_INNER;
  auto grid = [&](float n) { return wide ? max(kx_exponent(n), E - KX_FINEST) : E; };
#pragma unroll
  for (int k = 0; k < PB; ++k) {
    const int q = tid + 32 * KX_WARPS * k;
    if (q >= NB) continue;
    KxShared<CAP> &sm = smem[q / CAP];
    const int u = q % CAP;
    fx::Pos p;
    u64 M;
    int me;
    const int Eb = grid(nb[k]);
    fx::set_pos(p, odd ? 0.0 : bx[k], odd ? 0.0 : by[k], odd ? 0.0 : bz[k], Eb);
    fx::set_mass(odd ? 0.0 : bg[k], M, me);
    sm.h[u] = make_float4(p.hx, p.hy, p.hz, fx::mass_f(M, me, s_me[q / CAP]));
    sm.m[u] = make_float4(p.mx, p.my, p.mz, __int_as_float(me + ((E - Eb) << 16)));
    sm.xy[u] = make_longlong2(p.X, p.Y);
    sm.zM[u] = make_longlong2(p.Z, (long long)M);
    sm.lim[u] = kx_limit(bT[k], E, wide ? 0.0f : fx::FX_RMIN2);
  }
  fx::Pos pi;
  const int Ei = grid(ni);
  fx::set_pos(pi, odd ? 0.0 : xi, odd ? 0.0 : yi, odd ? 0.0 : zi, Ei);
  const float limi = odd ? __int_as_float(0x7f800000) : kx_limit(Ti, E, wide ? 0.0f : fx::FX_RMIN2);
  __syncthreads();
  ax = ay = az = 0.0;
  if (!on) return false;
  const KxShared<CAP> &sm = smem[cw];
  const int j0 = c0 * kchunk, cnt = min(kchunk, np - j0);  // at least one partner
  unsigned near[2] = {0u, 0u};
  if (wide && OUT) {
    unsigned nw[2] = {0u, 0u};
    double f[3];
    kx_far_wide(sm, cnt, pi, E - Ei, limi, s_me[cw], E, nw, f);
    near[0] = nw[0]; near[1] = nw[1];
    ax = f[0]; ay = f[1]; az = f[2];
  } else if (wide) {
    kx_far<true>(sm, cnt, pi, E - Ei, limi, s_me[cw], E, near, ax, ay, az);
  } else {
    kx_far<false>(sm, cnt, pi, 0, limi, s_me[cw], E, near, ax, ay, az);
  }
  // the near pairs in FP64: listed by (body, partner), one a lane, added per body in partner order
  {
    const unsigned self = I * 32 + lane - j0;  // the body itself is not a pair
    if (self < 32u) near[0] &= ~(1u << self);
    else if (self < 64u) near[1] &= ~(1u << (self - 32u));
    if (!ali) { near[0] = 0u; near[1] = 0u; }
  }
  const int nn = __popc(near[0]) + __popc(near[1]);
  int incl = nn;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  KxList &L = slist[wid];
  int at = incl - nn;
  for (int b0 = 0; b0 < total; b0 += KX_LIST) {
    const int first = at;
#pragma unroll
    for (int w = 0; w < 2; ++w)
      for (; near[w] && at < b0 + KX_LIST; near[w] &= near[w] - 1) L.e[at++ - b0] = lane << 8 | (32 * w + __ffs(near[w]) - 1);
    __syncwarp();
    for (int k = lane; k < min(total - b0, KX_LIST); k += 32) {
      double dx = 0.0, dy = 0.0, dz = 0.0;
      const double g = near_pair(base + I * 32 + (L.e[k] >> 8), base + j0 + (L.e[k] & 255), dx, dy, dz);
      L.f[0][k] = g * dx; L.f[1][k] = g * dy; L.f[2][k] = g * dz;
    }
    __syncwarp();
    for (int k = first; k < at; ++k) { ax += L.f[0][k - b0]; ay += L.f[1][k - b0]; az += L.f[2][k - b0]; }
    __syncwarp();
  }
  return true;
}

}  // namespace genga
