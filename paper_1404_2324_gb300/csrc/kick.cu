// kick.cu -- critical radii (Eq. rcrit), the K-weighted pairwise kick with the prechecker
// (Eq. Hb, Sect. 2.2 and 3.2 "Kick"), and its per-body finalisation (KickA/KickB reuse).
//
// Pair kernels. k_kick_fx (more than 64 bodies) evaluates each body's pull from every partner in 64-bit
// fixed point on the integer and FP32 pipes (fxpair.cuh). k_kick_small (up to 64 bodies) and k_kick_once
// (the same for the phase entry points, in one kernel with what follows) evaluate it in FP64, one warp
// per body. k_kick_precise (precise_div = 1: IEEE square root and division; any size) evaluates every
// unordered pair once in FP64. They leave partial sums per body tile in a fixed layout that the
// finalisation sums in a fixed order, so results are bitwise reproducible.
#include "fxforce.cuh"
#include "kick_fx.cuh"

namespace genga {

// ---------------------------------------------------------------------------------------------
// Critical radii, precheck thresholds and the kick-reuse test (once per full step)
// ---------------------------------------------------------------------------------------------
__global__ void k_rcrit(Sim S, DevParams P, double tau_abs, int check_reuse) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (check_reuse && i == 0) atomicAdd((unsigned long long *)&S.counters[C_STEPS], 1ULL);
  if (i >= S.npad) return;
  const int np = S.npad;
  if (!S.alive[i]) {
    S.rc[i] = 0.0; S.A[i] = 0.0; S.T[i] = 0ULL; S.rcsq[i] = 0ULL;
    return;
  }
  double x = S.x[i], y = S.x[np + i], z = S.x[2 * np + i];
  double vx = S.v[i], vy = S.v[np + i], vz = S.v[2 * np + i];
  double r2 = fma(z, z, fma(y, y, x * x));
  double ir = rsqrt_refined(r2);
  double v2 = fma(vz, vz, fma(vy, vy, vx * vx));
  double inva = fma(2.0, ir, -v2 * P.inv_mu);  // 1/a = 2/r - v^2/(G m0)
  double asemi = is_neg_or_zero(inva) ? r2 * ir : rcp_refined(inva);
  double rh = asemi * S.hill[i];               // Hill radius a (m/(3 m0))^(1/3)
  double vabs = (dbits(v2) == 0ULL) ? 0.0 : v2 * rsqrt_refined(v2);
  double rc = pmax(P.n1 * rh, (P.n2 * tau_abs) * vabs);
  if (check_reuse) {
    // reusing the last kick for non-candidate pairs is exact while rc_new <= pc * rc_old
    double lim = P.pc * S.rc[i];
    if (dbits(rc) > dbits(lim)) {
      S.flags[0] = 1;
      atomicOr(S.status, ST_REUSE_FULLKICK);
      atomicAdd((unsigned long long *)&S.counters[C_FULLKICK], 1ULL);
    }
  }
  S.rc[i] = rc;
  double t = __dmul_rn(P.pc, rc);
  S.T[i] = dbits(__dmul_rn(t, t));
  S.rcsq[i] = dbits(__dmul_rn(rc, rc));
  S.A[i] = (dbits(rc) == 0ULL) ? 0.0 : rcp_refined(0.9 * rc);
}

// ---------------------------------------------------------------------------------------------
// Pair kernel with IEEE square root and division (precise_div = 1). FULL: all pairs with inline
// changeover weights (used only when the critical radii grew too much for reuse); otherwise far
// pairs only, candidates recorded in the bitmap. Every unordered pair once (Newton's third law) on
// 32x32 body tiles: each lane holds one body i of tile I, the 32 bodies of tile J rotate through the
// lanes by warp shuffles, and the j-side sums rotate with them. A work item is half of a tile pair
// (16 ring steps); its partial sums go to a slot per (tile, partner tile, half).
// ---------------------------------------------------------------------------------------------
template <bool FULL>
__global__ void __launch_bounds__(128) k_kick_precise(Sim S, DevParams P, int force) {
  if (FULL && !force && S.flags[0] == 0) return;
  // a full opening kick after a new state also records the precheck candidates (flag 3)
  const bool record = FULL && !force && S.flags[3] != 0;
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int np = S.npad, nt = S.nt, W = S.W;
  const double *__restrict__ X = S.x;
  if ((!FULL || force) && warp < nt) {  // per-tile momentum before the closing kick (second Sun drift)
    int i = warp * 32 + lane;
    double mi = S.m[i];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      double p = warp_sum(mi * S.v[c * np + i]);
      if (lane < FIN_PER_TILE) S.pkick[(warp * FIN_PER_TILE + lane) * 3 + c] = lane == 0 ? p : 0.0;
    }
  }
  if (warp >= S.nwarps) return;
  const long it0 = (long)warp * S.nitems / S.nwarps, it1 = (long)(warp + 1) * S.nitems / S.nwarps;
  int curI = -1;
  double xi = 0, yi = 0, zi = 0, gmi = 0, Ai = 0;
  u64 Ti = 0, Qi = 0;
  for (long it = it0; it < it1; ++it) {
    const int code = S.items[it];
    const int I = code & 1023, J = (code >> 10) & 1023, h = code >> 20;
    const int i = I * 32 + lane;
    if (I != curI) {
      curI = I;
      xi = X[i]; yi = X[np + i]; zi = X[2 * np + i];
      gmi = S.gm[i]; Ti = S.T[i];
      if (FULL) { Qi = S.rcsq[i]; Ai = S.A[i]; }
    }
    const bool diag = (I == J);
    const int jl0 = diag ? lane : ((lane + 16 * h) & 31);
    const int j0 = J * 32 + jl0;
    double xj = X[j0], yj = X[np + j0], zj = X[2 * np + j0], gmj = S.gm[j0];
    u64 Tj = S.T[j0], Qj = 0;
    double Aj = 0;
    if (FULL) { Qj = S.rcsq[j0]; Aj = S.A[j0]; }
    double aix = 0, aiy = 0, aiz = 0, ajx = 0, ajy = 0, ajz = 0;
    const int src = (lane + 1) & 31;
#pragma unroll 4
    for (int s = 0; s < 16; ++s) {
      if (diag) {  // diagonal tile: rotate first, pair lane with lane + s + 1
        xj = __shfl_sync(0xffffffffu, xj, src); yj = __shfl_sync(0xffffffffu, yj, src);
        zj = __shfl_sync(0xffffffffu, zj, src); gmj = __shfl_sync(0xffffffffu, gmj, src);
        Tj = __shfl_sync(0xffffffffu, Tj, src);
        ajx = __shfl_sync(0xffffffffu, ajx, src); ajy = __shfl_sync(0xffffffffu, ajy, src);
        ajz = __shfl_sync(0xffffffffu, ajz, src);
        if (FULL) { Qj = __shfl_sync(0xffffffffu, Qj, src); Aj = __shfl_sync(0xffffffffu, Aj, src); }
      }
      const int jl = diag ? ((lane + s + 1) & 31) : ((lane + 16 * h + s) & 31);
      const bool act = !diag || s < 15 || lane < 16;
      const double dx = xj - xi, dy = yj - yi, dz = zj - zi;
      const double r2 = __fma_rn(dz, dz, __fma_rn(dy, dy, __dmul_rn(dx, dx)));
      const double w3 = 1.0 / (r2 * sqrt(r2));
      double gj = act ? gmj : 0.0, gi = act ? gmi : 0.0;
      const u64 rb = dbits(r2);
      if (FULL) {
        if (rb < umax64(Qi, Qj)) {  // inside the changeover zone: weight K (rare)
          double r = r2 * rsqrt_refined(r2), wB, wA;
          changeover_w(r, pmin(Ai, Aj), P.kmode, wB, wA);
          gj *= wB; gi *= wB;
        }
      }
      if ((!FULL || record) && act && rb < umax64(Ti, Tj)) {  // precheck candidate
        if (!FULL) { gj = 0.0; gi = 0.0; }  // handled by the near pass
        const int j = J * 32 + jl;
        atomicOr(&S.cbm[(size_t)i * W + (j >> 5)], 1u << (j & 31));
        atomicOr(&S.cbm[(size_t)j * W + (i >> 5)], 1u << (i & 31));
        atomicOr(&S.rowany[i >> 5], 1u << (i & 31));
        atomicOr(&S.rowany[j >> 5], 1u << (j & 31));
        const int ki = atomicAdd(&S.ccnt[i], 1), kj = atomicAdd(&S.ccnt[j], 1);
        if (ki < CCAP) S.clist[i * CCAP + ki] = j;
        if (kj < CCAP) S.clist[j * CCAP + kj] = i;
        atomicAdd((unsigned long long *)&S.counters[C_CAND], 1ULL);
      }
      const double fi = gj * w3, fj = gi * w3;
      aix = fma(fi, dx, aix); aiy = fma(fi, dy, aiy); aiz = fma(fi, dz, aiz);
      ajx = fma(-fj, dx, ajx); ajy = fma(-fj, dy, ajy); ajz = fma(-fj, dz, ajz);
      if (!diag && s < 15) {
        xj = __shfl_sync(0xffffffffu, xj, src); yj = __shfl_sync(0xffffffffu, yj, src);
        zj = __shfl_sync(0xffffffffu, zj, src); gmj = __shfl_sync(0xffffffffu, gmj, src);
        Tj = __shfl_sync(0xffffffffu, Tj, src);
        ajx = __shfl_sync(0xffffffffu, ajx, src); ajy = __shfl_sync(0xffffffffu, ajy, src);
        ajz = __shfl_sync(0xffffffffu, ajz, src);
        if (FULL) { Qj = __shfl_sync(0xffffffffu, Qj, src); Aj = __shfl_sync(0xffffffffu, Aj, src); }
      }
    }
    // return the j accumulators to the lane that owns body J*32 + lane
    const int home = diag ? ((lane + 16) & 31) : ((lane - 16 * h - 15) & 31);
    ajx = __shfl_sync(0xffffffffu, ajx, home);
    ajy = __shfl_sync(0xffffffffu, ajy, home);
    ajz = __shfl_sync(0xffffffffu, ajz, home);
    double *pi = S.part + ((size_t)(I * nt + J) * 2 + h) * 96 + lane;
    if (diag) {
      pi[0] = aix + ajx; pi[32] = aiy + ajy; pi[64] = aiz + ajz;
      pi[96] = 0.0; pi[128] = 0.0; pi[160] = 0.0;  // half 1 of a diagonal tile is empty
    } else {
      pi[0] = aix; pi[32] = aiy; pi[64] = aiz;
      double *pj = S.part + ((size_t)(J * nt + I) * 2 + h) * 96 + lane;
      pj[0] = ajx; pj[32] = ajy; pj[64] = ajz;
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Fixed-point pair kernel (kick_fx.cuh): FULL and the candidates as in k_kick_precise; every body records
// its own row of the bitmap. The sums of a (tile, chunk) go to its slot.
// ---------------------------------------------------------------------------------------------
// The pair (i, j) in FP64: records a candidate, returns the pull's factor (0: nothing to add here).
template <bool FULL>
__device__ __forceinline__ double kx_near(const Sim &S, const DevParams &P, int i, int j, bool record, double &dx,
                                          double &dy, double &dz) {
  const int np = S.npad;
  if (j == i || !S.alive[j]) return 0.0;
  dx = S.x[j] - S.x[i]; dy = S.x[np + j] - S.x[np + i]; dz = S.x[2 * np + j] - S.x[2 * np + i];
  const double r2 = __fma_rn(dz, dz, __fma_rn(dy, dy, __dmul_rn(dx, dx)));
  const u64 rb = dbits(r2);
  const bool cand = rb < umax64(S.T[i], S.T[j]);
  if (record && cand) {
    const int ki = atomicAdd(&S.ccnt[i], 1);
    atomicOr(&S.cbm[(size_t)i * S.W + (j >> 5)], 1u << (j & 31));
    atomicOr(&S.rowany[i >> 5], 1u << (i & 31));
    if (ki < CCAP) S.clist[i * CCAP + ki] = j;
    if (i < j) atomicAdd((unsigned long long *)&S.counters[C_CAND], 1ULL);
  }
  if (!FULL && cand) return 0.0;  // handled by the near pass
  double g = S.gm[j] * rcube_refined(r2);
  if (FULL && rb < umax64(S.rcsq[i], S.rcsq[j])) {  // inside the changeover zone: weight K
    double wB, wA;
    changeover_w(r2 * rsqrt_refined(r2), pmin(S.A[i], S.A[j]), P.kmode, wB, wA);
    g *= wB;
  }
  return g;
}

template <bool FULL, int TW>
__global__ void __launch_bounds__(32 * KX_WARPS, KX_CTAS) k_kick_fx(Sim S, DevParams P, int force) {
  wait_previous();
  if (FULL && !force && S.flags[0] == 0) return;
  const bool record = FULL ? (!force && S.flags[3] != 0) : true;
  const int lane = threadIdx.x & 31, np = S.npad, C = S.kch, nt = S.nt;
  const int gwarp = blockIdx.x * KX_WARPS + (threadIdx.x >> 5);
  if ((!FULL || force) && gwarp < nt) {  // per-tile momentum before the closing kick (second Sun drift)
    const int i = gwarp * 32 + lane;
    const double mi = S.m[i];
    const double p = segment_sum3<32>(mi * S.v[i], mi * S.v[np + i], mi * S.v[2 * np + i]);
    // the tile's total in the first of its slots (k_kick_small fills them all)
    if ((lane & 7) < FIN_PER_TILE && lane < 24)
      S.pkick[(gwarp * FIN_PER_TILE + (lane & 7)) * 3 + (lane >> 3)] = (lane & 7) == 0 ? p : 0.0;
  }
  const int tgroups = (nt + TW - 1) / TW;
  int I, c0;
  bool ali;
  double ax, ay, az;
  const bool on = kx_block<TW, true>(
      S.x, np, S.gm, S.alive, S.T, 0, np, nt, C, S.kchunk, blockIdx.x % tgroups, blockIdx.x / tgroups,
      [&](int i, int j, double &dx, double &dy, double &dz) { return kx_near<FULL>(S, P, i, j, record, dx, dy, dz); }, I, c0,
      ali, ax, ay, az);
  if (!on) return;
  double *p = S.part + ((size_t)I * C + c0) * 96 + lane;
  p[0] = ali ? ax : 0.0; p[32] = ali ? ay : 0.0; p[64] = ali ? az : 0.0;
}

// The fixed-point kernel's split of a tile's partners: chunks per tile, partners per chunk. About 8
// KX_CTAS warps per SM, at least 8 partners a chunk (below that the set-up of a warp outweighs its
// loop), at most 64 (the bit masks). Up to 1024 bodies at most 2048 chunks in all (the partial-sum
// slots of the static scratch). systems: equal systems summed by one launch.
void kick_split(int npad, int sms, int *chunks, int *chunk, int systems) {
  const int nt = npad / 32, lo = (npad + fx::FX_CHUNK - 1) / fx::FX_CHUNK, hi = npad / KX_SMALL;
  int C = (int)((long)KX_WARPS * KX_CTAS * sms / ((long)nt * systems));
  if (nt <= 32 && C > 2048 / nt) C = 2048 / nt;
  if (C > hi || nt < 8) C = hi;  // chunks of KX_SMALL
  if (C < lo) C = lo;
  *chunk = (npad + C - 1) / C;
  *chunks = (npad + *chunk - 1) / *chunk;
}

template <bool FULL>
static void launch_kick_fx(const Sim &S, const DevParams &P, int force, cudaStream_t st, bool after) {
  const int tw = S.nt >= 8 ? 8 : (S.nt >= 4 ? 4 : 2), cw = KX_WARPS / tw;  // at least three tiles
  const int grid = ((S.nt + tw - 1) / tw) * ((S.kch + cw - 1) / cw);
  auto *kernel = tw == 8 ? k_kick_fx<FULL, 8> : (tw == 4 ? k_kick_fx<FULL, 4> : k_kick_fx<FULL, 2>);
  if (after) launch_after(kernel, grid, 32 * KX_WARPS, st, S, P, force);
  else kernel<<<grid, 32 * KX_WARPS, 0, st>>>(S, P, force);
}

// r^-3 from r^2, on the integer pipes where r^2 is normal: rounded once, where the refined inverse root
// cubed carries four roundings.
__device__ __forceinline__ double inverse_cube(double r2) {
  const int ex = (int)(dbits(r2) >> 52);
  double y3, y5;
  if (ex > 0 && ex < 0x7ff) fx::inverse_powers(r2, y3, y5);
  else y3 = rcube_refined(r2);
  return y3;
}

// The near-pair pull of partner j on body i, per unit separation, with the current critical radii
// (the changeover weight as in the kick). ONCE: r^-3 rounded once, for the kick whose accelerations are
// the result (1000 bodies: error 2.7-3.2e-16 against 3.0-3.7e-16); a step keeps the shorter chain.
template <bool ONCE>
__device__ __forceinline__ double near_factor(const Sim &S, const DevParams &P, u64 Qi, double Ai, int j, double r2) {
  const double yr = rsqrt_refined(r2);
  double wB = 1.0, wA;
  if (dbits(r2) < umax64(Qi, S.rcsq[j])) changeover_w(r2 * yr, pmin(Ai, S.A[j]), P.kmode, wB, wA);
  return S.gm[j] * wB * (ONCE ? inverse_cube(r2) : yr * yr * yr);
}

// ---------------------------------------------------------------------------------------------
// Finalisation, LPB lanes per body, FIN_BODIES bodies per CTA:
//   CLOSE: a = sum of the pair partials (far field, stored for reuse) + near pairs;
//          v += h1 a (+ h2 a for the next substep's opening kick). The second Sun drift of the
//          substep (which the kick does not see: it shifts every body alike) is applied by the
//          next drift kernel, or by k_hc after the last substep, from the momentum the kick
//          kernel recorded before the velocities changed.
//   OPEN : first kick of a full step with the new critical radii: a = stored far field + near
//          pairs recomputed (KickA; KickB when there are none), or the full recompute's partials.
//   INIT : the very first kick: store the far field (and a = far + near into aout [3][ald] if given).
// The near partners are read from the body's row of the candidate bitmap, in ascending order, and
// evaluated one per lane, once for all three components; the sums have a fixed order. Also writes the
// CTA's momentum of the new velocities for the next Sun drift.
//
// Bound by latency (launch, the chain row -> positions -> FP64 terms -> sums) and by FP64 issue, 64-76
// cycles a warp instruction whatever its active lanes: LPB is the most (8, 16 or 32) that leaves one
// warp on each sub-partition. Measured against one CTA per tile and component, which gathered and
// ranked the candidate lists of 32 bodies and left rows of more than 32 partners to one lane each:
// 1024 bodies with wide radii 58 -> 10 us (opening 39 -> 8), 32 bodies 10.0 -> 7.4 us; against one warp
// per body at every size, 4 steps of 2048 bodies 1.69 -> 1.62 ms (with the cluster kernel's change).
// ---------------------------------------------------------------------------------------------
constexpr int FIN_BODIES = 32 / FIN_PER_TILE;

template <int MODE, int LPB>
__global__ void __launch_bounds__(FIN_BODIES * LPB) k_fin(Sim S, DevParams P, double h1, double h2, double *aout, int ald,
                                                          int nslot) {
  constexpr bool ALL = MODE == FIN_CLOSE_ALL;  // the pair kernel weighed every pair: no near pass
  __shared__ unsigned short s_j[FIN_BODIES][NMAX];  // near partners
  __shared__ double s_pm[3][FIN_BODIES];
  wait_previous();
  const int tid = threadIdx.x, bi = tid / LPB, sl = tid % LPB, np = S.npad;
  const int i = blockIdx.x * FIN_BODIES + bi;
  // this lane's component of the sums, held by the first lane of a quarter
  const int c = sl / (LPB / 4) < 2 ? sl / (LPB / 4) : 2;
  const bool own = sl % (LPB / 4) == 0 && sl < 3 * (LPB / 4);
  const bool use_part = (MODE != FIN_OPEN) || (S.flags[0] != 0);
  const bool near = !ALL && !(MODE == FIN_OPEN && use_part) && ((S.rowany[i >> 5] >> (i & 31)) & 1u);
  // the loads of the final update first, so that their latency passes under the sums
  const double a_far = !use_part ? S.afar[c * np + i] : 0.0;
  const double v_old = MODE != FIN_INIT ? S.v[c * np + i] : 0.0;
  const double m_i = S.m[i];
  const bool alive = S.alive[i] != 0;
  double a = a_far;
  if (use_part) {
    double f[3] = {0.0, 0.0, 0.0};
    const double *p = S.part + (size_t)(i >> 5) * nslot * 96 + (i & 31);
#pragma unroll 4
    for (int s = sl; s < nslot; s += LPB)
      for (int k = 0; k < 3; ++k) f[k] += p[(size_t)s * 96 + 32 * k];
    a = segment_sum3<LPB>(f[0], f[1], f[2]);
  }
  if (MODE != FIN_OPEN && !ALL && own) S.afar[c * np + i] = a;
  if (__any_sync(0xffffffffu, near)) {
    const int wl = (S.W + LPB - 1) / LPB, w0 = sl * wl, w1 = near ? (w0 + wl < S.W ? w0 + wl : S.W) : w0;
    const unsigned *row = S.cbm + (size_t)i * S.W;
    int mine = 0;
    for (int w = w0; w < w1; ++w) mine += __popc(row[w]);
    int incl = mine;
#pragma unroll
    for (int o = 1; o < LPB; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, o, LPB);
      if (sl >= o) incl += t;
    }
    const int cnt = __shfl_sync(0xffffffffu, incl, LPB - 1, LPB);
    if (mine) {
      int k = incl - mine;
      for (int w = w0; w < w1; ++w)
        for (unsigned bits = row[w]; bits; bits &= bits - 1) s_j[bi][k++] = (unsigned short)(w * 32 + __ffs(bits) - 1);
    }
    __syncwarp();
    const double xi = S.x[i], yi = S.x[np + i], zi = S.x[2 * np + i], Ai = S.A[i];
    const u64 Qi = S.rcsq[i];
    double nx = 0.0, ny = 0.0, nz = 0.0;
    for (int k = sl; k < cnt; k += LPB) {
      const int j = s_j[bi][k];
      const double dx = S.x[j] - xi, dy = S.x[np + j] - yi, dz = S.x[2 * np + j] - zi;
      const double f = near_factor<MODE == FIN_INIT>(S, P, Qi, Ai, j, r2_exact(dx, dy, dz));
      nx = fma(f, dx, nx); ny = fma(f, dy, ny); nz = fma(f, dz, nz);
    }
    a += segment_sum3<LPB>(nx, ny, nz);
  }
  if (aout && i < S.n && own) aout[(size_t)c * ald + i] = a;
  if (MODE == FIN_INIT) return;
  if (own) {
    double v = v_old;
    if (alive) {
      v = fma(h1, a, v);
      if (h2 != 0.0) v = fma(h2, a, v);
      S.v[c * np + i] = v;
    }
    s_pm[c][bi] = m_i * v;
  }
  __syncthreads();
  if (tid >= 32) return;
  double pm = tid < 3 * FIN_BODIES ? s_pm[tid / FIN_BODIES][tid % FIN_BODIES] : 0.0;
#pragma unroll
  for (int o = FIN_BODIES / 2; o > 0; o >>= 1) pm += __shfl_xor_sync(0xffffffffu, pm, o);
  if (tid < 3 * FIN_BODIES && tid % FIN_BODIES == 0) S.pfin[blockIdx.x * 3 + tid / FIN_BODIES] = pm;
}

// ---------------------------------------------------------------------------------------------
// The kick of few bodies: one warp per body, a partner a lane, every ordered pair in FP64, so that no
// sum has to wait for other warps. Bound by latency: at 32 bodies the fixed-point kernel's set-up (grid,
// chunks, bound pass) is most of its 10 us. Measured against it: 10 steps of 32 bodies 613 -> 570 us, 6
// of 64 bodies 399 -> 379; a kick of 64 bodies without allocation, here in one kernel, 20.0 -> 17-19 us
// (bound by submission). Beyond, the FP64 pairs cost more than the set-up (6 steps of 100 bodies 433 ->
// 440 us, of 200 bodies 512 -> 548).
// ---------------------------------------------------------------------------------------------
constexpr int KS_MAX = 64;

// The far sum of body i (all of it, weighted, if FULL) and, if NEAR, the weighted near sum, on the lanes
// of segment_sum3; records the candidates (the rows are clear).
template <bool FULL, bool NEAR>
__device__ __forceinline__ void small_sums(const Sim &S, const DevParams &P, int i, bool record, double &far, double &near) {
  const int lane = threadIdx.x & 31, np = S.npad;
  double fx = 0.0, fy = 0.0, fz = 0.0, nx = 0.0, ny = 0.0, nz = 0.0;
  if (S.alive[i]) {  // uniform within the warp, as the loop and its votes
    const double xi = S.x[i], yi = S.x[np + i], zi = S.x[2 * np + i], Ai = S.A[i];
    const u64 Ti = S.T[i], Qi = S.rcsq[i];
    int cnt = 0, pairs = 0;
    for (int w = 0; w < S.W; ++w) {
      const int j = w * 32 + lane;
      const bool act = j != i && S.alive[j];
      const double dx = S.x[j] - xi, dy = S.x[np + j] - yi, dz = S.x[2 * np + j] - zi;
      const double r2 = r2_exact(dx, dy, dz);
      const u64 rb = dbits(r2);
      const bool cand = act && rb < umax64(Ti, S.T[j]);
      if (act) {
        double g = S.gm[j] * (NEAR ? inverse_cube(r2) : rcube_refined(r2));
        if ((FULL || (NEAR && cand)) && rb < umax64(Qi, S.rcsq[j])) {
          double wB, wA;
          changeover_w(r2 * rsqrt_refined(r2), pmin(Ai, S.A[j]), P.kmode, wB, wA);
          g *= wB;
        }
        if (FULL || !cand) { fx = fma(g, dx, fx); fy = fma(g, dy, fy); fz = fma(g, dz, fz); }
        else if (NEAR) { nx = fma(g, dx, nx); ny = fma(g, dy, ny); nz = fma(g, dz, nz); }
      }
      const unsigned m = record ? __ballot_sync(0xffffffffu, cand) : 0u;
      if (m) {
        const int k = cnt + __popc(m & ((1u << lane) - 1u));
        if (cand && k < CCAP) S.clist[i * CCAP + k] = j;
        if (lane == 0) S.cbm[(size_t)i * S.W + w] = m;
        cnt += __popc(m);
        pairs += __popc(__ballot_sync(0xffffffffu, cand && j > i));
      }
    }
    if (lane == 0 && cnt) {
      S.ccnt[i] = cnt;
      atomicOr(&S.rowany[i >> 5], 1u << (i & 31));
      if (pairs) atomicAdd((unsigned long long *)&S.counters[C_CAND], (unsigned long long)pairs);
    }
  }
  far = segment_sum3<32>(fx, fy, fz);
  if (NEAR) near = segment_sum3<32>(nx, ny, nz);
}

// The pair kernel of a step (the arguments and the momentum as k_kick_fx); k_fin reads one sum a body.
template <bool FULL>
__global__ void __launch_bounds__(32 * FIN_BODIES) k_kick_small(Sim S, DevParams P, int force) {
  wait_previous();
  if (FULL && !force && S.flags[0] == 0) return;
  __shared__ double s_pm[3][FIN_BODIES];
  const int wi = threadIdx.x >> 5, lane = threadIdx.x & 31, np = S.npad, i = blockIdx.x * FIN_BODIES + wi;
  const int c = lane >> 3;  // lanes 0, 8, 16 hold the components of the sums
  const bool own = (lane & 7) == 0 && c < 3, moment = !FULL || force;
  if (moment && own) s_pm[c][wi] = S.m[i] * S.v[c * np + i];
  double far, near;
  small_sums<FULL, false>(S, P, i, FULL ? (!force && S.flags[3] != 0) : true, far, near);
  if (own) S.part[(size_t)(i >> 5) * 96 + c * 32 + (i & 31)] = far;
  if (!moment) return;  // uniform
  __syncthreads();
  if (wi != 0) return;
  double pm = c < 3 ? s_pm[c][lane & 7] : 0.0;
#pragma unroll
  for (int o = FIN_BODIES / 2; o > 0; o >>= 1) pm += __shfl_xor_sync(0xffffffffu, pm, o);
  if (own) S.pkick[blockIdx.x * 3 + c] = pm;
}

// The whole kick of the phase entry points: accelerations [3][ald] of the S.n bodies and the candidates.
__global__ void __launch_bounds__(32 * FIN_BODIES) k_kick_once(Sim S, DevParams P, double *aout, int ald) {
  wait_previous();
  const int lane = threadIdx.x & 31, i = blockIdx.x * FIN_BODIES + (threadIdx.x >> 5), c = lane >> 3;
  double far, near;
  small_sums<false, true>(S, P, i, true, far, near);
  if ((lane & 7) == 0 && c < 3 && i < S.n) aout[(size_t)c * ald + i] = far + near;
}

static bool kick_is_small(const Sim &S, bool precise) { return S.npad <= KS_MAX && !precise; }

// ---------------------------------------------------------------------------------------------
void launch_rcrit(const Sim &S, const DevParams &P, double tau_abs, int check_reuse, cudaStream_t st) {
  k_rcrit<<<(S.npad + 127) / 128, 128, 0, st>>>(S, P, tau_abs, check_reuse);
}

void launch_kick(const Sim &S, const DevParams &P, bool full, bool precise, cudaStream_t st, bool force, bool after) {
  const int f = force ? 1 : 0;
  if (precise) {
    const int grid = ((S.nwarps > S.nt ? S.nwarps : S.nt) * 32 + 127) / 128;
    if (full) k_kick_precise<true><<<grid, 128, 0, st>>>(S, P, f);
    else k_kick_precise<false><<<grid, 128, 0, st>>>(S, P, 0);
  } else if (kick_is_small(S, false)) {
    auto *kernel = full ? k_kick_small<true> : k_kick_small<false>;
    if (after) launch_after(kernel, S.nt * FIN_PER_TILE, 32 * FIN_BODIES, st, S, P, full ? f : 0);
    else kernel<<<S.nt * FIN_PER_TILE, 32 * FIN_BODIES, 0, st>>>(S, P, full ? f : 0);
  } else {
    if (full) launch_kick_fx<true>(S, P, f, st, after);
    else launch_kick_fx<false>(S, P, 0, st, after);
  }
}

// Lanes per body: about 600 sub-partitions, one warp each.
template <int MODE>
static void fin_lanes(const Sim &S, const DevParams &P, double h1, double h2, double *aout, int ald, int nslot,
                      cudaStream_t st, bool after) {
  const int lpb = S.npad > 1216 ? 8 : (S.npad > 608 ? 16 : 32), grid = S.nt * FIN_PER_TILE;
  auto *kernel = lpb == 8 ? k_fin<MODE, 8> : (lpb == 16 ? k_fin<MODE, 16> : k_fin<MODE, 32>);
  if (after) launch_after(kernel, grid, lpb * FIN_BODIES, st, S, P, h1, h2, aout, ald, nslot);
  else kernel<<<grid, lpb * FIN_BODIES, 0, st>>>(S, P, h1, h2, aout, ald, nslot);
}

void launch_fin(const Sim &S, const DevParams &P, FinMode mode, bool precise, double h1, double h2, double *aout,
                int ald, cudaStream_t st, bool after) {
  // partial-sum slots per tile of the pair kernel used
  const int nslot = precise ? 2 * S.nt : (kick_is_small(S, false) ? 1 : S.kch);
  if (mode == FIN_CLOSE) fin_lanes<FIN_CLOSE>(S, P, h1, h2, aout, ald, nslot, st, after);
  else if (mode == FIN_CLOSE_ALL) fin_lanes<FIN_CLOSE_ALL>(S, P, h1, h2, aout, ald, nslot, st, after);
  else if (mode == FIN_OPEN) fin_lanes<FIN_OPEN>(S, P, h1, h2, aout, ald, nslot, st, after);
  else fin_lanes<FIN_INIT>(S, P, h1, h2, aout, ald, nslot, st, after);
}

void launch_kick_init(const Sim &S, const DevParams &P, bool precise, double *aout, int ald, cudaStream_t st, bool after) {
  if (kick_is_small(S, precise)) {
    if (after) launch_after(k_kick_once, S.nt * FIN_PER_TILE, 32 * FIN_BODIES, st, S, P, aout, ald);
    else k_kick_once<<<S.nt * FIN_PER_TILE, 32 * FIN_BODIES, 0, st>>>(S, P, aout, ald);
    return;
  }
  launch_kick(S, P, false, precise, st, false, after);
  launch_fin(S, P, FIN_INIT, precise, 0.0, 0.0, aout, ald, st, true);
}

// Second Sun drift after the last substep: x += hcm * P, P the momentum before the closing kick.
__global__ void k_hc(Sim S, double hcm) {
  wait_previous();
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  double p[3] = {0.0, 0.0, 0.0};
  for (int t = lane; t < FIN_PER_TILE * S.nt; t += 32)
    for (int c = 0; c < 3; ++c) p[c] += S.pkick[t * 3 + c];
  const double ps = segment_sum3<32>(p[0], p[1], p[2]);
#pragma unroll
  for (int c = 0; c < 3; ++c) p[c] = __shfl_sync(0xffffffffu, ps, 8 * c);
  if (i >= S.npad || !S.alive[i]) return;
#pragma unroll
  for (int c = 0; c < 3; ++c) S.x[c * S.npad + i] = fma(hcm, p[c], S.x[c * S.npad + i]);
}

void launch_hc(const Sim &S, double hcm, cudaStream_t st) {
  launch_after(k_hc, (S.npad + 63) / 64, 64, st, S, hcm);
}

}  // namespace genga
