// bs_core.cuh -- the Bulirsch-Stoer of one encounter group by one CTA (Sect. 3.2), shared by the
// kernels of bs.cu and the persistent batched kernel (batch_persist.cu). Every translation unit
// that includes it holds its own copy of the Neville factors (bs_core_set_factors fills it).
#pragma once
#include "fxforce.cuh"
#include "genga_launch.h"

namespace genga {

// 1/((L/(L-j))^2 - 1) for the Neville extrapolation in h^2 with n_k = 2k
static __constant__ double c_facinv[BS_LEVELS + 1][BS_LEVELS];


// Fills this translation unit's c_facinv (host; once per device, before any capture).
static inline void bs_core_set_factors() {
  double h[BS_LEVELS + 1][BS_LEVELS] = {};
  for (int L = 2; L <= BS_LEVELS; ++L)
    for (int j = 1; j < L; ++j) {
      const double ratio = (double)L / (double)(L - j);
      h[L][j] = 1.0 / (ratio * ratio - 1.0);
    }
  cudaMemcpyToSymbol(c_facinv, h, sizeof(h));
}

// A group's state in shared memory, for groups of up to GM members.
template <int GM>
struct BsSharedT {
  int idx[GM], alive[GM];
  double gm[GM], m[GM], R[GM], A[GM];
  u64 rcsq[GM];
  double y[GM][6], yn[GM][6];
  double pos[2][BS_LEVELS][GM][3];
  double tab[BS_LEVELS][GM][6];
  unsigned bad;                         // not converged: bit r - 1 level r of the attempt at H, 7 + r of that at H/2
  unsigned char cont[GM * (GM - 1) / 2];
  double H, rem, U;
  int accept, next;
  int nseq, seq_base;          // recorded accepted substeps (adjoint engine only)
  long long y_base;
  double seqH[BS_SEQCAP];
  unsigned char seqk[BS_SEQCAP];
};
using BsShared = BsSharedT<BS_GMAX>;

// What a term of member q and partner p (p == q: the central mass) takes besides their positions; the
// thread's first one is formed once an attempt.
struct BsTerm {
  fx::Num gm, A;  // G m and 1/(0.9 rc) for the fixed-point factor
  u64 cut;        // r^2 below it: inside the critical radius
  int sign;       // the sign bit of G m
};
template <class SH>
__device__ __forceinline__ BsTerm bs_term(const SH &sh, double Gm0, int g, int q, int p) {
  BsTerm t;
  p = p < g ? p : q;
  const bool cen = p == q;
  const double gm = cen ? Gm0 : sh.gm[p];
  t.gm = fx::num(gm);
  t.A = fx::num(pmin(sh.A[q], sh.A[p]));
  t.cut = !cen && sh.alive[p] ? umax64(sh.rcsq[q], sh.rcsq[p]) : 0ULL;
  t.sign = __double2hiint(gm) & 0x80000000;
  return t;
}

// Acceleration of member q at positions pos by the slot's ttps threads (4, 2 or 1): thread tsub sums
// the terms p = tsub, tsub + ttps, ... (p == q: the central mass; any other p the (1 - K)-weighted pull
// of partner p, H_A, Eq. Ha) and is given the components it owns: thread c of 4 component c, threads 0
// and 1 of 2 the components 0, 1 and 2, one thread all three. Every lane runs the same straight-line
// code (the central mass is a partner at the origin with G m0 and weight 1; a partner outside rc gets
// weight 0): lanes of one warp that took different branches would each pay for both, and an FP64 warp
// instruction costs its sub-partition 64 cycles whatever its active lanes. The threads exchange what
// they do not own, so a slot of 4 issues 3 additions for the sum and 4 instructions for its chain
// step, where every thread holding every component took 6 and 6.
template <class SH>
__device__ __forceinline__ void bs_accel(const SH &sh, const DevParams &P, const BsTerm &t0, double Gm0, int g, int q, int tsub,
                                         int ttps, const double (*pos)[3], bool q_alive, double (&acc)[3]) {
  double a0 = 0.0, a1 = 0.0, a2 = 0.0;
  if (q_alive) {
    const double xq = pos[q][0], yq = pos[q][1], zq = pos[q][2];
    for (int p = tsub; p < g; p += ttps) {
      const bool cen = p == q;
      const double dx = (cen ? 0.0 : pos[p][0]) - xq, dy = (cen ? 0.0 : pos[p][1]) - yq,
                   dz = (cen ? 0.0 : pos[p][2]) - zq;
      const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
      BsTerm t = t0;
      if (p != tsub) t = bs_term(sh, Gm0, g, q, p);
      const bool inside = dbits(r2) < t.cut;
      double f = 0.0;
      if (cen || inside) {
        if (bs_factor_is_fixed(r2, P.kmode)) {
          f = fx::pull_factor(r2, t.gm, t.A, cen, inside);
          f = __hiloint2double(__double2hiint(f) | t.sign, __double2loint(f));
        } else {
          f = bs_factor_fp64(r2, cen ? Gm0 : sh.gm[p], pmin(sh.A[q], sh.A[p]), cen, P.kmode);
        }
      }
      a0 = fma(f, dx, a0); a1 = fma(f, dy, a1); a2 = fma(f, dz, a2);
    }
  }
  acc[0] = a0; acc[1] = a1; acc[2] = a2;
  if (ttps == 4) {
    const bool hi = (tsub & 2) != 0, odd = (tsub & 1) != 0;
    const double r0 = __shfl_xor_sync(0xffffffffu, hi ? a0 : a2, 2), r1 = __shfl_xor_sync(0xffffffffu, a1, 2);
    // threads 0, 1 now sum components 0 and 1 of the pair (tsub, tsub + 2), threads 2, 3 component 2
    const double s0 = (hi ? a2 : a0) + r0, s1 = a1 + r1;
    const double r = __shfl_xor_sync(0xffffffffu, hi || odd ? s0 : s1, 1);
    acc[0] = (hi || !odd ? s0 : s1) + r;
  } else if (ttps == 2) {
    const bool odd = (tsub & 1) != 0;
    const double r0 = __shfl_xor_sync(0xffffffffu, odd ? a0 : a2, 1), r1 = __shfl_xor_sync(0xffffffffu, a1, 1);
    acc[0] = (odd ? a2 : a0) + r0;
    acc[1] = a1 + r1;
  }
}

// Bulirsch-Stoer of one group (members S.gmem[g0 .. g0 + g - 1], ascending; central mass m0) over
// tau by the NT threads of the calling CTA: every level's modified-midpoint chain at once, each
// level's tableau row built and tested as soon as the level completes, the first converged level
// accepted (Sect. 3.2); contacts and mergers after every accepted substep; the result written back
// to S. step_no and substep label the collision reports (< 0: the counters of the step graph);
// rec_slot is the CTA's slot in the adjoint engine's recording scratch.
template <int NT, int GM>
__device__ void bs_group(BsSharedT<GM> &sh, const Sim &S, const DevParams &P, double tau, int gidx, int g0, int g,
                         double m0, int step_no, int substep, int rec_slot) {
  const int tid = threadIdx.x;
  const int np = S.npad;
  const double Gm0 = P.G * m0;
  const int tps = g <= 8 ? 4 : (g <= 16 ? 2 : 1);  // threads per (level, member) slot
  if (BS_LEVELS * g * tps > NT) {  // uniform; the queues route larger groups elsewhere
    if (tid == 0) atomicOr(S.status, ST_GROUP_TOO_LARGE);
    return;
  }
  // Wide speculation (groups of three or four members on 256 threads): the second half of the CTA runs
  // the attempt at H/2, as below, from the second attempt on (most groups accept the first). Measured
  // on 300 systems, whose longest groups of three set the BS phase: 2.41 -> 2.20 ms for 4 steps.
  const bool specw = (g == 3 || g == 4) && NT == 256 && GM >= 20;  // uniform
  const int stid = specw ? (tid & 127) : tid;
  const int slot = stid / tps, sub = stid % tps;
  const bool act = slot < BS_LEVELS * g;
  const int lev = act ? slot / g : 0;  // level k = lev + 1, n_k = 2k substeps
  const int q = act ? slot % g : 0;
  const int L = lev + 1, nk = 2 * L;
  // Speculation (groups of one or two members, whose slots leave two of their four threads idle):
  // threads 2, 3 of a slot run the attempt at H/2 from the same state, with the same arithmetic, in
  // the same warp instructions; its members sit at index 16 + q of the position and tableau arrays,
  // its tableau rows on threads 64 + (member, component). Its result is taken exactly when the
  // serial step control's next attempt would be that one (the attempt at H failed), so results and
  // decisions are the serial algorithm's, and a failed attempt no longer costs a round of its own.
  const bool spec = g <= 2 && tps == 4 && NT >= 128 && GM >= 18;  // uniform
  const int half = spec ? (sub >> 1) : (specw ? tid >> 7 : 0), tsub = spec ? (sub & 1) : sub, ttps = spec ? 2 : tps;
  const int qm = q + 16 * half;  // this thread's member in its attempt's position and tableau arrays
  const int oc = ttps == 4 ? tsub : 2 * tsub;  // this thread's components: oc .. oc + on - 1
  const int on = ttps == 4 ? (tsub < 3 ? 1 : 0) : (ttps == 2 ? 2 - tsub : 3);
  const int tb = spec ? 64 : (specw ? 128 : NT);  // tableau threads from tb on: the attempt at H/2
  const int thalf = tid >= tb ? 1 : 0, trow = thalf ? tid - tb : tid;
  if (tid < g) {
    const int i = S.gmem[g0 + tid];
    sh.idx[tid] = i;
    sh.alive[tid] = S.alive[i];
    sh.gm[tid] = S.gm[i]; sh.m[tid] = S.m[i]; sh.R[tid] = S.R[i]; sh.A[tid] = S.A[i];
    sh.rcsq[tid] = S.rcsq[i];
    for (int c = 0; c < 3; ++c) { sh.y[tid][c] = S.x0[c * np + i]; sh.y[tid][3 + c] = S.v0[c * np + i]; }
  }
  if (tid == 0) { sh.H = tau; sh.rem = tau; sh.U = 0.0; sh.nseq = 0; }
  __syncthreads();
  int halvings = 0, attempts = 0, steps = 0;
  while (true) {
    const double rem = sh.rem;
    double H = sh.H;
    if (absbits(rem) == 0ULL) break;
    if (absbits(H) > absbits(rem)) H = rem;
    if (++attempts > 200000) { if (tid == 0) atomicOr(S.status, ST_BS_FAILED); break; }
    // ---- one attempt of length H: all levels' modified-midpoint integrations at once ----
    // Level L finishes its chain at evaluation 2L; its tableau row and error are then computed
    // right away (thread (qc, cc) holds member qc's component cc of the previous row), and the
    // attempt stops at the first converged level: the same decision as building the whole
    // tableau first, but attempts that converge at level 4-6 (almost all) skip the deeper chains.
    const double h = __ddiv_rn(half ? 0.5 * H : H, (double)nk), h2 = 2.0 * h;
    const bool specn = spec || (specw && attempts > 1);  // uniform: this attempt has its twin at H/2
    const bool acta = act && (half == 0 || specn);
    const bool qa = acta && sh.alive[q];
    double xA[3], vA[3], xB[3], vB[3];  // the two newest states of the level's chain, own components
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      xA[k] = k < on ? sh.y[q][oc + k] : 0.0;
      vA[k] = k < on ? sh.y[q][3 + oc + k] : 0.0;
      if (acta && k < on) sh.pos[0][lev][qm][oc + k] = xA[k];
    }
    const int qc = trow / 6, cc = trow % 6;
    const bool rowth = qc < g && (thalf == 0 || specn);
    double scale = 0.0;  // error scale of (qc, cc): 1/|x| or 1/|v| at the start of the attempt
    if (rowth) {
      const double *yq = sh.y[qc] + (cc < 3 ? 0 : 3);
      const double s2 = fma(yq[2], yq[2], fma(yq[1], yq[1], yq[0] * yq[0]));
      scale = dbits(s2) == 0ULL ? 4.49423283715579e307 : rsqrt_refined(s2);
    }
    if (tid == 0) sh.bad = 0u;
    __syncthreads();
    double ac[3] = {0.0, 0.0, 0.0};
    const BsTerm t0 = bs_term(sh, Gm0, g, q, tsub);
    // every lane of a warp that holds any active slot takes part (the sums shuffle across lanes);
    // warps without active slots stay off the pipes
    if (__any_sync(0xffffffffu, acta)) bs_accel(sh, P, t0, Gm0, g, q, tsub, ttps, sh.pos[0][lev] + 16 * half, qa, ac);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (k >= on) continue;
      xB[k] = qa ? fma(h, vA[k], xA[k]) : xA[k];
      vB[k] = qa ? fma(h, ac[k], vA[k]) : vA[k];
    }
    const int lmax = P.bs_kmax < BS_LEVELS ? P.bs_kmax : BS_LEVELS;
    const u64 eps = dbits(P.bs_eps);
    double prev[BS_LEVELS], tlast = 0.0;  // previous tableau row; T_{Lc,Lc} of the current one
    int acc = 0, accB = 0;
    int b = 1;
    for (int e = 1; e <= 2 * lmax; ++e) {
      const bool lv = acta && e <= nk;
      if (lv) {
#pragma unroll
        for (int k = 0; k < 3; ++k)
          if (k < on) sh.pos[b][lev][qm][oc + k] = xB[k];
      }
      __syncthreads();
      if (__any_sync(0xffffffffu, lv)) bs_accel(sh, P, t0, Gm0, g, q, tsub, ttps, sh.pos[b][lev] + 16 * half, qa, ac);
      if (lv) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          if (k >= on) continue;
          if (e < nk) {
            if (qa) {
              const double xn = fma(h2, vB[k], xA[k]), vn = fma(h2, ac[k], vA[k]);
              xA[k] = xB[k]; vA[k] = vB[k];
              xB[k] = xn; vB[k] = vn;
            }
          } else {  // T_{L,1}
            sh.tab[lev][qm][oc + k] = qa ? 0.5 * fma(h, vB[k], xB[k] + xA[k]) : xA[k];
            sh.tab[lev][qm][3 + oc + k] = qa ? 0.5 * fma(h, ac[k], vB[k] + vA[k]) : vA[k];
          }
        }
      }
      b ^= 1;
      if (e & 1) continue;
      // level Lc = e/2 is complete: its tableau row (polynomial extrapolation in h^2, Neville)
      const int Lc = e >> 1;
      __syncthreads();
      bool bad = false;
      if (rowth) {
        double before;
        tlast = neville_row(sh.tab[Lc - 1][qc + 16 * thalf][cc], Lc, [&](int j) { return c_facinv[Lc][j]; }, prev, before);
        if (Lc >= 2 && sh.alive[qc]) bad = absbits((tlast - before) * scale) > eps;
      }
      if (Lc >= 2) warp_flag(&sh.bad, 1u << (Lc - 1 + 8 * thalf), bad);  // thalf is uniform per warp
      __syncthreads();
      if (specn && !accB && Lc >= 2 && !((sh.bad >> (Lc + 7)) & 1u)) {  // the attempt at H/2 converged (uniform)
        accB = Lc;
        if (thalf && rowth) sh.yn[qc + 16][cc] = tlast;
      }
      if (Lc >= 2 && !((sh.bad >> (Lc - 1)) & 1u)) { acc = Lc; break; }  // uniform: every thread reads the same bits
    }
    if (acc && rowth && !thalf) sh.yn[qc][cc] = tlast;  // the accepted row is the last one built
    double Hs = H;  // length of the accepted substep
    if (!acc && specn) {  // the serial control halves H; its next attempt is the one at H/2
      if (++halvings > P.bs_max_halvings) {
        if (tid == 0) atomicOr(S.status, ST_BS_FAILED);
        __syncthreads();
        break;
      }
      ++attempts;
      if (accB) {
        acc = accB;
        Hs = 0.5 * H;
        __syncthreads();
        if (tid < 6 * g) sh.yn[tid / 6][tid % 6] = sh.yn[tid / 6 + 16][tid % 6];
      } else {  // that attempt failed too: the serial control halves again
        if (tid == 0) sh.H = 0.25 * H;
        if (++halvings > P.bs_max_halvings) {
          if (tid == 0) atomicOr(S.status, ST_BS_FAILED);
          __syncthreads();
          break;
        }
        __syncthreads();
        continue;
      }
    }
    if (acc) {
      __syncthreads();
      if (P.collisions) {  // contact test over the accepted substep (Hermite, threshold (R_a + R_b)^2)
        const int npair = g * (g - 1) / 2;
        int anyhit = 0;
        for (int pi = tid; pi < npair; pi += NT) {
          int a = 0, rest = pi;
          while (rest >= g - 1 - a) { rest -= g - 1 - a; a++; }
          const int bq = a + 1 + rest;
          unsigned char hit = 0;
          if (sh.alive[a] && sh.alive[bq]) {
            const double rr = sh.R[a] + sh.R[bq];
            const double dmin = hermite_min_capped(
                __dsub_rn(sh.y[bq][0], sh.y[a][0]), __dsub_rn(sh.y[bq][1], sh.y[a][1]), __dsub_rn(sh.y[bq][2], sh.y[a][2]),
                __dsub_rn(sh.y[bq][3], sh.y[a][3]), __dsub_rn(sh.y[bq][4], sh.y[a][4]), __dsub_rn(sh.y[bq][5], sh.y[a][5]),
                __dsub_rn(sh.yn[bq][0], sh.yn[a][0]), __dsub_rn(sh.yn[bq][1], sh.yn[a][1]), __dsub_rn(sh.yn[bq][2], sh.yn[a][2]),
                __dsub_rn(sh.yn[bq][3], sh.yn[a][3]), __dsub_rn(sh.yn[bq][4], sh.yn[a][4]), __dsub_rn(sh.yn[bq][5], sh.yn[a][5]), Hs, rr * rr);
            hit = dmin < rr * rr;
          }
          sh.cont[pi] = hit;
          anyhit |= hit;
        }
        if (__syncthreads_or(anyhit) && tid == 0) {  // mergers in ascending pair order, post-substep states (none without contact)
          int pi = 0;
          for (int a = 0; a < g; ++a)
            for (int bq = a + 1; bq < g; ++bq, ++pi) {
              if (!sh.cont[pi] || !sh.alive[a] || !sh.alive[bq]) continue;
              const int ia = sh.idx[a], ib = sh.idx[bq];
              const double ma = sh.m[a], mb = sh.m[bq], M = ma + mb;
              const double dx = sh.yn[bq][0] - sh.yn[a][0], dy = sh.yn[bq][1] - sh.yn[a][1], dz = sh.yn[bq][2] - sh.yn[a][2];
              const double dvx = sh.yn[bq][3] - sh.yn[a][3], dvy = sh.yn[bq][4] - sh.yn[a][4], dvz = sh.yn[bq][5] - sh.yn[a][5];
              const double r = sqrt(dx * dx + dy * dy + dz * dz);
              const double v2 = dvx * dvx + dvy * dvy + dvz * dvz;
              sh.U += 0.5 * ma * mb / M * v2 - P.G * ma * mb / r;
              const bool keep_a = ma > mb || (ma == mb && ia < ib);
              merger_report(S, ia, ib, sh.y[a], sh.y[bq], sh.yn[a], sh.yn[bq], ma, mb, keep_a, tau - rem, step_no, substep);
              const int s = keep_a ? a : bq, d = keep_a ? bq : a;
              for (int c = 0; c < 6; ++c) sh.yn[s][c] = (ma * sh.yn[a][c] + mb * sh.yn[bq][c]) / M;
              const double Ra = sh.R[a], Rb = sh.R[bq];
              sh.R[s] = cbrt(Ra * Ra * Ra + Rb * Rb * Rb);
              sh.m[s] = M; sh.gm[s] = P.G * M;
              sh.m[d] = 0.0; sh.gm[d] = 0.0; sh.R[d] = 0.0; sh.alive[d] = 0;
              const int is = sh.idx[s], idd = sh.idx[d];
              S.m[is] = M; S.gm[is] = P.G * M; S.R[is] = sh.R[s]; S.hill[is] = cbrt(M / (3.0 * m0));
              S.m[idd] = 0.0; S.gm[idd] = 0.0; S.R[idd] = 0.0; S.hill[idd] = 0.0; S.alive[idd] = 0;
              S.T[idd] = 0ULL; S.rcsq[idd] = 0ULL;
              atomicAdd((unsigned long long *)&S.counters[C_MERGE], 1ULL);
            }
        }
        __syncthreads();
      }
      if (tid < g) for (int c = 0; c < 6; ++c) sh.y[tid][c] = sh.yn[tid][c];
      if (S.seq_len && tid < g && steps < BS_SEQCAP)  // adjoint engine: the state after this substep
        for (int c = 0; c < 6; ++c)
          S.y_scratch[(((size_t)rec_slot * BS_SEQCAP + steps) * BS_GMAX + tid) * 6 + c] = sh.yn[tid][c];
      if (tid == 0) {
        sh.rem = rem - Hs; sh.H = 2.0 * Hs;
        if (sh.nseq < BS_SEQCAP) { sh.seqH[sh.nseq] = Hs; sh.seqk[sh.nseq] = (unsigned char)acc; }
        sh.nseq++;
      }
      halvings = 0;
      steps++;
    } else {
      if (tid == 0) sh.H = 0.5 * H;
      if (++halvings > P.bs_max_halvings) {
        if (tid == 0) atomicOr(S.status, ST_BS_FAILED);
        __syncthreads();
        break;
      }
    }
    __syncthreads();
  }
  // write back: live members take the integrated state, ghosts are parked far out
  if (tid < g && S.bsn) S.bsn[sh.idx[tid]] = (unsigned char)(steps < 255 ? steps : 255);
  if (tid < g) {
    const int i = sh.idx[tid];
    if (sh.alive[tid]) {
      for (int c = 0; c < 3; ++c) { S.x[c * np + i] = sh.y[tid][c]; S.v[c * np + i] = sh.y[tid][3 + c]; }
    } else {
      S.x[i] = PARK + 1.0e4 * i; S.x[np + i] = 0.0; S.x[2 * np + i] = 0.0;
      for (int c = 0; c < 3; ++c) S.v[c * np + i] = 0.0;
    }
  }
  if (tid == 0) {
    atomicAdd((unsigned long long *)&S.counters[C_BSSTEPS], (unsigned long long)steps);
    if (dbits(sh.U) != 0ULL) atomicAdd(S.U, sh.U);
    if (S.seq_len) {  // the adjoint engine records the accepted sequence
      int n = sh.nseq, base = -1;
      if (n <= BS_SEQCAP) {
        base = atomicAdd(S.seq_count, n);
        if (base + n > S.seq_cap) base = -1;
      }
      long long ybase = 0;
      if (base >= 0 && n > 1) {  // states after substeps 1 .. n-1 (the last one is the result)
        ybase = atomicAdd((unsigned long long *)S.y_count, (unsigned long long)((n - 1) * g * 6));
        if (ybase + (long long)(n - 1) * g * 6 > S.y_cap) base = -1;
      }
      if (base < 0) { atomicOr(S.status, ST_RECORD_OVERFLOW); n = 0; base = 0; ybase = 0; }
      S.seq_off[gidx] = base;
      S.seq_len[gidx] = n;
      S.y_off[gidx] = ybase;
      sh.seq_base = base;
      sh.y_base = ybase;
      sh.nseq = n;
    }
  }
  __syncthreads();
  if (S.seq_len) {
    for (int k = tid; k < sh.nseq; k += NT) S.seq_pool[sh.seq_base + k] = make_double2(sh.seqH[k], (double)sh.seqk[k]);
    const int ny = (sh.nseq > 1 ? sh.nseq - 1 : 0) * g * 6;
    for (int k = tid; k < ny; k += NT) {
      const int s = k / (g * 6), r = k % (g * 6);
      S.y_pool[sh.y_base + k] = S.y_scratch[(((size_t)rec_slot * BS_SEQCAP + s) * BS_GMAX + r / 6) * 6 + r % 6];
    }
  }
  __syncthreads();
}

}  // namespace genga
