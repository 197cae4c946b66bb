// bs_cluster.cu -- Bulirsch-Stoer of the larger encounter groups (Sect. 3.2) on a thread-block
// cluster of 8 CTAs: CTA r integrates extrapolation level r + 1 (n = 2(r + 1) midpoint substeps).
//
// A group of g members costs 8 levels x g members x g terms per force evaluation; on one SM (the
// one-CTA kernel in bs.cu) that saturates the FP64 pipes once g reaches a handful. Here each level
// has an SM of its own. After every second evaluation the CTAs meet at a cluster barrier; level Lc
// is then complete in CTA Lc - 1, every CTA reads its T_{Lc,1} from that CTA's shared memory
// (distributed shared memory), extends its own copy of the Neville tableau and tests level Lc, with
// the same arithmetic and order in every CTA. Each pair is evaluated once (Newton's third law); of
// large groups only the pairs that may be inside their critical radius. All CTAs therefore take the
// same decision and follow the same control flow: every cluster barrier is reached by all 8 CTAs the
// same number of times. Level results are double-buffered by attempt parity. Cluster k takes the k-th entry of
// the large-group list that the grouping kernel writes.
#include <cooperative_groups.h>

#include "fxforce.cuh"
#include "genga_launch.h"

namespace cg = cooperative_groups;

namespace genga {

constexpr int CL_SIZE = BS_LEVELS;  // CTAs per cluster, one per level
constexpr int CL_THREADS = 256;
constexpr int CL_TPS = CL_THREADS / BS_GMAX;  // lanes per member that list pairs (8)
constexpr int CL_PAIRS = BS_GMAX * (BS_GMAX - 1) / 2;
// the first level whose convergence is tested: groups of five or more members converge at level 5
// or later in practice, and a level below it that converges is still found (its row is kept), at
// the cost of the evaluations up to this level
constexpr int CL_FIRST_CHECK = 4;

// 1/((L/(L-j))^2 - 1), the Neville factors (same values as the one-CTA kernel's table)
__constant__ double c_facinv_cl[BS_LEVELS + 1][BS_LEVELS];

struct BsClShared {
  int idx[BS_GMAX], alive[BS_GMAX];
  double gm[BS_GMAX], m[BS_GMAX], R[BS_GMAX], A[BS_GMAX];
  u64 rcsq[BS_GMAX];
  double y[BS_GMAX][6], yn[BS_GMAX][6];
  double isc[BS_GMAX][2];                // 1/|x|, 1/|v| at the start of the attempt
  double pos[2][BS_GMAX][3];             // chain positions, double-buffered by evaluation
  float fp[2][BS_GMAX][3];               // the same in single precision
  double term[BS_GMAX][BS_GMAX][3];      // this evaluation's factors of partner [j] on member [i] ([i][i]: central pull)
  float rcf[BS_GMAX];                    // critical radii, rounded up
  unsigned mask[2][BS_GMAX];             // partners inside the critical radius, by evaluation
  int cnt[2];                            // pairs listed, by evaluation
  unsigned short pair[CL_PAIRS];         // the listed pairs i << 8 | j, i < j
  double T1[2][BS_GMAX][6];              // this level's result, double-buffered by attempt
  unsigned bad;                          // bit r - 1: level r has not converged
  unsigned char cont[BS_GMAX * (BS_GMAX - 1) / 2];
  double H, rem, U;
  int accept, nseq;
  long long y_base;
  int seq_base;
  double seqH[BS_SEQCAP];
  unsigned char seqk[BS_SEQCAP];
};

// Single precision by truncation, on the integer pipe (a conversion takes an FP64 slot): within 2^-23,
// 0 below 2^-126, infinite from 2^128 on.
__device__ __forceinline__ float cl_float(double x) {
  const u64 b = dbits(x);
  const unsigned hi = (unsigned)(b >> 32), ex = (hi >> 20) & 0x7ffu;
  const unsigned m = ex < 897u ? 0u : (ex > 1150u ? 0x7f800000u : ((hi & 0x7fffffffu) - (896u << 20)) << 3 | (unsigned)b >> 29);
  return __uint_as_float(m | (hi & 0x80000000u));
}

// One force evaluation at the positions pos (fp: the same in single precision) by all threads of the
// CTA; returns the acceleration of member a, component c, on the thread of (a, c).
//  1. Groups whose pairs are more than the threads: eight lanes a member list the pairs that may be
//     inside the pair's critical radius, from the single-precision distance with a bound on its error
//     (outside, the weight 1 - K is zero). Smaller groups list every pair, once for the group.
//  2. One item per thread (Newton's third law): item t < g is member t's central pull G m0 d / r^3, then
//     the factor w d / r^3 of each listed pair (i < j), d = x_j - x_i, w the weight. A pair inside the
//     radius (decided in FP64) leaves the factor for both members and marks each for the other.
//  3. Member a sums its central pull and G m_b times the factors of its marked partners in ascending
//     order (whatever the order of the list).
// Bound by latency, the instructions of one item and of one sum after the other (levels of a small
// group), and by FP64 issue, 64-76 cycles a warp instruction, where a group has many pairs inside.
// Measured against every pair a term, summed over all partners with barriers between: 1024 bodies with
// wide radii 89 -> 56 us a launch, 2048 bodies (groups of 5-12) 59.5 -> 51.7 us.
__device__ __forceinline__ double cl_eval(BsClShared &sh, const DevParams &P, double Gm0, int g, const double (*pos)[3],
                                          const float (*fp)[3], int &par, int a, int c) {
  const int tid = threadIdx.x;
  int nitems = g + g * (g - 1) / 2;
  if (nitems > CL_THREADS) {
    const int m = tid / CL_TPS, sub = tid % CL_TPS;
    if (m < g && sh.alive[m]) {
      const float x = fp[m][0], y = fp[m][1], z = fp[m][2], rc = sh.rcf[m], e = fabsf(x) + fabsf(y) + fabsf(z);
      for (int q = m + 1 + sub; q < g; q += CL_TPS) {
        const float qx = fp[q][0], qy = fp[q][1], qz = fp[q][2], dx = qx - x, dy = qy - y, dz = qz - z;
        const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
        // truncation moves a coordinate by at most 2^-23 of itself
        const float lim = fmaxf(rc, sh.rcf[q]) + 4.0e-7f * (e + (fabsf(qx) + fabsf(qy) + fabsf(qz)));
        if (!(r2 > fmaxf(lim * lim, 1.0e-30f) && r2 < 3.0e38f)) sh.pair[atomicAdd(&sh.cnt[par], 1)] = (unsigned short)(m << 8 | q);
      }
    }
    __syncthreads();
    nitems = g + sh.cnt[par];
  }
  if (tid < g) sh.mask[par ^ 1][tid] = 0u;  // the next evaluation's marks and list
  if (tid == 0) sh.cnt[par ^ 1] = 0;
  for (int t = tid; t < nitems; t += CL_THREADS) {
    const bool cen = t < g;
    const int pr = cen ? t << 8 | t : sh.pair[t - g], i = pr >> 8, j = pr & 255;
    const double dx = (cen ? 0.0 : pos[j][0]) - pos[i][0], dy = (cen ? 0.0 : pos[j][1]) - pos[i][1],
                 dz = (cen ? 0.0 : pos[j][2]) - pos[i][2];
    const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
    const bool inside = !cen && sh.alive[i] && sh.alive[j] && dbits(r2) < umax64(sh.rcsq[i], sh.rcsq[j]);
    const double f = bs_factor(r2, cen ? Gm0 : 1.0, pmin(sh.A[i], sh.A[j]), cen && sh.alive[i], inside, P.kmode);
    const double fx = f * dx, fy = f * dy, fz = f * dz;
    if (cen || inside) { sh.term[i][j][0] = fx; sh.term[i][j][1] = fy; sh.term[i][j][2] = fz; }
    if (inside) {
      sh.term[j][i][0] = -fx; sh.term[j][i][1] = -fy; sh.term[j][i][2] = -fz;
      atomicOr(&sh.mask[par][i], 1u << j);
      atomicOr(&sh.mask[par][j], 1u << i);
    }
  }
  __syncthreads();
  double v = 0.0;
  if (a < g) {
    v = sh.term[a][a][c];
    for (unsigned bits = sh.mask[par][a]; bits; bits &= bits - 1) {
      const int q = __ffs(bits) - 1;
      v = fma(sh.gm[q], sh.term[a][q][c], v);
    }
  }
  par ^= 1;
  return v;
}

__global__ void __cluster_dims__(CL_SIZE, 1, 1) __launch_bounds__(CL_THREADS, 2)
    k_bs_cluster(Sim S, DevParams P, double tau, int gmin) {
  __shared__ BsClShared sh;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int L = rank + 1, nk = 2 * L;
  const int tid = threadIdx.x;
  const int np = S.npad;
  const int ngroups = *S.ngroups;
  const int ncl = gridDim.x / CL_SIZE, cid = blockIdx.x / CL_SIZE;
  // the groups listed by size (one per cluster while there are no more than clusters), else all
  const int nwork = S.big ? *S.nbig : ngroups;
  for (int k = cid; k < nwork; k += ncl) {
    const int gidx = S.big ? S.big[k] : k;
    const int g0 = S.gstart[gidx], g = S.gsize ? S.gsize[gidx] : S.gstart[gidx + 1] - g0;
    if (g < gmin || g > BS_GMAX) continue;  // the same for all CTAs of the cluster (g < gmin: one-CTA kernel)
    const double m0 = S.sys_of ? S.sys_m0[S.sys_of[S.gmem[g0]]] : P.m0;
    const double Gm0 = P.G * m0;
    const int q = tid / 3, c = tid % 3;  // chain threads: one per (member, component)
    const bool act = q < g;
    int par = 0;
    if (tid < g) {
      const int i = S.gmem[g0 + tid];
      sh.idx[tid] = i;
      sh.alive[tid] = S.alive[i];
      sh.gm[tid] = S.gm[i]; sh.m[tid] = S.m[i]; sh.R[tid] = S.R[i]; sh.A[tid] = S.A[i];
      sh.rcsq[tid] = S.rcsq[i];
      sh.rcf[tid] = 1.0001f * sqrtf(__double2float_ru(__longlong_as_double((long long)S.rcsq[i])));
      for (int c = 0; c < 3; ++c) { sh.y[tid][c] = S.x0[c * np + i]; sh.y[tid][3 + c] = S.v0[c * np + i]; }
    }
    if (tid == 0) { sh.H = tau; sh.rem = tau; sh.U = 0.0; sh.nseq = 0; }
    if (tid < 2) sh.cnt[tid] = 0;
    if (tid < 2 * BS_GMAX) sh.mask[tid / BS_GMAX][tid % BS_GMAX] = 0u;
    if (g + g * (g - 1) / 2 <= CL_THREADS && tid < g)  // every pair, row by row
      for (int j = tid + 1, k = tid * (g - 1) - tid * (tid - 1) / 2; j < g; ++j, ++k) sh.pair[k] = (unsigned short)(tid << 8 | j);
    __syncthreads();
    int halvings = 0, attempts = 0, steps = 0, buf = 0;
    while (true) {
      const double rem = sh.rem;
      double H = sh.H;
      if (absbits(rem) == 0ULL) break;
      if (absbits(H) > absbits(rem)) H = rem;
      if (++attempts > 200000) { if (tid == 0 && rank == 0) atomicOr(S.status, ST_BS_FAILED); break; }
      const double h = __ddiv_rn(H, (double)nk), h2 = 2.0 * h;
      const bool qa = act && sh.alive[q];
      if (tid < g) {  // error scales at the start of the attempt
        const double *yq = sh.y[tid];
        const double sx2 = fma(yq[2], yq[2], fma(yq[1], yq[1], yq[0] * yq[0]));
        const double sv2 = fma(yq[5], yq[5], fma(yq[4], yq[4], yq[3] * yq[3]));
        sh.isc[tid][0] = dbits(sx2) == 0ULL ? 4.49423283715579e307 : rsqrt_refined(sx2);
        sh.isc[tid][1] = dbits(sv2) == 0ULL ? 4.49423283715579e307 : rsqrt_refined(sv2);
      }
      // ---- this level's modified-midpoint integration; levels checked as they complete ----
      // Level Lc finishes at evaluation 2 Lc. At every even evaluation all CTAs meet at a cluster
      // barrier, read T_{Lc,1} from its CTA, extend their tableau rows (thread (qc, cc): member
      // qc, component cc) and test level Lc; the first converged level ends the attempt in every
      // CTA at once (the same data, the same arithmetic, so the same decision).
      double xA = act ? sh.y[q][c] : 0.0, vA = act ? sh.y[q][3 + c] : 0.0, xB = xA, vB = vA;
      if (act) { sh.pos[0][q][c] = xA; sh.fp[0][q][c] = cl_float(xA); }
      const int qc = tid / 6, cc = tid % 6;
      const bool rowth = qc < g;
      if (tid == 0) sh.bad = 0u;
      __syncthreads();
      double acc_c = cl_eval(sh, P, Gm0, g, sh.pos[0], sh.fp[0], par, q, c);
      if (qa) {
        xB = fma(h, vA, xA);
        vB = fma(h, acc_c, vA);
      }
      const int lmax = P.bs_kmax < BS_LEVELS ? P.bs_kmax : BS_LEVELS;
      const u64 eps = dbits(P.bs_eps);
      const double scale = rowth ? sh.isc[qc][cc < 3 ? 0 : 1] : 0.0;
      double prev[BS_LEVELS], tlast = 0.0;  // previous tableau row; T_{Lc,Lc} of the current one
      int acc = 0;
      int b = 1;
      for (int e = 1; e <= 2 * lmax; ++e) {
        const bool lv = e <= nk;  // this CTA's level is still integrating
        if (lv) {
          if (act) { sh.pos[b][q][c] = xB; sh.fp[b][q][c] = cl_float(xB); }
          __syncthreads();
          acc_c = cl_eval(sh, P, Gm0, g, sh.pos[b], sh.fp[b], par, q, c);
          if (qa && e < nk) {
            const double xn = fma(h2, vB, xA), vn = fma(h2, acc_c, vA);
            xA = xB; vA = vB;
            xB = xn; vB = vn;
          }
          if (e == nk && act) {  // T_{L,1}
            sh.T1[buf][q][c] = qa ? 0.5 * fma(h, vB, xB + xA) : xA;
            sh.T1[buf][q][3 + c] = qa ? 0.5 * fma(h, acc_c, vB + vA) : vA;
          }
          b ^= 1;
        }
        if (e & 1) continue;
        const int Lc = e >> 1;
        // the rows of the levels below the first check are built with it: the same rows and the same
        // first converged level as a check per level, one cluster barrier instead of CL_FIRST_CHECK
        const int fc = lmax < CL_FIRST_CHECK ? lmax : CL_FIRST_CHECK;
        if (Lc < fc) continue;
        cluster.sync();  // T_{r,1} is complete in CTA r - 1 for every r <= Lc
        const int r0 = Lc == fc ? 1 : Lc;
        double tk[CL_FIRST_CHECK + 1];  // T_{r,r} of the rows built at the first check
#pragma unroll
        for (int r = 1; r <= BS_LEVELS; ++r) {
          if (r < r0 || r > Lc) continue;  // uniform
          bool bad = false;
          if (rowth) {
            const double *rt = cluster.map_shared_rank(&sh.T1[buf][0][0], (unsigned)(r - 1));
            double before;
            tlast = neville_row(rt[qc * 6 + cc], r, [&](int j) { return c_facinv_cl[r][j]; }, prev, before);
            if (r >= 2 && sh.alive[qc]) bad = absbits((tlast - before) * scale) > eps;
            if (r <= CL_FIRST_CHECK) tk[r] = tlast;
          }
          if (r >= 2) warp_flag(&sh.bad, 1u << (r - 1), bad);
        }
        __syncthreads();
        for (int r = r0 < 2 ? 2 : r0; r <= Lc; ++r)  // uniform: every thread reads the same bits
          if (!((sh.bad >> (r - 1)) & 1u)) { acc = r; break; }
        if (acc) {
          if (acc < Lc && rowth) tlast = tk[acc];
          break;
        }
      }
      if (acc && rowth) sh.yn[qc][cc] = tlast;  // the accepted row is the last one built
      buf ^= 1;
      if (acc) {
        __syncthreads();
        if (P.collisions) {  // contact test and mergers, redundantly in every CTA; globals by rank 0
          const int npair = g * (g - 1) / 2;
          int anyhit = 0;
          for (int pi = tid; pi < npair; pi += CL_THREADS) {
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
                  __dsub_rn(sh.yn[bq][3], sh.yn[a][3]), __dsub_rn(sh.yn[bq][4], sh.yn[a][4]), __dsub_rn(sh.yn[bq][5], sh.yn[a][5]), H, rr * rr);
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
                if (rank == 0) merger_report(S, ia, ib, sh.y[a], sh.y[bq], sh.yn[a], sh.yn[bq], ma, mb, keep_a, tau - rem);
                const int s = keep_a ? a : bq, d = keep_a ? bq : a;
                for (int c = 0; c < 6; ++c) sh.yn[s][c] = (ma * sh.yn[a][c] + mb * sh.yn[bq][c]) / M;
                const double Ra = sh.R[a], Rb = sh.R[bq];
                sh.R[s] = cbrt(Ra * Ra * Ra + Rb * Rb * Rb);
                sh.m[s] = M; sh.gm[s] = P.G * M;
                sh.m[d] = 0.0; sh.gm[d] = 0.0; sh.R[d] = 0.0; sh.alive[d] = 0;
                if (rank == 0) {
                  const int is = sh.idx[s], idd = sh.idx[d];
                  S.m[is] = M; S.gm[is] = P.G * M; S.R[is] = sh.R[s]; S.hill[is] = cbrt(M / (3.0 * m0));
                  S.m[idd] = 0.0; S.gm[idd] = 0.0; S.R[idd] = 0.0; S.hill[idd] = 0.0; S.alive[idd] = 0;
                  S.T[idd] = 0ULL; S.rcsq[idd] = 0ULL;
                  atomicAdd((unsigned long long *)&S.counters[C_MERGE], 1ULL);
                }
              }
          }
          __syncthreads();
        }
        if (tid < g) for (int c = 0; c < 6; ++c) sh.y[tid][c] = sh.yn[tid][c];
        if (rank == 0 && S.seq_len && tid < g && steps < BS_SEQCAP)  // adjoint engine: state after this substep
          for (int c = 0; c < 6; ++c)
            S.y_scratch[(((size_t)cid * BS_SEQCAP + steps) * BS_GMAX + tid) * 6 + c] = sh.yn[tid][c];
        if (tid == 0) {
          sh.rem = rem - H; sh.H = 2.0 * H;
          if (sh.nseq < BS_SEQCAP) { sh.seqH[sh.nseq] = H; sh.seqk[sh.nseq] = (unsigned char)acc; }
          sh.nseq++;
        }
        halvings = 0;
        steps++;
      } else {
        if (tid == 0) sh.H = 0.5 * H;
        if (++halvings > P.bs_max_halvings) {
          if (tid == 0 && rank == 0) atomicOr(S.status, ST_BS_FAILED);
          __syncthreads();
          break;
        }
      }
      __syncthreads();
    }
    // write-back, counters and the adjoint recording by rank 0
    if (rank == 0) {
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
        if (S.seq_len) {
          int n = sh.nseq, base = -1;
          if (n <= BS_SEQCAP) {
            base = atomicAdd(S.seq_count, n);
            if (base + n > S.seq_cap) base = -1;
          }
          long long ybase = 0;
          if (base >= 0 && n > 1) {
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
        for (int k = tid; k < sh.nseq; k += CL_THREADS) S.seq_pool[sh.seq_base + k] = make_double2(sh.seqH[k], (double)sh.seqk[k]);
        const int ny = (sh.nseq > 1 ? sh.nseq - 1 : 0) * g * 6;
        for (int k = tid; k < ny; k += CL_THREADS) {
          const int s = k / (g * 6), r = k % (g * 6);
          S.y_pool[sh.y_base + k] = S.y_scratch[(((size_t)cid * BS_SEQCAP + s) * BS_GMAX + r / 6) * 6 + r % 6];
        }
      }
    }
    cluster.sync();  // no CTA starts the next group while another may still read its results
  }
}

void bs_cluster_init_constants() {
  double h[BS_LEVELS + 1][BS_LEVELS] = {};
  for (int Lv = 2; Lv <= BS_LEVELS; ++Lv)
    for (int j = 1; j < Lv; ++j) {
      const double ratio = (double)Lv / (double)(Lv - j);
      h[Lv][j] = 1.0 / (ratio * ratio - 1.0);
    }
  cudaMemcpyToSymbol(c_facinv_cl, h, sizeof(h));
}

// As many clusters as can be resident at once (the scheduler's answer for this kernel's resources);
// one cluster per 8 SMs if the query fails.
int bs_cluster_grid() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int clusters = sms > CL_SIZE ? sms / CL_SIZE : 1;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = CL_SIZE; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
  cfg.gridDim = dim3(CL_SIZE * clusters, 1, 1);
  cfg.blockDim = dim3(CL_THREADS, 1, 1);
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int active = 0;
  if (cudaOccupancyMaxActiveClusters(&active, k_bs_cluster, &cfg) == cudaSuccess && active > 0) clusters = active;
  cudaGetLastError();
  return clusters * CL_SIZE;
}

void launch_bs_cluster(const Sim &S, const DevParams &P, double tau, int gmin, int grid, cudaStream_t st) {
  k_bs_cluster<<<grid, CL_THREADS, 0, st>>>(S, P, tau, gmin);
}

}  // namespace genga
