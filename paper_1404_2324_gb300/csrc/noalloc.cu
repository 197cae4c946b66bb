// noalloc.cu -- genga_kick_noalloc: the kick phase (accelerations + precheck candidates) for
// callers that must not allocate device memory.
//
// cudaMalloc can block on the driver's allocator and cudaFree synchronises the whole device, so
// code that runs inside a latency-critical loop, or that lives in a process whose device memory
// is owned by another allocator (a framework's caching allocator, an embedding application with
// a fixed memory budget), cannot call entry points that allocate. This variant keeps all of its
// scratch in one file-scope __device__ array instead: every GPU that loads the library holds it
// (about 2 MB) until the process exits. The caller still provides the inputs and outputs.
#include <atomic>
#include <cstring>

#include "../../include/genga.h"
#include "genga_launch.h"

using namespace genga;

namespace {

constexpr int NA_NMAX = 1024;              // largest n accepted by genga_kick_noalloc
constexpr int NA_NT = NA_NMAX / 32;        // tiles
constexpr int NA_W = NA_NMAX / 32;         // bitmap words per row
constexpr size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

// byte offsets of the sub-arrays inside the scratch array
constexpr size_t O_X = 0;
constexpr size_t O_V = O_X + align256(3 * NA_NMAX * sizeof(double));
constexpr size_t O_M = O_V + align256(3 * NA_NMAX * sizeof(double));
constexpr size_t O_GM = O_M + align256(NA_NMAX * sizeof(double));
constexpr size_t O_RC = O_GM + align256(NA_NMAX * sizeof(double));
constexpr size_t O_A = O_RC + align256(NA_NMAX * sizeof(double));
constexpr size_t O_ALIVE = O_A + align256(NA_NMAX * sizeof(double));
constexpr size_t O_T = O_ALIVE + align256(NA_NMAX * sizeof(int));
constexpr size_t O_RCSQ = O_T + align256(NA_NMAX * sizeof(u64));
constexpr size_t O_AFAR = O_RCSQ + align256(NA_NMAX * sizeof(u64));
constexpr size_t O_PART = O_AFAR + align256(3 * NA_NMAX * sizeof(double));
constexpr size_t O_PKICK = O_PART + align256((size_t)NA_NT * NA_NT * 2 * 96 * sizeof(double));
constexpr size_t O_PFIN = O_PKICK + align256(NA_NT * FIN_PER_TILE * 3 * sizeof(double));
constexpr size_t O_CBM = O_PFIN + align256(NA_NT * FIN_PER_TILE * 3 * sizeof(double));
constexpr size_t O_ROWANY = O_CBM + align256((size_t)NA_NMAX * NA_W * sizeof(unsigned));
constexpr size_t O_CCNT = O_ROWANY + align256(NA_W * sizeof(unsigned));
constexpr size_t O_CLIST = O_CCNT + align256(NA_NMAX * sizeof(int));
constexpr size_t O_ITEMS = O_CLIST + align256((size_t)NA_NMAX * CCAP * sizeof(int));
constexpr size_t O_FLAGS = O_ITEMS + align256((size_t)NA_NT * NA_NT * sizeof(int));
constexpr size_t O_STATUS = O_FLAGS + align256(4 * sizeof(int));
constexpr size_t O_COUNTERS = O_STATUS + align256(sizeof(int));
constexpr size_t NA_BYTES = O_COUNTERS + align256(NCOUNTERS * sizeof(long long));

}  // namespace

// The scratch shared by every call. In host code this name is only a stand-in for the device
// symbol; its device address comes from cudaGetSymbolAddress below.
static __device__ __align__(256) unsigned char g_kick_scratch[NA_BYTES];

namespace {

constexpr int NA_MAXDEV = 64;
std::atomic<unsigned char *> g_scratch_ptr[NA_MAXDEV] = {};  // device address of g_kick_scratch, per device

// Set-up, once per device, with that device current. Threads that get here first at the same time
// look the address up alike and store the same value.
int scratch_address(unsigned char **out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NA_MAXDEV) return GENGA_ECUDA;
  unsigned char *p = g_scratch_ptr[dev].load(std::memory_order_acquire);
  if (!p) {
    void *q = nullptr;
    if (cudaGetSymbolAddress(&q, g_kick_scratch) != cudaSuccess || !q) return GENGA_ECUDA;
    p = (unsigned char *)q;
    g_scratch_ptr[dev].store(p, std::memory_order_release);
  }
  *out = p;
  return GENGA_OK;
}

// What the pair kernel and its finalisation read, from the caller's arrays: padded positions, G m,
// critical radii and their squares. Clears what must start at zero (the array keeps the previous
// call's contents): the candidate bitmap, row bits and counts, flags, status and counters. One launch
// for what six fills, a copy and a set-up kernel took: the call was bound by the gaps between its
// launches (n = 64: 32.6 -> 23.6 us; n = 1000: 62.5 -> 41.0 us, also from the pair list reading only
// rows that have candidates; 17-19 and 32.8 us with dependent launches and the one-kernel kick of few
// bodies).
__global__ void k_kick_setup(Sim S, double G, double pc, const double *m, const int *alive, const double *x,
                             const double *rc, int n) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x, nthr = gridDim.x * blockDim.x, np = S.npad;
  for (int k = t; k < np * S.W; k += nthr) S.cbm[k] = 0u;
  if (t < S.W) S.rowany[t] = 0u;
  if (t < 4) S.flags[t] = 0;
  if (t < NCOUNTERS) S.counters[t] = 0;
  if (t == 0) *S.status = 0;
  if (t >= np) return;
  const int i = t;
  const bool in = i < n && alive[i];
  for (int c = 0; c < 3; ++c) {
    S.x[c * np + i] = in ? x[c * n + i] : (c == 0 ? PARK + 1.0e4 * i : 0.0);
    S.v[c * np + i] = 0.0;
  }
  const double mi = in ? m[i] : 0.0, r = in ? rc[i] : 0.0, tq = __dmul_rn(pc, r);
  S.m[i] = mi; S.gm[i] = G * mi;
  S.alive[i] = in ? 1 : 0;
  S.ccnt[i] = 0;
  S.rc[i] = r;
  S.T[i] = in ? dbits(__dmul_rn(tq, tq)) : 0ULL;
  S.rcsq[i] = in ? dbits(__dmul_rn(r, r)) : 0ULL;
  S.A[i] = dbits(r) != 0ULL ? rcp_refined(0.9 * r) : 0.0;
}

// kick work list: for tile I the diagonal item, then both halves of every J > I
__global__ void k_items(int *items, int nt) {
  const int I = threadIdx.x;
  if (I >= nt) return;
  int k = I * (2 * nt - I);
  items[k++] = I | (I << 10);
  for (int J = I + 1; J < nt; ++J) {
    items[k++] = I | (J << 10);
    items[k++] = I | (J << 10) | (1 << 20);
  }
}

}  // namespace

extern "C" int genga_kick_noalloc(int n, double G, double pc, int kmode, int precise_div, const double *m,
                                  const int *alive, const double *x, const double *rc, double *a, int *cand,
                                  int cap, int *ncand, void *stream) {
  if (n > NA_NMAX) return GENGA_ESIZE;
  if (n < 1 || !m || !alive || !x || !rc || !a || !ncand || cap < 0 || (cap > 0 && !cand) || !(G > 0.0) ||
      !(pc >= 1.0) || (kmode != 0 && kmode != 1))
    return GENGA_EINVAL;
  unsigned char *base = nullptr;
  int rc0 = scratch_address(&base);
  if (rc0 != GENGA_OK) return rc0;
  cudaStream_t st = (cudaStream_t)stream;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return GENGA_ECUDA;

  Sim S;
  memset(&S, 0, sizeof(S));
  S.n = n;
  S.npad = ((n + 31) / 32) * 32;
  S.nt = S.npad / 32;
  S.W = S.npad / 32;
  S.x = (double *)(base + O_X); S.v = (double *)(base + O_V);
  S.m = (double *)(base + O_M); S.gm = (double *)(base + O_GM); S.rc = (double *)(base + O_RC); S.A = (double *)(base + O_A);
  S.alive = (int *)(base + O_ALIVE); S.T = (u64 *)(base + O_T); S.rcsq = (u64 *)(base + O_RCSQ);
  S.afar = (double *)(base + O_AFAR); S.part = (double *)(base + O_PART);
  S.pkick = (double *)(base + O_PKICK); S.pfin = (double *)(base + O_PFIN);
  S.cbm = (unsigned *)(base + O_CBM); S.rowany = (unsigned *)(base + O_ROWANY);
  S.ccnt = (int *)(base + O_CCNT); S.clist = (int *)(base + O_CLIST);
  S.items = (int *)(base + O_ITEMS);
  S.nitems = S.nt * S.nt;
  S.nwarps = S.nitems < 8 * sms ? S.nitems : 8 * sms;  // the allocating kick's configuration
  kick_split(S.npad, sms, &S.kch, &S.kchunk);
  S.flags = (int *)(base + O_FLAGS); S.status = (int *)(base + O_STATUS);
  S.counters = (long long *)(base + O_COUNTERS);

  genga_params prm;
  genga_default_params(&prm);
  prm.pc = pc;
  prm.kmode = kmode;
  DevParams P;
  memset(&P, 0, sizeof(P));
  P.G = G; P.m0 = 1.0; P.Gm0 = G; P.inv_m0 = 1.0; P.mu2 = 2.0 * G; P.inv_mu = 1.0 / G;
  P.n1 = prm.n1; P.n2 = prm.n2; P.pc = prm.pc; P.bs_eps = prm.bs_eps; P.bs_kmax = prm.bs_kmax;
  P.bs_max_halvings = prm.bs_max_halvings; P.kepler_maxit = prm.kepler_maxit; P.kmode = kmode;
  P.collisions = prm.collisions;

  if (precise_div) k_items<<<1, 32, 0, st>>>(S.items, S.nt);
  // 8 threads a body: the bitmap's words, up to 32 a body, are most of what there is to clear
  k_kick_setup<<<(8 * S.npad + 127) / 128, 128, 0, st>>>(S, G, pc, m, alive, x, rc, n);
  launch_kick_init(S, P, precise_div != 0, a, n, st, true);
  launch_bitmap_pairs(S.cbm, S.rowany, S.npad, S.W, cand, cap, ncand, st, true);
  return cudaGetLastError() == cudaSuccess ? GENGA_OK : GENGA_ECUDA;
}
