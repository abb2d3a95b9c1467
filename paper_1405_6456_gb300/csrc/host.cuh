// Host-side infrastructure shared by the translation units of the library:
// the context (device workspaces, reduction scratch, trace counters), error
// handling, stencil weights of Sec. 4, and kernel launch configuration.
#pragma once
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <functional>
#include <new>
#include <string>
#include <thread>
#include <type_traits>
#include <vector>

#include "../../include/ofdft.h"
#include "fastdiag.cuh"
#include "kernels.cuh"


// ----------------------------------------------------------------- context --
struct DevBuf {
  void* p = nullptr;
  size_t bytes = 0;
};

using ofd::CgScalars;

// Eigenvectors and eigenvalues of one axis of the fast diagonalisation (node
// count n, stencil radius R, spacing 1), kept for the context's lifetime.
struct FdTable {
  int n = 0, R = 0;
  void* dev = nullptr;
  ofd::FdAxis ax;
  const float *mu = nullptr, *mul = nullptr;  // eigenvalues, even modes first
  const float *mx = nullptr, *mxl = nullptr;  // ... in the order of a scratch row
};

struct ofdft_ctx {
  int device = 0;
  cudaStream_t stream = nullptr;
  std::string err;
  int sms = 152;
  // reduction scratch
  DevBuf partials;
  unsigned int* counter = nullptr;
  // small device scalars: CG scalars (2 sets), functional outputs, dot outputs
  CgScalars* sc = nullptr;
  CgScalars* sc32 = nullptr;
  double* scal = nullptr;  // 64 doubles
  double* host_scal = nullptr;  // pinned mirror
  // named vector workspaces
  DevBuf v[32];
  // launch counters and optional CUDA-event timing of every launch
  long long launches = 0;
  long long kind_launches[OFDFT_K_COUNT] = {0};
  long long timed_launches[OFDFT_K_COUNT] = {0};
  double timed_ms[OFDFT_K_COUNT] = {0};
  int prof = 0;
  struct Pending {
    cudaEvent_t a, b;
    int kind;
  };
  std::vector<Pending> pending;
  std::vector<cudaEvent_t> free_events;
  // pinned double buffer for polling CG flags without draining the stream
  CgScalars* ring = nullptr;
  cudaEvent_t ring_ev[2] = {nullptr, nullptr};
  // CUDA graphs of a chunk of CG iterations, keyed by everything they bake in
  struct GraphEntry {
    std::vector<long long> key;
    cudaGraphExec_t exec = nullptr;
  };
  std::vector<GraphEntry> graphs;
  int use_graphs = 1;
  cudaStream_t gstream = nullptr;  // private stream used only to capture graphs
  cudaEvent_t gev[2][2] = {{nullptr, nullptr}, {nullptr, nullptr}};  // sampling events recorded by CG graphs
  // autotuned z-splits of the z-streaming passes: key -> number of z chunks
  std::vector<std::pair<std::vector<long long>, int>> ztune;
  std::vector<std::vector<long long>> ztuned;  // (type, radius, grid, 16-byte staging) already tuned
  std::vector<long long> last_zkey;            // key of the last z-streaming launch
  int force_nz = -1;                           // >= 0: z-split of the next launches (autotuner)
  int pw_per_sm = 4;                           // blocks per SM of the pointwise passes
  int coop = 0;                                // persistent cooperative CG iterations (opt-in)
  unsigned int* coop_bar = nullptr;            // arrival counter of its grid barriers
  long long coop_iters = 0;                    // CG iterations run by it (trace counter)
  long long tma_launches = 0;                  // z-streaming passes staged by TMA (trace counter)
  int coop_nz = 0;                             // z-chunks of its grid (0: the default rule)
  int precond = 1;                             // Poisson CG preconditioner (OFDFT_PRECOND_*)
  int trace = 0;                               // OFDFT_TRACE=1: diagnostic lines on stderr
  double mg_omega = 0.9;                       // multigrid Jacobi weight (0 < omega < 1)
  int mg_sweeps = 20;                          // Jacobi sweeps on the multigrid bottom level
  DevBuf mgbuf;                                // multigrid levels below the finest
  int autotune = 1;
  double cg_fold_bytes = 96.0 * (1 << 20);     // fold the CG iterate update above this CG working set
  long long mg_fuse_nodes = -1;                // multigrid levels of at least this many nodes: two fused launches (-1: none)
  int ff_residual = 1;                         // mixed residual pass in float-float (else FP64)
  int cond_graphs = 1;                         // CG loops as one graph with a device-side WHILE node
  int mixed_ff = 0;                            // the last mixed Poisson solve ran the float-float residual pass
  int tma = 0;                                 // FP32 z-streaming passes stage planes by TMA where they can
  int pdl = 0;                                 // programmatic dependent launch for the CG-loop kernels
  int mg_finest_smooth = 1;                    // damped-Jacobi smoothing on the finest multigrid level
  long long mg_fuse_below = -1;                // coarser multigrid levels of at most this many nodes: fused
  int mg_cluster = 0;                          // coarse levels on one thread-block cluster (mg_cluster_kernel)
  int func_split_dots = 0;                     // G.d and G.s_old by a pass after the functional
  int mg_zstream = 0;                          // level smoothing passes as z-streaming radius-1 stencils
  long long mg_zstream_nodes = -1;             // ... on the levels of at least this many nodes (-1: none)
  int fd = 1;                                  // fast diagonalisation on the grids it covers (else V-cycles)
  std::vector<FdTable> fdtab;                  // its axis tables
  // the b_J tables in V_BTAB belong to this geometry (atoms, charges, grid,
  // sigma, r_c, stencil radius); empty: none kept
  std::vector<double> btab_key;
};

namespace ofd {

enum Vec {
  V_R = 0, V_P0, V_P1, V_AP,           // CG vectors (prec type)
  V_R64, V_PHI64, V_B64, V_E32,        // mixed refinement (FP64 r, phi, b; FP32 correction)
  V_U, V_UT, V_PHI, V_B,               // solve state
  V_G, V_GT, V_S, V_ST, V_SN, V_D,     // NLCG vectors
  V_ATOM0, V_ATOM1, V_ATOM2,           // atom scratch
  V_W,                                 // u / Jacobi diagonal (rank-one preconditioner)
  V_PHI0,                              // FP64 potential at the origin of the current line search
  V_Z, V_T,                            // PCG: z = M r and the multigrid's finest-level scratch
  V_PHI2,                              // mixed: the FP64 potential as float-float pairs (residual pass)
  V_BACC,                              // FP64 running sums of the pseudocharge over atom ranges
  V_B2,                                // mixed: the FP64 pseudocharge as float-float pairs (residual pass)
  V_BTAB,                              // b_J tables of every atom, kept from the pseudocharge for the forces
  V_OC,                                // overlap correction: b, b~, V, V~ (FP64)
  V_GTAB,                              // coefficients of the nuclear potential (gtab_v)
  V_COUNT
};

inline int fail(ofdft_ctx* c, int code, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  if (c) c->err = buf;
  return code;
}

#define CU(call)                                                                   \
  do {                                                                             \
    cudaError_t e_ = (call);                                                       \
    if (e_ != cudaSuccess)                                                         \
      return fail(c, e_ == cudaErrorMemoryAllocation ? OFDFT_ENOMEM : OFDFT_ECUDA, \
                  "%s: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, __LINE__); \
  } while (0)

#define TRY(expr)            \
  do {                       \
    int rc_ = (expr);        \
    if (rc_ != OFDFT_OK) return rc_; \
  } while (0)

inline int ensure(ofdft_ctx* c, DevBuf& b, size_t bytes) {
  if (b.bytes >= bytes && b.p) return OFDFT_OK;
  if (b.p) {
    CU(cudaStreamSynchronize(c->stream));
    CU(cudaFree(b.p));
    b.p = nullptr;
    b.bytes = 0;
  }
  const size_t want = std::max<size_t>(bytes, 256);
  CU(cudaMalloc(&b.p, want));
  b.bytes = want;
  return OFDFT_OK;
}

template <typename T>
T* vec(ofdft_ctx* c, int which) {
  return static_cast<T*>(c->v[which].p);
}

inline cudaEvent_t take_event(ofdft_ctx* c) {
  if (!c->free_events.empty()) {
    cudaEvent_t e = c->free_events.back();
    c->free_events.pop_back();
    return e;
  }
  cudaEvent_t e = nullptr;
  if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
  return e;
}

// Folds the durations of completed timed launches into the totals (call after
// the stream has been synchronised) and recycles their events.
inline void harvest(ofdft_ctx* c) {
  for (auto& p : c->pending) {
    float ms = 0.0f;
    if (cudaEventElapsedTime(&ms, p.a, p.b) == cudaSuccess) {
      c->timed_ms[p.kind] += ms;
      c->timed_launches[p.kind] += 1;
    }
    c->free_events.push_back(p.a);
    c->free_events.push_back(p.b);
  }
  c->pending.clear();
}

// Counts a kernel launch of `kind`; with profiling on, brackets it with events.
struct ProfScope {
  ofdft_ctx* c;
  int kind;
  cudaEvent_t a = nullptr, b = nullptr;
  ProfScope(ofdft_ctx* c_, int k) : c(c_), kind(k) {
    c->launches++;
    c->kind_launches[k]++;
    if (c->prof & (1 << k)) {
      a = take_event(c);
      b = take_event(c);
      if (a && b) cudaEventRecord(a, c->stream);
    }
  }
  ~ProfScope() {
    if (a && b) {
      cudaEventRecord(b, c->stream);
      c->pending.push_back({a, b, kind});
      if (c->pending.size() > 4096) {
        cudaEventSynchronize(b);
        harvest(c);
      }
    }
  }
};

inline RedBuf red(ofdft_ctx* c) { return RedBuf{static_cast<double*>(c->partials.p), c->counter}; }

inline int ensure_partials(ofdft_ctx* c, long long nblocks, int K) {
  return ensure(c, c->partials, (size_t)nblocks * K * sizeof(double) + 64);
}

inline GridDev gdev(const ofdft_grid* g) {
  GridDev d;
  d.n1 = g->n[0];
  d.n2 = g->n[1];
  d.n3 = g->n[2];
  d.G = (long long)d.n1 * d.n2 * d.n3;
  return d;
}

inline int check_grid(ofdft_ctx* c, const ofdft_grid* g) {
  if (!g) return fail(c, OFDFT_EINVAL, "grid is NULL");
  for (int d = 0; d < 3; ++d)
    if (g->n[d] < 1 || g->n[d] > (1 << 16)) return fail(c, OFDFT_EINVAL, "grid dimension %d is %d", d, g->n[d]);
  if (!(g->h > 0.0) || !isfinite(g->h)) return fail(c, OFDFT_EINVAL, "grid spacing must be positive");
  // the stencil kernels hold in-plane offsets in 32 bits
  if ((long long)g->n[0] * (g->n[1] + 2 * kMaxR) >= (1LL << 31))
    return fail(c, OFDFT_EINVAL, "grid plane of %d x %d nodes is too large", g->n[0], g->n[1]);
  return OFDFT_OK;
}

inline int check_order(ofdft_ctx* c, int fd_order) {
  if (fd_order < 2 || fd_order > 2 * kMaxR || (fd_order & 1))
    return fail(c, OFDFT_EINVAL, "fd_order must be even in [2, %d], got %d", 2 * kMaxR, fd_order);
  return OFDFT_OK;
}

inline int check_prec(ofdft_ctx* c, int prec) {
  if (prec != OFDFT_PREC_FP64 && prec != OFDFT_PREC_MIXED)
    return fail(c, OFDFT_EINVAL, "precision must be OFDFT_PREC_FP64 or OFDFT_PREC_MIXED");
  return OFDFT_OK;
}

// Laplacian weights of Sec. 4 (Eq. FD:Laplacian) in FP64, scaled by `scale`;
// c = 6 w_0 (the p = 0 term counts the centre six times).
inline Weights<double> lap_weights(int R, double h, double scale) {
  Weights<double> W;
  memset(&W, 0, sizeof(W));
  double s = 0.0;
  for (int q = 1; q <= R; ++q) s += 1.0 / ((double)q * q);
  W.c = scale * 6.0 * (-s / (h * h));
  // (R!)^2 / ((R-p)! (R+p)!) as a running product
  for (int p = 1; p <= R; ++p) {
    double ratio = 1.0;
    for (int i = 1; i <= p; ++i) ratio *= (double)(R - p + i) / (double)(R + i);
    const double sign = (p & 1) ? 1.0 : -1.0;
    W.w[p] = scale * 2.0 * sign * ratio / (h * h * (double)p * p);
  }
  return W;
}

// Gradient weights of Sec. 4: w~_p = (-1)^{p+1} (R!)^2 / (h p (R-p)! (R+p)!).
inline Weights<double> grad_weights(int R, double h) {
  Weights<double> W;
  memset(&W, 0, sizeof(W));
  for (int p = 1; p <= R; ++p) {
    double ratio = 1.0;
    for (int i = 1; i <= p; ++i) ratio *= (double)(R - p + i) / (double)(R + i);
    const double sign = (p & 1) ? 1.0 : -1.0;
    W.w[p] = sign * ratio / (h * (double)p);
  }
  return W;
}

template <typename T>
Weights<T> cast_weights(const Weights<double>& W) {
  Weights<T> o;
  o.c = (T)W.c;
  for (int p = 0; p <= kMaxR; ++p) o.w[p] = (T)W.w[p];
  return o;
}
// float-float weights: hi = nearest float, lo = nearest float of the remainder
inline float2 ff_of(double v) {
  const float hi = (float)v;
  return make_float2(hi, (float)(v - (double)hi));
}
template <>
inline Weights<float2> cast_weights<float2>(const Weights<double>& W) {
  Weights<float2> o;
  o.c = ff_of(W.c);
  for (int p = 0; p <= kMaxR; ++p) o.w[p] = ff_of(W.w[p]);
  return o;
}

inline int pointwise_blocks(ofdft_ctx* c, long long G) {
  long long b = (G + 1023) / 1024;
  return (int)std::max<long long>(1, std::min<long long>(b, (long long)c->sms * c->pw_per_sm));
}

// Poisson tolerance inside a solve's NLCG at a point with h^3 r.s = rs (see
// ofdft_params.poisson_adapt): the gradient's error from an inexact potential
// only has to stay small against the gradient itself.
inline double adaptive_poisson_tol(const ofdft_params* p, double rs, int M) {
  if (!(p->poisson_adapt > 0.0) || !(rs > 0.0) || !isfinite(rs)) return p->tol_poisson;
  const double t = p->poisson_adapt * p->tol_poisson * sqrt(rs / (p->tol_inner * M));
  return std::max(p->tol_poisson, std::min(1e-4, t));
}

// Poisson tolerance of a secant trial point (ofdft_params.trial_poisson_loosen).
inline double trial_poisson_tol(const ofdft_params* p, double tol) {
  if (!(p->trial_poisson_loosen > 1.0)) return tol;
  return std::max(tol, std::min(1e-4, tol * p->trial_poisson_loosen));
}

// Resolution of L in a MIXED evaluation: the FP32 energy densities (TF, vW
// with the FP32 stencil, XC) carry rounding noise that measured about 1e-9 of the
// summed magnitudes of the energy terms on the 666-atom cluster; a secant step
// whose L rises by less than that is not a rise the evaluation can resolve.
// FP64 evaluations resolve far below any step the NLCG takes: 0.
inline double l_resolution(const ofdft_energy& e, bool mixed) {
  if (!mixed) return 0.0;
  return 1e-9 * (fabs(e.E_tf) + fabs(e.E_vw) + fabs(e.E_xc) + fabs(e.E_es));
}

// Relative tolerance of one FP32 round of the mixed Poisson CG: cut the FP32
// residual by 1e-4 (the reduction FP32 recurrences track faithfully), but not
// below half of what the FP64 stopping test still asks for (||r|| <= tol ||b||),
// so that the last round does not over-solve.  rr = ||r64||^2, bb = ||b||^2.
inline double mixed_inner_tol(double rr, double bb, double tol) {
  const double want = (rr > 0.0) ? 0.5 * tol * sqrt(bb / rr) : 1e-4;
  return std::max(1e-4, std::min(want, 0.5));
}

// z-streaming launch shape: tiles of columns times chunks of z planes.
struct ZShape {
  dim3 grid;
  int zchunk;
  long long nblocks;
};

template <typename T>
ZShape zshape(ofdft_ctx* c, const GridDev& g, int blocks_per_sm = 2, int force_nz = 0) {
  ZShape s;
  const int gx = (g.n1 + BX - 1) / BX, gy = (g.n2 + ZCfg<T>::TY - 1) / ZCfg<T>::TY;
  const long long tiles = (long long)gx * gy;
  const int per_sm = std::max(blocks_per_sm, 1);
  int best = 1;
  if (force_nz > 0) {
    best = std::min(force_nz, g.n3);
  } else {
    // a block's chunk of zc planes costs zc + c0 plane times, k blocks on an SM
    // slow each other down to 1 + a (k - 1) of that: FP64 passes share a pipe that
    // one block fills (a = 0.95, c0 = 0.7), FP32 and float-float ones mostly wait
    // (a = 0.45, c0 = 2.3).  Fitted to sweeps of 1 to 64 chunks on 48^3 to 192^3;
    // the chosen split is within 4% of the best measured one; one wave in chunks of at
    // least 2 R planes is 10 to 75% slower below 160^3 (functional, us, that | this:
    // FP64 48^3 245 | 61, 80^3 283 | 173; FP32 64^3 68 | 33, 128^3 92 | 71) and the same
    // above.
    const double a = sizeof(T) == 8 && std::is_same<T, double>::value ? 0.95 : 0.45;
    const double c0 = std::is_same<T, double>::value ? 0.7 : 2.3;
    double least = 1e300;
    for (int zc = g.n3; zc >= 1; --zc) {
      const int nz = (g.n3 + zc - 1) / zc;
      const long long blocks = tiles * nz, wave = (long long)c->sms * per_sm;
      const long long last = blocks % wave;
      double cost = (double)(blocks / wave) * (1.0 + a * (per_sm - 1));
      if (last) cost += 1.0 + a * (double)((last + c->sms - 1) / c->sms - 1);
      cost *= zc + c0;
      if (cost < least * (1.0 - 1e-9)) {
        least = cost;
        best = nz;
      }
    }
  }
  const int zc = (g.n3 + best - 1) / best;
  const int nz = (g.n3 + zc - 1) / zc;
  s.grid = dim3(gx, gy, nz);
  s.zchunk = zc;
  s.nblocks = tiles * nz;
  return s;
}

// Key of an autotuned z-split: the kernel instantiation and the grid.
inline std::vector<long long> ztune_key(const void* fn, const GridDev& g) {
  return {(long long)(uintptr_t)fn, g.n1, g.n2, g.n3};
}

// True when a pass can stage 16-byte copies: rows of a whole number of copies
// (n1 % (16 / sizeof(T)) == 0) and 16-byte aligned stencil and epilogue inputs.
template <typename T, class L, class E>
bool zvec_ok(const GridDev& g, const L& ld, const E& ep) {
  if (g.n1 % (16 / (int)sizeof(T))) return false;
  auto aligned = [](const void* p) { return ((uintptr_t)p & 15u) == 0; };
  if (!aligned(ld.f)) return false;
  for (int j = 0; j < E::NIN; ++j)
    if (ep.input(j) && !aligned(ep.input(j))) return false;
  return true;
}

// Fast diagonalisation of one grid (kernels and the method: fastdiag.cuh).
struct FdPlan {
  bool on = false;
  FdAxis ax[3];                       // x, y, z
  const float *mu[3], *mul[3];        // eigenvalues of h^2 T, high and low parts
  int pitch = 0;                      // floats of a scratch row
  double h2 = 0.0;                    // h^2
};

// Multigrid preconditioner of the Poisson CG (S3): the levels of a grid (kernels
// and the cycle's steps: mg_* in kernels.cuh).
constexpr int kMgCoarseNodes = 4096;  // levels from this size down run in one block
constexpr int kMgSweeps = 20;         // Jacobi sweeps from zero on the bottom level
constexpr double kMgOmega = 0.9;      // Jacobi weight (the cycle is SPD for 0 < omega < 1)

struct MgPlan {
  int nlev = 0;  // levels from the grid itself down to the bottom (smallest extent below 4)
  int lc = -1;   // first level handled by the one-block kernel
  MgLevel d[kMgMaxLevels];
  long long off[kMgMaxLevels] = {0};  // element offset of level l's r, z, t (l = 1 .. lc) in mgbuf
  long long elems = 0;                // mgbuf elements
  size_t smem = 0;                    // shared memory of the one-block kernel
  double s0 = 0.0;                    // omega h^2 / 6 of the finest level
  bool ok = false;
  // the cluster end (mg_cluster_kernel): levels lq .. lc-1 in the distributed
  // shared memory of one thread-block cluster (lq < 0: none fits)
  int lq = -1;
  MgSlab slab[kMgMaxLevels];
  size_t csmem = 0;       // dynamic shared memory per block of the cluster kernel
  unsigned tail_off = 0;  // byte offset of block 0's coarse-end arrays
  FdPlan fd;              // fd.on: z = M r by fast diagonalisation instead of the cycle
};
constexpr size_t kMgClusterSmem = 220 * 1024;  // dynamic shared memory per cluster block (of 227 KB)

inline long long mg_nodes(const MgLevel& d) { return (long long)d.n1 * d.n2 * d.n3; }

inline MgPlan mg_plan(const GridDev& g, double h, size_t es, double omega = kMgOmega) {
  MgPlan P;
  MgLevel d{g.n1, g.n2, g.n3};
  P.d[0] = d;
  P.nlev = 1;
  while (std::min(d.n1, std::min(d.n2, d.n3)) >= 4 && P.nlev < kMgMaxLevels) {
    d = MgLevel{d.n1 / 2, d.n2 / 2, d.n3 / 2};
    P.d[P.nlev++] = d;
  }
  for (int l = 0; l < P.nlev; ++l)
    if (mg_nodes(P.d[l]) <= kMgCoarseNodes) {
      P.lc = l;
      break;
    }
  if (P.lc < 0) return P;  // the bottom level is too large for one block: plain CG
  if (mg_nodes(P.d[0]) >= (1LL << 31)) return P;  // the level kernels index with 32-bit integers
  long long e = 0;
  for (int l = 1; l <= P.lc; ++l) {
    P.off[l] = e;
    e += 3 * mg_nodes(P.d[l]);
  }
  P.elems = e;
  size_t sm = 0;
  for (int l = P.lc; l < P.nlev; ++l) sm += 3 * (size_t)mg_nodes(P.d[l]) * es;
  P.smem = sm;
  P.s0 = omega * h * h / 6.0;
  P.ok = sm <= 200 * 1024;
  if (!P.ok) return P;
  // the cluster end: the most levels above lc (level 0 excluded: its pass forms
  // r.z) whose z-plane slabs, with the coarse end's arrays in block 0, fit
  for (int lq = 1; lq < P.lc && P.lq < 0; ++lq) {
    size_t off = 0;  // bytes
    for (int l = lq; l < P.lc; ++l) {
      const MgLevel& d = P.d[l];
      const int pl = (d.n3 + kMgClusterCtas - 1) / kMgClusterCtas;
      P.slab[l] = MgSlab{d, pl, (unsigned)(off / es)};
      off += ((3 * (size_t)pl * d.n1 * d.n2 * es + 15) / 16) * 16;
    }
    P.slab[P.lc] = MgSlab{P.d[P.lc], 0, 0};
    if (off + sm <= kMgClusterSmem) {
      P.lq = lq;
      P.tail_off = (unsigned)off;
      P.csmem = off + sm;
    }
  }
  return P;
}

// Launches kern on the context's stream.  With c->pdl the launch allows
// programmatic dependent launch: the grid may be scheduled while the previous
// kernel of the stream is still finishing, and holds at pdl_wait() (the first
// statement of every kernel launched here) until that kernel has completed and
// its writes are visible; the previous kernel releases it early with
// pdl_launch_dependents().  Only the launch latency overlaps, never the work.
template <typename... KArgs, typename... Args>
cudaError_t launch_k(ofdft_ctx* c, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, Args... args) {
  if (c->pdl) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = c->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
  }
  kern<<<grid, block, smem, c->stream>>>(args...);
  return cudaGetLastError();
}

// ------------------------------------------------------ fast diagonalisation --
// Eigenpairs of a symmetric m x m matrix a (row-major, destroyed): Householder
// tridiagonalisation and the implicit symmetric QR iteration with Wilkinson's
// shift (Golub and Van Loan, Matrix Computations, sec. 8.3).  On return d holds
// the eigenvalues and row k of v the eigenvector of d[k].  Returns false when an
// eigenvalue does not settle.
inline bool sym_eigen(int m, std::vector<double>& a, std::vector<double>& d, std::vector<double>& v) {
  d.assign(m, 0.0);
  v.assign((size_t)m * m, 0.0);
  for (int i = 0; i < m; ++i) v[(size_t)i * m + i] = 1.0;
  std::vector<double> e(m, 0.0), h(m), p(m);
  for (int k = 0; k + 2 < m; ++k) {  // reflect column k below the subdiagonal away
    double nrm = 0.0;
    for (int i = k + 1; i < m; ++i) nrm += a[(size_t)i * m + k] * a[(size_t)i * m + k];
    nrm = sqrt(nrm);
    if (nrm == 0.0) continue;
    const double x0 = a[(size_t)(k + 1) * m + k], al = x0 > 0.0 ? -nrm : nrm;
    for (int i = k + 1; i < m; ++i) h[i] = a[(size_t)i * m + k];
    h[k + 1] -= al;
    double hh = 0.0;
    for (int i = k + 1; i < m; ++i) hh += h[i] * h[i];
    const double be = 2.0 / hh;
    double hp = 0.0;
    for (int i = k + 1; i < m; ++i) {
      double t = 0.0;
      for (int j = k + 1; j < m; ++j) t += a[(size_t)i * m + j] * h[j];
      p[i] = be * t;
      hp += h[i] * p[i];
    }
    for (int i = k + 1; i < m; ++i) p[i] -= 0.5 * be * hp * h[i];
    for (int i = k + 1; i < m; ++i)
      for (int j = k + 1; j < m; ++j) a[(size_t)i * m + j] -= h[i] * p[j] + p[i] * h[j];
    a[(size_t)(k + 1) * m + k] = a[(size_t)k * m + k + 1] = al;
    std::fill(p.begin(), p.end(), 0.0);  // v = (I - be h h^T) v
    for (int i = k + 1; i < m; ++i)
      for (int j = 0; j < m; ++j) p[j] += h[i] * v[(size_t)i * m + j];
    for (int i = k + 1; i < m; ++i)
      for (int j = 0; j < m; ++j) v[(size_t)i * m + j] -= be * h[i] * p[j];
  }
  for (int i = 0; i < m; ++i) {
    d[i] = a[(size_t)i * m + i];
    if (i + 1 < m) e[i] = a[(size_t)(i + 1) * m + i];
  }
  int hi = m - 1, its = 0;
  while (hi > 0) {
    for (int k = 0; k < hi; ++k)
      if (fabs(e[k]) <= 1.2e-16 * (fabs(d[k]) + fabs(d[k + 1]))) e[k] = 0.0;
    if (e[hi - 1] == 0.0) {
      --hi;
      its = 0;
      continue;
    }
    if (++its > 80) return false;
    int lo = hi - 1;
    while (lo > 0 && e[lo - 1] != 0.0) --lo;
    const double g = 0.5 * (d[hi - 1] - d[hi]), q = e[hi - 1];
    const double den = g + (g >= 0.0 ? 1.0 : -1.0) * hypot(g, q);
    const double mu = d[hi] - q * q / den;
    double x = d[lo] - mu, z = e[lo];
    for (int k = lo; k < hi; ++k) {  // chase the bulge with plane rotations
      const double r = hypot(x, z);
      const double cs = r > 0.0 ? x / r : 1.0, sn = r > 0.0 ? z / r : 0.0;
      if (k > lo) e[k - 1] = r;
      const double dk = d[k], dn = d[k + 1], ek = e[k];
      d[k] = cs * cs * dk + 2.0 * cs * sn * ek + sn * sn * dn;
      d[k + 1] = sn * sn * dk - 2.0 * cs * sn * ek + cs * cs * dn;
      e[k] = (cs * cs - sn * sn) * ek + cs * sn * (dn - dk);
      if (k + 1 < hi) {
        x = e[k];
        z = sn * e[k + 1];
        e[k + 1] *= cs;
      }
      double* v0 = &v[(size_t)k * m];
      double* v1 = v0 + m;
      for (int j = 0; j < m; ++j) {
        const double t = v0[j];
        v0[j] = cs * t + sn * v1[j];
        v1[j] = cs * v1[j] - sn * t;
      }
    }
  }
  return true;
}

// fn(0) .. fn(n - 1) on up to eight threads; what threads cannot be had for runs here.
template <class Fn>
void host_parallel(int n, Fn fn) {
  std::atomic<int> next{0};
  auto work = [&]() {
    for (int i = next.fetch_add(1); i < n; i = next.fetch_add(1)) fn(i);
  };
  std::vector<std::thread> ts;
  try {
    const int nt = std::min(n, (int)std::min(8u, std::thread::hardware_concurrency())) - 1;
    ts.reserve(std::max(nt, 0));
    for (int k = 0; k < nt; ++k) ts.emplace_back(work);
  } catch (...) {
  }
  work();
  for (std::thread& t : ts) t.join();
}

// The same for a matrix of half-bandwidth b, whose lower band a[j (b + 2) + i - j]
// holds (i - j <= b; the last place is for the bulge): plane rotations reduce the band
// to a tridiagonal matrix (Schwarz 1968), and the same iteration diagonalises that.
// The rotations are only recorded, as runs on consecutive rows; rotate() then applies
// them to the identity, eight columns at a time in cache and on several threads, which
// is most of the work: 6 m operations for each of about 1.4 m^2 rotations.  512 nodes
// in 5 ms where sym_eigen takes 29, 400 in 2.7 against 13.5 (Grace, 8 threads).
struct BandEigen {
  struct Run {
    int row, n;
    size_t at;
  };
  int m = 0;
  std::vector<double> a, d;
  std::vector<Run> runs;
  std::vector<double> cs, sn;
  bool ok = false;

  void turn(int row, double c, double s, bool joins) {
    if (!joins || runs.empty()) runs.push_back(Run{row, 0, cs.size()});
    ++runs.back().n;
    cs.push_back(c);
    sn.push_back(s);
  }

  void tridiagonal(int b) {
    const int w = b + 2;
    auto L = [&](int i, int j) -> double& { return a[(size_t)j * w + (i - j)]; };
    for (int k = 0; k + 2 < m; ++k)
      for (int p = std::min(b, m - 1 - k); p >= 2; --p)
        for (int col = k, i = k + p - 1; i + 1 < m; col = i, i += b) {  // rows i, i + 1 clear (i + 1, col)
          const double x = L(i, col), y = L(i + 1, col);
          if (y == 0.0) break;
          const double r = sqrt(x * x + y * y), c = x / r, s = y / r;
          L(i, col) = r;
          L(i + 1, col) = 0.0;
          for (int j = col + 1; j < i; ++j) {
            const double u = L(i, j), v = L(i + 1, j);
            L(i, j) = c * u + s * v;
            L(i + 1, j) = c * v - s * u;
          }
          const double p0 = L(i, i), q = L(i + 1, i), p1 = L(i + 1, i + 1);
          L(i, i) = c * c * p0 + 2.0 * c * s * q + s * s * p1;
          L(i + 1, i + 1) = s * s * p0 - 2.0 * c * s * q + c * c * p1;
          L(i + 1, i) = (c * c - s * s) * q + c * s * (p1 - p0);
          for (int j = i + 2; j <= std::min(m - 1, i + 1 + b); ++j) {
            const double u = j - i <= b ? L(j, i) : 0.0, v = L(j, i + 1);
            L(j, i) = c * u + s * v;  // (j = i + 1 + b: the bulge, cleared next)
            L(j, i + 1) = c * v - s * u;
          }
          turn(i, c, s, false);
        }
  }

  // a as above; false when an eigenvalue does not settle
  bool solve(int m_, int b, std::vector<double>& band) {
    m = m_;
    a.swap(band);
    tridiagonal(b);
    d.assign(m, 0.0);
    std::vector<double> e(m, 0.0);
    for (int i = 0; i < m; ++i) {
      d[i] = a[(size_t)i * (b + 2)];
      if (i + 1 < m) e[i] = a[(size_t)i * (b + 2) + 1];
    }
    int hi = m - 1, its = 0;
    while (hi > 0) {
      for (int k = 0; k < hi; ++k)
        if (fabs(e[k]) <= 1.2e-16 * (fabs(d[k]) + fabs(d[k + 1]))) e[k] = 0.0;
      if (e[hi - 1] == 0.0) {
        --hi;
        its = 0;
        continue;
      }
      if (++its > 80) return false;
      int lo = hi - 1;
      while (lo > 0 && e[lo - 1] != 0.0) --lo;
      const double g = 0.5 * (d[hi - 1] - d[hi]), q = e[hi - 1];
      const double den = g + (g >= 0.0 ? 1.0 : -1.0) * hypot(g, q);
      const double mu = d[hi] - q * q / den;
      double x = d[lo] - mu, z = e[lo];
      for (int k = lo; k < hi; ++k) {  // chase the bulge with plane rotations
        const double r = sqrt(x * x + z * z);
        const double c = r > 0.0 ? x / r : 1.0, s = r > 0.0 ? z / r : 0.0;
        if (k > lo) e[k - 1] = r;
        const double dk = d[k], dn = d[k + 1], ek = e[k];
        d[k] = c * c * dk + 2.0 * c * s * ek + s * s * dn;
        d[k + 1] = s * s * dk - 2.0 * c * s * ek + c * c * dn;
        e[k] = (c * c - s * s) * ek + c * s * (dn - dk);
        if (k + 1 < hi) {
          x = e[k];
          z = s * e[k + 1];
          e[k + 1] *= c;
        }
        turn(k, c, s, k > lo);
      }
    }
    return true;
  }

  // Columns [8 q, 8 q + 8) of v, whose row k becomes the eigenvector of d[k]; buf: 8 m doubles.
  void rotate(int q, double* buf, double* v) const {
    constexpr int W = 8;
    for (int i = 0; i < m * W; ++i) buf[i] = 0.0;
    for (int l = 0; l < W && q * W + l < m; ++l) buf[(size_t)(q * W + l) * W + l] = 1.0;
    for (const Run& run : runs) {
      double* p = buf + (size_t)run.row * W;
      double cur[W];
      for (int l = 0; l < W; ++l) cur[l] = p[l];
      for (int t = 0; t < run.n; ++t, p += W) {
        const double c = cs[run.at + t], s = sn[run.at + t];
        for (int l = 0; l < W; ++l) {
          const double nx = p[W + l];
          p[l] = c * cur[l] + s * nx;
          cur[l] = c * nx - s * cur[l];
        }
      }
      for (int l = 0; l < W; ++l) p[l] = cur[l];
    }
    for (int i = 0; i < m; ++i)
      for (int l = 0; l < W && q * W + l < m; ++l) v[(size_t)i * m + q * W + l] = buf[(size_t)i * W + l];
  }
};

// Axes up to this long take the dense eigenproblem: 0.6 ms at 128 nodes, 1.7 at 192,
// 3.8 at 256 in a context's first solve on such an axis.  Beyond, the banded one: with
// the dense one first solves on long thin grids took longer than they had with V-cycles
// (512 x 48 x 48 MIXED 31 ms against 7.0; 6.1 to 7.0 so).
constexpr int kFdDense = 256;

// The axis table of n nodes at stencil radius R, in host memory: `mat` holds
// forwards high, low, backwards high, low (each the even half's ne x pe and the
// odd half's no x po elements), `mu` the n eigenvalues at spacing 1 (even modes
// first).  The half problems: in the basis (delta_i +- delta_{n-1-i}) / sqrt 2
// (and the middle node of an odd axis) the Toeplitz matrix t(|i - j|) reads
// t(|i - j|) +- t(n - 1 - i - j).
inline bool fd_axis_host(int n, int R, FdAxis* ax, std::vector<float>* mat, std::vector<double>* mu) {
  ax->n = n;
  ax->ne = (n + 1) / 2;
  ax->no = n / 2;
  ax->pe = (ax->ne + kFdTile - 1) / kFdTile * kFdTile;
  ax->po = (ax->no + kFdTile - 1) / kFdTile * kFdTile;
  const size_t se = (size_t)ax->ne * ax->pe, so = (size_t)ax->no * ax->po, sz = se + so;
  mat->assign(4 * sz, 0.0f);
  mu->assign(n, 0.0);
  const Weights<double> W = lap_weights(R, 1.0, -1.0);
  auto t = [&](int q) { return q == 0 ? W.c / 3.0 : q <= R ? W.w[q] : 0.0; };
  const double r2 = sqrt(0.5);
  // element (i, j) of a half's matrix
  auto element = [&](int odd, int i, int j) {
    const int m = odd ? ax->no : ax->ne;
    const bool mid = !odd && (n & 1);
    const double x = t(abs(i - j)), y = t(n - 1 - i - j);
    const int mids = (mid && i == m - 1) + (mid && j == m - 1);
    if (mids == 1) return 2.0 * r2 * x;  // sqrt 2 t(|i - m|): both mirror images couple to the middle
    return mids ? x : x + (odd ? -y : y);
  };
  std::vector<double> d[2], v[2];
  if (n <= kFdDense) {
    for (int odd = 0; odd < 2; ++odd) {
      const int m = odd ? ax->no : ax->ne;
      std::vector<double> a((size_t)m * m);
      for (int i = 0; i < m; ++i)
        for (int j = 0; j < m; ++j) a[(size_t)i * m + j] = element(odd, i, j);
      if (!sym_eigen(m, a, d[odd], v[odd])) return false;
    }
  } else {
    BandEigen eig[2];
    std::vector<double> buf[2];
    host_parallel(2, [&](int odd) {
      const int m = odd ? ax->no : ax->ne, w = R + 2;
      try {
        std::vector<double> a((size_t)m * w, 0.0);
        for (int j = 0; j < m; ++j)
          for (int i = j; i < std::min(m, j + R + 1); ++i) a[(size_t)j * w + (i - j)] = element(odd, i, j);
        v[odd].resize((size_t)m * m);
        buf[odd].resize((size_t)(m + 7) / 8 * 8 * m);
        eig[odd].ok = eig[odd].solve(m, R, a);
      } catch (const std::bad_alloc&) {
        eig[odd].ok = false;
      }
    });
    if (!eig[0].ok || !eig[1].ok) return false;
    const int q0 = (ax->ne + 7) / 8, q1 = (ax->no + 7) / 8;
    host_parallel(q0 + q1, [&](int q) {
      const int odd = q >= q0, k = odd ? q - q0 : q;
      eig[odd].rotate(k, buf[odd].data() + (size_t)k * 8 * eig[odd].m, v[odd].data());
    });
    d[0].swap(eig[0].d);
    d[1].swap(eig[1].d);
  }
  for (int odd = 0; odd < 2; ++odd) {
    const int m = odd ? ax->no : ax->ne, wp = odd ? ax->po : ax->pe;
    const bool mid = !odd && (n & 1);
    for (int k = 0; k < m; ++k) (*mu)[(odd ? ax->ne : 0) + k] = d[odd][k];
    for (int k = 0; k < m; ++k)
      for (int i = 0; i < m; ++i) {
        const double x = v[odd][(size_t)k * m + i] * ((mid && i == m - 1) ? 1.0 : r2);
        const float h = (float)x, l = (float)(x - (double)h);
        const size_t f = (odd ? se : 0) + (size_t)i * wp + k, b = (odd ? se : 0) + (size_t)k * wp + i;
        (*mat)[f] = h;
        (*mat)[sz + f] = l;
        (*mat)[2 * sz + b] = h;
        (*mat)[3 * sz + b] = l;
      }
  }
  return true;
}

// The context's table for (n, R), built and copied to the device on first use.
inline int fd_table(ofdft_ctx* c, int n, int R, const FdTable** out) {
  for (const FdTable& t : c->fdtab)
    if (t.n == n && t.R == R) {
      *out = &t;
      return OFDFT_OK;
    }
  FdTable t;
  t.n = n;
  t.R = R;
  std::vector<float> mat;
  std::vector<double> mu;
  *out = nullptr;
  if (!fd_axis_host(n, R, &t.ax, &mat, &mu)) return OFDFT_OK;  // not settled: the caller keeps the V-cycle
  // the eigenvalues twice: in order (as the z axis uses them) and laid out as the
  // scratch rows are (x), where the padding's ones only ever divide zeros
  const size_t sz = mat.size() / 4, np = (size_t)n + 16;
  mat.resize(4 * sz + 4 * np, 1.0f);
  for (int k = 0; k < n; ++k) {
    const float h = (float)mu[k], l = (float)(mu[k] - (double)h);
    const size_t x = k < t.ax.ne ? k : fd_up4(t.ax.ne) + k - t.ax.ne;
    mat[4 * sz + k] = h;
    mat[4 * sz + np + k] = l;
    mat[4 * sz + 2 * np + x] = h;
    mat[4 * sz + 3 * np + x] = l;
  }
  CU(cudaMalloc(&t.dev, mat.size() * sizeof(float)));
  const cudaError_t e = cudaMemcpyAsync(t.dev, mat.data(), mat.size() * sizeof(float), cudaMemcpyHostToDevice, c->stream);
  if (e != cudaSuccess || cudaStreamSynchronize(c->stream) != cudaSuccess) {
    cudaFree(t.dev);
    return fail(c, OFDFT_ECUDA, "fast diagonalisation: copying an axis table failed");
  }
  const float* p = static_cast<const float*>(t.dev);
  t.ax.fwd = p;
  t.ax.fwdl = p + sz;
  t.ax.inv = p + 2 * sz;
  t.ax.invl = p + 3 * sz;
  t.mu = p + 4 * sz;
  t.mul = p + 4 * sz + np;
  t.mx = p + 4 * sz + 2 * np;
  t.mxl = p + 4 * sz + 3 * np;
  c->fdtab.push_back(t);
  *out = &c->fdtab.back();
  return OFDFT_OK;
}

// Whether a grid takes the fast diagonalisation: every axis of kFdMinN to
// kFdMaxN nodes.  Measured against the V-cycle on whole Poisson solves of a random
// density, order 12 (us; FP64 to 1e-10, MIXED to 1e-8; V-cycle | here):
//   32^3       FP64   2,444 |    115    MIXED   1,248 |    148
//   64^3              4,167 |    178            1,782 |    180
//   512x48^2         11,911 |    636            3,793 |    411
//   160^3            28,141 |  1,787            5,053 |    680
//   512^2x64        128,135 | 10,388           18,334 |  3,337
//   400^3           424,080 | 48,156           59,099 | 13,738
// and to 1e-4 (the loosest a solve asks for) 3 to 9 times faster, so nothing
// inside the limits goes to the V-cycle.  The upper limit is what one block's
// panel holds; the work grows with n1 + n2 + n3 per node.  The lower one is not where
// the V-cycle becomes faster (30^3 takes it 1,900 us in FP64 and 1,040 in MIXED): below
// it the V-cycle keeps the iteration counts that callers who cap them see (a cap of a
// few steps ends a 24^3 solve with OFDFT_ENOTCONV).
inline bool fd_usable(const ofdft_ctx* c, const GridDev& g, int nmax = kFdMaxN) {
  const int lo = std::min(g.n1, std::min(g.n2, g.n3)), hi = std::max(g.n1, std::max(g.n2, g.n3));
  return c->fd && lo >= kFdMinN && hi <= nmax;
}

// Floats of a scratch row, and elements of the scratch array.
inline int fd_pitch(int n1) { return fd_up4((n1 + 1) / 2) + fd_up4(n1 / 2); }
inline long long fd_scratch(const GridDev& g) { return (long long)fd_pitch(g.n1) * g.n2 * g.n3; }

inline int fd_plan(ofdft_ctx* c, const GridDev& g, int R, double h, FdPlan* P) {
  *P = FdPlan{};
  const int n[3] = {g.n1, g.n2, g.n3};
  for (int d = 0; d < 3; ++d) {
    const FdTable* t = nullptr;
    TRY(fd_table(c, n[d], R, &t));
    if (!t) return OFDFT_OK;
    P->ax[d] = t->ax;
    P->mu[d] = d == 0 ? t->mx : t->mu;
    P->mul[d] = d == 0 ? t->mxl : t->mul;
  }
  P->pitch = fd_pitch(g.n1);
  P->h2 = h * h;
  P->on = true;
  return OFDFT_OK;
}

// The job of pass p (0 .. 4: x, y, z, y, x) of z = M r.
template <typename T>
FdJob fd_job(const GridDev& g, const FdPlan& P, int p, const T* r, T* z, void* scratch, CgScalars* sc) {
  FdJob J = {};
  const int d = p == 2 ? 2 : (p == 1 || p == 3) ? 1 : 0;
  J.ax = P.ax[d];
  J.in = r;
  J.out = z;
  J.s = static_cast<float*>(scratch);
  J.sl = J.s + fd_scratch(g);
  J.pitch = P.pitch;
  J.ncols = d == 0 ? (long long)g.n2 * g.n3 : d == 1 ? (long long)P.pitch * g.n3 : (long long)P.pitch * g.n2;
  J.cw = d == 1 ? P.pitch : (int)((long long)P.pitch * g.n2);
  J.is = d == 1 ? P.pitch : P.pitch * g.n2;
  J.cs = (long long)P.pitch * g.n2;
  J.mx = P.mu[0], J.my = P.mu[1], J.mz = P.mu[2];
  J.mxl = P.mul[0], J.myl = P.mul[1], J.mzl = P.mul[2];
  const double h2 = sizeof(T) == 8 ? frexp(P.h2, &J.eh) : P.h2;
  J.h2 = make_float2((float)h2, (float)(h2 - (double)(float)h2));
  J.vec = g.n1 % 8 == 0 && (((uintptr_t)r | (uintptr_t)z) & 15u) == 0;
  J.sc = sc;
  return J;
}

template <typename T, bool XAX, int MODE, int CT, int TPW>
int fd_launch(ofdft_ctx* c, FdJob J, int warps) {
  constexpr int TC = 16 * CT;
  const size_t smem = (size_t)fd_panel_floats(J.ax, XAX, TC) * sizeof(T) + (size_t)warps * fd_ring_floats<sizeof(T) == 8>() * sizeof(float);
  static bool attr_dev[64] = {false};
  if (c->device < 0 || c->device >= 64) return fail(c, OFDFT_EINVAL, "device index out of range");
  if (!attr_dev[c->device]) {
    CU(cudaFuncSetAttribute(fd_kernel<T, XAX, MODE, CT, TPW>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFdSmem));
    attr_dev[c->device] = true;
  }
  const long long nb = (J.ncols + TC - 1) / TC;
  if (MODE == FD_SOLVE && J.sc) {
    TRY(ensure_partials(c, nb, 1));
    J.red = red(c);
    J.nblocks = (int)nb;
  }
  ProfScope ps_(c, OFDFT_K_MG);
  CU(launch_k(c, fd_kernel<T, XAX, MODE, CT, TPW>, dim3((unsigned)nb), dim3(warps * 32), smem, J));
  return OFDFT_OK;
}

template <typename T, bool XAX, int MODE>
int fd_pass(ofdft_ctx* c, const FdJob& J) {
  const int tiles = J.ax.pe / kFdTile + J.ax.po / kFdTile;
  const int tpw = tiles > 16 ? 2 : 1, warps = (tiles + tpw - 1) / tpw;
  // Panel width.  Float-float passes keep an SM's FP32 pipes busy with one block, so
  // the width (16 or 32 columns) that leaves the busiest SM the least columns is
  // taken, the wider where within a tenth (us per application, 16 | 32: 48^3 56 | 68,
  // 80^3 123 | 145, 112^3 309 | 296, 192^3 1790 | 1684).  FP32 passes wait more than
  // they compute on small grids: 64 columns from 128 an SM on (32 | 64: 80^3 60 | 67,
  // 112^3 92 | 104, 160^3 212 | 200, 192^3 329 | 307, with the correction in the last pass).
  constexpr int HI = sizeof(T) == 4 ? 4 : 2, LO = HI / 2;
  auto most = [&](int ct) { return (J.ncols + 16LL * ct * c->sms - 1) / (16LL * ct * c->sms) * ct; };
  const bool wide = sizeof(T) == 4 ? J.ncols >= 128LL * c->sms : most(HI) * 10 <= most(LO) * 11;
  if (wide) return tpw == 1 ? fd_launch<T, XAX, MODE, HI, 1>(c, J, warps) : fd_launch<T, XAX, MODE, HI, 2>(c, J, warps);
  return tpw == 1 ? fd_launch<T, XAX, MODE, LO, 1>(c, J, warps) : fd_launch<T, XAX, MODE, LO, 2>(c, J, warps);
}

// The five passes: z = M r with r.z and the PCG scalars as the V-cycle's last pass
// forms them, or (phi64 given) phi64 += M r with its other forms.  scratch:
// fd_scratch(g) elements of T.
template <typename T>
int fd_passes(ofdft_ctx* c, const GridDev& g, const FdPlan& P, const T* r, T* z, void* scratch, CgScalars* sc,
              double* phi64 = nullptr, float2* phi2 = nullptr, float* phi32 = nullptr,
              const CgScalars* gate = nullptr) {
  auto job = [&](int p) {
    FdJob J = fd_job<T>(g, P, p, r, z, scratch, sc);
    J.phi64 = phi64;
    J.phi2 = phi2;
    J.phi32 = phi32;
    J.gate = gate;
    if (phi64 && (((uintptr_t)phi64 | (uintptr_t)phi2 | (uintptr_t)phi32) & 15u)) J.vec = 0;
    return J;
  };
  TRY((fd_pass<T, true, FD_FWD>(c, job(0))));
  TRY((fd_pass<T, false, FD_FWD>(c, job(1))));
  TRY((fd_pass<T, false, FD_SOLVE>(c, job(2))));
  TRY((fd_pass<T, false, FD_INV>(c, job(3))));
  return fd_pass<T, true, FD_INV>(c, job(4));
}

// One correction of a mixed Poisson solve: phi64 += M r, with its pairs and its FP32
// rounding, in the last pass; nothing when gate->done.
inline int fd_correction(ofdft_ctx* c, const GridDev& g, const FdPlan& P, const float* r, void* scratch,
                         double* phi64, float2* phi2, float* phi32, const CgScalars* gate) {
  return fd_passes<float>(c, g, P, r, nullptr, scratch, nullptr, phi64, phi2, phi32, gate);
}

template <typename T, int R, int V, class L, class E>
int launch_zv(ofdft_ctx* c, const GridDev& g, const Weights<double>& W, L ld, E ep, int kind) {
  constexpr int smem = zsmem_bytes<T, R, V, E>();
  // resident blocks per SM of this kernel, per device (dynamic shared memory above
  // 48 KB needs an opt-in, a per-device setting)
  static int per_sm_dev[64] = {0};
  if (c->device < 0 || c->device >= 64) return fail(c, OFDFT_EINVAL, "device index out of range");
  int& per_sm = per_sm_dev[c->device];
  if (!per_sm) {
    CU(cudaFuncSetAttribute(zstream_kernel<T, R, V, L, E>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    int nb = 0;
    CU(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, zstream_kernel<T, R, V, L, E>, NT, smem));
    per_sm = std::max(nb, 1);
  }
  const std::vector<long long> key = ztune_key((const void*)zstream_kernel<T, R, V, L, E>, g);
  int nz = 0;
  if (c->force_nz >= 0) {
    nz = c->force_nz;
  } else {
    for (auto& t : c->ztune)
      if (t.first == key) {
        nz = t.second;
        break;
      }
  }
  c->last_zkey = key;
  const ZShape s = zshape<T>(c, g, per_sm, nz);
  if (E::K > 0) TRY(ensure_partials(c, s.nblocks, E::K));
  {
    ProfScope ps_(c, kind);
    CU(launch_k(c, zstream_kernel<T, R, V, L, E>, s.grid, dim3(BX, BY), smem, g, cast_weights<T>(W), s.zchunk, ld,
                ep, red(c)));
  }
  return OFDFT_OK;
}

// cuTensorMapEncodeTiled of the driver, found through the runtime (no link
// against libcuda); nullptr when the driver does not offer it.
inline PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// Tensor map of an FP32 grid array (x-fastest, n1 x n2 x n3) read in boxes of
// bx x by x 1 elements; out-of-grid elements read as zero.
inline bool fp32_grid_map(CUtensorMap* m, const void* base, const GridDev& g, int bx, int by) {
  auto enc = tensor_map_encoder();
  if (!enc) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)g.n1, (cuuint64_t)g.n2, (cuuint64_t)g.n3};
  const cuuint64_t strides[2] = {(cuuint64_t)g.n1 * 4, (cuuint64_t)g.n1 * g.n2 * 4};
  const cuuint32_t box[3] = {(cuuint32_t)bx, (cuuint32_t)by, 1};
  const cuuint32_t es[3] = {1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(base), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The z-streaming pass with TMA staging (zstream_tma_kernel).  Returns false
// (nothing launched) when the pass cannot take it: another element type or
// staging width, a slot size off the 128-byte grid, an epilogue input that is
// NULL, or no tensor-map encoder.
template <typename T, int R, int V, class L, class E>
int launch_zv_tma(ofdft_ctx* c, const GridDev& g, const Weights<double>& W, L ld, E ep, int kind, bool* done) {
  *done = false;
  if constexpr (!ztma_fits<T, R, V>() || E::NIN > 3) {
    return OFDFT_OK;
  } else {
    if (!c->tma) return OFDFT_OK;
    constexpr int TY = ZCfg<T>::TY, RA = zhalo_x<T, R, V>();
    CUtensorMap mf, mi[3];
    if (!fp32_grid_map(&mf, ld.f, g, BX + 2 * RA, TY + 2 * R)) return OFDFT_OK;
    for (int j = 0; j < 3; ++j) mi[j] = mf;
    for (int j = 0; j < E::NIN; ++j) {
      const void* in = ep.input(j);
      if (!in || !fp32_grid_map(&mi[j], in, g, BX, TY)) return OFDFT_OK;
    }
    constexpr int smem = zsmem_bytes<T, R, V, E>() + 128;
    static int per_sm_dev[64] = {0};
    if (c->device < 0 || c->device >= 64) return fail(c, OFDFT_EINVAL, "device index out of range");
    int& per_sm = per_sm_dev[c->device];
    if (!per_sm) {
      CU(cudaFuncSetAttribute(zstream_tma_kernel<T, R, V, L, E>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
      int nb = 0;
      CU(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, zstream_tma_kernel<T, R, V, L, E>, NT, smem));
      per_sm = std::max(nb, 1);
    }
    const std::vector<long long> key = ztune_key((const void*)zstream_tma_kernel<T, R, V, L, E>, g);
    int nz = 0;
    if (c->force_nz >= 0) {
      nz = c->force_nz;
    } else {
      for (auto& t : c->ztune)
        if (t.first == key) {
          nz = t.second;
          break;
        }
    }
    c->last_zkey = key;
    const ZShape s = zshape<T>(c, g, per_sm, nz);
    if (E::K > 0) TRY(ensure_partials(c, s.nblocks, E::K));
    {
      ProfScope ps_(c, kind);
      CU(launch_k(c, zstream_tma_kernel<T, R, V, L, E>, s.grid, dim3(BX, BY), smem, mf, mi[0], mi[1], mi[2], g,
                  cast_weights<T>(W), s.zchunk, ld, ep, red(c)));
    }
    c->tma_launches++;
    *done = true;
    return OFDFT_OK;
  }
}

template <typename T, int R, class L, class E>
int launch_z(ofdft_ctx* c, const GridDev& g, const Weights<double>& W, L ld, E ep, int kind) {
  if (zvec_ok<T>(g, ld, ep)) {
    bool done = false;
    TRY((launch_zv_tma<T, R, 16 / (int)sizeof(T)>(c, g, W, ld, ep, kind, &done)));
    if (done) return OFDFT_OK;
    return launch_zv<T, R, 16 / (int)sizeof(T)>(c, g, W, ld, ep, kind);
  }
  return launch_zv<T, R, 1>(c, g, W, ld, ep, kind);
}

// Runtime radius -> template radius.
template <typename T, class L, class E>
int launch_z_r(ofdft_ctx* c, int R, const GridDev& g, const Weights<double>& W, L ld, E ep, int kind) {
  switch (R) {
    case 1: return launch_z<T, 1>(c, g, W, ld, ep, kind);
    case 2: return launch_z<T, 2>(c, g, W, ld, ep, kind);
    case 3: return launch_z<T, 3>(c, g, W, ld, ep, kind);
    case 4: return launch_z<T, 4>(c, g, W, ld, ep, kind);
    case 5: return launch_z<T, 5>(c, g, W, ld, ep, kind);
    case 6: return launch_z<T, 6>(c, g, W, ld, ep, kind);
  }
  return fail(c, OFDFT_EINVAL, "stencil radius %d not supported", R);
}


inline int sync_scalars(ofdft_ctx* c, const void* dev, size_t bytes, void* host) {
  // through the context's pinned block: a copy to pageable memory is staged by the
  // driver (5 us more a call)
  void* to = bytes <= 32 * sizeof(double) ? (void*)c->host_scal : host;
  CU(cudaMemcpyAsync(to, dev, bytes, cudaMemcpyDeviceToHost, c->stream));
  CU(cudaStreamSynchronize(c->stream));
  if (to != host) memcpy(host, to, bytes);
  if (!c->pending.empty()) harvest(c);
  return OFDFT_OK;
}

struct EvalOut {
  double sums[12];
};

// What a Poisson solve launches behind its last expected kernel, before it knows
// whether it has converged, so that both are waited for together: launch(gate)
// enqueues it and the `sums` (12 doubles at c->scal) come with the solve's scalars.
// It writes nothing where the solve has not converged by then (`anyway`, for calls
// that take the potential as it is: where the residual is not finite).  done: it
// ran; otherwise the caller launches it again (launch(NULL)) or reports the error.
struct Behind {
  std::function<int(const CgScalars* gate)> launch;
  EvalOut* out = nullptr;
  bool anyway = false;
  bool done = false;
  void ended(const CgScalars& s) {  // the scalars that the device's test saw
    done = anyway ? std::isfinite(s.rr) : s.rr <= s.tol2 * (s.bb > 0.0 ? s.bb : 1.0);
  }
};

// sync_scalars for the CG scalars and, with b, its sums.
inline int sync_behind(ofdft_ctx* c, const CgScalars* dev, CgScalars* host, Behind* b) {
  if (!b) return sync_scalars(c, dev, sizeof(CgScalars), host);
  double* sums = c->host_scal + 32;
  CU(cudaMemcpyAsync(sums, c->scal, 12 * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  TRY(sync_scalars(c, dev, sizeof(CgScalars), host));
  memcpy(b->out->sums, sums, 12 * sizeof(double));
  return OFDFT_OK;
}

inline void fill_energy(const EvalOut& o, double h, const ofdft_params* p, double E_self, double ezz, double eta,
                 double mu, ofdft_energy* e) {
  const double h3 = h * h * h;
  const bool es = p->terms & OFDFT_TERM_ES;
  e->E_tf = h3 * o.sums[0];
  e->E_vw = -0.5 * p->lambda * h3 * o.sums[1];
  e->E_xc = h3 * o.sums[2];
  e->E_self = es ? E_self : 0.0;
  e->E_es = es ? h3 * (0.5 * o.sums[3] + o.sums[4] / (8.0 * kPi)) - E_self : 0.0;
  e->E_zz_corr = ezz;
  e->E = e->E_tf + e->E_vw + e->E_xc + e->E_es + ezz;
  e->C = o.sums[9];
  e->L = e->E - eta * e->C + 0.5 * e->C * e->C / mu;
  e->gd = h3 * o.sums[5];
  e->gs_old = h3 * o.sums[6];
  e->rs = h3 * o.sums[7];
  e->rs_pc = e->rs;
  e->gnorm2 = h3 * o.sums[8];
}

// Coefficients of gtab_v, [power][interval]: the Taylor series of
// g(s) = erf(sqrt s)/sqrt s around c = (middle of the interval of s + 1) - 1.  Up to
// c = 3 from g's power series (2/sqrt pi) sum (-s)^j / (j! (2j + 1)); beyond from
// 2 s g' + g = (2/sqrt pi) e^{-s}, whose recurrence for the coefficients,
//   a_{k+1} = ((2/sqrt pi) e^{-c} (-1)^k / k! - (2k + 1) a_k) / (2 c (k + 1)),
// is stable forwards there (a_k ~ c^{-k} is its dominant solution).
inline const std::vector<double>& gtab_host() {
  static const std::vector<double> tab = [] {
    std::vector<double> t((size_t)kGtabN * kGtabC);
    const long double tsp = 2.0L / sqrtl(acosl(-1.0L));
    for (int i = 0; i < kGtabN; ++i) {
      const long double c = ldexpl(1.0L + ((i % 64) + 0.5L) / 64.0L, i / 64) - 1.0L;
      long double a[kGtabC];
      if (c < 3.0L) {
        for (int k = 0; k < kGtabC; ++k) {
          long double s = 0.0L, f = 1.0L;  // f = C(j, k) c^{j-k} / j!, from j = k on
          for (int m = 1; m <= k; ++m) f /= m;
          for (int j = k; j < k + 60; ++j) {
            s += ((j & 1) ? -f : f) / (2 * j + 1);
            f *= c / (j + 1 - k);
          }
          a[k] = tsp * s;
        }
      } else {
        a[0] = erfl(sqrtl(c)) / sqrtl(c);
        long double f = tsp * expl(-c);
        for (int k = 0; k + 1 < kGtabC; ++k) {
          a[k + 1] = (f - (2 * k + 1) * a[k]) / (2.0L * c * (k + 1));
          f *= -1.0L / (k + 1);
        }
      }
      for (int k = 0; k < kGtabC; ++k) t[(size_t)k * kGtabN + i] = (double)a[k];
    }
    return t;
  }();
  return tab;
}
// The smallest d2 whose rounded square root is not below rc: r < rc is d2 < rc2
// exactly, without a square root per node.  No distance is below an rc <= 0.
inline double sq_threshold(double rc) {
  if (!(rc > 0.0)) return 0.0;
  double x = rc * rc;
  while (sqrt(x) >= rc) x = nextafter(x, 0.0);
  while (sqrt(x) < rc) x = nextafter(x, INFINITY);
  return x;
}

// Routines of api.cu used by the batched engine (instantiated for double and float).
int check_atoms(ofdft_ctx* c, const double* R, const double* Z, int M);
int check_params(ofdft_ctx* c, const ofdft_params* p);
template <typename T>
int device_pseudocharge(ofdft_ctx* c, const ofdft_grid* gr, int R, const double* R_host, const double* Z_host,
                        int M, double sigma, double rc, T* b, double* E_self, bool keep_tables = false);
template <typename T>
int device_guess(ofdft_ctx* c, const ofdft_grid* gr, const double* R_host, const double* Z_host, int M,
                 double gsig, double gcut, double N, T* u);
template <typename T>
int device_forces(ofdft_ctx* c, const ofdft_grid* gr, int R, const double* R_host, const double* Z_host, int M,
                  double sigma, double rc, int variant, const T* phi, double* F);
int device_ezz(ofdft_ctx* c, const double* R_host, const double* Z_host, int M, double sigma, double* E,
               double* F);

}  // namespace ofd
