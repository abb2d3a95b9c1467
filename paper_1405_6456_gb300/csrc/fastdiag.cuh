// Fast diagonalisation of the discrete Poisson operator: the preconditioner of
// the Poisson CG on grids whose axes it covers.
//
// With zero Dirichlet values -L_h is a Kronecker sum, T_x (+) T_y (+) T_z, of one
// symmetric banded Toeplitz matrix per axis (the weights of Eq. FD:Laplacian).
// With T = Q diag(mu) Q^T for every axis (Lynch, Rice and Thomas 1964),
//   z = (Q_x Q_y Q_z) diag(1 / (mu_x + mu_y + mu_z)) (Q_x Q_y Q_z)^T r
// inverts it up to rounding, so a CG that would take 20 to 35 V-cycles takes one
// or two steps.  A symmetric Toeplitz matrix commutes with the reversal of its
// axis, so every eigenvector is even or odd: on the sums and differences
// f_i +- f_{n-1-i} a transform is two products with matrices of half the size,
// n / 2 multiply-adds per node and transform instead of n.
//
// One pass per axis and direction, the z axis forwards, divided and backwards in
// one: x, y, z, y, x, five launches, all but the first and the last in place in
// one scratch array (rows padded to whole 16-byte vectors).  A block holds a
// panel, all n nodes of the axis times TC columns, in shared memory; a warp owns
// a tile of 16 outputs x TC columns (8 x CT per thread, in register pairs: the
// packed FP32 FMA takes two outputs at a time) and walks the contraction without
// any block barrier: the panel's row comes from shared memory, the matrix's row
// from the warp's own ring (each matrix element is read by one warp of a block).
//
// What bounds it: the FMA pipes.  At 192^3 in FP32 the five passes need 576
// multiply-adds a node, 101 us at the pipes' rate, and move 283 MB through L2; they
// take 48 + 39 + 81 + 40 + 44 = 252 us (40% of the pipes' rate; a V-cycle takes
// 158 us but 16 to 30 times as many of them are needed).  The same passes with the
// matrix rows read through L1 took 475 us (42% of them missed); with the x panels
// transposed on the way in 300 us.  The last pass of a correction takes 95 us instead
// of 44 (303 us the five).  At 128^3 in float-float: 63 + 62 + 128 + 62 + 67 us, 59% of
// the rate of its 12 operations.
//
// Element types: FP32 fields compute in FP32.  FP64 fields compute in float-float
// pairs (ff, about 2^-46 relative): 12 packed FP32 operations per multiply-add
// against the 64 FP32 slots that one FP64 FMA costs on this GPU.  Pairs have FP32's
// exponents, so the first pass divides r by 2^k ~ ||r|| (from the CG's r.r) and the
// last one, and r.z, put 2^k back: integer operations on the exponents, exact, and
// a source of any size FP64 holds is solved alike.
#pragma once

#include "kernels.cuh"

namespace ofd {

constexpr int kFdTile = 16;     // outputs per warp tile
constexpr int kFdMaxN = 512;    // longest axis: 16 warps of two tiles each
constexpr int kFdMinN = 32;     // shortest axis (see fd_usable)
constexpr int kFdSmem = 216 * 1024;  // dynamic shared memory limit of its kernels (n = 512, float-float: 193 KB)

// One axis: matrices [contraction][output], outputs padded with zeros to whole
// tiles, the even half first (ne rows of pe) and then the odd one (no rows of po).
struct FdAxis {
  const float* fwd;   // contraction over nodes, outputs are modes
  const float* fwdl;  // ... low parts (float-float)
  const float* inv;   // contraction over modes, outputs are nodes
  const float* invl;
  int n, ne, no, pe, po;
};

enum { FD_FWD = 0, FD_INV = 1, FD_SOLVE = 2 };

// One pass over one grid.  Column c of a strided axis (y, z) starts at element
// (c / cw) cs + c % cw and its node i lies is further on; a column of the x axis
// is a row of n contiguous nodes.
struct FdJob {
  FdAxis ax;
  const void* in;   // x forwards: r
  void* out;        // x backwards: z, or (corrections of a mixed solve) NULL and
  double* phi64;    // phi64 += z,
  float2* phi2;     // with its pairs (may be NULL)
  float* phi32;     // and its FP32 rounding
  float* s;         // scratch, high parts
  float* sl;        // scratch, low parts (float-float)
  long long ncols;
  int cw, is;
  long long cs;
  int pitch;        // scratch row: x modes, the odd ones from fd_up4(ne) on, zeros in between and behind
  int vec;          // x axis: n1 a multiple of 8 and r, z on 16 bytes: rows move as whole vectors
  const float *mx, *my, *mz;     // eigenvalues of h^2 T by axis
  const float *mxl, *myl, *mzl;  // ... low parts
  float2 h2;        // h^2 = h2 2^eh
  int eh;           // (0 for FP32 fields)
  CgScalars* sc;    // the CG this serves (NULL: none; r.z is then not formed)
  const CgScalars* gate;  // a correction launched ahead: nothing to do when its solve is done
  RedBuf red;       // z: r.z
  int nblocks;
};

// Sum of a double over a block of `nt` threads (a multiple of 32, at most 512).
__device__ __forceinline__ double fd_block_sum(double v, double* smem, int tid, int nt) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((tid & 31) == 0) smem[tid >> 5] = v;
  __syncthreads();
  double s = 0.0;
  if (tid < 32) {
    s = tid < nt / 32 ? smem[tid] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  }
  __syncthreads();
  return s;
}

__device__ __forceinline__ float2 fd_neg(float2 a) { return make_float2(-a.x, -a.y); }
// a - b, lane by lane
__device__ __forceinline__ float2 fd_sub(float2 a, float2 b) { return __fadd2_rn(a, fd_neg(b)); }

// acc += w f for two outputs (w) and one column (f), in FP32 or float-float.
template <bool FF>
struct FdAcc;
template <>
struct FdAcc<false> {
  float2 h;
  __device__ __forceinline__ void zero() { h = make_float2(0.0f, 0.0f); }
  __device__ __forceinline__ void add(float2 w, float2, float2 f, float2, float2) { h = __ffma2_rn(w, f, h); }
  __device__ __forceinline__ void finish() {}
};
template <>
struct FdAcc<true> {
  float2 h, l;
  __device__ __forceinline__ void zero() { h = l = make_float2(0.0f, 0.0f); }
  // (the packed instructions have no operand signs: a difference a - b is the FMA
  // b (-1) + a, and the product enters with its sign turned through f, nf = -f)
  __device__ __forceinline__ void add(float2 w, float2 wl, float2 f, float2 fl, float2 nf) {
    const float2 m1 = make_float2(-1.0f, -1.0f);
    const float2 np = __fmul2_rn(w, nf);        // -p
    const float2 e = __ffma2_rn(w, f, np);      // exact rounding error of the product
    const float2 s = __ffma2_rn(np, m1, h);     // TwoSum(h, p)
    const float2 b = __ffma2_rn(h, m1, s);
    const float2 t = __ffma2_rn(__ffma2_rn(b, m1, s), m1, h);
    const float2 u = __ffma2_rn(__fadd2_rn(np, b), m1, t);
    h = s;
    l = __fadd2_rn(l, __fadd2_rn(u, e));
    l = __ffma2_rn(w, fl, l);
    l = __ffma2_rn(wl, f, l);
  }
  __device__ __forceinline__ void finish() {  // renormalise (|h| >= |l|)
    const float2 s = __fadd2_rn(h, l);
    l = fd_sub(l, fd_sub(s, h));
    h = s;
  }
};

// A warp's private ring of matrix rows: kFdStages chunks of kFdChunk rows of its
// tile's 16 outputs, copied asynchronously kFdStages - 1 chunks ahead of use, so
// the contraction neither waits for L2 nor meets a block barrier.  (Read straight
// from global memory the rows cost 17 of 19 stall cycles per issue and left the
// FMA pipe 73% idle: 83 us a pass at 192^3 in FP32.)
constexpr int kFdChunk = 8, kFdStages = 4;
template <bool FF>
constexpr int fd_ring_floats() {  // per warp
  return kFdStages * kFdChunk * kFdTile * (FF ? 2 : 1);
}

template <bool FF>
struct FdRing {
  float* base;         // this warp's ring
  const float *w, *wl; // the tile's first output, row 0
  int wp, rows, lane;
  // chunk ch into its slot: each lane copies 16 bytes of one row; rows past the
  // end read as zeros
  __device__ __forceinline__ void stage(int ch) const {
    const int r = lane >> 2, o = (lane & 3) * 4, row = ch * kFdChunk + r;
    const bool ok = row < rows;
    float* d = base + (ch & (kFdStages - 1)) * (kFdChunk * kFdTile * (FF ? 2 : 1)) + r * kFdTile + o;
    const size_t so = ok ? (size_t)row * wp + o : 0;
    cp_async_bytes<16>(d, w + so, ok);
    if constexpr (FF) cp_async_bytes<16>(d + kFdChunk * kFdTile, wl + so, ok);
    cp_async_commit();
  }
  __device__ __forceinline__ void start() const {
#pragma unroll
    for (int ch = 0; ch < kFdStages - 1; ++ch) stage(ch);
  }
};

// The contraction of one warp tile: acc[q][c] (outputs 2q, 2q + 1 of the
// thread's eight, column c) over the ring's rows and the panel's, which start at
// sh (sl).  The ring has been started.  Node-major panels (XAX false) hold a
// node's columns together, the thread's CT columns adjacent; column-major ones
// (the x axis) hold a column's nodes together, the thread's columns 16 apart, and
// are read four nodes at a time (zeros fill them up to a multiple of four).
template <bool FF, bool XAX, int CT>
__device__ __forceinline__ void fd_contract(FdAcc<FF> (&acc)[4][CT], const FdRing<FF>& ring, int kq, const float* sh,
                                            const float* sl, int pitch) {
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int c = 0; c < CT; ++c) acc[q][c].zero();
  // one node: matrix row wr, the thread's values f (fl)
  auto row = [&](const float* wr, const float (&f)[CT], const float (&fl)[CT]) {
    const float4 a = *reinterpret_cast<const float4*>(wr);
    const float4 b = *reinterpret_cast<const float4*>(wr + 4);
    const float2 wv[4] = {make_float2(a.x, a.y), make_float2(a.z, a.w), make_float2(b.x, b.y), make_float2(b.z, b.w)};
    float2 wlv[4] = {};
    if constexpr (FF) {
      const float4 al = *reinterpret_cast<const float4*>(wr + kFdChunk * kFdTile);
      const float4 bl = *reinterpret_cast<const float4*>(wr + kFdChunk * kFdTile + 4);
      wlv[0] = make_float2(al.x, al.y);
      wlv[1] = make_float2(al.z, al.w);
      wlv[2] = make_float2(bl.x, bl.y);
      wlv[3] = make_float2(bl.z, bl.w);
    }
#pragma unroll
    for (int c = 0; c < CT; ++c) {
      const float2 fv = make_float2(f[c], f[c]);
      float2 flv = make_float2(0.0f, 0.0f), nfv = flv;
      if constexpr (FF) flv = make_float2(fl[c], fl[c]), nfv = make_float2(-f[c], -f[c]);
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q][c].add(wv[q], wlv[q], fv, flv, nfv);
    }
  };
  auto node = [&](const float* wr, int i) {  // node-major
    float f[CT], fl[CT];
#pragma unroll
    for (int c = 0; c < CT; c += CT) {
      if constexpr (CT == 1) {
        f[0] = sh[i * pitch];
        if constexpr (FF) fl[0] = sl[i * pitch];
      } else if constexpr (CT == 4) {
        const float4 v = *reinterpret_cast<const float4*>(sh + i * pitch);
        f[0] = v.x, f[1] = v.y, f[2] = v.z, f[3] = v.w;
        if constexpr (FF) {
          const float4 u = *reinterpret_cast<const float4*>(sl + i * pitch);
          fl[0] = u.x, fl[1] = u.y, fl[2] = u.z, fl[3] = u.w;
        }
      } else {
        const float2 v = *reinterpret_cast<const float2*>(sh + i * pitch);
        f[0] = v.x, f[1] = v.y;
        if constexpr (FF) {
          const float2 u = *reinterpret_cast<const float2*>(sl + i * pitch);
          fl[0] = u.x, fl[1] = u.y;
        }
      }
    }
    row(wr, f, fl);
  };
  auto nodes4 = [&](const float* wr, int i) {  // column-major, nodes i .. i + 3
    float v[CT][4], u[CT][4];
#pragma unroll
    for (int c = 0; c < CT; ++c) {
      const float4 t = *reinterpret_cast<const float4*>(sh + 16 * c * pitch + i);
      v[c][0] = t.x, v[c][1] = t.y, v[c][2] = t.z, v[c][3] = t.w;
      if constexpr (FF) {
        const float4 x = *reinterpret_cast<const float4*>(sl + 16 * c * pitch + i);
        u[c][0] = x.x, u[c][1] = x.y, u[c][2] = x.z, u[c][3] = x.w;
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float f[CT], fl[CT];
#pragma unroll
      for (int c = 0; c < CT; ++c) {
        f[c] = v[c][k];
        if constexpr (FF) fl[c] = u[c][k];
      }
      row(wr + k * kFdTile, f, fl);
    }
  };
  const int nch = (ring.rows + kFdChunk - 1) / kFdChunk;
  for (int ch = 0; ch < nch; ++ch) {
    cp_async_wait<kFdStages - 2>();  // chunk ch has landed (this lane's copies)
    __syncwarp();                    // ... and every lane's; the slot of chunk ch - 1 is free
    ring.stage(ch + kFdStages - 1);
    const float* wr = ring.base + (ch & (kFdStages - 1)) * (kFdChunk * kFdTile * (FF ? 2 : 1)) + kq;
    const int i0 = ch * kFdChunk;
    if constexpr (XAX) {
      nodes4(wr, i0);
      if (i0 + 4 < ring.rows) nodes4(wr + 4 * kFdTile, i0 + 4);
    } else {
      if (i0 + kFdChunk <= ring.rows) {
#pragma unroll
        for (int r = 0; r < kFdChunk; ++r) node(wr + r * kFdTile, i0 + r);
      } else {
        for (int r = 0; i0 + r < ring.rows; ++r) node(wr + r * kFdTile, i0 + r);
      }
    }
  }
  cp_async_wait<0>();  // the ring is free again
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int c = 0; c < CT; ++c) acc[q][c].finish();
}

// k with 2^k <= ||r|| < 2^(k+1) for the residual r the job reads (0: no CG).
__device__ __forceinline__ int fd_exponent(const CgScalars* sc) {
  return sc ? ((int)(((unsigned)__double2hiint(sc->rr) >> 20) & 0x7ffu) - 1023) >> 1 : 0;
}

// Float-float helpers on single values.
__device__ __forceinline__ float2 fd_ff_add(float2 a, float2 b) {
  const float2 s = ff_two_sum(a.x, b.x);
  return ff_fast_two_sum(s.x, s.y + (a.y + b.y));
}
// 1 / d for a positive pair: one Newton step from the FP32 reciprocal, the
// residual 1 - d y formed exactly
__device__ __forceinline__ float2 fd_ff_rcp(float2 d) {
  const float y = 1.0f / d.x;
  const float e = fmaf(-d.y, y, fmaf(-d.x, y, 1.0f));
  return ff_fast_two_sum(y, y * e);
}

// Column-major panels (x axis): a column's even nodes, then its odd ones, each
// padded to a multiple of four; the pitch is an odd multiple of four, so that
// eight columns' 16-byte reads meet no bank twice.
__host__ __device__ __forceinline__ int fd_up4(int n) { return (n + 3) & ~3; }
__host__ __device__ __forceinline__ int fd_xpitch(int ne, int no) {
  const int w = fd_up4(ne) + fd_up4(no);
  return (w & 4) ? w : w + 4;
}
// Floats of one panel (one of two in float-float) of TC columns.
__host__ __device__ __forceinline__ int fd_panel_floats(const FdAxis& ax, bool xax, int tc) {
  return xax ? tc * fd_xpitch(ax.ne, ax.no) : ax.n * tc;
}

__device__ __forceinline__ float4 f4(float a, float b, float c, float d) { return make_float4(a, b, c, d); }

// 16 aligned bytes of a field, and the same number of elements of a panel.
__device__ __forceinline__ void fd_load16(const float* p, float (&v)[4]) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
}
__device__ __forceinline__ void fd_load16(const double* p, double (&v)[2]) {
  const double2 a = *reinterpret_cast<const double2*>(p);
  v[0] = a.x, v[1] = a.y;
}
__device__ __forceinline__ void fd_store16(float* p, const float (&v)[4]) { *reinterpret_cast<float4*>(p) = f4(v[0], v[1], v[2], v[3]); }
__device__ __forceinline__ void fd_store16(double* p, const double (&v)[2]) { *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]); }
__device__ __forceinline__ void fd_put(float* p, const float (&v)[4]) { *reinterpret_cast<float4*>(p) = f4(v[0], v[1], v[2], v[3]); }
__device__ __forceinline__ void fd_put(float* p, const float (&v)[2]) { *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]); }
__device__ __forceinline__ void fd_get(const float* p, float (&v)[4]) { fd_load16(p, v); }
__device__ __forceinline__ void fd_get(const float* p, float (&v)[2]) {
  const float2 a = *reinterpret_cast<const float2*>(p);
  v[0] = a.x, v[1] = a.y;
}

// phi64 += z with the potential's other forms (v: phi64's old values).
__device__ __forceinline__ void fd_correct(const FdJob& J, long long i, float z) {
  const double v = J.phi64[i] + double_of_float(z);
  const float2 p = ff_of_double(v);
  J.phi64[i] = v;
  if (J.phi2) J.phi2[i] = p;
  J.phi32[i] = ff_nearest(p);
}
__device__ __forceinline__ void fd_correct2(const FdJob& J, long long i, double2 v, const float (&z)[2]) {
  v.x += double_of_float(z[0]);
  v.y += double_of_float(z[1]);
  const float2 p = ff_of_double(v.x), q = ff_of_double(v.y);
  *reinterpret_cast<double2*>(J.phi64 + i) = v;
  if (J.phi2) *reinterpret_cast<float4*>(J.phi2 + i) = f4(p.x, p.y, q.x, q.y);
  *reinterpret_cast<float2*>(J.phi32 + i) = make_float2(ff_nearest(p), ff_nearest(q));
}

// One block's panel of a pass: columns [c0, c0 + TC) of the job.  T is the field
// type (float, or double computed in float-float).  XAX: the x axis (columns are
// contiguous rows); MODE: forwards, backwards, or the z axis' whole solve.
template <typename T, bool XAX, int MODE, int CT, int TPW>
__device__ __forceinline__ void fd_panel(const FdJob& J, long long c0, int bid, float* sm) {
  constexpr bool FF = sizeof(T) == 8;
  constexpr int TC = 16 * CT;
  const int n = J.ax.n, ne = J.ax.ne, no = J.ax.no;
  const int P = XAX ? fd_xpitch(ne, no) : TC;          // panel pitch
  const int oo = XAX ? fd_up4(ne) : ne;                // where the odd part starts (nodes of a column, or rows)
  const int pf = XAX ? TC * P : n * TC;
  float* ph = sm;
  float* pl = FF ? sm + pf : sm;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const int te = J.ax.pe / kFdTile, tiles = te + J.ax.po / kFdTile;
  // this warp's ring over the matrix rows of a tile
  float* rbase = sm + (size_t)pf * (FF ? 2 : 1) + warp * fd_ring_floats<FF>();
  auto ring_of = [&](int tile, bool fwd) {
    const bool odd = tile >= te;
    const size_t mo = (odd ? (size_t)ne * J.ax.pe : 0) + (size_t)(odd ? tile - te : tile) * kFdTile;
    return FdRing<FF>{rbase, (fwd ? J.ax.fwd : J.ax.inv) + mo, (fwd ? J.ax.fwdl : J.ax.invl) + mo,
                      odd ? J.ax.po : J.ax.pe, odd ? no : ne, lane};
  };

  // ---- the panel into shared memory (forwards: sums and differences) ----
  if constexpr (XAX && MODE == FD_FWD) {
    const T* src = static_cast<const T*>(J.in);
    const int ke = FF ? fd_exponent(J.sc) : 0;
    if (J.vec) {
      constexpr int GS = 16 / (int)sizeof(T);  // elements of a lane's 16 bytes
      const int gr = ne / GS;                  // groups of a half row
#pragma unroll 4
      for (int q = tid; q < TC * gr; q += nt) {
        const int c = q / gr, x = (q - c * gr) * GS;
        const long long row = c0 + c;
        T a[GS] = {}, b[GS] = {};
        if (row < J.ncols) {
          fd_load16(src + row * n + x, a);
          fd_load16(src + row * n + n - GS - x, b);
        }
        float s[GS], d[GS], sl[GS], dl[GS];
#pragma unroll
        for (int k = 0; k < GS; ++k) {
          if constexpr (FF) {
            const float2 fa = ff_of_double(a[k], ke), fb = ff_of_double(b[GS - 1 - k], ke);
            const float2 sv = fd_ff_add(fa, fb), dv = fd_ff_add(fa, fd_neg(fb));
            s[k] = sv.x, sl[k] = sv.y, d[k] = dv.x, dl[k] = dv.y;
          } else {
            s[k] = a[k] + b[GS - 1 - k];
            d[k] = a[k] - b[GS - 1 - k];
          }
        }
        fd_put(ph + c * P + x, s);
        fd_put(ph + c * P + oo + x, d);
        if constexpr (FF) {
          fd_put(pl + c * P + x, sl);
          fd_put(pl + c * P + oo + x, dl);
        }
      }
    } else {
      for (int c = warp; c < TC; c += nw) {
        const long long row = c0 + c;
        const bool ok = row < J.ncols;
        const long long o = (ok ? row : 0) * n;
#pragma unroll 4
        for (int x = lane; x < oo; x += 32) {
          T a = T(0), b = T(0);
          if (ok && x < ne) a = src[o + x];
          if (ok && x < no) b = src[o + n - 1 - x];
          float2 s, d;
          if constexpr (FF) {
            const float2 fa = ff_of_double(a, ke), fb = ff_of_double(b, ke);
            s = fd_ff_add(fa, fb);
            d = fd_ff_add(fa, fd_neg(fb));
          } else {
            s = make_float2(a + b, 0.0f);
            d = make_float2(a - b, 0.0f);
          }
          ph[c * P + x] = s.x;
          if constexpr (FF) pl[c * P + x] = s.y;
          if (oo + x < P) {  // (the padding with zeros)
            ph[c * P + oo + x] = x < no ? d.x : 0.0f;
            if constexpr (FF) pl[c * P + oo + x] = x < no ? d.y : 0.0f;
          }
        }
      }
    }
  } else if constexpr (XAX) {
    // rows of modes, laid out as the panel's columns are
    const int gr = J.pitch / 4;
#pragma unroll 4
    for (int q = tid; q < TC * gr; q += nt) {
      const int c = q / gr, x = (q - c * gr) * 4;
      const bool ok = c0 + c < J.ncols;
      const long long o = ok ? (c0 + c) * J.pitch + x : 0;
      cp_async_bytes<16>(ph + c * P + x, J.s + o, ok);
      if constexpr (FF) cp_async_bytes<16>(pl + c * P + x, J.sl + o, ok);
    }
    cp_async_commit();
  } else if constexpr (MODE == FD_INV) {
    constexpr int CG = TC / 4;  // 16-byte column groups
#pragma unroll 4
    for (int q = tid; q < n * CG; q += nt) {
      const int i = q / CG, c = (q % CG) * 4;
      const long long col = c0 + c;
      const bool ok = col < J.ncols;
      const long long o = ok ? (col / J.cw) * J.cs + col % J.cw + (long long)i * J.is : 0;
      cp_async_bytes<16>(ph + i * P + c, J.s + o, ok);
      if constexpr (FF) cp_async_bytes<16>(pl + i * P + c, J.sl + o, ok);
    }
    cp_async_commit();
  } else {
    constexpr int CG = TC / 4;
#pragma unroll 2
    for (int q = tid; q < ne * CG; q += nt) {
      const int i = q / CG, c = (q % CG) * 4;
      const long long col = c0 + c;
      float4 a = f4(0.f, 0.f, 0.f, 0.f), b = a, al = a, bl = a;
      if (col < J.ncols) {
        const long long o = (col / J.cw) * J.cs + col % J.cw;
        a = *reinterpret_cast<const float4*>(J.s + o + (long long)i * J.is);
        if constexpr (FF) al = *reinterpret_cast<const float4*>(J.sl + o + (long long)i * J.is);
        if (i < no) {
          b = *reinterpret_cast<const float4*>(J.s + o + (long long)(n - 1 - i) * J.is);
          if constexpr (FF) bl = *reinterpret_cast<const float4*>(J.sl + o + (long long)(n - 1 - i) * J.is);
        }
      }
      float4 s, d, sl = al, dl = al;
      if constexpr (FF) {
        const float2 s0 = fd_ff_add(make_float2(a.x, al.x), make_float2(b.x, bl.x));
        const float2 s1 = fd_ff_add(make_float2(a.y, al.y), make_float2(b.y, bl.y));
        const float2 s2 = fd_ff_add(make_float2(a.z, al.z), make_float2(b.z, bl.z));
        const float2 s3 = fd_ff_add(make_float2(a.w, al.w), make_float2(b.w, bl.w));
        const float2 d0 = fd_ff_add(make_float2(a.x, al.x), make_float2(-b.x, -bl.x));
        const float2 d1 = fd_ff_add(make_float2(a.y, al.y), make_float2(-b.y, -bl.y));
        const float2 d2 = fd_ff_add(make_float2(a.z, al.z), make_float2(-b.z, -bl.z));
        const float2 d3 = fd_ff_add(make_float2(a.w, al.w), make_float2(-b.w, -bl.w));
        s = f4(s0.x, s1.x, s2.x, s3.x), sl = f4(s0.y, s1.y, s2.y, s3.y);
        d = f4(d0.x, d1.x, d2.x, d3.x), dl = f4(d0.y, d1.y, d2.y, d3.y);
      } else {
        s = f4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
        d = f4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
      }
      *reinterpret_cast<float4*>(ph + i * P + c) = s;
      if constexpr (FF) *reinterpret_cast<float4*>(pl + i * P + c) = sl;
      if (i < no) {
        *reinterpret_cast<float4*>(ph + (ne + i) * P + c) = d;
        if constexpr (FF) *reinterpret_cast<float4*>(pl + (ne + i) * P + c) = dl;
      }
    }
  }
  if (MODE == FD_INV) cp_async_wait<0>();
  if (warp < tiles) ring_of(warp, MODE != FD_INV).start();
  __syncthreads();

  // ---- the products: warp tiles of 16 outputs, thread tiles of 8 x CT ----
  FdAcc<FF> acc[TPW][4][CT];
  const int kq = (lane >> 4) * 8;
  const int cl = XAX ? (lane & 15) : (lane & 15) * CT;  // the thread's first column (x axis: the others 16 apart)
  const int po = XAX ? cl * P : cl;                     // its panel offset
  // (the first tile's ring is started by the caller)
  auto product = [&](bool fwd) {
#pragma unroll
    for (int t = 0; t < TPW; ++t) {
      const int tile = warp + t * nw;
      if (tile >= tiles) break;
      const FdRing<FF> ring = ring_of(tile, fwd);
      if (t > 0) ring.start();
      const int odd0 = (tile >= te ? oo : 0) * (XAX ? 1 : P);
      fd_contract<FF, XAX, CT>(acc[t], ring, kq, ph + odd0 + po, pl + odd0 + po, P);
    }
  };
  auto hi = [](const FdAcc<FF>& a, int l) { return l ? a.h.y : a.h.x; };
  auto lo = [](const FdAcc<FF>& a, int l) {
    if constexpr (FF)
      return l ? a.l.y : a.l.x;
    else
      return 0.0f;
  };
  // the thread's outputs to panel (or scratch) d, dl: node-major, row k of a part
  // at k * stride, the columns adjacent
  auto put_rows = [&](float* d0, float* dl0, long long stride) {
#pragma unroll
    for (int t = 0; t < TPW; ++t) {
      const int tile = warp + t * nw;
      if (tile >= tiles) break;
      const bool odd = tile >= te;
      const int k0 = (odd ? tile - te : tile) * kFdTile + kq, half = odd ? no : ne, row0 = odd ? ne : 0;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        if (k0 + k >= half) continue;
        float* d = d0 + (row0 + k0 + k) * stride;
        float* dl = dl0 + (row0 + k0 + k) * stride;
        const FdAcc<FF>(&a)[CT] = acc[t][k >> 1];
        if constexpr (CT == 4) {
          *reinterpret_cast<float4*>(d) = f4(hi(a[0], k & 1), hi(a[1], k & 1), hi(a[2], k & 1), hi(a[3], k & 1));
          if constexpr (FF)
            *reinterpret_cast<float4*>(dl) = f4(lo(a[0], k & 1), lo(a[1], k & 1), lo(a[2], k & 1), lo(a[3], k & 1));
        } else if constexpr (CT == 2) {
          *reinterpret_cast<float2*>(d) = make_float2(hi(a[0], k & 1), hi(a[1], k & 1));
          if constexpr (FF) *reinterpret_cast<float2*>(dl) = make_float2(lo(a[0], k & 1), lo(a[1], k & 1));
        } else {
          *d = hi(a[0], k & 1);
          if constexpr (FF) *dl = lo(a[0], k & 1);
        }
      }
    }
  };
  // column-major panel: eight consecutive outputs of each of the thread's columns
  // (outputs past the half land in the padding or are dropped)
  auto put_cols = [&]() {
#pragma unroll
    for (int t = 0; t < TPW; ++t) {
      const int tile = warp + t * nw;
      if (tile >= tiles) break;
      const bool odd = tile >= te;
      const int k0 = (odd ? tile - te : tile) * kFdTile + kq, half4 = fd_up4(odd ? no : ne);
#pragma unroll
      for (int c = 0; c < CT; ++c) {
        float* d = ph + (cl + 16 * c) * P + (odd ? oo : 0) + k0;
        float* dl = pl + (cl + 16 * c) * P + (odd ? oo : 0) + k0;
#pragma unroll
        for (int q = 0; q < 4; q += 2) {
          if (k0 + 2 * q >= half4) continue;
          *reinterpret_cast<float4*>(d + 2 * q) = f4(acc[t][q][c].h.x, acc[t][q][c].h.y, acc[t][q + 1][c].h.x,
                                                     acc[t][q + 1][c].h.y);
          if constexpr (FF)
            *reinterpret_cast<float4*>(dl + 2 * q) = f4(acc[t][q][c].l.x, acc[t][q][c].l.y, acc[t][q + 1][c].l.x,
                                                        acc[t][q + 1][c].l.y);
        }
      }
    }
  };

  product(MODE != FD_INV);
  if constexpr (MODE == FD_FWD) {
    if constexpr (XAX) {
      __syncthreads();  // every warp has read the panel
      put_cols();
      __syncthreads();
      const int gr = J.pitch / 4;
#pragma unroll 4
      for (int q = tid; q < TC * gr; q += nt) {
        const int c = q / gr, x = (q - c * gr) * 4;
        if (c0 + c >= J.ncols) break;
        const long long o = (c0 + c) * J.pitch + x;
        *reinterpret_cast<float4*>(J.s + o) = *reinterpret_cast<const float4*>(ph + c * P + x);
        if constexpr (FF) *reinterpret_cast<float4*>(J.sl + o) = *reinterpret_cast<const float4*>(pl + c * P + x);
      }
    } else {
      const long long col = c0 + cl;
      if (col < J.ncols) {
        const long long o = (col / J.cw) * J.cs + col % J.cw;
        put_rows(J.s + o, J.sl + o, J.is);
      }
    }
    return;
  }

  if constexpr (MODE == FD_SOLVE) {
    if (warp < tiles) ring_of(warp, false).start();  // ahead of the division and the barriers
    // divide by the eigenvalues; r.z is the sum of c^2 / lambda over the modes
    const long long col = c0 + cl;
    const bool ok = col < J.ncols;
    const int kx = ok ? (int)(col % J.pitch) : 0, ky = ok ? (int)(col / J.pitch) : 0;
    const float2 h2 = J.h2;
    DotAcc<float> dot;
#pragma unroll
    for (int t = 0; t < TPW; ++t) {
      const int tile = warp + t * nw;
      if (tile >= tiles) break;
      const bool odd = tile >= te;
      const int k0 = (odd ? tile - te : tile) * kFdTile + kq, half = odd ? no : ne, row0 = odd ? ne : 0;
#pragma unroll
      for (int c = 0; c < CT; ++c) {
        float2 xy = make_float2(J.mx[kx + c] + J.my[ky], 0.0f);
        if constexpr (FF) xy = fd_ff_add(make_float2(J.mx[kx + c], J.mxl[kx + c]), make_float2(J.my[ky], J.myl[ky]));
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int kz = row0 + min(k0 + k, half - 1);  // outputs past the half are zero
          FdAcc<FF>& a = acc[t][k >> 1][c];
          const float ch = hi(a, k & 1);
          if constexpr (FF) {
            const float cw = lo(a, k & 1);
            const float2 y = fd_ff_rcp(fd_ff_add(xy, make_float2(J.mz[kz], J.mzl[kz])));
            const float2 v = ff_mul(ff_mul(h2, y), make_float2(ch, cw));
            dot.add(ch, v.x);
            dot.lo += fmaf(ch, v.y, cw * v.x);
            if (k & 1)
              a.h.y = v.x, a.l.y = v.y;
            else
              a.h.x = v.x, a.l.x = v.y;
          } else {
            const float v = ch * (h2.x / (xy.x + J.mz[kz]));
            dot.add(ch, v);
            if (k & 1)
              a.h.y = v;
            else
              a.h.x = v;
          }
        }
      }
    }
    __syncthreads();  // every warp has read the panel
    put_rows(ph + cl, pl + cl, P);
    __syncthreads();
    product(false);
    // the blocks' parts of r.z: the last block sums them in order and sets beta,
    // as the V-cycle's last pass does
    __shared__ double dsm[16];
    __shared__ bool last;
    if (J.sc) {
      const double v = fd_block_sum(dot.value(), dsm, tid, nt);
      if (tid == 0) {
        J.red.partials[bid] = v;
        __threadfence();
        last = atomicAdd(J.red.counter, 1u) == (unsigned)(J.nblocks - 1);
      }
      __syncthreads();
      if (last) {
        __threadfence();
        double s = 0.0;
        for (int b = tid; b < J.nblocks; b += nt) s += __ldcg(&J.red.partials[b]);
        s = fd_block_sum(s, dsm, tid, nt);
        if (tid == 0) {
          if constexpr (FF) s = scalbn(s, 2 * fd_exponent(J.sc) + J.eh);
          MgFin{J.sc}(&s);
          *J.red.counter = 0u;
        }
      }
    }
  }
  __syncthreads();
  if constexpr (XAX)
    put_cols();
  else
    put_rows(ph + cl, pl + cl, P);
  __syncthreads();

  // ---- f_i and f_{n-1-i} from the even and odd parts ----
  if constexpr (XAX) {
    T* out = static_cast<T*>(J.out);
    const int kz = FF ? fd_exponent(J.sc) + J.eh : 0;
    auto value = [&](float e, float el, float d, float dl) -> T {
      if constexpr (FF) {
        const float2 v = fd_ff_add(make_float2(e, el), make_float2(d, dl));
        return double_of_float(v.x, kz) + double_of_float(v.y, kz);
      } else {
        return e + d;
      }
    };
    if (J.vec) {
      // a lane stores 16 bytes of its widest array at a time (with 32 the sectors of a
      // store are half filled: 98 against 45 us for the correcting pass at 192^3)
      const int cols = (int)min((long long)TC, J.ncols - c0);
      auto halves = [&](auto gs, int c, int x, T* up, T* dn) {
        constexpr int GS = decltype(gs)::value;
        float e[GS], d[GS], el[GS] = {}, dl[GS] = {};
        fd_get(ph + c * P + x, e);
        fd_get(ph + c * P + oo + x, d);
        if constexpr (FF) {
          fd_get(pl + c * P + x, el);
          fd_get(pl + c * P + oo + x, dl);
        }
#pragma unroll
        for (int k = 0; k < GS; ++k) {
          up[k] = value(e[k], el[k], d[k], dl[k]);
          dn[GS - 1 - k] = value(e[k], el[k], -d[k], -dl[k]);
        }
      };
      if (FF || out) {  // (only FP32 passes correct)
        constexpr int GS = 16 / (int)sizeof(T);
        const int gr = ne / GS, items = cols * gr;
#pragma unroll 2
        for (int q = tid; q < items; q += nt) {
          const int c = q / gr, x = (q - c * gr) * GS;
          T up[GS], dn[GS];
          halves(std::integral_constant<int, GS>{}, c, x, up, dn);
          const long long o = (c0 + c) * n;
          fd_store16(out + o + x, up);
          fd_store16(out + o + n - GS - x, dn);
        }
      } else if constexpr (!FF) {
        // the potential's old values of four items in flight together
        const int gr = ne / 2, items = cols * gr;
        for (int q0 = tid; q0 < items; q0 += 4 * nt) {
          double2 pu[4], pd[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int q = q0 + k * nt, c = q / gr, x = (q - c * gr) * 2;
            const long long o = (c0 + c) * n;
            if (q < items) {
              pu[k] = *reinterpret_cast<const double2*>(J.phi64 + o + x);
              pd[k] = *reinterpret_cast<const double2*>(J.phi64 + o + n - 2 - x);
            }
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int q = q0 + k * nt, c = q / gr, x = (q - c * gr) * 2;
            const long long o = (c0 + c) * n;
            if (q < items) {
              T up[2], dn[2];
              halves(std::integral_constant<int, 2>{}, c, x, up, dn);
              fd_correct2(J, o + x, pu[k], up);
              fd_correct2(J, o + n - 2 - x, pd[k], dn);
            }
          }
        }
      }
    } else {
      for (int c = warp; c < TC; c += nw) {
        if (c0 + c >= J.ncols) break;
        const long long o = (c0 + c) * n;
#pragma unroll 4
        for (int x = lane; x < n; x += 32) {
          const int i = x < ne ? x : n - 1 - x;
          const float sg = x < ne ? 1.0f : -1.0f;
          const float d = i < no ? sg * ph[c * P + oo + i] : 0.0f;
          float el = 0.0f, dl = 0.0f;
          if constexpr (FF) {
            el = pl[c * P + i];
            dl = i < no ? sg * pl[c * P + oo + i] : 0.0f;
          }
          const T v = value(ph[c * P + i], el, d, dl);
          if (FF || out)
            out[o + x] = v;
          else if constexpr (!FF)
            fd_correct(J, o + x, v);
        }
      }
    }
  } else {
    constexpr int CG = TC / 4;
#pragma unroll 2
    for (int q = tid; q < ne * CG; q += nt) {
      const int i = q / CG, c = (q % CG) * 4;
      const long long col = c0 + c;
      if (col >= J.ncols) continue;
      const long long o = (col / J.cw) * J.cs + col % J.cw;
      const float4 e = *reinterpret_cast<const float4*>(ph + i * P + c);
      float4 el = e, d = f4(0.f, 0.f, 0.f, 0.f), dl = d;
      if constexpr (FF) el = *reinterpret_cast<const float4*>(pl + i * P + c);
      if (i < no) {
        d = *reinterpret_cast<const float4*>(ph + (ne + i) * P + c);
        if constexpr (FF) dl = *reinterpret_cast<const float4*>(pl + (ne + i) * P + c);
      }
      float* up = J.s + o + (long long)i * J.is;
      float* dn = J.s + o + (long long)(n - 1 - i) * J.is;
      if constexpr (FF) {
        float* upl = J.sl + o + (long long)i * J.is;
        float* dnl = J.sl + o + (long long)(n - 1 - i) * J.is;
        const float2 a0 = fd_ff_add(make_float2(e.x, el.x), make_float2(d.x, dl.x));
        const float2 a1 = fd_ff_add(make_float2(e.y, el.y), make_float2(d.y, dl.y));
        const float2 a2 = fd_ff_add(make_float2(e.z, el.z), make_float2(d.z, dl.z));
        const float2 a3 = fd_ff_add(make_float2(e.w, el.w), make_float2(d.w, dl.w));
        *reinterpret_cast<float4*>(up) = f4(a0.x, a1.x, a2.x, a3.x);
        *reinterpret_cast<float4*>(upl) = f4(a0.y, a1.y, a2.y, a3.y);
        if (i < no) {
          const float2 b0 = fd_ff_add(make_float2(e.x, el.x), make_float2(-d.x, -dl.x));
          const float2 b1 = fd_ff_add(make_float2(e.y, el.y), make_float2(-d.y, -dl.y));
          const float2 b2 = fd_ff_add(make_float2(e.z, el.z), make_float2(-d.z, -dl.z));
          const float2 b3 = fd_ff_add(make_float2(e.w, el.w), make_float2(-d.w, -dl.w));
          *reinterpret_cast<float4*>(dn) = f4(b0.x, b1.x, b2.x, b3.x);
          *reinterpret_cast<float4*>(dnl) = f4(b0.y, b1.y, b2.y, b3.y);
        }
      } else {
        *reinterpret_cast<float4*>(up) = f4(e.x + d.x, e.y + d.y, e.z + d.z, e.w + d.w);
        if (i < no) *reinterpret_cast<float4*>(dn) = f4(e.x - d.x, e.y - d.y, e.z - d.z, e.w - d.w);
      }
    }
  }
}

template <typename T, bool XAX, int MODE, int CT, int TPW>
__global__ void __maxnreg__(TPW == 1 ? 80 : 128) fd_kernel(const __grid_constant__ FdJob J) {
  pdl_enter();
  extern __shared__ __align__(16) float fd_sm[];
  if ((J.sc && J.sc->done) || (J.gate && J.gate->done)) return;
  fd_panel<T, XAX, MODE, CT, TPW>(J, (long long)blockIdx.x * (16 * CT), blockIdx.x, fd_sm);
}

// The same pass for several grids of a batch: block b takes panel tiles[b].panel
// of job tiles[b].job, always with eight warps, so that a grid's sums do not
// depend on the others.
struct FdTile {
  int job, panel;
};
constexpr int kFdBatchWarps = 8;
template <typename T, bool XAX, int MODE, int CT, int TPW>
__global__ void __maxnreg__(TPW == 1 ? 80 : 128)
    fd_batch_kernel(const FdTile* __restrict__ tiles, const FdJob* __restrict__ jobs) {
  extern __shared__ __align__(16) float fd_sm[];
  const FdTile t = tiles[blockIdx.x];
  const FdJob J = jobs[t.job];
  if ((J.sc && J.sc->done) || (J.gate && J.gate->done)) return;
  fd_panel<T, XAX, MODE, CT, TPW>(J, (long long)t.panel * (16 * CT), t.panel, fd_sm);
}

}  // namespace ofd
