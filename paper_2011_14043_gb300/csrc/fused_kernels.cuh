// One launch per updating procedure: the three pairs (lines along y, z and x,
// disjoint arrays) share a grid, each pair a range of blocks.
//
// What bound the one-launch-per-pair kernels (ncu, GB300): instruction issue,
// not arithmetic.  A 256^3 launch issued 46-50 warp instructions per node
// (FP32, homogeneous) and 112-127 (per-node media) for 18 and 25 FMAs:
// 64-bit addresses and line numbers, per-node bounds, products shuffled
// through the carry scans.  Small grids waited on three launches forked and
// joined in every procedure.  Here
//  - y/z lines: a warp holds 8 columns x 4 segments of L = 8 nodes; an FP32
//    column is two adjacent x lines, moved as 8-byte vectors and computed
//    with packed FP32 FMAs (same rounding as the scalar ones).  Carries join
//    by two shuffles in the warp, then over the warps of the tile through
//    shared memory with one barrier per sweep.
//  - homogeneous media: a segment's carry product is the constant (-m)^L, so
//    the scans move values only (and the tiles' stop where the product is
//    below 2^-50 of the carry).
//  - 32-bit element offsets; a node's address is formed once for all arrays.
//  - the point source is added by the thread that owns its sample.
// FADI 128^3 FP32: 37.3 -> 30.8 us per step, 64^3 16.5 -> 9.9, 32^3 13.6 -> 7.0
// (16 steps to a graph, programmatic edges), 219x101x75 45.7 -> 30.3 (the TMA
// kernel's blocks held 3-4 warps there).  What bounds it now: 24 warps per SM
// (80 registers) waiting on the loads of their own tile; at 128^3 it moves
// 6.5 TB/s of algorithmic bytes out of L2.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "line_kernels.cuh"

namespace fdtd {

constexpr int kFusedL = 8;         // nodes per segment
constexpr int kFusedMaxN = 256;    // 8 warps x 4 segments x 8 nodes
constexpr int kFusedThreads = 256;

// A y/z thread's column (FP32 fields): V = 2 adjacent x lines, one operation on
// both of them.
template <typename T>
struct Wide;
template <>
struct Wide<float> {
  using type = float2;
  static constexpr int V = 2;
};

__device__ __forceinline__ float2 wset(float2, float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 wfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 wmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 wadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 wsub(float2 a, float2 b) {
  return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a);  // one rounding, as a - b
}
__device__ __forceinline__ float2 wup(float2 a, int d) {
  return make_float2(__shfl_up_sync(0xffffffffu, a.x, d), __shfl_up_sync(0xffffffffu, a.y, d));
}
__device__ __forceinline__ float2 wdown(float2 a, int d) {
  return make_float2(__shfl_down_sync(0xffffffffu, a.x, d), __shfl_down_sync(0xffffffffu, a.y, d));
}
__device__ __forceinline__ float2 wfrom(float2 a, int l) {
  return make_float2(__shfl_sync(0xffffffffu, a.x, l), __shfl_sync(0xffffffffu, a.y, l));
}
__device__ __forceinline__ float2 wsel(bool c, float2 a, float2 b) { return make_float2(c ? a.x : b.x, c ? a.y : b.y); }

// (hi + lo) x + c, the coefficient a scalar of the field precision
template <typename T, typename W>
__device__ __forceinline__ W wfma2(T hi, T lo, W x, W c) {
  return wfma(wset(x, hi), x, wfma(wset(x, lo), x, c));
}

// A point source on one E sample, added by the thread that owns it: before
// the solve (pre) and to the new E (post); each term is coef f(n + off) with
// f read from a device table at the device step counter (plus the step's
// place in the graph), rounded before the add as the host path forms it.
struct FusedSource {
  const double* table;
  const long long* step;
  long long len;
  int sub;                 // steps since the counter's value
  int ec;                  // component (0..2), -1: none
  int i, j, k;
  double pre[2], post[2];
  int pre_off[2], post_off[2];
};

template <typename T>
__device__ __noinline__ T source_add(const FusedSource& s, const double (&coef)[2], const int (&off)[2], T v) {
  for (int q = 0; q < 2; ++q) {
    if (coef[q] == 0.0) continue;
    const long long n = *s.step + s.sub + off[q];
    const double f = (n >= 0 && n < s.len) ? s.table[n] : 0.0;
    v = (T)__dadd_rn((double)v, __dmul_rn(coef[q], f));
  }
  return v;
}

template <typename T>
struct FusedParams {
  PairParams<T> p[3];      // lines along y, z, x
  int ec[3];               // E component of each pair
  int nb[3];               // blocks of each pair
  int wpt[2];              // y, z: warps per tile of 8 columns
  int tpb[2];              // y, z: tiles per block
  int tiles_x[2];          // y, z: tiles per outer index
  unsigned ntiles[2];
  int lpl;                 // x: lanes per line
  unsigned div[3];         // ceil(2^32 / d) of d = tiles_x (y, z), n_o (x); 0: d = 1
  FusedSource src;
};

// n / d by the precomputed reciprocal: exact while n (d - 1) < 2^32 (n: lines
// or tiles, at most 2^20; d at most 1024).
__device__ __forceinline__ unsigned fast_div(unsigned n, unsigned m) { return m ? __umulhi(n, m) : n; }

template <typename T>
__device__ __forceinline__ T* at_bytes(T* base, unsigned byte_off) {
  return reinterpret_cast<T*>(reinterpret_cast<uintptr_t>(base) + byte_off);
}

__device__ __forceinline__ void tile_barrier(int id, int threads) {
  __syncwarp();
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Shared memory of a block: the warps' carries and (per-node media) products
// of both sweeps, and what the wall correction of a tile needs of its first
// two segments.  Indexed by the warp in the block, then the column.
template <typename W>
struct TileShare {
  W fa[8][8], fp[8][8], ba[8][8], bp[8][8], y1[8][8], b1[8][8];
};

// The columns of one tile on its nw warps; this is warp w of them.
template <typename T, bool PN>
__device__ __forceinline__ void fused_strided_warp(const FusedParams<T>& fp, int dir, unsigned tile, int w, int nw,
                                                   int w0, int bar, TileShare<typename Wide<T>::type>& sh) {
  using W = typename Wide<T>::type;
  constexpr int V = Wide<T>::V, L = kFusedL;
  const PairParams<T>& p = fp.p[dir];
  const int lane = threadIdx.x & 31;
  const int c = lane & 7, sl = lane >> 3;
  const unsigned oo = fast_div(tile, fp.div[dir]);
  const int o = p.o_lo + (int)oo;
  const int x = (int)(tile - oo * (unsigned)fp.tiles_x[dir]) * (8 * V) + V * c;
  const int N = p.N;
  const int j0 = (w * 4 + sl) * L;
  const unsigned line = (unsigned)o * (unsigned)p.os + (unsigned)x;
  const bool in_grid = FDTD_IN_RANGE((long long)line, (long long)line + (long long)(N - 1) * p.ls + V, p.n_elem);
  const bool a0 = x >= p.lane_lo && x < p.lane_hi && in_grid;
  const bool a1 = x + 1 >= p.lane_lo && x + 1 < p.lane_hi && in_grid;
  const bool any = a0 || a1;
  const unsigned lsb = (unsigned)p.ls * (unsigned)sizeof(T);
  const unsigned off = line * (unsigned)sizeof(T) + (unsigned)j0 * lsb;
  const bool full = (w + 1) * 4 * L <= N;  // the same for the whole warp
  const W zero = wset(W(), T(0));

  W E[L], H[L], y[L], ib[PN ? L : 1], il[PN ? L : 1];
  W hm1 = zero, ibp = zero, ilp = zero;
#pragma unroll
  for (int t = 0; t < L; ++t) E[t] = H[t] = y[t] = zero;
  if constexpr (PN) {
#pragma unroll
    for (int t = 0; t < L; ++t) ib[t] = il[t] = zero;
  }
  if (any) {
#pragma unroll
    for (int t = 0; t < L; ++t) {
      if (full || j0 + t < N) {
        const unsigned at = off + (unsigned)t * lsb;
        E[t] = *reinterpret_cast<const W*>(at_bytes(p.e_in, at));
        H[t] = *reinterpret_cast<const W*>(at_bytes(p.h_in, at));
        if constexpr (PN) {
          y[t] = *reinterpret_cast<const W*>(at_bytes(p.nq, at));
          ib[t] = *reinterpret_cast<const W*>(at_bytes(p.nib, at));
          il[t] = *reinterpret_cast<const W*>(at_bytes(p.nibl, at));
        }
      }
    }
    if (j0 > 0 && j0 <= N) {
      const unsigned at = off - lsb;
      hm1 = *reinterpret_cast<const W*>(at_bytes(p.h_in, at));
      if constexpr (PN) {
        ibp = *reinterpret_cast<const W*>(at_bytes(p.nib, at));
        ilp = *reinterpret_cast<const W*>(at_bytes(p.nibl, at));
      }
    }
  }
  // the source's node in this thread's column, or -1
  int src_t = -1;
  bool src_hi = false;
  if (fp.src.ec == fp.ec[dir] && fp.src.ec >= 0) {
    const int so = dir == 0 ? fp.src.k : fp.src.j, sj = dir == 0 ? fp.src.j : fp.src.k;
    if (so == o && sj >= j0 && sj < j0 + L && fp.src.i >= x && fp.src.i < x + V) {
      src_t = sj - j0;
      src_hi = fp.src.i != x;
    }
  }
  auto source = [&](const double(&coef)[2], const int(&offs)[2]) {
#pragma unroll
    for (int t = 0; t < L; ++t)
      if (t == src_t) {
        if (src_hi) E[t].y = source_add<T>(fp.src, coef, offs, E[t].y);
        else E[t].x = source_add<T>(fp.src, coef, offs, E[t].x);
      }
  };
  if (src_t >= 0) source(fp.src.pre, fp.src.pre_off);

  // right-hand side and forward sweep from a zero carry
  W win;
  if constexpr (!PN) {
    const T nmh = -p.cv[2], nml = -p.cv[3];
    W hp = hm1;
#pragma unroll
    for (int t = 0; t < L; ++t) {
      W r = wfma(wset(zero, p.kb), wsub(H[t], hp), E[t]);
      hp = H[t];
      if (t == 0 && j0 == 0) r = zero;  // node 0: the wall
      y[t] = t == 0 ? r : wfma2(nmh, nml, y[t - 1], r);
    }
    W a = y[L - 1];
    {
      const W u1 = wup(a, 8);
      if (sl >= 1) a = wfma2(p.qf[0][L - 1], p.qf[1][L - 1], u1, a);
      const W u2 = wup(a, 16);
      if (sl >= 2) a = wfma2(p.qf[0][2 * L - 1], p.qf[1][2 * L - 1], u2, a);
    }
    W yin = wup(a, 8);
    if (sl == 0) yin = zero;
    if (nw > 1) {
      if (sl == 3) sh.fa[w0 + w][c] = a;
      tile_barrier(bar, nw * 32);
      W cx = zero;
      for (int k = max(0, w - p.kx); k < w; ++k)
        cx = wfma2(p.qf[0][4 * L - 1], p.qf[1][4 * L - 1], cx, sh.fa[w0 + k][c]);
      const T sh_ = sl == 0 ? T(1) : p.qf[0][sl * L - 1], sl_ = sl == 0 ? T(0) : p.qf[1][sl * L - 1];
      yin = wfma2(sh_, sl_, cx, yin);
    }
#pragma unroll
    for (int t = 0; t < L; ++t) y[t] = wfma2(p.qf[0][t], p.qf[1][t], yin, y[t]);
    if (!full) {
      // nodes from N on hold no unknown: a zero value there makes their w zero
#pragma unroll
      for (int t = 0; t < L; ++t) y[t] = wsel(j0 + t < N, y[t], zero);
    }
    W wn = zero;
#pragma unroll
    for (int t = L - 1; t >= 0; --t) {
      const W u = wfma(wset(zero, nmh), wn, wfma(wset(zero, nml), wn, wmul(y[t], wset(zero, p.cv[1]))));
      y[t] = wfma(y[t], wset(zero, p.cv[0]), u);
      wn = y[t];
    }
    W b = y[0];
    {
      const W d1 = wdown(b, 8);
      if (sl <= 2) b = wfma2(p.qf[0][L - 1], p.qf[1][L - 1], d1, b);
      const W d2 = wdown(b, 16);
      if (sl <= 1) b = wfma2(p.qf[0][2 * L - 1], p.qf[1][2 * L - 1], d2, b);
    }
    win = wdown(b, 8);
    if (sl == 3) win = zero;
    const bool corr = w * 4 * L < p.kg_len;  // the same for the whole warp
    W w1 = zero;
    if (nw > 1) {
      if (sl == 0) sh.ba[w0 + w][c] = b;
      if (w == 0 && sl == 0) sh.y1[w0][c] = y[1];
      if (w == 0 && sl == 1) sh.b1[w0][c] = b;
      tile_barrier(bar, nw * 32);
      W cx = zero;
      for (int k = min(nw - 1, w + p.kx); k > w; --k)
        cx = wfma2(p.qf[0][4 * L - 1], p.qf[1][4 * L - 1], cx, sh.ba[w0 + k][c]);
      const int r = 3 - sl;
      const T rh = r == 0 ? T(1) : p.qf[0][r * L - 1], rl = r == 0 ? T(0) : p.qf[1][r * L - 1];
      win = wfma2(rh, rl, cx, win);
      if (corr) {
        W c0 = zero;  // the carry into warp 0
        for (int k = min(nw - 1, p.kx); k > 0; --k)
          c0 = wfma2(p.qf[0][4 * L - 1], p.qf[1][4 * L - 1], c0, sh.ba[w0 + k][c]);
        const W win0 = wfma2(p.qf[0][3 * L - 1], p.qf[1][3 * L - 1], c0, sh.b1[w0][c]);
        w1 = wfma2(p.qf[0][L - 2], p.qf[1][L - 2], win0, sh.y1[w0][c]);
      }
    } else {
      const W win0 = wfrom(b, 8 + c);
      w1 = wfma2(p.qf[0][L - 2], p.qf[1][L - 2], win0, wfrom(y[1], c));
    }
#pragma unroll
    for (int t = 0; t < L; ++t) y[t] = wfma2(p.qf[0][L - 1 - t], p.qf[1][L - 1 - t], win, y[t]);
    if (j0 == 0) y[0] = zero;
    if (corr) {
      // rank-one wall correction (as in strided_solve_wall)
      const T* kgh = p.tab + TB_KGH * p.tlen + j0;
      const T* kgl = p.tab + TB_KGL * p.tlen + j0;
#pragma unroll
      for (int t = 0; t < L; ++t) y[t] = wfma2(__ldg(kgh + t), __ldg(kgl + t), w1, y[t]);
      win = wfma2(__ldg(kgh + L), __ldg(kgl + L), w1, win);
    }
  } else {
    // rows scaled by 1/b_j; y holds q_j until the right-hand side is formed.
    // Multipliers as in phase_forward / phase_backward: 1/beta and the
    // off-diagonal, each as hi + lo, one after the other.
    const W nh = wset(zero, -p.offh), nl = wset(zero, -p.offl), ks = wset(zero, p.ks);
    const W one = wset(zero, T(1));
    W pr = one, hp = hm1;
#pragma unroll
    for (int t = 0; t < L; ++t) {
      const W r = wfma(y[t], E[t], wmul(ks, wsub(H[t], hp)));
      hp = H[t];
      const W bp = t == 0 ? ibp : ib[t == 0 ? 0 : t - 1];
      const W m = wmul(nh, bp);
      if (t == 0) {
        y[t] = r;
      } else {
        const W v = wfma(bp, y[t - 1], wmul(il[t - 1], y[t - 1]));
        y[t] = wfma(nh, v, wfma(nl, v, r));
      }
      pr = wmul(pr, m);
    }
    W a = y[L - 1];
    {
      const W u1 = wup(a, 8), q1 = wup(pr, 8);
      if (sl >= 1) {
        a = wfma(pr, u1, a);
        pr = wmul(pr, q1);
      }
      const W u2 = wup(a, 16), q2 = wup(pr, 16);
      if (sl >= 2) {
        a = wfma(pr, u2, a);
        pr = wmul(pr, q2);
      }
    }
    W yin = wup(a, 8), pe = wup(pr, 8);
    if (sl == 0) {
      yin = zero;
      pe = one;
    }
    if (nw > 1) {
      if (sl == 3) {
        sh.fa[w0 + w][c] = a;
        sh.fp[w0 + w][c] = pr;
      }
      tile_barrier(bar, nw * 32);
      W cx = zero;
      for (int k = 0; k < w; ++k) cx = wfma(sh.fp[w0 + k][c], cx, sh.fa[w0 + k][c]);
      yin = wfma(pe, cx, yin);
    }
    // the carry, run through the segment's own multipliers (hi + lo, as in the
    // sweep: products of their hi parts alone bias the first node of
    // every segment by up to 2^-24 of its carry, the same way at every step)
    W q = yin;
#pragma unroll
    for (int t = 0; t < L; ++t) {
      const W bp = t == 0 ? ibp : ib[t == 0 ? 0 : t - 1];
      const W v = wfma(bp, q, wmul(t == 0 ? ilp : il[t == 0 ? 0 : t - 1], q));
      q = wfma(nh, v, wmul(nl, v));
      y[t] = wadd(q, y[t]);
    }
    W wn = zero;
    pr = one;
#pragma unroll
    for (int t = L - 1; t >= 0; --t) {
      const W m = wmul(nh, ib[t]);
      const W u = wfma(nh, wn, wfma(nl, wn, y[t]));
      y[t] = wfma(ib[t], u, wmul(il[t], u));
      pr = wmul(pr, m);
      wn = y[t];
    }
    W b = y[0];
    {
      const W d1 = wdown(b, 8), q1 = wdown(pr, 8);
      if (sl <= 2) {
        b = wfma(pr, d1, b);
        pr = wmul(pr, q1);
      }
      const W d2 = wdown(b, 16), q2 = wdown(pr, 16);
      if (sl <= 1) {
        b = wfma(pr, d2, b);
        pr = wmul(pr, q2);
      }
    }
    win = wdown(b, 8);
    pe = wdown(pr, 8);
    if (sl == 3) {
      win = zero;
      pe = one;
    }
    if (nw > 1) {
      if (sl == 0) {
        sh.ba[w0 + w][c] = b;
        sh.bp[w0 + w][c] = pr;
      }
      tile_barrier(bar, nw * 32);
      W cx = zero;
      for (int k = nw - 1; k > w; --k) cx = wfma(sh.bp[w0 + k][c], cx, sh.ba[w0 + k][c]);
      win = wfma(pe, cx, win);
    }
    q = win;
#pragma unroll
    for (int t = L - 1; t >= 0; --t) {
      const W u = wfma(nh, q, wmul(nl, q));
      q = wfma(ib[t], u, wmul(il[t], u));
      y[t] = wadd(q, y[t]);
    }
  }

  // H += kd (w_{f+1} - w_f), E <- alpha w + beta E
#pragma unroll
  for (int t = 0; t < L; ++t) {
    const W wnext = (t + 1 < L) ? y[t + 1] : win;
    H[t] = wfma(wset(zero, p.kd), wsub(wnext, y[t]), H[t]);
    E[t] = wfma(wset(zero, p.beta), E[t], wmul(wset(zero, p.alpha), y[t]));
  }
  if (src_t >= 0) source(fp.src.post, fp.src.post_off);
  if (!any) return;
  const bool both = a0 && a1;
#pragma unroll
  for (int t = 0; t < L; ++t) {
    if (full || j0 + t < N) {
      const unsigned at = off + (unsigned)t * lsb;
      if (both) {
        *reinterpret_cast<W*>(at_bytes(p.e_out, at)) = E[t];
        *reinterpret_cast<W*>(at_bytes(p.h_out, at)) = H[t];
      } else {
        // one of the two lines is a wall's or past the last one
        const unsigned a1b = at + (a0 ? 0u : (unsigned)sizeof(T));
        *at_bytes(p.e_out, a1b) = a0 ? E[t].x : E[t].y;
        *at_bytes(p.h_out, a1b) = a0 ? H[t].x : H[t].y;
      }
    }
  }
}

// x lines, LPL lanes per line, L = 8 nodes per lane (32 / LPL lines per warp).
template <typename T, bool PN, int LPL>
__device__ __forceinline__ void fused_rows_warp(const FusedParams<T>& fp, unsigned gwarp) {
  constexpr int L = kFusedL, LPW = 32 / LPL;
  const PairParams<T>& p = fp.p[2];
  const int lane = threadIdx.x & 31;
  const int sl = lane % LPL;
  const unsigned n = (unsigned)p.n_o * (unsigned)p.n_o2;
  if (gwarp * LPW >= n) return;  // the whole warp
  const unsigned gl = gwarp * LPW + (unsigned)(lane / LPL);
  const unsigned line = min(gl, n - 1u);
  const unsigned kk = fast_div(line, fp.div[2]);
  const int jo = p.o_lo + (int)(line - kk * (unsigned)p.n_o), ko = p.o2_lo + (int)kk;
  const unsigned base = (unsigned)ko * (unsigned)p.os2 + (unsigned)jo * (unsigned)p.os;
  const int j0 = sl * L;
  const int N = p.N;
  const bool in_grid = gl < n && FDTD_IN_RANGE((long long)base, (long long)base + (N + L - 1) / L * L, p.n_elem);
  const unsigned at = (base + (unsigned)j0) * (unsigned)sizeof(T);
  T E[L], H[L];
#pragma unroll
  for (int t = 0; t < L; ++t) E[t] = H[t] = T(0);
  const bool mine = in_grid && j0 < N;
  if (mine) {
    // whole segments: the row pitch covers 32 segments, padding holds zeros
    load_seg<T, L>(at_bytes(p.e_in, at), E);
    load_seg<T, L>(at_bytes(p.h_in, at), H);
  }
  int src_t = -1;
  if (fp.src.ec == fp.ec[2] && fp.src.ec >= 0 && mine && fp.src.j == jo && fp.src.k == ko && fp.src.i >= j0 &&
      fp.src.i < j0 + L)
    src_t = fp.src.i - j0;
  if (src_t >= 0) {
#pragma unroll
    for (int t = 0; t < L; ++t)
      if (t == src_t) E[t] = source_add<T>(fp.src, fp.src.pre, fp.src.pre_off, E[t]);
  }
  if constexpr (PN) {
    T q[L], ib[L], il[L];
#pragma unroll
    for (int t = 0; t < L; ++t) q[t] = ib[t] = il[t] = T(0);
    if (mine) {
      load_seg<T, L>(at_bytes(p.nq, at), q);
      load_seg<T, L>(at_bytes(p.nib, at), ib);
      load_seg<T, L>(at_bytes(p.nibl, at), il);
    }
    row_solve_pn<T, L, LPL>(p, sl, E, H, q, ib, il);
  } else {
    row_solve_wall<T, L, LPL>(p, sl, E, H);
  }
  if (src_t >= 0) {
#pragma unroll
    for (int t = 0; t < L; ++t)
      if (t == src_t) E[t] = source_add<T>(fp.src, fp.src.post, fp.src.post_off, E[t]);
  }
  if (!mine) return;
  if (j0 + L <= N) {
    store_seg<T, L>(at_bytes(p.e_out, at), E);
    store_seg<T, L>(at_bytes(p.h_out, at), H);
  } else {
#pragma unroll
    for (int t = 0; t < L; ++t)
      if (j0 + t < N) {
        *at_bytes(p.e_out, at + t * (unsigned)sizeof(T)) = E[t];
        *at_bytes(p.h_out, at + t * (unsigned)sizeof(T)) = H[t];
      }
  }
}

// Block b of a procedure: [0, nb0) take the y lines, the next nb1 the z lines,
// the rest the x lines (LPL = 0: 8, 16 or 32 lanes per x line by fp.lpl).
template <typename T, bool PN, int LPL>
__device__ __forceinline__ void fused_block(const FusedParams<T>& fp, unsigned b,
                                            TileShare<typename Wide<T>::type>& sh) {
  const int warp = threadIdx.x >> 5;
  if (b < (unsigned)(fp.nb[0] + fp.nb[1])) {
    const int dir = b < (unsigned)fp.nb[0] ? 0 : 1;
    if (dir) b -= (unsigned)fp.nb[0];
    const int nw = fp.wpt[dir];
    const int g = warp / nw;
    const unsigned tile = b * (unsigned)fp.tpb[dir] + (unsigned)g;
    if (g >= fp.tpb[dir] || tile >= fp.ntiles[dir]) return;  // whole tiles leave together
    fused_strided_warp<T, PN>(fp, dir, tile, warp - g * nw, nw, g * nw, 1 + g, sh);
  } else {
    b -= (unsigned)(fp.nb[0] + fp.nb[1]);
    const unsigned gw = b * (blockDim.x >> 5) + (unsigned)warp;
    if constexpr (LPL != 0) {
      fused_rows_warp<T, PN, LPL>(fp, gw);
    } else {
      if (fp.lpl == 8) fused_rows_warp<T, PN, 8>(fp, gw);
      else if (fp.lpl == 16) fused_rows_warp<T, PN, 16>(fp, gw);
      else fused_rows_warp<T, PN, 32>(fp, gw);
    }
  }
}

// In a captured step the launches are chained by programmatic edges: the next
// procedure's blocks start while this one's last blocks drain, and wait for
// its stores before their first load.
template <typename T, bool PN, int LPL>
__global__ void __launch_bounds__(kFusedThreads, PN ? 2 : 3)
    proc_fused_kernel(const __grid_constant__ FusedParams<T> fp) {
  __shared__ TileShare<typename Wide<T>::type> sh;
  cudaTriggerProgrammaticLaunchCompletion();
  cudaGridDependencySynchronize();
  fused_block<T, PN, LPL>(fp, blockIdx.x, sh);
}

// The same for many grids: blocks[b] names the grid and the block within it;
// its parameters are copied to shared memory.  Ten cavities (5.9 M cells,
// eps_r blocks): 312 -> 280 us per FADI step against 16 launches per step on
// four branches, homogeneous ones 345 -> 217; 64 cavities (34 M cells) stay
// with the launches (1.35 ms against 1.73).
template <typename T, bool PN>
__global__ void __launch_bounds__(kFusedThreads, PN ? 2 : 3)
    proc_fused_batch_kernel(const FusedParams<T>* __restrict__ grids, const int2* __restrict__ blocks) {
  __shared__ TileShare<typename Wide<T>::type> sh;
  __shared__ FusedParams<T> fp;
  cudaTriggerProgrammaticLaunchCompletion();
  const int2 at = blocks[blockIdx.x];
  static_assert(sizeof(FusedParams<T>) % 4 == 0, "word copy");
  for (int k = threadIdx.x; k < (int)(sizeof(FusedParams<T>) / 4); k += blockDim.x)
    reinterpret_cast<int*>(&fp)[k] = reinterpret_cast<const int*>(grids + at.x)[k];
  __syncthreads();
  cudaGridDependencySynchronize();
  fused_block<T, PN, 0>(fp, (unsigned)at.y, sh);
}

}  // namespace fdtd
