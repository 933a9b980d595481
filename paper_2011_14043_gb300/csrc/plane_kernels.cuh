// Small 2-D grids (nz = 1: Ez, Hx, Hy): any number of steps in one launch, the
// state held in the shared memory of one cluster of 16 thread blocks.
//
// A step of such a grid is two line solves of a few microseconds of work:
// launched one by one (or as graph nodes) they cost their launches, their
// loads and, in FP64, the pipe of the few SMs their blocks land on (an FP64
// warp instruction holds its scheduler's pipe for 64 cycles, measured).  Here
// a block owns R rows (Ez and Hy, for the x lines of A) and C columns (Ez and
// Hx, for the y lines of B); Hy and Hx never leave it.  A procedure reads its
// lines from the block's own shared memory, solves them one warp to a line
// (L = 2, 4 or 8 nodes per lane, so that 64 lines keep 64 schedulers busy),
// and pushes the new Ez to the blocks that own its columns (or rows) in
// 16-byte stores; a cluster barrier (380 cycles) separates the two.  Probes and
// the source are handled in the loop.
// 64 x 64 FP64 FADI with a probe: 30.7 us per step before, 6.1 now (6.3 with
// the columns pulled from the row owners element by element).  Of a
// procedure's 5,800 cycles the solve takes 3,700: 33 FP64 instructions in a
// dependent chain at 64 cycles each, and the scans' shuffles.
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "line_kernels.cuh"

namespace fdtd {

constexpr int kPlaneBlocks = 16;   // blocks of the cluster
constexpr int kPlaneProbes = 16;

template <typename T>
struct PlaneParams {
  PairParams<T> p[2];      // A: (Ez, Hy) along x; B: (Ez, Hx) along y
  T* ez;
  T* hx;
  T* hy;
  int nx, ny;
  int R, RP, C, CP;        // rows and columns per block, their padded counts in shared memory
  int ld, ldc;             // elements per row (Hy) and per column (Hx)
  long long pitch;
  int nproc, seq[3];       // procedures of a step
  long long n0, nsteps;    // first step's index, steps of this launch
  // the source: sample (si, sj), -1: none; terms before and after each procedure
  int si, sj;
  const double* table;
  long long len;
  double pre[3][2], post[3][2];
  int pre_off[3][2], post_off[3][2];
  // probes: kind 0..2: Ez, Hx, Hy at (i, j); 3: a sample that no procedure
  // changes (value at ptr)
  int nprobes, average;    // average: (value after A + value after B - added source) / 2
  int pk[kPlaneProbes], pi[kPlaneProbes], pj[kPlaneProbes], pat_src[kPlaneProbes];
  const T* pptr[kPlaneProbes];
  double* out;             // [probe][cap], column n0 + step
  long long cap;
};

template <typename T>
__device__ __forceinline__ double plane_source(const PlaneParams<T>& p, double coef, long long n) {
  const double f = (n >= 0 && n < p.len) ? p.table[n] : 0.0;
  return __dmul_rn(coef, f);
}

template <typename T, int L>
__global__ void __launch_bounds__(512) plane_steps_kernel(const __grid_constant__ PlaneParams<T> p) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) unsigned char plane_smem[];
  T* row_e = reinterpret_cast<T*>(plane_smem);     // [i][row], RP rows
  T* col_e = row_e + (p.nx + 1) * p.RP;            // [j][column], CP columns
  T* hy = col_e + (p.ny + 1) * p.CP;               // [row][i]
  T* hx = hy + p.R * p.ld;                         // [column][j]
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nw = blockDim.x >> 5;
  const int row0 = rank * p.R, col0 = rank * p.C;
  const int j0 = lane * L;

  // the walls (row and column 0) are never pushed: they stay zero
  for (int k = threadIdx.x; k < (p.ny + 1) * p.CP; k += blockDim.x) col_e[k] = T(0);
  for (int k = threadIdx.x; k < (p.nx + 1) * p.RP; k += blockDim.x) {
    const int i = k / p.RP, r = k % p.RP, j = row0 + r;
    const long long at = (long long)j * p.pitch + i;
    const bool in = r < p.R && j < p.ny && FDTD_IN_RANGE(at, at + 1, p.p[0].n_elem);
    row_e[k] = in ? p.ez[at] : T(0);
    if (r < p.R) hy[r * p.ld + i] = in ? p.hy[at] : T(0);
  }
  for (int k = threadIdx.x; k < p.C * p.ny; k += blockDim.x) {
    const int c = k % p.C, j = k / p.C, i = col0 + c;
    const long long at = (long long)j * p.pitch + i;
    hx[c * p.ldc + j] = (i < p.nx && FDTD_IN_RANGE(at, at + 1, p.p[0].n_elem)) ? p.hx[at] : T(0);
  }
  // where this lane's L nodes of an x line (y line) go: the block that owns
  // those columns (rows; R and C are multiples of L), and the place in it
  T* to_cols = cl.map_shared_rank(col_e, min(j0, p.nx - 1) / p.C) + min(j0, p.nx - 1) % p.C;
  T* to_rows = cl.map_shared_rank(row_e, min(j0, p.ny - 1) / p.R) + min(j0, p.ny - 1) % p.R;
  const int my_probe = (int)threadIdx.x < p.nprobes ? (int)threadIdx.x : -1;
  bool probe_mine = false;
  const T* probe_at = nullptr;
  if (my_probe >= 0) {
    const int kind = p.pk[my_probe], i = p.pi[my_probe], j = p.pj[my_probe];
    if (kind == 3) {
      probe_mine = rank == 0;
      probe_at = p.pptr[my_probe];
    } else if (kind == 1) {
      probe_mine = i >= col0 && i < col0 + p.C;
      probe_at = hx + (i - col0) * p.ldc + j;
    } else {
      probe_mine = j >= row0 && j < row0 + p.R;
      probe_at = kind == 0 ? row_e + i * p.RP + (j - row0) : hy + (j - row0) * p.ld + i;
    }
  }
  cl.sync();

  // line q of this block in procedure k (operator OP): solve, push
  auto solve_line = [&](auto op_c, int k, int q, long long n) {
    constexpr int OP = decltype(op_c)::value;
    const PairParams<T>& pp = p.p[OP];
    const int N = pp.N;
    const int line = (OP == 0 ? row0 : col0) + q;
    if (line < 1 || line >= (OP == 0 ? p.ny : p.nx)) return;  // the whole warp
    const T* e = OP == 0 ? row_e + j0 * p.RP + q : col_e + j0 * p.CP + q;
    const int es = OP == 0 ? p.RP : p.CP;
    T* h = OP == 0 ? hy + q * p.ld + j0 : hx + q * p.ldc + j0;
    T E[L], H[L];
#pragma unroll
    for (int t = 0; t < L; ++t) {
      const bool in = j0 + t < N;
      E[t] = in ? e[t * es] : T(0);
      H[t] = in ? h[t] : T(0);
    }
    const int src_t = (p.si >= 0 && line == (OP == 0 ? p.sj : p.si)) ? (OP == 0 ? p.si : p.sj) - j0 : -1;
    const bool src = src_t >= 0 && src_t < L;
    auto add = [&](const double(&coef)[2], const int(&off)[2]) {
#pragma unroll
      for (int t = 0; t < L; ++t)
        if (t == src_t)
          for (int m = 0; m < 2; ++m)
            if (coef[m] != 0.0) E[t] = (T)__dadd_rn((double)E[t], plane_source(p, coef[m], n + off[m]));
    };
    if (src) add(p.pre[k], p.pre_off[k]);
    __syncwarp();
    row_solve_wall<T, L, 32>(pp, lane, E, H);
    if (src) add(p.post[k], p.post_off[k]);
    if (j0 >= N) return;
    T* to = OP == 0 ? to_cols + line * p.CP : to_rows + line * p.RP;
    if (j0 + L <= N) {
      store_seg<T, L>(to, E);
    } else {
#pragma unroll
      for (int t = 0; t < L; ++t)
        if (j0 + t < N) to[t] = E[t];
    }
#pragma unroll
    for (int t = 0; t < L; ++t)
      if (j0 + t < N) {
        h[t] = H[t];
        // (the next procedure may be A again, and probes read the rows)
        if (OP == 0) row_e[(j0 + t) * p.RP + q] = E[t];
      }
  };

  for (long long st = 0; st < p.nsteps; ++st) {
    const long long n = p.n0 + st;
    double stash = 0.0;
    for (int k = 0; k < p.nproc; ++k) {
      if (p.seq[k] == 0) {
        for (int q = warp; q < p.R; q += nw) solve_line(std::integral_constant<int, 0>(), k, q, n);
      } else {
        for (int q = warp; q < p.C; q += nw) solve_line(std::integral_constant<int, 1>(), k, q, n);
      }
      if (p.nprobes && p.average && k == 0) {
        // after A (rows of this block only): what the average needs of it
        __syncthreads();
        if (probe_mine) stash = (double)*probe_at;
      }
      cl.sync();
    }
    if (p.nprobes) {
      if (probe_mine) {
        double v = (double)*probe_at;
        if (p.average) {
          const double sub = p.pat_src[my_probe] ? plane_source(p, p.post[1][0], n + p.post_off[1][0]) : 0.0;
          v = 0.5 * (stash + v - sub);
        }
        p.out[(long long)my_probe * p.cap + n] = v;
      }
      __syncthreads();  // before this block's rows change again
    }
  }

  for (int k = threadIdx.x; k < (p.nx + 1) * p.R; k += blockDim.x) {
    const int i = k % (p.nx + 1), r = k / (p.nx + 1), j = row0 + r;
    const long long at = (long long)j * p.pitch + i;
    if (j >= p.ny || !FDTD_IN_RANGE(at, at + 1, p.p[0].n_elem)) continue;
    p.ez[at] = row_e[i * p.RP + r];
    p.hy[at] = hy[r * p.ld + i];
  }
  for (int k = threadIdx.x; k < p.C * p.ny; k += blockDim.x) {
    const int c = k % p.C, j = k / p.C, i = col0 + c;
    const long long at = (long long)j * p.pitch + i;
    if (i >= p.nx || !FDTD_IN_RANGE(at, at + 1, p.p[0].n_elem)) continue;
    p.hx[at] = hx[c * p.ldc + j];
  }
}

}  // namespace fdtd
