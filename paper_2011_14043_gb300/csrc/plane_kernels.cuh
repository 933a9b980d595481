// Small 2-D grids (nz = 1: Ez, Hx, Hy): any number of steps in one launch, the
// state held in the shared memory of one cluster of 16 thread blocks.
//
// A step of such a grid is two line solves of a few microseconds of work:
// launched one by one (or as graph nodes) they cost their launches, their
// loads and, in FP64, the pipe of the few SMs their blocks land on (an FP64
// warp instruction holds its scheduler's pipe for 64 cycles, measured).  Here
// a block owns a strip of R rows of the three arrays.  The x lines of a
// procedure are its own rows; the y lines are dealt out over all warps of the
// cluster, each reading its column from the 16 blocks and writing it back
// (distributed shared memory, 200 cycles a load); a cluster barrier (380
// cycles) separates the two.  A warp takes one line, L = 2 (lines of up to
// 64 cells), 4 or 8 nodes per lane, so that 64 lines keep 64 schedulers busy.
// Probes and the source are handled in the loop.
// 64 x 64 FP64 FADI with a probe: 30.7 -> 6.3 us per step (of its 13,000 cycles
// the two solves take 8,000: about 35 FP64 instructions each at 64 cycles, and
// the scans' shuffles; the columns' scattered remote loads 2,500, the
// barriers with the stores behind them 2,700).
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

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
  int nx, ny, R, ld;       // R rows per block, ld elements per row in shared memory
  long long pitch;
  int nproc, seq[3];       // procedures of a step
  long long n0, nsteps;    // first step's index, steps of this launch
  // the source: sample (si, sj), -1: none; terms before and after each procedure
  int si, sj;
  const double* table;
  long long len;
  double pre[3][2], post[3][2];
  int pre_off[3][2], post_off[3][2];
  // probes: kind 0..2: Ez, Hx, Hy at (i, j) of the strips; 3: a sample that
  // no procedure changes (value at ptr)
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
  T* s_ez = reinterpret_cast<T*>(plane_smem);
  const int strip = p.R * p.ld;
  T* s_h[2] = {s_ez + 2 * strip, s_ez + strip};  // of A: Hy; of B: Hx
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nw = blockDim.x >> 5;
  const int row0 = rank * p.R;
  const int j0 = lane * L;

  for (int k = threadIdx.x; k < strip; k += blockDim.x) {
    const int r = k / p.ld, i = k % p.ld, j = row0 + r;
    const long long at = (long long)j * p.pitch + i;
    const bool in = j < p.ny && i <= p.nx && FDTD_IN_RANGE(at, at + 1, p.p[0].n_elem);
    s_ez[k] = in ? p.ez[at] : T(0);
    s_h[1][k] = in ? p.hx[at] : T(0);
    s_h[0][k] = in ? p.hy[at] : T(0);
  }
  // this lane's nodes of a y line: the block and row that hold them
  T* col[L];
#pragma unroll
  for (int t = 0; t < L; ++t) {
    const int j = j0 + t < p.ny ? j0 + t : 0;
    col[t] = cl.map_shared_rank(s_ez, j / p.R) + (j % p.R) * p.ld;
  }
  const int my_probe = (int)threadIdx.x < p.nprobes ? (int)threadIdx.x : -1;
  bool probe_mine = false;
  const T* probe_at = nullptr;
  if (my_probe >= 0) {
    const int kind = p.pk[my_probe];
    probe_mine = kind == 3 ? rank == 0 : (p.pj[my_probe] >= row0 && p.pj[my_probe] < row0 + p.R);
    if (probe_mine)
      probe_at = kind == 3 ? p.pptr[my_probe]
                           : (kind == 0 ? s_ez : s_h[kind == 1 ? 1 : 0]) + (p.pj[my_probe] - row0) * p.ld + p.pi[my_probe];
  }
  cl.sync();

  for (long long st = 0; st < p.nsteps; ++st) {
    const long long n = p.n0 + st;
    double stash = 0.0;
    for (int k = 0; k < p.nproc; ++k) {
      const int op = p.seq[k];
      const int lines = op == 0 ? p.R : p.nx - 1;
      const int first = op == 0 ? warp : rank * nw + warp, step = op == 0 ? nw : nw * kPlaneBlocks;
      for (int q = first; q < lines; q += step) {
        // A: row row0 + q of this block; B: column 1 + q
        const int line = op == 0 ? row0 + q : 1 + q;
        const PairParams<T>& pp = p.p[op];
        const int N = pp.N;
        if (op == 0 && (line < 1 || line >= p.ny)) continue;  // the whole warp
        T E[L], H[L];
#pragma unroll
        for (int t = 0; t < L; ++t) {
          const bool in = j0 + t < N;
          const T* e = op == 0 ? s_ez + q * p.ld + j0 + t : col[t] + line;
          E[t] = in ? *e : T(0);
          H[t] = in ? e[op == 0 ? 2 * strip : strip] : T(0);
        }
        const int src_t = (p.si >= 0 && line == (op == 0 ? p.sj : p.si)) ? (op == 0 ? p.si : p.sj) - j0 : -1;
        if (src_t >= 0 && src_t < L) {
#pragma unroll
          for (int t = 0; t < L; ++t)
            if (t == src_t)
              for (int m = 0; m < 2; ++m)
                if (p.pre[k][m] != 0.0)
                  E[t] = (T)__dadd_rn((double)E[t], plane_source(p, p.pre[k][m], n + p.pre_off[k][m]));
        }
        __syncwarp();
        row_solve_wall<T, L, 32>(pp, lane, E, H);
        if (src_t >= 0 && src_t < L) {
#pragma unroll
          for (int t = 0; t < L; ++t)
            if (t == src_t)
              for (int m = 0; m < 2; ++m)
                if (p.post[k][m] != 0.0)
                  E[t] = (T)__dadd_rn((double)E[t], plane_source(p, p.post[k][m], n + p.post_off[k][m]));
        }
#pragma unroll
        for (int t = 0; t < L; ++t) {
          if (j0 + t < N) {
            T* e = op == 0 ? s_ez + q * p.ld + j0 + t : col[t] + line;
            *e = E[t];
            e[op == 0 ? 2 * strip : strip] = H[t];
          }
        }
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

  for (int k = threadIdx.x; k < strip; k += blockDim.x) {
    const int r = k / p.ld, i = k % p.ld, j = row0 + r;
    if (j >= p.ny || i > p.nx) continue;
    const long long at = (long long)j * p.pitch + i;
    if (!FDTD_IN_RANGE(at, at + 1, p.p[0].n_elem)) continue;
    p.ez[at] = s_ez[k];
    p.hx[at] = s_h[1][k];
    p.hy[at] = s_h[0][k];
  }
}

}  // namespace fdtd
