// Coefficients of per-node media, formed on the device in FP64: the means of
// the per-cell media at the Yee samples, and the pivots of every grid line
// ("precomputed bidiagonally factorized elements", Sec. IV).
//
// A gradient or a sweep over media forms them once per evaluation, so their
// cost counts beside the steps.  On the host (one thread, six pairs of lines,
// a conversion pass and a pageable copy of every array) they took 53 ms of
// a 66 ms gradient evaluation on 96^3 cells and 1.25 s on 256^3; here one
// thread per line walks the pivot recurrence, bound by the FP64 pipe (one
// division per node).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "line_kernels.cuh"

namespace fdtd {

// Means of a per-cell array (compact [k][j][i]) at the samples of a component:
// over the in-domain cells among the offsets {-1, 0} along the axes with
// wx / wy / wz set (E edges: the two axes across; H faces: the axis of the
// component), added in the order k-offset fastest along the last averaged
// axis.  Samples outside the component's extent keep `fill`.
__global__ void cell_mean_kernel(const double* __restrict__ cell, double* __restrict__ out, int nx, int ny, int nz,
                                 int sx, int sy, int sz, int wx, int wy, int wz, long long pitch, long long plane,
                                 double fill) {
  const long long rows = (long long)(ny + 1) * (nz + 1);
  for (long long r = blockIdx.x; r < rows; r += gridDim.x) {
    const int j = (int)(r % (ny + 1));
    const int k = (int)(r / (ny + 1));
    const long long at = (long long)k * plane + (long long)j * pitch;
    if (!FDTD_IN_RANGE(at, at + pitch, plane * (nz + 1))) continue;
    for (int i = threadIdx.x; i < (int)pitch; i += blockDim.x) {
      double v = fill;
      if (i < sx && j < sy && k < sz) {
        double s = 0.0;
        int n = 0;
        for (int c = -wx; c <= 0; ++c)
          for (int b = -wy; b <= 0; ++b)
            for (int a = -wz; a <= 0; ++a) {
              const int ci = i + c, cj = j + b, ck = k + a;
              if (ci < 0 || cj < 0 || ck < 0 || ci >= nx || cj >= ny || ck >= nz) continue;
              s += cell[((long long)ck * ny + cj) * nx + ci];
              ++n;
            }
        v = n ? s / n : 1.0;
      }
      out[at + i] = v;
    }
  }
}

// One line per thread: rows scaled by 1/b_j (a symmetric matrix),
//   q_j w_j / 2 - (|ks| |kd| / 2) (w_{j+1} - 2 w_j + w_{j-1}) = q_j E_j + ks (H_j - H_{j-1}),
// q_j = 1/|b_j|, b_j = h / (2 eps), ks = s sign(h) / d_eta, plus loss sigma_j / 4
// on the diagonal.  Factored in FP64 from exactly the q_j, ks, kd the line
// kernels use (rounded to the field precision first), so each procedure is
// an exact Cayley transform of the medium those rounded values describe.
// Per-node mu (mr != nullptr): each face f (between nodes f and f+1) has its
// own coupling kd_f = s h / (2 mu d_eta) and off-diagonal -|ks| |kd_f| / 2.
// T is the field precision; FP32 fields keep 1/beta and the off-diagonals
// as hi + lo pairs.
struct FactorParams {
  long long ls, os, os2;
  int lane_lo, lane_hi, o_lo, n_o, o2_lo, n_o2, rows, N;
  const double* er;   // eps_r at the E samples
  const double* sr;   // sigma at the E samples (nullptr: sigma_u everywhere)
  const double* mr;   // mu_r at the H samples (nullptr: uniform mu)
  double sigma_u, loss_sign, h, eps2, mu2, sign, de, kk, off, ks_abs;  // eps2 = 2 eps0, mu2 = 2 mu0
  long long n_elem;
};

template <typename T>
__global__ void __launch_bounds__(64) factor_lines_kernel(const FactorParams p, T* __restrict__ nq, T* __restrict__ nib,
                                                          T* __restrict__ nibl, T* __restrict__ nkd,
                                                          T* __restrict__ noffh, T* __restrict__ noffl) {
  const long long line = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long nlx = p.rows ? p.n_o : p.lane_hi - p.lane_lo;
  const long long n_lines = p.rows ? nlx * p.n_o2 : nlx * p.n_o;
  if (line >= n_lines) return;
  long long base;
  if (p.rows) base = (long long)(p.o2_lo + (int)(line / nlx)) * p.os2 + (long long)(p.o_lo + (int)(line % nlx)) * p.os;
  else base = (long long)(p.o_lo + (int)(line / nlx)) * p.os + p.lane_lo + (int)(line % nlx);
  if (!FDTD_IN_RANGE(base, base + (long long)(p.N - 1) * p.ls + 1, p.n_elem)) return;
  constexpr bool hilo = sizeof(T) == 4;
  double ibm = 0.0;
  double kkm = p.kk, offm = p.off;  // of the face before the node
  if (p.mr) {
    const T kdf = (T)(p.sign * (p.h / (p.mu2 * p.mr[base])) / p.de);
    kkm = p.ks_abs * fabs((double)kdf);
    offm = -kkm / 2.0;
    nkd[base] = kdf;
    noffh[base] = (T)offm;
    if (hilo) noffl[base] = (T)(offm - (double)(T)offm);
  }
  for (int j = 1; j <= p.N - 1; ++j) {
    const long long at = base + (long long)j * p.ls;
    double kkj = p.kk, offj = p.off;
    if (p.mr) {
      const T kdf = (T)(p.sign * (p.h / (p.mu2 * p.mr[at])) / p.de);
      kkj = p.ks_abs * fabs((double)kdf);
      offj = -kkj / 2.0;
      nkd[at] = kdf;
      noffh[at] = (T)offj;
      if (hilo) noffl[at] = (T)(offj - (double)(T)offj);
    }
    const T q = (T)(1.0 / (fabs(p.h) / (p.eps2 * p.er[at])));
    const double loss = p.loss_sign != 0.0 ? p.loss_sign * (p.sr ? p.sr[at] : p.sigma_u) / 4.0 : 0.0;
    const double diag = (double)q / 2.0 + (p.mr ? (kkj + kkm) / 2.0 : p.kk) + loss;
    const double beta = diag - offm * offm * ibm;
    const double ib = 1.0 / beta;
    nq[at] = q;
    nib[at] = (T)ib;
    if (hilo) nibl[at] = (T)(ib - (double)(T)ib);
    ibm = ib;
    kkm = kkj;
    offm = offj;
  }
}

}  // namespace fdtd
