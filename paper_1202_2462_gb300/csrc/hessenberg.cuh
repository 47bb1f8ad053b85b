// The least squares of fixed-step GMRES by one warp.
#pragma once
#include "common.cuh"

namespace sapmg {

// argmin || beta e1 - H y || for the (m+1) x m Hessenberg H held by columns in
// shared memory (hr, hi: entry (i, k) at i + 33 k, zero below the subdiagonal;
// overwritten): column k on lane k; step j's rotation
// [conj a, conj b; -b, a] / sqrt(|a|^2 + |b|^2) is formed by every lane from the
// pivot column and applied to the lane's own, then the back substitution takes
// y_i out of all rows above at once.  A vanishing pivot column is left as it is and
// a zero diagonal entry gives y_i = 0.  m <= 32; every lane calls, lane i returns y_i.
__device__ __forceinline__ Cplx<double> hessenberg_warp(double* hr, double* hi, int m, double beta) {
  const int lane = threadIdx.x & 31;
  double gr = lane == 0 ? beta : 0.0, gi = 0.0;          // g_lane; g_32 only closes the residual
  __syncwarp();
  for (int j = 0; j < m; ++j) {
    const double ar = hr[j + j * 33], ai = hi[j + j * 33];
    const double br = hr[j + 1 + j * 33], bi = hi[j + 1 + j * 33];
    const double d2 = ar * ar + ai * ai + br * br + bi * bi;
    const double inv = rsqrt(d2);
    const double cr = d2 > 0.0 ? ar * inv : 1.0, ci = d2 > 0.0 ? ai * inv : 0.0;
    const double sr = d2 > 0.0 ? br * inv : 0.0, si = d2 > 0.0 ? bi * inv : 0.0;
    __syncwarp();                                         // every lane has read column j
    if (lane >= j && lane < m) {
      const double xr = hr[j + lane * 33], xi = hi[j + lane * 33];
      const double zr = hr[j + 1 + lane * 33], zi = hi[j + 1 + lane * 33];
      hr[j + lane * 33] = cr * xr + ci * xi + sr * zr + si * zi;
      hi[j + lane * 33] = cr * xi - ci * xr + sr * zi - si * zr;
      hr[j + 1 + lane * 33] = cr * zr - ci * zi - sr * xr + si * xi;
      hi[j + 1 + lane * 33] = cr * zi + ci * zr - sr * xi - si * xr;
    }
    const double xr = __shfl_sync(0xffffffffu, gr, j), xi = __shfl_sync(0xffffffffu, gi, j);
    if (lane == j) {                                      // g_{j+1} was 0
      gr = cr * xr + ci * xi;
      gi = cr * xi - ci * xr;
    } else if (lane == j + 1) {
      gr = -(sr * xr - si * xi);
      gi = -(sr * xi + si * xr);
    }
    __syncwarp();
  }
  double wr = 0.0, wi = 0.0;                              // the reciprocals of the diagonal, one a lane
  if (lane < m) {
    const double dr = hr[lane + lane * 33], di = hi[lane + lane * 33];
    const double d2 = dr * dr + di * di;
    if (d2 > 0.0) {
      const double q = 1.0 / d2;
      wr = dr * q;
      wi = -di * q;
    }
  }
  Cplx<double> y = cmk(0.0, 0.0);
  for (int i = m - 1; i >= 0; --i) {
    const double tr = gr * wr - gi * wi, ti = gr * wi + gi * wr;
    const double sr = __shfl_sync(0xffffffffu, tr, i), si = __shfl_sync(0xffffffffu, ti, i);
    if (lane == i) y = cmk(sr, si);
    if (lane < i) {
      const double ur = hr[lane + i * 33], ui = hi[lane + i * 33];
      gr -= ur * sr - ui * si;
      gi -= ur * si + ui * sr;
    }
  }
  return y;
}

}  // namespace sapmg
