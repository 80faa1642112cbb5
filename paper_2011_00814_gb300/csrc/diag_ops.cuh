// diag_ops.cuh -- the FP64 diagnostics of one grid by a set of blocks, shared by
// the single-problem and the batched kernels (see diag.cu).
#pragma once

#include "gpe2p_dev.cuh"

namespace gpe2p {

constexpr int DIAG_THREADS = 256;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// the partial sums of block bid of nb over one grid, into partial[0..3]
template <typename real, int DIM>
__device__ __forceinline__ void diag_block(const KParams<real>& P, const real* p, const real* u0, const real* u1,
                                           const real* u2, const real* phi, const real* phi_lo, int bid, int nb,
                                           double* partial) {
  // blocks stride over the rows (j, k), threads along x; per cell, in FP64:
  // phi, and for each face the face density (the mean of the two cells'
  // rho(phi) = (rhoL + rhoG)/2 + phi (rhoL - rhoG)/2) times u^2; the factor
  // 1/2 of the kinetic energy is applied once per thread
  const int nx = P.n[0], ny = P.n[1];
  const long long rows = (long long)ny * P.n[2];
  const double rm = 0.5 * ((double)P.rhoL + (double)P.rhoG), rd = 0.25 * ((double)P.rhoL - (double)P.rhoG);
  double sphi = 0.0, ke = 0.0;
  real umax = real(0);
  bool bad = false;
  const real* U[3] = {u0, u1, u2};
  for (long long r = bid; r < rows; r += nb) {
    const int j = (int)(r % ny), k = (int)(r / ny);
    const long long q0 = lin(P, 0, j, k);
    for (int i = threadIdx.x; i < nx; i += blockDim.x) {
      const long long q = q0 + i;
      const real fr = phi[q];
      const double f = (double)fr + (phi_lo ? (double)phi_lo[q] : 0.0);
      sphi += f;
      bad = bad || !isfinite(fr) || !isfinite(p[q]);
#pragma unroll
      for (int c = 0; c < DIM; ++c) {
        const double fm = (double)ld_cen(phi, P, i - (c == 0), j - (c == 1), k - (c == 2));
        const real uc = U[c][q];
        const double ud = (double)uc;
        ke = fma(fma(rd, fm + f, rm), ud * ud, ke);
        umax = fmax(umax, fabs(uc));
        bad = bad || !isfinite(uc);
      }
    }
  }
  ke *= 0.5;
  double umaxd = (double)umax, badd = bad ? 1.0 : 0.0;
  __shared__ double red[4][DIAG_THREADS / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  sphi = warp_sum(sphi);
  ke = warp_sum(ke);
  umaxd = warp_max(umaxd);
  badd = warp_max(badd);
  if (lane == 0) {
    red[0][wid] = sphi;
    red[1][wid] = ke;
    red[2][wid] = umaxd;
    red[3][wid] = badd;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0, c = 0.0, d = 0.0;
    for (int w = 0; w < DIAG_THREADS / 32; ++w) {
      a += red[0][w];
      b += red[1][w];
      c = fmax(c, red[2][w]);
      d = fmax(d, red[3][w]);
    }
    partial[0] = a;
    partial[1] = b;
    partial[2] = c;
    partial[3] = d;
  }
}

// the fixed-order sum of nblocks partials by one block
__device__ __forceinline__ void diag_sum(const double* partial, int nblocks, double vol, double* out) {
  __shared__ double red[4][DIAG_THREADS];
  double a = 0.0, b = 0.0, c = 0.0, d = 0.0;
  for (int q = threadIdx.x; q < nblocks; q += blockDim.x) {
    a += partial[4 * q + 0];
    b += partial[4 * q + 1];
    c = fmax(c, partial[4 * q + 2]);
    d = fmax(d, partial[4 * q + 3]);
  }
  red[0][threadIdx.x] = a;
  red[1][threadIdx.x] = b;
  red[2][threadIdx.x] = c;
  red[3][threadIdx.x] = d;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      red[0][threadIdx.x] += red[0][threadIdx.x + s];
      red[1][threadIdx.x] += red[1][threadIdx.x + s];
      red[2][threadIdx.x] = fmax(red[2][threadIdx.x], red[2][threadIdx.x + s]);
      red[3][threadIdx.x] = fmax(red[3][threadIdx.x], red[3][threadIdx.x + s]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[0] = red[0][0] * vol;
    out[1] = red[1][0] * vol;
    out[2] = red[2][0];
    out[3] = red[3][0];
  }
}

}  // namespace gpe2p
