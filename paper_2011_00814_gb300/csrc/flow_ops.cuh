// flow_ops.cuh -- staging of a 2D tile, and the 2D FP64 flow stage (Sec. 3) on one
// tile, shared by the single-instance and the batched kernels so that both
// compute bit-identical results.
//
//   out = a q^n + b (q + dt L(q)),  q = (p, u, v[, w]),
// with L of Eq. p-u-v-semidiscrete-2d built from Eqs. div-v-discretization,
// diff-p-discretization, conv-u-discretization, u-stress-discretization
// (a)-(d), st-u-discretization, gradp-u-discretization and gradp-u-p-ave-3d,
// phi and mu frozen (Sec. 3, after Eq. tvd-rk3).
//
// The axisymmetric form (2D, KParams::axisym; x = r, y = z, cell column i
// centred at r = (i + 1/2) dx, u face i at r = i dx) adds, as printed in
// Eqs. div-v-axisym, gpe-pressure-two-phase-axisym and
// gpe-momentum-two-phase-axisym-r/-z: u_r / r to the divergence (u_r at the
// centre = mean of its faces), (nu / r) dp/dr to the pressure rate,
// (eta / r)(du_r/dr - u_r / r) to the radial and (eta / r) du_z/dr to the
// axial momentum, with central differences and the face viscosity the mean
// of the two cells the face separates.
#pragma once

#include "gpe2p_dev.cuh"
#include "gpe2p_launch.h"

namespace gpe2p {

// 2D tile accessor: NF staged fields of (TXv+2) x (TYv+2) elements
template <typename real, int SXv, int PLv>
struct Tile2 {
  const real* sm;
  int c;   // the thread's cell within a staged field
  int gi;  // its global column index (the radius of the axisymmetric form)
  __device__ __forceinline__ real operator()(int f, int dx, int dy, int) const {
    return sm[f * PLv + c + dy * SXv + dx];
  }
};

// Whether the one-cell halo of the TXv x TYv tile at (i0, j0) lies inside
// the domain, so that its staged values need no boundary map: every staged
// cell (gi, gj) then has 0 <= gi < nx and 0 <= gj < ny, and a face value on
// it is the stored one (the wall faces 0 of a walled axis lie outside such a
// halo, since i0, j0 >= 1).
template <typename real, int TXv, int TYv>
__device__ __forceinline__ bool tile_interior(const KParams<real>& P, int i0, int j0) {
  return i0 >= 1 && i0 + TXv + 1 <= P.n[0] && j0 >= 1 && j0 + TYv + 1 <= P.n[1];
}

// The staged region of a 2D tile, (TXv + 2) x (TYv + 2) cells, spread over
// the block's threads.  fn(e, lx, ly, off) is called for every staged cell
// e = ly (TXv + 2) + lx, i.e. the cell (i0 - 1 + lx, j0 - 1 + ly); off is its
// element offset when the tile is interior (every staged cell inside the
// domain; formed from one per-tile base in 32-bit arithmetic), else -1.
template <typename real, int TXv, int TYv, int NT = TXv * TYv / 2, typename Fn>
__device__ __forceinline__ void stage2d(const KParams<real>& P, int i0, int j0, bool interior, Fn fn) {
  constexpr int SXv = TXv + 2, PLv = SXv * (TYv + 2);
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  const long long base = interior ? lin(P, i0 - 1, j0 - 1, 0) : -1LL;
  const int sy = (int)P.sy;
  for (int e = tid; e < PLv; e += NT) {
    const int ly = e / SXv, lx = e - ly * SXv;
    fn(e, lx, ly, interior ? base + (ly * sy + lx) : -1LL);
  }
}

// The FP64 flow stage on one tile, by NT threads.  GB300's FP64 pipe takes two
// lanes a cycle and SM, so this stage is bound by the number of FP64
// operations (and on a small grid by their latency) and nothing else:
//   - every term that two cells share (a corner's viscous stress, a face's
//     diffusive pressure flux, a cell's normal stress and divergence) is formed
//     once and read back from shared memory;
//   - what is frozen over the three stages (corner viscosities, face sums of
//     nu, surface tension and gravity, 1 / rho on the faces: all the divisions)
//     is formed by the first stage (MODE 1) and stored in the fields Z for the
//     others (MODE 2): 7 words per cell, which stay in L2 or cost less than
//     the 50 operations they replace (without CORNERS, as in a batch, which has
//     no free field for them, the corner viscosities are formed in every stage:
//     three additions of staged values, the same bits);
//   - pressure, u and v of a cell are separate work items, so that a small
//     tile's chains run side by side.
// MODE 0: A.out = L(q).  sm: flow64_smem bytes.
// 256 x 1024 Rayleigh-Taylor: the three stages 71, 49 and 48 us (129, 84 and 84
// FP64 instructions a cell), the step 269 us; 385 us with every
// term formed per cell, two cells a thread.
enum { Z_NX, Z_NY, Z_E4, Z_FX, Z_FY, Z_RX, Z_RY, Z_N };  // the frozen fields
enum { D_P, D_U, D_V, D_ETA, D_TX, D_TY, D_DIV, D_TAU, D_FX, D_FY, D_PHI, D_MU, D_NU, F64_N };
template <int TXv, int TYv>
constexpr size_t flow64_smem(int mode) {
  return sizeof(double) * ((size_t)(mode == 2 ? (int)D_PHI : (int)F64_N) * (TXv + 2) * (TYv + 2) + 2 * (TXv + 2));
}

template <int MODE, int TXv, int TYv, int NT, bool CORNERS = true>
__device__ __forceinline__ void flow2d_tile64(const KParams<double>& P, const FlowArgs<double>& A, int i0, int j0,
                                              double* sm) {
  using real = double;
  constexpr int SXv = TXv + 2, PLv = SXv * (TYv + 2);
  constexpr bool FROZEN = MODE == 2;
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  const int nx = P.n[0], ny = P.n[1];
  stage2d<real, TXv, TYv, NT>(P, i0, j0, tile_interior<real, TXv, TYv>(P, i0, j0),
                              [&](int e, int lx, int ly, long long q) {
    real pv, uv, vv, phi, muv = real(0);
    if (q >= 0) {
      pv = A.q[0][q];
      uv = A.q[1][q];
      vv = A.q[2][q];
      phi = A.phi[q];
      if (!FROZEN) muv = A.mu[q];
    } else {
      const int gi = clampi(i0 - 1 + lx, -1, nx), gj = clampi(j0 - 1 + ly, -1, ny);
      pv = ld_cen(A.q[0], P, gi, gj, 0);
      uv = ld_face<0>(A.q[1], P, gi, gj, 0);
      vv = ld_face<1>(A.q[2], P, gi, gj, 0);
      phi = ld_cen(A.phi, P, gi, gj, 0);
      if (!FROZEN) muv = ld_cen(A.mu, P, gi, gj, 0);
    }
    real* b = sm + e;
    b[D_P * PLv] = pv;
    b[D_U * PLv] = uv;
    b[D_V * PLv] = vv;
    const real eta = eta_of(P, phi);
    b[D_ETA * PLv] = eta;
    if (!FROZEN) {
      b[D_PHI * PLv] = phi;
      b[D_MU * PLv] = muv;
      b[D_NU * PLv] = fdiv(eta, rho_of(P, phi));
    }
  });
  // axisymmetric form: dx / (2 r) at a staged column's centre and dx / r at its low face
  real* axc = sm + (size_t)(FROZEN ? (int)D_PHI : (int)F64_N) * PLv;
  real* axf = axc + SXv;
  if (P.axisym)
    for (int lx = tid; lx < SXv; lx += NT) {
      const int gi = i0 - 1 + lx;
      axc[lx] = fdiv(real(1), real(2 * gi + 1));
      axf[lx] = gi == 0 ? real(0) : fdiv(real(1), real(gi));  // (face 0, on the axis, is never updated)
    }
  __syncthreads();
  constexpr int NP = (TXv + 1) * (TYv + 1);
  for (int e = tid; e < 2 * NP; e += NT) {
    const bool corner = e >= NP;
    const int k = corner ? e - NP : e;
    const int ly = k / (TXv + 1), lx = k - ly * (TXv + 1);
    real* c = sm + ly * SXv + lx;
    if (!corner) {
      // the cell's normal stresses and divergence
      const real u0 = c[D_U * PLv], up = c[D_U * PLv + 1], v0 = c[D_V * PLv], vp = c[D_V * PLv + SXv];
      const real du = up - u0, dv = vp - v0;
      real D = du + dv;
      if (P.axisym) D = fma(u0 + up, axc[lx], D);
      const real eta = c[D_ETA * PLv], b = P.bulk ? D : real(0);
      c[D_TX * PLv] = mul_rn(eta, fma(real(2), du, b));
      c[D_TY * PLv] = mul_rn(eta, fma(real(2), dv, b));
      c[D_DIV * PLv] = D;
    } else {
      // of the cell up and right: the viscous stress at its low corner, the
      // diffusive pressure fluxes through its low faces
      c += SXv + 1;
      auto corner4 = [&]() {
        return (c[D_ETA * PLv] + c[D_ETA * PLv - 1]) + (c[D_ETA * PLv - SXv] + c[D_ETA * PLv - SXv - 1]);
      };
      real e4, nx2, ny2;
      const int i = i0 + lx, j = j0 + ly;
      if (FROZEN && i < nx && j < ny) {
        const long long id = lin(P, i, j, 0);
        e4 = CORNERS ? A.z[Z_E4][id] : corner4();
        nx2 = A.z[Z_NX][id];
        ny2 = A.z[Z_NY][id];
      } else if (FROZEN) {
        // past the domain's high end: the wrapped cell's (or, at a wall, the ghosts')
        const int ci = clampi(i, 0, nx), cj = clampi(j, 0, ny);
        const bool wi = ci == nx && P.bc[0] != BC_PERIODIC, wj = cj == ny && P.bc[1] != BC_PERIODIC;
        if (wi || wj) {
          // the corner sums of the ghost cells; the flux through a wall is zero
          // (equal pressures on its sides), whatever the viscosity
          e4 = corner4();
          const long long id = lin(P, ci == nx ? nx - 1 : ci, cj == ny ? ny - 1 : cj, 0);
          nx2 = A.z[Z_NX][id];
          ny2 = A.z[Z_NY][id];
        } else {
          const long long id = lin(P, ci == nx ? 0 : ci, cj == ny ? 0 : cj, 0);
          e4 = CORNERS ? A.z[Z_E4][id] : corner4();
          nx2 = A.z[Z_NX][id];
          ny2 = A.z[Z_NY][id];
        }
      } else {
        e4 = corner4();
        const real nu = c[D_NU * PLv];
        nx2 = add_rn(nu, c[D_NU * PLv - 1]);
        ny2 = add_rn(nu, c[D_NU * PLv - SXv]);
        if (MODE == 1 && lx < TXv && ly < TYv && i < nx && j < ny) {
          const long long id = lin(P, i, j, 0);
          if (CORNERS) A.z[Z_E4][id] = e4;
          A.z[Z_NX][id] = nx2;
          A.z[Z_NY][id] = ny2;
        }
      }
      const real S = (c[D_U * PLv] - c[D_U * PLv - SXv]) + (c[D_V * PLv] - c[D_V * PLv - 1]);
      c[D_TAU * PLv] = mul_rn(e4, S);
      const real p = c[D_P * PLv];
      c[D_FX * PLv] = mul_rn(nx2, p - c[D_P * PLv - 1]);
      c[D_FY * PLv] = mul_rn(ny2, p - c[D_P * PLv - SXv]);
    }
  }
  __syncthreads();
  const real gfac = P.pavg ? mul_rn(P.inv_dx, real(1.0 / 6.0)) : P.inv_dx;
  constexpr int NC = TXv * TYv;
  for (int e = tid; e < 3 * NC; e += NT) {
    const int f = e / NC, k = e - f * NC;
    const int ly = k / TXv, lx = k - ly * TXv;
    const int i = i0 + lx, j = j0 + ly;
    if (i >= nx || j >= ny) continue;
    const long long id = lin(P, i, j, 0);
    const real* c = sm + (ly + 1) * SXv + lx + 1;
    real qn = real(0);
    if (MODE == 2) qn = A.q0[f][id];
    real L, q;
    if (f == 0) {
      q = c[D_P * PLv];
      real diff = (c[D_FX * PLv + 1] - c[D_FX * PLv]) + (c[D_FY * PLv + SXv] - c[D_FY * PLv]);
      real rho;
      if (P.axisym || !FROZEN) {
        const real phi = FROZEN ? A.phi[id] : c[D_PHI * PLv];
        rho = rho_of(P, phi);
        if (P.axisym) {
          const real nu = fdiv(c[D_ETA * PLv], rho);
          diff = fma(mul_rn(mul_rn(real(2), nu), c[D_P * PLv + 1] - c[D_P * PLv - 1]), axc[lx + 1], diff);
        }
      } else {
        rho = rho_of(P, A.phi[id]);
      }
      L = fma(diff, mul_rn(real(0.5), P.inv_dx2), -mul_rn(mul_rn(rho, P.cs2), mul_rn(c[D_DIV * PLv], P.inv_dx)));
    } else {
      // the u face (f = 1): low neighbour one column left; the v face: one row down
      const int lo = f == 1 ? 1 : SXv, tr = f == 1 ? SXv : 1;
      const real* U = c + (f == 1 ? (int)D_U : (int)D_V) * PLv;  // the component
      const real* T = c + (f == 1 ? (int)D_V : (int)D_U) * PLv;  // the transverse one
      const real* N = c + (f == 1 ? (int)D_TX : (int)D_TY) * PLv;
      q = U[0];
      const real dn = U[lo] - U[-lo], dt = U[tr] - U[-tr];
      real visc = fma(real(0.25), c[D_TAU * PLv + tr] - c[D_TAU * PLv], N[0] - N[-lo]);
      if (P.axisym) {
        const real et = mul_rn(real(0.5), c[D_ETA * PLv - lo] + c[D_ETA * PLv]);
        if (f == 1) {
          const real ir = axf[lx + 1];
          visc = fma(mul_rn(et, ir), fma(real(0.5), dn, -mul_rn(q, ir)), visc);
        } else {
          visc = fma(mul_rn(et, dt), axc[lx + 1], visc);
        }
      }
      const real* p = c + D_P * PLv;
      real gp = p[0] - p[-lo];
      if (P.pavg) gp = fma(real(4), gp, (p[tr] + p[-tr]) - (p[tr - lo] + p[-tr - lo]));
      const real T4 = (T[0] + T[-lo]) + (T[tr] + T[tr - lo]);
      const real conv = fma(q, dn, mul_rn(real(0.25), mul_rn(T4, dt)));
      real fs, ri;
      if (FROZEN) {
        fs = A.z[f == 1 ? Z_FX : Z_FY][id];
        ri = A.z[f == 1 ? Z_RX : Z_RY][id];
      } else {
        const real ph0 = c[D_PHI * PLv], phl = c[D_PHI * PLv - lo];
        const real rb2 = rho_of(P, phl) + rho_of(P, ph0);
        const real st = mul_rn(mul_rn(-P.sigma, ph0 + phl), c[D_MU * PLv] - c[D_MU * PLv - lo]);
        fs = fma(st, P.inv_2dx, mul_rn(fma(real(0.5), rb2, -P.rho_ref), P.g[f - 1]));
        ri = fdiv(real(2), rb2);
        if (MODE == 1) {
          A.z[f == 1 ? Z_FX : Z_FY][id] = fs;
          A.z[f == 1 ? Z_RX : Z_RY][id] = ri;
        }
      }
      const real F = fma(visc, P.inv_dx2, fma(-gp, gfac, fs));
      L = fma(ri, F, -mul_rn(conv, P.inv_2dx));
      // faces on a wall are never updated
      if ((f == 1 && i == 0 && P.bc[0] != BC_PERIODIC) || (f == 2 && j == 0 && P.bc[1] != BC_PERIODIC)) L = real(0);
    }
    real out = L;
    if (MODE != 0) {
      out = fma(P.dt, L, q);
      if (MODE == 2) {
        out = fma(A.a, qn, mul_rn(A.b, out));
        if (f > 0 && A.usum[0]) A.usum[f - 1][id] = qn + out;
      }
    }
    A.out[f][id] = out;
  }
  __syncthreads();
}

}  // namespace gpe2p
