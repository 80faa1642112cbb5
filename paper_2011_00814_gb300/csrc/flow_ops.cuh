// flow_ops.cuh -- the semi-discrete flow operators of one cell (Sec. 3) and
// the 2D flow stage on one tile, shared by the single-instance and the
// batched 2D kernels so that both compute bit-identical results.
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

enum { F_P = 0, F_U = 1, F_V = 2, F_W = 3, F_PHI = 4, F_RHO = 5, F_ETA = 6, F_NU = 7, F_MU = 8, F_N = 9 };

// The rates below gather every term with its grid factor applied once:
// sums of the four edge viscosities, face velocities and transverse
// pressures are formed unnormalised and scaled together at the end.  Every
// sum of two products is written as the fused multiply-add it is meant to be
// (the compiler could otherwise fuse either product, and two kernels that
// inline this code could round differently).
template <typename real, int DIM, typename T>
struct FlowOps {
  // dx / (2 r) at the centre of the cell column at x offset ox (axisymmetric form, 2D tiles)
  __device__ __forceinline__ static real dx_2r(const T& S, int ox) {
    return fdiv(real(1), real(2 * (S.gi + ox) + 1));
  }

  // velocity divergence of the cell at offset (ox,oy,oz) times dx, Eq. div-v-discretization
  // (plus dx u_r / r, Eq. div-v-axisym, in the axisymmetric form)
  __device__ __forceinline__ static real divsum(const T& S, const KParams<real>& P, int ox, int oy, int oz) {
    real d = (S(F_U, ox + 1, oy, oz) - S(F_U, ox, oy, oz)) + (S(F_V, ox, oy + 1, oz) - S(F_V, ox, oy, oz));
    if constexpr (DIM == 3) {
      d += S(F_W, ox, oy, oz + 1) - S(F_W, ox, oy, oz);
    } else {
      if (P.axisym) d += (S(F_U, ox, oy, oz) + S(F_U, ox + 1, oy, oz)) * dx_2r(S, ox);
    }
    return d;
  }

  // 4 x (eta averaged over the four cells around the edge shared by the faces
  // of components C and t), Eq. u-stress-discretization (eta bar at i, j+-1/2):
  // the edge on the +t side (e4p) and on the -t side (e4m) of the C face
  template <int C>
  __device__ __forceinline__ static void edge_eta4(const T& S, int t, real& e4p, real& e4m) {
    const int cx = C == 0, cy = C == 1, cz = C == 2;
    const int tx = t == 0, ty = t == 1, tz = t == 2;
    if constexpr (DIM == 3) {
      // summed in one order per edge whichever face asks (pairs along the
      // lower axis first), so that the rates of the two components and the
      // two cells that share an edge share its sum
      const int a = C < t ? C : t, b = C < t ? t : C;
      auto e4 = [&](int ox, int oy, int oz) {
        const int ax = a == 0, ay = a == 1, az = a == 2, bx = b == 0, by = b == 1, bz = b == 2;
        return (S(F_ETA, ox, oy, oz) + S(F_ETA, ox + ax, oy + ay, oz + az)) +
               (S(F_ETA, ox + bx, oy + by, oz + bz) + S(F_ETA, ox + ax + bx, oy + ay + by, oz + az + bz));
      };
      e4p = e4(-cx, -cy, -cz);
      e4m = e4(-cx - tx, -cy - ty, -cz - tz);
    } else {
      e4p = (S(F_ETA, 0, 0, 0) + S(F_ETA, tx, ty, tz)) + (S(F_ETA, -cx, -cy, -cz) + S(F_ETA, tx - cx, ty - cy, tz - cz));
      e4m = (S(F_ETA, 0, 0, 0) + S(F_ETA, -tx, -ty, -tz)) +
            (S(F_ETA, -cx, -cy, -cz) + S(F_ETA, -tx - cx, -ty - cy, -tz - cz));
    }
  }

  // whether the pressure gradient averages transversally (Eq. gradp-u-p-ave-3d)
  __device__ __forceinline__ static bool averaged(const KParams<real>& P) {
    if constexpr (T::PAVG == 0) return false;
    else if constexpr (T::PAVG > 0) return true;
    else return P.pavg != 0;
  }

  // the averaged pressure of the cell at offset o for the gradient along C,
  // unnormalised: 6 pbar in 2D (Eq. gradp-u-discretization), 36 pbar in 3D
  template <int C>
  __device__ __forceinline__ static real psum(const T& S, int ox, int oy, int oz) {
    if (DIM == 2) {
      constexpr int tx = C == 1, ty = C == 0;
      return real(4) * S(F_P, ox, oy, oz) + (S(F_P, ox + tx, oy + ty, oz) + S(F_P, ox - tx, oy - ty, oz));
    } else {
      constexpr int T1 = (C + 1) % 3, T2 = (C + 2) % 3;
      constexpr int ax = T1 == 0, ay = T1 == 1, az = T1 == 2;  // unit vector t1
      constexpr int bx = T2 == 0, by = T2 == 1, bz = T2 == 2;  // unit vector t2
      const real s4 = (S(F_P, ox + ax, oy + ay, oz + az) + S(F_P, ox - ax, oy - ay, oz - az)) +
                      (S(F_P, ox + bx, oy + by, oz + bz) + S(F_P, ox - bx, oy - by, oz - bz));
      const real s1 = (S(F_P, ox + ax + bx, oy + ay + by, oz + az + bz) +
                       S(F_P, ox - ax - bx, oy - ay - by, oz - az - bz)) +
                      (S(F_P, ox - ax + bx, oy - ay + by, oz - az + bz) +
                       S(F_P, ox + ax - bx, oy + ay - by, oz + az - bz));
      return real(16) * S(F_P, ox, oy, oz) + (real(4) * s4 + s1);
    }
  }

  // pressure rate at the cell centre: -rho c_s^2 div u + div(nu grad p); d0 = dx div u
  __device__ __forceinline__ static real rate_p(const T& S, const KParams<real>& P, real d0) {
    real diff = real(0);
    const real nu0 = S(F_NU, 0, 0, 0), p0 = S(F_P, 0, 0, 0);
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      const int ex = a == 0, ey = a == 1, ez = a == 2;
      diff = fma(nu0 + S(F_NU, ex, ey, ez), S(F_P, ex, ey, ez) - p0, diff);
      diff = fma(nu0 + S(F_NU, -ex, -ey, -ez), S(F_P, -ex, -ey, -ez) - p0, diff);
    }
    if constexpr (DIM == 2) {
      // (nu / r) dp/dr, Eq. gpe-pressure-two-phase-axisym
      if (P.axisym) diff = fma(real(2) * nu0 * (S(F_P, 1, 0, 0) - S(F_P, -1, 0, 0)), dx_2r(S, 0), diff);
    }
    return fma(diff, real(0.5) * P.inv_dx2, -(S(F_RHO, 0, 0, 0) * P.cs2 * mul_rn(d0, P.inv_dx)));
  }

  // rate of velocity component C on the cell's low face along C; d0 = dx div u of the cell
  template <int C>
  __device__ __forceinline__ static real rate_vel(const T& S, const KParams<real>& P, real d0) {
    constexpr int cx = C == 0, cy = C == 1, cz = C == 2;
    const int FC = F_U + C;
    const real rb2 = S(F_RHO, -cx, -cy, -cz) + S(F_RHO, 0, 0, 0);   // 2 rho on the face
    real gradp;
    if (averaged(P))
      gradp = (psum<C>(S, 0, 0, 0) - psum<C>(S, -cx, -cy, -cz)) *
              (P.inv_dx * real(DIM == 2 ? 1.0 / 6.0 : 1.0 / 36.0));
    else
      gradp = (S(F_P, 0, 0, 0) - S(F_P, -cx, -cy, -cz)) * P.inv_dx;
    const real uc0 = S(FC, 0, 0, 0);
    const real tcc = fma(S(F_ETA, -cx, -cy, -cz), S(FC, -cx, -cy, -cz) - uc0,
                         mul_rn(S(F_ETA, 0, 0, 0), S(FC, cx, cy, cz) - uc0));
    real edge = real(0), conv4 = real(0);
#pragma unroll
    for (int t = 0; t < DIM; ++t) {
      if (t == C) continue;
      const int tx = t == 0, ty = t == 1, tz = t == 2;
      const int FT = F_U + t;
      real e4p, e4m;
      edge_eta4<C>(S, t, e4p, e4m);
      const real ucp = S(FC, tx, ty, tz), ucm = S(FC, -tx, -ty, -tz);
      const real ut0 = S(FT, 0, 0, 0), utc = S(FT, -cx, -cy, -cz);
      const real utp = S(FT, tx, ty, tz), utpc = S(FT, tx - cx, ty - cy, tz - cz);
      edge = fma(e4p, (ucp - uc0) + (utp - utpc), edge);
      edge = fma(e4m, (ucm - uc0) + (utc - ut0), edge);
      conv4 = fma((ut0 + utc) + (utp + utpc), ucp - ucm, conv4);
    }
    real visc = fma(real(2), tcc, mul_rn(real(0.25), edge));
    if (P.bulk) {
      visc = fma(S(F_ETA, 0, 0, 0), d0, visc);
      visc = fma(-S(F_ETA, -cx, -cy, -cz), divsum(S, P, -cx, -cy, -cz), visc);
    }
    if constexpr (DIM == 2) {
      if (P.axisym) {
        const real eta_f = real(0.5) * (S(F_ETA, -cx, -cy, 0) + S(F_ETA, 0, 0, 0));
        const real dudr2 = S(FC, 1, 0, 0) - S(FC, -1, 0, 0);  // 2 dx du_c/dr
        if (C == 0) {
          // (eta / r)(du_r/dr - u_r / r) on the u face i, r = i dx (i >= 1)
          const real ir = fdiv(real(1), real(S.gi));
          visc = fma(mul_rn(eta_f, ir), fma(real(0.5), dudr2, -mul_rn(uc0, ir)), visc);
        } else {
          // (eta / r) du_z/dr on the v face of column i, r = (i + 1/2) dx
          visc = fma(mul_rn(eta_f, dudr2), dx_2r(S, 0), visc);
        }
      }
    }
    const real st = -P.sigma * (S(F_PHI, 0, 0, 0) + S(F_PHI, -cx, -cy, -cz)) *
                    (S(F_MU, 0, 0, 0) - S(F_MU, -cx, -cy, -cz));
    const real grav = fma(real(0.5), rb2, -P.rho_ref);
    real force = fma(visc, P.inv_dx2, -gradp);
    force = fma(st, P.inv_2dx, force);
    force = fma(grav, P.g[C], force);
    const real conv = fma(uc0, S(FC, cx, cy, cz) - S(FC, -cx, -cy, -cz), mul_rn(real(0.25), conv4));
    return fma(-conv, P.inv_2dx, fdiv(real(2) * force, rb2));
  }
};

// 2D tile accessor: NF staged fields of (TXv+2) x (TYv+2) elements
template <typename real, int SXv, int PLv>
struct Tile2 {
  static constexpr int PAVG = -1;  // pressure averaging decided at run time
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

// The FP32 rates L(q) on the tile of TXv x TYv cells at (i0, j0) into A.out, by a
// block of TXv*TYv/2 threads (the operator-level check; the FP32 step runs in
// the fused passes of step2d.cuh): thread t computes the cells
// (t % TXv, 2 (t / TXv) + r), r = 0, 1.  The block stages p, u, v, phi, rho,
// eta, nu = eta/rho and mu with a one-cell halo in sm, F_N * (TXv+2)*(TYv+2)
// reals: straight from the fields on an interior tile, through the boundary
// maps (ghosts) on a tile at the domain's edge.
template <typename real, int TXv, int TYv>
__device__ __forceinline__ void rates2d_tile(const KParams<real>& P, const FlowArgs<real>& A, int i0, int j0,
                                             real* sm) {
  constexpr int SXv = TXv + 2, SYv = TYv + 2, PLv = SXv * SYv;
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  const int tx = tid % TXv, ty = tid / TXv;
  const int nx = P.n[0], ny = P.n[1];
  const int i = i0 + tx;
  stage2d<real, TXv, TYv>(P, i0, j0, tile_interior<real, TXv, TYv>(P, i0, j0),
                          [&](int e, int lx, int ly, long long q) {
    real pv, uv, vv, phi, muv;
    if (q >= 0) {
      pv = A.q[0][q];
      uv = A.q[1][q];
      vv = A.q[2][q];
      phi = A.phi[q];
      muv = A.mu[q];
    } else {
      const int gi = clampi(i0 - 1 + lx, -1, nx), gj = clampi(j0 - 1 + ly, -1, ny);
      pv = ld_cen(A.q[0], P, gi, gj, 0);
      uv = ld_face<0>(A.q[1], P, gi, gj, 0);
      vv = ld_face<1>(A.q[2], P, gi, gj, 0);
      phi = ld_cen(A.phi, P, gi, gj, 0);
      muv = ld_cen(A.mu, P, gi, gj, 0);
    }
    const real rho = rho_of(P, phi), eta = eta_of(P, phi);
    real* b = sm + e;
    b[F_P * PLv] = pv;
    b[F_U * PLv] = uv;
    b[F_V * PLv] = vv;
    b[F_PHI * PLv] = phi;
    b[F_RHO * PLv] = rho;
    b[F_ETA * PLv] = eta;
    b[F_NU * PLv] = fdiv(eta, rho);
    b[F_MU * PLv] = muv;
  });
  __syncthreads();
  using Ops = FlowOps<real, 2, Tile2<real, SXv, PLv>>;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int j = j0 + 2 * ty + r;
    Tile2<real, SXv, PLv> S;
    S.sm = sm;
    S.c = (2 * ty + r + 1) * SXv + (tx + 1);
    S.gi = i;
    const real D0 = Ops::divsum(S, P, 0, 0, 0);
    if (i < nx && j < ny) {
      const long long id = lin(P, i, j, 0);
      A.out[0][id] = Ops::rate_p(S, P, D0);
      A.out[1][id] = (P.bc[0] != BC_PERIODIC && i == 0) ? real(0) : Ops::template rate_vel<0>(S, P, D0);
      A.out[2][id] = (P.bc[1] != BC_PERIODIC && j == 0) ? real(0) : Ops::template rate_vel<1>(S, P, D0);
    }
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
//     the 50 operations they replace;
//   - pressure, u and v of a cell are separate work items, so that a small
//     tile's chains run side by side.
// Results differ from FlowOps by rounding (the order of the sums) only.
// MODE 0: A.out = L(q).  sm: flow64_smem bytes.
// 256 x 1024 Rayleigh-Taylor: the three stages 71, 49 and 48 us (129, 84 and 84
// FP64 instructions a cell), the step 269 us; 385 us with FlowOps at two cells a thread.
enum { Z_NX, Z_NY, Z_E4, Z_FX, Z_FY, Z_RX, Z_RY, Z_N };  // the frozen fields
enum { D_P, D_U, D_V, D_ETA, D_TX, D_TY, D_DIV, D_TAU, D_FX, D_FY, D_PHI, D_MU, D_NU, F64_N };
template <int TXv, int TYv>
constexpr size_t flow64_smem(int mode) {
  return sizeof(double) * ((size_t)(mode == 2 ? (int)D_PHI : (int)F64_N) * (TXv + 2) * (TYv + 2) + 2 * (TXv + 2));
}

template <int MODE, int TXv, int TYv, int NT>
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
      real e4, nx2, ny2;
      const int i = i0 + lx, j = j0 + ly;
      if (FROZEN && i < nx && j < ny) {
        const long long id = lin(P, i, j, 0);
        e4 = A.z[Z_E4][id];
        nx2 = A.z[Z_NX][id];
        ny2 = A.z[Z_NY][id];
      } else if (FROZEN) {
        // past the domain's high end: the wrapped cell's (or, at a wall, the ghosts')
        const int ci = clampi(i, 0, nx), cj = clampi(j, 0, ny);
        const bool wi = ci == nx && P.bc[0] != BC_PERIODIC, wj = cj == ny && P.bc[1] != BC_PERIODIC;
        if (wi || wj) {
          // the corner sums of the ghost cells; the flux through a wall is zero
          // (equal pressures on its sides), whatever the viscosity
          e4 = (c[D_ETA * PLv] + c[D_ETA * PLv - 1]) + (c[D_ETA * PLv - SXv] + c[D_ETA * PLv - SXv - 1]);
          const long long id = lin(P, ci == nx ? nx - 1 : ci, cj == ny ? ny - 1 : cj, 0);
          nx2 = A.z[Z_NX][id];
          ny2 = A.z[Z_NY][id];
        } else {
          const long long id = lin(P, ci == nx ? 0 : ci, cj == ny ? 0 : cj, 0);
          e4 = A.z[Z_E4][id];
          nx2 = A.z[Z_NX][id];
          ny2 = A.z[Z_NY][id];
        }
      } else {
        e4 = (c[D_ETA * PLv] + c[D_ETA * PLv - 1]) + (c[D_ETA * PLv - SXv] + c[D_ETA * PLv - SXv - 1]);
        const real nu = c[D_NU * PLv];
        nx2 = add_rn(nu, c[D_NU * PLv - 1]);
        ny2 = add_rn(nu, c[D_NU * PLv - SXv]);
        if (MODE == 1 && lx < TXv && ly < TYv && i < nx && j < ny) {
          const long long id = lin(P, i, j, 0);
          A.z[Z_E4][id] = e4;
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
