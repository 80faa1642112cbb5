// step2d.cuh -- a 2D step in two tile passes: the three TVD-RK3 flow stages on
// one tile, and the TVD-RK2 Cahn-Hilliard step with both chemical potentials on
// one tile.  Shared by the single-problem and the batched FP32 kernels; every
// sum of two products is written as the fused operation it is meant to be, so
// that each kernel that inlines this code gives the same bits.
//
// Why fused: a stage per launch moves 49 words per cell and step between L2 or
// HBM and the SMs and re-forms everything frozen over the stages (phi, mu,
// rho, eta and nu do not change during the flow step).  A tile here
// reads phi, mu, p, u, v once and writes p, u, v and the two face sums; the
// second pass reads phi, mu and the face sums and writes phi and mu: 16 words.
// The price is a halo of three (flow) or four (CH) cells that neighbouring
// tiles compute too, 1.4 and 1.5 times the cells at 32 rows.  The arithmetic is
// the same, operation by operation, in every tile shape and in the batched
// kernels.
//
// A block is NW warps; lane = column, each thread R adjacent rows.  The rows'
// face and edge terms (normal stresses, corner stresses, diffusive pressure
// fluxes, averaged pressures) are formed once and handed to the left or
// right neighbour by a shuffle, to the row above in registers.  The terms
// frozen over the stages (corner and face viscosities, surface tension and
// gravity, 1 / rho on the faces) are formed once and stay in registers.
#pragma once

#include "ch_ops.cuh"
#include "gpe2p_dev.cuh"
#include "gpe2p_launch.h"

namespace gpe2p {

// output columns and rows of a fused tile whose first stage computes NR rows
constexpr int FUSED_X = 26;
constexpr int flow_rows(int NR) { return NR - 4; }
constexpr int ch_rows(int NR) { return NR - 6; }
// shared memory: flow keeps p, u, v three times (q^n and two stage results,
// the second in place of phi and mu) in rows of 32 columns
// (neighbouring lanes' reads at the ends of the planes stay inside the pad);
// CH keeps phi, mu and phi_1 in rows of 34 columns
constexpr int FUSED_PAD = 8;
template <typename real>
constexpr size_t flow_fused_smem(int NR) { return sizeof(real) * (size_t)(9 * (NR + 2) * 32 + 2 * FUSED_PAD); }
template <typename real>
constexpr size_t ch_fused_smem(int NR) { return sizeof(real) * (size_t)(3 * (NR + 2) * 34 + 2 * FUSED_PAD); }

// The tiles: tall ones (32 rows computed by eight warps of four rows a thread,
// 1.4 to 1.5 times the cells) where there are enough of them for two blocks on
// every SM, else short ones (16 rows by eight warps of two rows a thread, 1.6 to 2
// times) that spread a small grid over the chip.  Measured (both passes):
//   400 x 1200, 20 steps        tall 919 us, short 1017 us
//   256 x 256, 64 steps         tall 789 us (as 16 rows of four), short 655 us
//   96 uneven instances, 8 steps  tall 5.45 ms, short 6.86 ms
// (24 rows by twelve warps of two: 933 us and 5.91 ms; 24 rows by eight of
// three: 930 us and 5.87 ms).
constexpr int FUSED_R = 2, FUSED_NW = 8, FUSED_R_TALL = 4, FUSED_NW_TALL = 8;
// blocks per SM the passes are compiled for: 80 registers a thread at two rows, 128 at four (flow)
constexpr int flow_blocks(int NW, int R) { return (R <= 2 ? 24 : 16) / NW; }
constexpr int ch_blocks(int NW, int R) { return (R <= 2 ? 36 : 24) / NW; }
inline long long fused_tiles(int nx, int ny) {
  const long long rows = flow_rows(FUSED_NW_TALL * FUSED_R_TALL);
  return ((nx + FUSED_X - 1) / FUSED_X) * ((ny + rows - 1) / rows);
}
inline bool fused_tall(int nx, int ny) { return fused_tiles(nx, ny) >= 2 * 152; }

// Where a coordinate x of one axis is stored: c for a cell-centred value or a
// face value tangential to the axis (negative with neg_t), f for the velocity
// component along the axis (negative with neg_f, zero with zero_f).  On a wall
// axis x is first clamped to the ghost layer [-1, n]; on a periodic one
// it may lie any distance outside.  The rules of ld_cen and ld_face.
struct Map1 {
  int c, f;
  bool neg_t, neg_f, zero_f;
};
__device__ __forceinline__ Map1 map1(int x, int n, int bc, bool even_low) {
  Map1 m;
  m.neg_t = m.neg_f = m.zero_f = false;
  if (bc == BC_PERIODIC) {
    if (x < 0) x += n;
    if (x >= n) x -= n;
    if (x < 0 || x >= n) {  // a grid narrower than the tile's halo
      x %= n;
      if (x < 0) x += n;
    }
    m.c = m.f = x;
  } else {
    x = clampi(x, -1, n);
    m.c = clampi(x, 0, n - 1);
    m.neg_t = bc == BC_NOSLIP && ((x < 0 && !even_low) || x >= n);
    m.neg_f = x < 0;
    m.f = x < 0 ? 1 : x;
    m.zero_f = m.f == 0 || m.f >= n;
    if (m.zero_f) m.f = 0;
  }
  return m;
}

// Whether a tile whose staged region is [a, a + len) on an axis of n cells meets
// no ghost there (a periodic axis has none) and wraps at most once: its
// staged cells are then plain loads at wrap1 of their coordinate, without
// the maps' signs and zeros (a third of the CH pass's instructions).
__device__ __forceinline__ bool plain_axis(int a, int len, int n, int bc) {
  return bc == BC_PERIODIC ? n >= 2 * len : (a >= 0 && a + len <= n);
}

// The ghost cells of a fused flow tile after a stage: the cells at -1 and n of
// every walled axis, set from the staged cells they mirror.  q: p, u, v planes.
template <typename real, int NR, int NT>
__device__ __forceinline__ void flow_ghosts(const KParams<real>& P, real* q, int gi0, int gj0, int tid) {
  constexpr int ROWS = NR + 2, PLN = ROWS * 32;
  const int nx = P.n[0], ny = P.n[1];
  const bool wx = P.bc[0] != BC_PERIODIC, wy = P.bc[1] != BC_PERIODIC;
  for (int e = tid; e < 2 * ROWS + 64; e += NT) {
    int lx, ly;
    if (e < 2 * ROWS) {
      if (!wx) continue;
      ly = e >> 1;
      lx = ((e & 1) ? nx : -1) - gi0;
    } else {
      if (!wy) continue;
      lx = (e - 2 * ROWS) >> 1;
      ly = ((e & 1) ? ny : -1) - gj0;
    }
    const int gi = gi0 + lx, gj = gj0 + ly;
    if (lx < 0 || lx >= 32 || ly < 0 || ly >= ROWS) continue;
    if ((wx && (gi < -1 || gi > nx)) || (wy && (gj < -1 || gj > ny))) continue;
    // a periodic axis needs no map: the cell's own column or row is staged
    Map1 mx, my;
    mx.c = mx.f = gi;
    my.c = my.f = gj;
    mx.neg_t = mx.neg_f = mx.zero_f = my.neg_t = my.neg_f = my.zero_f = false;
    if (wx) mx = map1(gi, nx, P.bc[0], P.axisym != 0);
    if (wy) my = map1(gj, ny, P.bc[1], false);
    const int cx = mx.c - gi0, cy = my.c - gj0, fx = mx.f - gi0, fy = my.f - gj0;
    const int d = ly * 32 + lx;
    // a mirrored cell outside the staged region belongs to a ghost that no valid cell reads
    auto at = [&](int f, int x, int y) -> real {
      return (x >= 0 && x < 32 && y >= 0 && y < ROWS) ? q[f * PLN + y * 32 + x] : real(0);
    };
    const real pv = at(0, cx, cy);
    real uv = mx.zero_f ? real(0) : at(1, fx, cy);
    real vv = my.zero_f ? real(0) : at(2, cx, fy);
    if (mx.neg_f != my.neg_t) uv = -uv;
    if (mx.neg_t != my.neg_f) vv = -vv;
    q[d] = pv;
    q[PLN + d] = uv;
    q[2 * PLN + d] = vv;
  }
}

// the step's flow arguments on one grid
template <typename real>
struct FlowStepArgs {
  const real* q[3];   // p, u, v at t^n
  real* out[3];       // at t^{n+1}
  const real* phi;
  const real* mu;
  real* usum[2];      // u^n + u^{n+1} per face, or nullptr
};

// Three flow stages on the tile of FUSED_X x flow_rows(NW R) cells at (i0, j0)
// by NW warps.  sm: flow_fused_smem reals.  With RATES the first stage alone, its
// rates L(q) in A.out and u + u in A.usum (the operator-level check runs the code
// that steps).
template <typename real, int NW, int R, bool AXI, bool RATES = false>
__device__ __forceinline__ void flow2d_fused_tile(const KParams<real>& P, const FlowStepArgs<real>& A, int i0, int j0,
                                                  real* sm) {
  constexpr int NR = NW * R, ROWS = NR + 2, PLN = ROWS * 32, NT = 32 * NW;
  constexpr unsigned FULL = 0xffffffffu;
  const int tid = threadIdx.y * blockDim.x + threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int nx = P.n[0], ny = P.n[1];
  const bool wx = P.bc[0] != BC_PERIODIC, wy = P.bc[1] != BC_PERIODIC;
  const int gi0 = i0 - 3, gj0 = j0 - 3;
  real* qa = sm + FUSED_PAD;      // p, u, v at t^n
  real* qb = qa + 3 * PLN;        // ... after stage 1
  real* qc = qb + 3 * PLN;        // ... after stage 2; phi and mu until the frozen terms are formed
  real* sphi = qc;
  real* smu = qc + PLN;
  const int gi = gi0 + lane;
  if (plain_axis(gi0, 32, nx, P.bc[0]) && plain_axis(gj0, ROWS, ny, P.bc[1])) {
    const int cx = wrap1(gi, nx);
#pragma unroll
    for (int k = 0; k < (ROWS + NW - 1) / NW; ++k) {
      const int ly = w + k * NW;
      if (ly < ROWS) {
        const long long id = (long long)wrap1(gj0 + ly, ny) * P.sy + cx;
        const int d = ly * 32 + lane;
        qa[d] = A.q[0][id];
        qa[PLN + d] = A.q[1][id];
        qa[2 * PLN + d] = A.q[2][id];
        sphi[d] = A.phi[id];
        smu[d] = A.mu[id];
      }
    }
  } else {
    const Map1 mx = map1(gi, nx, P.bc[0], AXI);
    for (int ly = w; ly < ROWS; ly += NW) {
      const Map1 my = map1(gj0 + ly, ny, P.bc[1], false);
      const long long rc = (long long)my.c * P.sy, rf = (long long)my.f * P.sy;
      const int d = ly * 32 + lane;
      const real pv = A.q[0][rc + mx.c];
      real uv = A.q[1][rc + mx.f];
      real vv = A.q[2][rf + mx.c];
      const real fv = A.phi[rc + mx.c];
      const real mv = A.mu[rc + mx.c];
      if (mx.neg_f != my.neg_t) uv = -uv;
      if (mx.neg_t != my.neg_f) vv = -vv;
      if (mx.zero_f) uv = real(0);
      if (my.zero_f) vv = real(0);
      qa[d] = pv;
      qa[PLN + d] = uv;
      qa[2 * PLN + d] = vv;
      sphi[d] = fv;
      smu[d] = mv;
    }
  }
  __syncthreads();

  const int rb = w * R + 1;            // staged row of the thread's first row
  const int gj = gj0 + rb;             // its global row
  const bool live = gj <= ny + 2;      // (uniform per warp) some row of the warp is needed
  const int c0 = rb * 32 + lane;
  // ---- the terms frozen over the stages ----
  real eta[R + 1];                     // rows -1 .. R-1
  real etl[R];                         // eta(i-1)
  real e4u[R + 1], e4v[R], e4vr[R];    // corner viscosity sums: u's order at rows 0 .. R, v's at i and i+1
  real nxl[R], nxr[R], nfy[R + 1];     // sums of nu over the faces
  real stx[R], sty[R], rbx[R], rby[R]; // surface tension, 2 rho on the faces
  real rc[R];                          // rho c_s^2
  real axc = real(0), irx = real(0), nu2[R], eax[R], efy[R];  // axisymmetric terms
  const real gp = P.inv_dx * real(1.0 / 6.0);
  if (live) {
    real ph[R + 2], et[R + 2], rh[R + 2], nu[R + 2], mm[R + 1];
#pragma unroll
    for (int r = -1; r <= R; ++r) {
      ph[r + 1] = sphi[c0 + 32 * r];
      et[r + 1] = eta_of(P, ph[r + 1]);
      rh[r + 1] = rho_of(P, ph[r + 1]);
      nu[r + 1] = fdiv(et[r + 1], rh[r + 1]);
      if (r < R) mm[r + 1] = smu[c0 + 32 * r];
      if (r < R) eta[r + 1] = et[r + 1];
    }
    if (AXI) {
      axc = fdiv(real(1), real(2 * gi + 1));
      irx = fdiv(real(1), real(gi));
    }
#pragma unroll
    for (int r = 0; r <= R; ++r) {
      const real sy = et[r + 1] + et[r];  // the column's pair of the corner
      e4u[r] = sy + __shfl_up_sync(FULL, sy, 1);
      // (add_rn: rounded by itself in every kernel that inlines this)
      nfy[r] = add_rn(nu[r + 1], nu[r]);
    }
    real sx[R + 1];  // eta(i) + eta(i-1), rows -1 .. R-1
#pragma unroll
    for (int r = -1; r < R; ++r) {
      const real el = __shfl_up_sync(FULL, et[r + 1], 1);
      sx[r + 1] = et[r + 1] + el;
      if (r >= 0) etl[r] = el;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      e4v[r] = sx[r + 1] + sx[r];
      e4vr[r] = __shfl_down_sync(FULL, e4v[r], 1);
      nxl[r] = add_rn(nu[r + 1], __shfl_up_sync(FULL, nu[r + 1], 1));
      nxr[r] = __shfl_down_sync(FULL, nxl[r], 1);
      rbx[r] = __shfl_up_sync(FULL, rh[r + 1], 1) + rh[r + 1];
      rby[r] = rh[r] + rh[r + 1];
      const real px = ph[r + 1] + __shfl_up_sync(FULL, ph[r + 1], 1), py = ph[r + 1] + ph[r];
      const real mx = mm[r + 1] - __shfl_up_sync(FULL, mm[r + 1], 1), my = mm[r + 1] - mm[r];
      stx[r] = mul_rn(mul_rn(-P.sigma, px), mx);
      sty[r] = mul_rn(mul_rn(-P.sigma, py), my);
      rc[r] = mul_rn(rh[r + 1], P.cs2);
      if (AXI) {
        nu2[r] = mul_rn(real(2), nu[r + 1]);
        eax[r] = mul_rn(mul_rn(real(0.5), sx[r + 1]), irx);
        efy[r] = mul_rn(real(0.5), et[r] + et[r + 1]);
      }
    }
  }
  const bool bulk = P.bulk != 0, pavg = P.pavg != 0;
  const real half_dx2 = mul_rn(real(0.5), P.inv_dx2);
  const bool wall_tile = (wx && (gi0 < 0 || gi0 + 31 >= nx)) || (wy && (gj0 < 0 || gj0 + ROWS > ny));

  constexpr int NST = RATES ? 1 : 3;
#pragma unroll
  for (int st = 1; st <= NST; ++st) {
    const real* q = st == 1 ? qa : (st == 2 ? qb : qc);
    real* qo = st == 1 ? qb : qc;
    real out[R][3];
    if (live) {
      real u[R + 2], v[R + 2], p[R + 2];
#pragma unroll
      for (int r = -1; r <= R; ++r) {
        p[r + 1] = q[c0 + 32 * r];
        u[r + 1] = q[PLN + c0 + 32 * r];
        v[r + 1] = q[2 * PLN + c0 + 32 * r];
      }
      real ur[R + 1], D[R + 1], px[R + 1], pr[R + 1], pl[R + 1];  // rows -1 .. R-1
      real vl[R + 1], S[R + 1];                                   // rows 0 .. R; S: strain at the corner (i-1/2, j-1/2)
#pragma unroll
      for (int r = -1; r < R; ++r) {
        const int k = r + 1;
        ur[k] = q[PLN + c0 + 32 * r + 1];
        pr[k] = q[c0 + 32 * r + 1];
        pl[k] = q[c0 + 32 * r - 1];
        D[k] = (ur[k] - u[k]) + (v[k + 1] - v[k]);
        if (AXI) D[k] = fma(u[k] + ur[k], axc, D[k]);
        px[k] = pavg ? fma(real(4), p[k], pr[k] + pl[k]) : p[k];
      }
#pragma unroll
      for (int r = 0; r <= R; ++r) {
        vl[r] = q[2 * PLN + c0 + 32 * r - 1];
        S[r] = (u[r + 1] - u[r]) + (v[r + 1] - vl[r]);
      }
      const real gfac = pavg ? gp : P.inv_dx;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int k = r + 1;
        const real ul = q[PLN + c0 + 32 * r - 1], vr = q[2 * PLN + c0 + 32 * r + 1];
        // pressure
        real diff = mul_rn(nxr[r], pr[k] - p[k]);
        diff = fma(nxl[r], pl[k] - p[k], diff);
        diff = fma(nfy[r + 1], p[k + 1] - p[k], diff);
        diff = fma(nfy[r], p[k - 1] - p[k], diff);
        if (AXI) diff = fma(mul_rn(nu2[r], pr[k] - pl[k]), axc, diff);
        const real Lp = fma(diff, half_dx2, -mul_rn(rc[r], mul_rn(D[k], P.inv_dx)));
        // u on the low x face
        const real Dl = __shfl_up_sync(FULL, D[k], 1);
        real tcc = fma(etl[r], ul - u[k], mul_rn(eta[k], ur[k] - u[k]));
        real edge = fma(e4u[r], -S[r], mul_rn(e4u[r + 1], S[r + 1]));
        real visc = fma(real(2), tcc, mul_rn(real(0.25), edge));
        if (bulk) visc = fma(-etl[r], Dl, fma(eta[k], D[k], visc));
        if (AXI) visc = fma(eax[r], fma(real(0.5), ur[k] - ul, -mul_rn(u[k], irx)), visc);
        const real py = pavg ? fma(real(4), p[k], p[k + 1] + p[k - 1]) : p[k];
        real F = fma(visc, P.inv_dx2, -mul_rn(py - __shfl_up_sync(FULL, py, 1), gfac));
        F = fma(stx[r], P.inv_2dx, F);
        F = fma(fma(real(0.5), rbx[r], -P.rho_ref), P.g[0], F);
        const real V4 = (v[k] + vl[r]) + (v[k + 1] + vl[r + 1]);
        real conv = fma(u[k], ur[k] - ul, mul_rn(real(0.25), mul_rn(V4, u[k + 1] - u[k - 1])));
        real Lu = fma(-conv, P.inv_2dx, fdiv(mul_rn(real(2), F), rbx[r]));
        // v on the low y face
        tcc = fma(eta[k - 1], v[k - 1] - v[k], mul_rn(eta[k], v[k + 1] - v[k]));
        edge = fma(e4v[r], -S[r], mul_rn(e4vr[r], __shfl_down_sync(FULL, S[r], 1)));
        visc = fma(real(2), tcc, mul_rn(real(0.25), edge));
        if (bulk) visc = fma(-eta[k - 1], D[k - 1], fma(eta[k], D[k], visc));
        if (AXI) visc = fma(mul_rn(efy[r], vr - vl[r]), axc, visc);
        F = fma(visc, P.inv_dx2, -mul_rn(px[k] - px[k - 1], gfac));
        F = fma(sty[r], P.inv_2dx, F);
        F = fma(fma(real(0.5), rby[r], -P.rho_ref), P.g[1], F);
        const real uy = u[k] + u[k - 1];
        const real U4 = uy + __shfl_down_sync(FULL, uy, 1);
        conv = fma(v[k], v[k + 1] - v[k - 1], mul_rn(real(0.25), mul_rn(U4, vr - vl[r])));
        real Lv = fma(-conv, P.inv_2dx, fdiv(mul_rn(real(2), F), rby[r]));
        // faces on a wall are never updated
        if (wx && gi == 0) Lu = real(0);
        if (wy && gj + r == 0) Lv = real(0);
        if constexpr (RATES) {
          out[r][0] = Lp;
          out[r][1] = Lu;
          out[r][2] = Lv;
          continue;
        }
        const real a0 = fma(P.dt, Lp, p[k]), a1 = fma(P.dt, Lu, u[k]), a2 = fma(P.dt, Lv, v[k]);
        if (st == 1) {
          out[r][0] = a0;
          out[r][1] = a1;
          out[r][2] = a2;
        } else {
          const real a = st == 2 ? real(0.75) : real(1.0 / 3.0), b = st == 2 ? real(0.25) : real(2.0 / 3.0);
          const real* q0 = qa + c0 + 32 * r;
          out[r][0] = fma(a, q0[0], mul_rn(b, a0));
          out[r][1] = fma(a, q0[PLN], mul_rn(b, a1));
          out[r][2] = fma(a, q0[2 * PLN], mul_rn(b, a2));
        }
      }
    }
    if (st < NST) {
      // another buffer than any this stage reads (phi and mu are last read
      // before the first barrier of this loop)
      if (live && (!wx || (gi >= 0 && gi < nx))) {
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (!wy || (gj + r >= 0 && gj + r < ny)) {
#pragma unroll
            for (int f = 0; f < 3; ++f) qo[f * PLN + c0 + 32 * r] = out[r][f];
          }
      }
      __syncthreads();
      if (wall_tile) {
        flow_ghosts<real, NR, NT>(P, qo, gi0, gj0, tid);
        __syncthreads();
      }
    } else if (live && lane >= 3 && lane < 3 + FUSED_X && gi < nx) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int ly = rb + r;
        if (ly >= 3 && ly < 3 + flow_rows(NR) && gj + r < ny) {
          const long long id = (long long)(gj + r) * P.sy + gi;
#pragma unroll
          for (int f = 0; f < 3; ++f) A.out[f][id] = out[r][f];
          if (A.usum[0]) {
            const real un = qa[PLN + c0 + 32 * r], vn = qa[2 * PLN + c0 + 32 * r];
            A.usum[0][id] = un + (RATES ? un : out[r][1]);
            A.usum[1][id] = vn + (RATES ? vn : out[r][2]);
          }
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// the Cahn-Hilliard step
// ---------------------------------------------------------------------------

template <typename real>
struct CHStepArgs {
  const real* phi;
  const real* mu;
  const real* usum[2];  // u^n + u^{n+1} per face
  real* phi_out;
  real* mu_out;
  const real* lo;       // low part of phi (compensated accumulation), or nullptr
  real* lo_out;
};

// even ghosts of a walled tile's plane f (rows of 34 columns)
template <typename real, int NR, int NT>
__device__ __forceinline__ void ch_ghosts(const KParams<real>& P, real* f, int gi0, int gj0, int tid) {
  constexpr int ROWS = NR + 2;
  const int nx = P.n[0], ny = P.n[1];
  const bool wx = P.bc[0] != BC_PERIODIC, wy = P.bc[1] != BC_PERIODIC;
  for (int e = tid; e < 2 * ROWS + 68; e += NT) {
    int lx, ly;
    if (e < 2 * ROWS) {
      if (!wx) continue;
      ly = e >> 1;
      lx = ((e & 1) ? nx : -1) - gi0;
    } else {
      if (!wy) continue;
      lx = (e - 2 * ROWS) >> 1;
      ly = ((e & 1) ? ny : -1) - gj0;
    }
    if (lx < 0 || lx >= 34 || ly < 0 || ly >= ROWS) continue;
    const int gi = gi0 + lx, gj = gj0 + ly;
    if ((wx && (gi < -1 || gi > nx)) || (wy && (gj < -1 || gj > ny))) continue;
    const int cx = (wx ? clampi(gi, 0, nx - 1) : gi) - gi0, cy = (wy ? clampi(gj, 0, ny - 1) : gj) - gj0;
    if (cx >= 0 && cx < 34 && cy >= 0 && cy < ROWS) f[ly * 34 + lx] = f[cy * 34 + cx];
  }
}

// The whole TVD-RK2 CH step of the advective form on the tile of FUSED_X x
// ch_rows(NW R) cells at (i0, j0): phi_1, mu(phi_1), phi^{n+3/2} and its mu,
// each on one cell less on every side.  sm: ch_fused_smem reals.  With RATES the
// rate of phi alone, in A.phi_out.
template <typename real, int NW, int R, bool RATES = false>
__device__ __forceinline__ void ch2d_fused_tile(const KParams<real>& P, const CHStepArgs<real>& A, int i0, int j0,
                                                real* sm) {
  constexpr int NR = NW * R, ROWS = NR + 2, PLN = ROWS * 34, NT = 32 * NW;
  const int tid = threadIdx.y * blockDim.x + threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int nx = P.n[0], ny = P.n[1];
  const bool wx = P.bc[0] != BC_PERIODIC, wy = P.bc[1] != BC_PERIODIC;
  const int gi0 = i0 - 4, gj0 = j0 - 4;
  real* sa = sm + FUSED_PAD;   // phi, then phi^{n+3/2}
  real* sb = sa + PLN;         // phi_1
  real* sc = sb + PLN;         // mu, then mu(phi_1)
  const int rb = w * R + 1;
  const int gi = gi0 + 1 + lane, gj = gj0 + rb;  // the thread's column and first row
  const bool live = gj <= ny + 2;
  const int c0 = rb * 34 + lane + 1;
  // the time-centred velocity of the thread's cells (Eq. u-center-2d), frozen over the stages
  real uh[R][2], lo[R];
  if (plain_axis(gi0, 35, nx, P.bc[0]) && plain_axis(gj0, ROWS + 1, ny, P.bc[1])) {
    const int cx = wrap1(gi0 + lane, nx);
    if (live) {
      const int ux = wrap1(gi, nx), ux1 = wrap1(gi + 1, nx);
      real s0[R], s0n[R], s1[R + 1];
#pragma unroll
      for (int r = 0; r <= R; ++r) {
        const long long row = (long long)wrap1(gj + r, ny) * P.sy;
        s1[r] = A.usum[1][row + ux];
        if (r < R) {
          s0[r] = A.usum[0][row + ux];
          s0n[r] = A.usum[0][row + ux1];
          lo[r] = A.lo ? A.lo[row + ux] : real(0);
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        uh[r][0] = real(0.25) * (s0[r] + s0n[r]);
        uh[r][1] = real(0.25) * (s1[r] + s1[r + 1]);
      }
    }
#pragma unroll
    for (int k = 0; k < (ROWS + NW - 1) / NW; ++k) {
      const int ly = w + k * NW;
      if (ly < ROWS) {
        const long long id = (long long)wrap1(gj0 + ly, ny) * P.sy + cx;
        sa[ly * 34 + lane] = A.phi[id];
        sc[ly * 34 + lane] = A.mu[id];
      }
    }
    if (tid < 2 * ROWS) {  // the last two columns
      const int ly = tid >> 1, lx = 32 + (tid & 1);
      const long long id = (long long)wrap1(gj0 + ly, ny) * P.sy + wrap1(gi0 + lx, nx);
      sa[ly * 34 + lx] = A.phi[id];
      sc[ly * 34 + lx] = A.mu[id];
    }
  } else {
    const Map1 m0 = map1(gi0 + lane, nx, P.bc[0], false);
    for (int ly = w; ly < ROWS; ly += NW) {
      const long long row = (long long)map1(gj0 + ly, ny, P.bc[1], false).c * P.sy;
      sa[ly * 34 + lane] = A.phi[row + m0.c];
      sc[ly * 34 + lane] = A.mu[row + m0.c];
    }
    if (tid < 2 * ROWS) {
      const int ly = tid >> 1, lx = 32 + (tid & 1);
      const long long id = (long long)map1(gj0 + ly, ny, P.bc[1], false).c * P.sy + map1(gi0 + lx, nx, P.bc[0], false).c;
      sa[ly * 34 + lx] = A.phi[id];
      sc[ly * 34 + lx] = A.mu[id];
    }
    if (live) {
      const Map1 mx = map1(gi, nx, P.bc[0], false), mx1 = map1(gi + 1, nx, P.bc[0], false);
      real s1[R + 1];
#pragma unroll
      for (int r = 0; r <= R; ++r) {
        const Map1 my = map1(gj + r, ny, P.bc[1], false);
        s1[r] = my.zero_f ? real(0) : A.usum[1][(long long)my.f * P.sy + mx.c];
        if (r < R) {
          const long long row = (long long)my.c * P.sy;
          const real a = mx.zero_f ? real(0) : A.usum[0][row + mx.f];
          const real b = mx1.zero_f ? real(0) : A.usum[0][row + mx1.f];
          uh[r][0] = real(0.25) * (a + b);
          lo[r] = A.lo ? A.lo[row + mx.c] : real(0);
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) uh[r][1] = real(0.25) * (s1[r] + s1[r + 1]);
    }
  }
  static_assert(2 * (NR + 2) <= 32 * NW, "a thread stages at most one cell of the last two columns");
  __syncthreads();
  const bool inx = !wx || (gi >= 0 && gi < nx);
  const bool wall_tile = (wx && (gi0 < 0 || gi0 + 33 >= nx)) || (wy && (gj0 < 0 || gj0 + ROWS > ny));
  auto store = [&](real* f, const real* val) {
    if (live && inx) {
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (!wy || (gj + r >= 0 && gj + r < ny)) f[c0 + 34 * r] = val[r];
    }
    __syncthreads();
    if (wall_tile) {
      ch_ghosts<real, NR, NT>(P, f, gi0, gj0, tid);
      __syncthreads();
    }
  };
  // the stencil neighbourhood of the thread's column: rows -1 .. R of three columns
  auto window = [&](const real* f, real L[R + 2], real C[R + 2], real Rt[R + 2]) {
#pragma unroll
    for (int r = -1; r <= R; ++r) {
      L[r + 1] = f[c0 + 34 * r - 1];
      C[r + 1] = f[c0 + 34 * r];
      Rt[r + 1] = f[c0 + 34 * r + 1];
    }
  };
  auto rate = [&](const real* fphi, real L[R], real centre[R]) {
    real a[R + 2], b[R + 2], c[R + 2];
    window(sc, a, b, c);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      real lap = lap9<real>(P, a + r, b + r, c + r);
      if (P.axisym) lap = add_rn(lap, axis9_over_r<real>(P, a + r, c + r, gi));
      L[r] = lap;
    }
    window(fphi, a, b, c);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int k = r + 1;
      // the isotropic gradient, term by term in the order of grad_iso
      real sx = mul_rn(-P.w2, a[k - 1]), sy = sx;
      sy = fma(-P.w1, b[k - 1], sy);
      sx = fma(P.w2, c[k - 1], sx);
      sy = fma(-P.w2, c[k - 1], sy);
      sx = fma(-P.w1, a[k], sx);
      sx = fma(P.w1, c[k], sx);
      sx = fma(-P.w2, a[k + 1], sx);
      sy = fma(P.w2, a[k + 1], sy);
      sy = fma(P.w1, b[k + 1], sy);
      sx = fma(P.w2, c[k + 1], sx);
      sy = fma(P.w2, c[k + 1], sy);
      const real adv = fma(uh[r][1], mul_rn(P.grad_c, sy), mul_rn(uh[r][0], mul_rn(P.grad_c, sx)));
      L[r] = fma(P.M, L[r], -adv);
      centre[r] = b[k];
    }
  };
  auto chem = [&](const real* f, real out[R]) {
    real a[R + 2], b[R + 2], c[R + 2];
    window(f, a, b, c);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      real lap = lap9<real>(P, a + r, b + r, c + r);
      if (P.axisym) lap = add_rn(lap, axis9_over_r<real>(P, a + r, c + r, gi));
      out[r] = chem_pot<real>(P, b[r + 1], lap);
    }
  };
  real pn[R], L[R], d1[R], val[R], f1[R];
  if constexpr (RATES) {
    if (live) {
      rate(sa, L, pn);
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (lane >= 3 && lane < 3 + FUSED_X && gi < nx && rb + r >= 4 && rb + r < 4 + ch_rows(NR) && gj + r < ny)
          A.phi_out[(long long)(gj + r) * P.sy + gi] = L[r];
    }
    return;
  }
  if (live) {
    rate(sa, L, pn);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      val[r] = fma(P.dt, L[r], pn[r]);
      d1[r] = mul_rn(P.dt, L[r]);
    }
  }
  store(sb, val);
  if (live) chem(sb, val);
  // (sc: every thread is past its reads of mu)
  store(sc, val);
  real hi[R], low[R];
  if (live) {
    rate(sb, L, f1);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (A.lo) {
        pair_half(pn[r], lo[r], d1[r], mul_rn(P.dt, L[r]), hi[r], low[r]);
      } else {
        hi[r] = fma(real(0.5), pn[r], mul_rn(real(0.5), fma(P.dt, L[r], f1[r])));
        low[r] = real(0);
      }
    }
  }
  store(sa, hi);
  if (live && lane >= 3 && lane < 3 + FUSED_X && gi < nx) {
    chem(sa, val);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int ly = rb + r;
      if (ly >= 4 && ly < 4 + ch_rows(NR) && gj + r < ny) {
        const long long id = (long long)(gj + r) * P.sy + gi;
        A.phi_out[id] = hi[r];
        A.mu_out[id] = val[r];
        if (A.lo) A.lo_out[id] = low[r];
      }
    }
  }
}

// the passes of one problem; rates: the rates of the current state in their place
cudaError_t launch_flow_fused(const KParams<float>& P, const FlowStepArgs<float>& A, bool rates, cudaStream_t s);
cudaError_t launch_ch_fused(const KParams<float>& P, const CHStepArgs<float>& A, bool rates, cudaStream_t s);

}  // namespace gpe2p
