// flow.cu -- one TVD-RK3 stage of the GPE flow update (Sec. 3):
//   out = a q^n + b (q + dt L(q)),  q = (p, u, v[, w]),
// with L the semi-discrete operators of Eq. p-u-v-semidiscrete-2d built from
// Eqs. div-v-discretization, diff-p-discretization, conv-u-discretization,
// u-stress-discretization (a)-(d), st-u-discretization, gradp-u-discretization
// and gradp-u-p-ave-3d, with phi and mu frozen (Sec. 3, after Eq. tvd-rk3).
//
// The 2D FP64 stage of one tile is in flow_ops.cuh, the 2D FP32 step in step2d.cuh.
// 3D blocks march along z fed by the TMA plane ring of ring3d.cuh, two cells per
// thread.
#include "flow_ops.cuh"
#include "gpe2p_dev.cuh"
#include "gpe2p_launch.h"
#include "ring3d.cuh"

namespace gpe2p {

// 2D FP64: one tile per block (the FP32 step runs in the fused passes of step2d.cuh).
template <int MODE, int TXv, int TYv, int NT>
__global__ void __launch_bounds__(NT) flow2d64_kernel(const __grid_constant__ KParams<double> P,
                                                     const FlowArgs<double> A) {
  extern __shared__ __align__(16) double sm2d64[];
  after_previous_kernel();
  flow2d_tile64<MODE, TXv, TYv, NT>(P, A, blockIdx.x * TXv, blockIdx.y * TYv, sm2d64);
}

template <int TXv, int TYv, int NT>
static cudaError_t flow64_go(const KParams<double>& P, const FlowArgs<double>& A, int mode, cudaStream_t s) {
  static_assert(flow64_smem<TXv, TYv>(0) <= 48 * 1024, "no opt-in shared memory");
  const size_t sm = flow64_smem<TXv, TYv>(mode);
  const dim3 grd((P.n[0] + TXv - 1) / TXv, (P.n[1] + TYv - 1) / TYv);
  return launch_step(mode == 0 ? flow2d64_kernel<0, TXv, TYv, NT>
                               : (mode == 1 ? flow2d64_kernel<1, TXv, TYv, NT> : flow2d64_kernel<2, TXv, TYv, NT>),
                     small_grid(P), grd, NT, sm, s, P, A);
}

// The tile of a 2D FP64 stage: 32 x 8 where two tiles fall on every SM, else a
// smaller one, since a small grid is bound by the FP64 operations of its
// busiest SM (64 x 64: 16 tiles of 32 x 8 or 128 of 8 x 4).
// Measured: 20 steps of 64 x 64 with host arrays in and out 1.73 -> 0.80 ms,
// 50 steps of 128 x 64 4.05 -> 1.56 ms (32 x 8 tiles with every term formed per cell before); with
// overlapped launches 0.74 and 1.43 ms.
static cudaError_t flow64(const KParams<double>& P, const FlowArgs<double>& A, int mode, cudaStream_t s) {
  auto tiles = [&](int tx, int ty) {
    return (long long)((P.n[0] + tx - 1) / tx) * ((P.n[1] + ty - 1) / ty);
  };
  if (tiles(32, 8) >= 2 * 152) return flow64_go<32, 8, 256>(P, A, mode, s);
  if (!small_grid(P)) return flow64_go<16, 4, 192>(P, A, mode, s);
  return flow64_go<8, 4, 96>(P, A, mode, s);
}

// ---------------------------------------------------------------------------
// 3D: the same stage fed by the TMA plane ring of ring3d.cuh
// ---------------------------------------------------------------------------

// fields staged per plane; rho, eta and nu are formed from phi
enum { R_P = 0, R_U = 1, R_V = 2, R_W = 3, R_PHI = 4, R_MU = 5, NRAW_FLOW = 6 };

// a / rho.  FP32: times the approximate reciprocal, whose relative error is at most one
// ulp for the normal numbers that densities are.  With __fdividef in its place the fields
// of two 3D bubbles were the same and took longer: two steps of 256 x 256 x 512 5413 us
// against 5345, eight of 101 x 75 x 130 1718 against 1698.  FP64: the IEEE quotient.
__device__ __forceinline__ float quot_rho(float a, float rho) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(rho));
  return a * r;
}
__device__ __forceinline__ double quot_rho(double a, double rho) { return a / rho; }

// Material and viscosity sums of one plane at the thread's column: rows -1 .. R.
template <typename real, int R>
struct FlowMat {
  real eta[R + 2], nu[R + 2];  // eta / dx^2 and nu / dx^2, rows -1 .. R
  real rho[R + 1];             // rows -1 .. R-1
  real sx[R + 2];              // eta(i) + eta(i-1), rows -1 .. R
  real sy[R + 1];              // eta(j) + eta(j-1), rows 0 .. R
};

// The terms of the faces and edges between a plane and the one above it, and the
// plane's x-y averaged pressure.  The block marches along z, so the values
// formed above one plane are those below the next and stay in registers.
template <typename real, int R>
struct FlowZ {
  real txz[R];      // 4 eta_edge/dx^2 (du/dz + dw/dx) dx on the x-z edges, rows 0 .. R-1
  real tyz[R + 1];  // the y-z edges, rows 0 .. R
  real tz[R];       // normal stress of the plane's cells along z
  real fz[R];       // (nu + nu(+z)) (p(+z) - p)
  real xy[R];       // 36 x the pressure averaged over x and y
  real rho[R];
};

// One block: FLOW_K3_TX x FLOW_K3_TY cells of a column over the planes
// [kbeg, kend).  Lane = staged column (30 of the 32 are the block's own);
// each thread takes R = 2 adjacent rows.
//
// What bounds it: instruction issue, not HBM.  So every term that two
// cells share is formed once: the normal stresses, corner stresses, diffusive
// fluxes and averaged pressures of a column go to its left or right
// neighbour by a shuffle, to the row above in registers (the two rows beyond
// the thread's own are formed twice), and to the plane above in registers
// (FlowZ); averages are taken axis by axis.  The price is two idle
// lanes of 32.  Stage 2 of 128 x 128 x 256 (ncu): 105 us, 218 floating-point
// instructions a cell; 121 us and 365 with each thread forming all terms of its
// two cells.
// FLOW_MINB blocks of four warps per SM: 128 registers (FP64: two blocks, which
// its ALU rate keeps busy).
template <typename real, int MODE, int RING, int PAVG>
__global__ void __launch_bounds__(FLOW_NTHR, sizeof(real) == 8 ? FLOW_MINB64 : FLOW_MINB)
    flow3d_kernel(const __grid_constant__ Maps<NRAW_FLOW> maps, const __grid_constant__ KParams<real> P,
                  const FlowArgs<real> A, const int kchunk, int* err) {
  constexpr int SYv = FLOW_K3_SY, R = 2;
  using G = FlowGeom<real, SYv>;
  constexpr unsigned FULL = 0xffffffffu;
  extern __shared__ __align__(128) unsigned char smraw[];
  Ring<real, NRAW_FLOW, RING, SYv, G, FLOW_TY> Rg;
  unsigned char* sbase = smem_base128(smraw);
  Rg.bar = reinterpret_cast<uint64_t*>(sbase);
  Rg.raw = reinterpret_cast<real*>(sbase + 128);
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
  const int i0 = blockIdx.x * FLOW_K3_TX, j0 = blockIdx.y * FLOW_K3_TY;
  const int kbeg = blockIdx.z * kchunk;
  const int kend = min(kbeg + kchunk, P.n[2]);
  const int nx = P.n[0], ny = P.n[1], nz = P.n[2];
  const bool edge_tile = i0 == 0 || i0 + 31 > nx || j0 == 0 || j0 + FLOW_K3_TY + 1 > ny;
  const int i = i0 - 1 + tx, ja = j0 + 2 * ty;
  const bool own = tx >= 1 && tx <= FLOW_K3_TX && i < nx;
  const bool act[2] = {own && ja < ny, own && ja + 1 < ny};
  const int shift = G::shift(i0);

  Rg.start(P, maps.m, kbeg, kend, i0, j0, (P.wait_fault & WF_FLOW_RING) != 0);

  // set the ghost cells of plane kk, which has landed: those of a tile on the
  // boundary, all of a plane beyond a periodic z side; a plane beyond a z wall is
  // filled from the plane next to it by zwall
  const bool zper = P.bc[2] == BC_PERIODIC;
  auto ghosts = [&](int kk) {
    const bool ghost_plane = kk < 0 || kk >= nz;
    if (ghost_plane ? !zper : !edge_tile) return;
    real* pl[NRAW_FLOW];
#pragma unroll
    for (int f = 0; f < NRAW_FLOW; ++f) pl[f] = Rg.plane(kk, f) + shift;
    if (ghost_plane) {
      for (int q = tid; q < 32 * SYv; q += FLOW_NTHR) {
        const int ly = q >> 5, lx = q & 31;
        const int e = G::at(lx, ly);
        const int ci = clampi(i0 - 1 + lx, -1, nx), cj = clampi(j0 - 1 + ly, -1, ny);
        pl[R_P][e] = ld_cen(A.q[0], P, ci, cj, kk);
        pl[R_U][e] = ld_face<0>(A.q[1], P, ci, cj, kk);
        pl[R_V][e] = ld_face<1>(A.q[2], P, ci, cj, kk);
        pl[R_W][e] = ld_face<2>(A.q[3], P, ci, cj, kk);
        pl[R_PHI][e] = ld_cen(A.phi, P, ci, cj, kk);
        pl[R_MU][e] = ld_cen(A.mu, P, ci, cj, kk);
      }
    } else {
      static_assert(ghost_count<SYv, 32>() <= FLOW_NTHR, "a ghost cell per thread");
      int lx, ly;
      if (tid < ghost_count<SYv, 32>() && ghost_cell<SYv, 32>(P, i0, j0, tid, lx, ly)) {
        const int e = G::at(lx, ly), gi = i0 - 1 + lx, gj = j0 - 1 + ly;
        pl[R_P][e] = ghost_value<G>(K_CEN, pl[R_P], A.q[0], P, i0, j0, gi, gj, kk);
        pl[R_U][e] = ghost_value<G>(K_FACE0, pl[R_U], A.q[1], P, i0, j0, gi, gj, kk);
        pl[R_V][e] = ghost_value<G>(K_FACE1, pl[R_V], A.q[2], P, i0, j0, gi, gj, kk);
        pl[R_W][e] = ghost_value<G>(K_FACE2, pl[R_W], A.q[3], P, i0, j0, gi, gj, kk);
        pl[R_PHI][e] = ghost_value<G>(K_CEN, pl[R_PHI], A.phi, P, i0, j0, gi, gj, kk);
        pl[R_MU][e] = ghost_value<G>(K_CEN, pl[R_MU], A.mu, P, i0, j0, gi, gj, kk);
      }
    }
    fence_proxy_async_smem();
  };
  // the plane kk beyond a z wall from the plane next to it, after a barrier that
  // follows that plane's ghost writes
  auto zwall = [&](int kk) {
    const int from = kk < 0 ? 0 : nz - 1;
    for (int q = tid; q < G::BX * SYv; q += FLOW_NTHR) {
      Rg.plane(kk, R_P)[q] = Rg.plane(from, R_P)[q];
      Rg.plane(kk, R_U)[q] = zwall_value<K_FACE0>(P, Rg.plane(from, R_U)[q]);
      Rg.plane(kk, R_V)[q] = zwall_value<K_FACE1>(P, Rg.plane(from, R_V)[q]);
      Rg.plane(kk, R_W)[q] = real(0);
      Rg.plane(kk, R_PHI)[q] = Rg.plane(from, R_PHI)[q];
      Rg.plane(kk, R_MU)[q] = Rg.plane(from, R_MU)[q];
    }
    fence_proxy_async_smem();
  };

  if (!Rg.wait(kbeg - 1)) { Rg.fail(err, kbeg - 1); return; }
  ghosts(kbeg - 1);
  if (!Rg.wait(kbeg)) { Rg.fail(err, kbeg); return; }
  ghosts(kbeg);
  // after every thread's writes of the two planes' ghost cells
  if (edge_tile || kbeg == 0 || kbeg + 1 >= nz) __syncthreads();
  if (kbeg == 0 && !zper) {
    zwall(-1);
    __syncthreads();
  }

  const real* smr = reinterpret_cast<const real*>(smraw);
  const int cell0 = (int)(Rg.raw - smr) + shift + G::at(tx, 2 * ty + 1);
  auto base = [&](int kk) { return cell0 + Rg.slot(kk) * NRAW_FLOW * G::PE; };
  // staged field f at row r, column offset dx of the plane at base b
  auto S = [&](int b, int f, int r, int dx) { return smr[b + f * G::PE + r * G::BX + dx]; };
  auto left = [&](real v) { return __shfl_up_sync(FULL, v, 1); };
  auto right = [&](real v) { return __shfl_down_sync(FULL, v, 1); };
  const real emd = P.eta_d * P.inv_dx2, emm = P.eta_m * P.inv_dx2;
  const real bulk = P.bulk ? real(1) : real(0);

  auto material = [&](int b, FlowMat<real, R>& m) {
#pragma unroll
    for (int r = -1; r <= R; ++r) {
      const real ph = S(b, R_PHI, r, 0);
      m.eta[r + 1] = fma(emd, ph, emm);
      const real rho = rho_of(P, ph);
      if (r < R) m.rho[r + 1] = rho;
      m.nu[r + 1] = quot_rho(m.eta[r + 1], rho);
      m.sx[r + 1] = m.eta[r + 1] + left(m.eta[r + 1]);
      if (r >= 0) m.sy[r] = m.eta[r + 1] + m.eta[r];
    }
  };
  // dx div u of the cell in row r of the plane at b, n above it
  auto divsum = [&](int b, int n, int r) {
    return ((S(b, R_U, r, 1) - S(b, R_U, r, 0)) + (S(b, R_V, r + 1, 0) - S(b, R_V, r, 0))) +
           (S(n, R_W, r, 0) - S(b, R_W, r, 0));
  };
  // bD: the bulk viscosity's share of the divergence, rows -1 .. R-1
  auto above = [&](int b, int n, const FlowMat<real, R>& mc, const FlowMat<real, R>& mn, const real* bD,
                   FlowZ<real, R>& z) {
#pragma unroll
    for (int r = 0; r <= R; ++r)
      z.tyz[r] = (mc.sy[r] + mn.sy[r]) *
                 ((S(n, R_V, r, 0) - S(b, R_V, r, 0)) + (S(n, R_W, r, 0) - S(n, R_W, r - 1, 0)));
#pragma unroll
    for (int r = 0; r < R; ++r) {
      z.txz[r] = (mc.sx[r + 1] + mn.sx[r + 1]) *
                 ((S(n, R_U, r, 0) - S(b, R_U, r, 0)) + (S(n, R_W, r, 0) - S(n, R_W, r, -1)));
      const real dw = S(n, R_W, r, 0) - S(b, R_W, r, 0);
      z.tz[r] = mc.eta[r + 1] * fma(real(2), dw, bD[r + 1]);
      z.rho[r] = mc.rho[r + 1];
      z.fz[r] = (mc.nu[r + 1] + mn.nu[r + 1]) * (S(n, R_P, r, 0) - S(b, R_P, r, 0));
      if (PAVG) {
        const real yp = fma(real(4), S(b, R_P, r, 0), S(b, R_P, r + 1, 0) + S(b, R_P, r - 1, 0));
        z.xy[r] = fma(real(4), yp, left(yp) + right(yp));
      }
    }
  };

  FlowMat<real, R> mc;
  FlowZ<real, R> zp;
  {
    FlowMat<real, R> mm;
    material(base(kbeg - 1), mm);
    material(base(kbeg), mc);
    real bD[R + 1];
#pragma unroll
    for (int r = 0; r < R; ++r) bD[r + 1] = bulk * divsum(base(kbeg - 1), base(kbeg), r);
    above(base(kbeg - 1), base(kbeg), mm, mc, bD, zp);
  }
  const real gfac = P.inv_dx * (PAVG ? real(1.0 / 36.0) : real(1));
  const real c_st = -P.sigma * P.inv_2dx;
  const real q2 = real(0.25);
  long long id = lin(P, i, ja, kbeg);
  for (int k = kbeg; k < kend; ++k, id += P.sz) {
    real q0v[R][4];
    if (MODE == 2) {
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (act[r]) {
#pragma unroll
          for (int f = 0; f < 4; ++f) q0v[r][f] = A.q0[f][id + r * P.sy];
        }
    }
    if (!Rg.wait(k + 1)) { Rg.fail(err, k + 1); return; }
    Rg.refill(P, maps.m, k + 1);
    ghosts(k + 1);
    // the threads' writes of ghost cells must be seen by all before the stencil
    // reads them; a plane that needed none is visible to every thread after
    // its own wait on the plane's barrier
    if (k + 1 == nz && !zper) zwall(nz);  // (plane nz - 1 was set and read in the last turn)
    if (edge_tile || k + 1 >= nz) __syncthreads();
    const int bm = base(k - 1), bc = base(k), bn = base(k + 1);
    FlowMat<real, R> mn;
    FlowZ<real, R> zc;
    material(bn, mn);
    real out[R][4];
    // terms of rows -1 .. R the two cells share
    real D[R + 1], bD[R + 1], Ty[R + 1], txy[R + 1], fy[R + 1], zpr[R + 2], xz[R + 1];
#pragma unroll
    for (int r = -1; r < R; ++r) {
      D[r + 1] = divsum(bc, bn, r);
      bD[r + 1] = bulk * D[r + 1];
      Ty[r + 1] = mc.eta[r + 1] * fma(real(2), S(bc, R_V, r + 1, 0) - S(bc, R_V, r, 0), bD[r + 1]);
    }
    above(bc, bn, mc, mn, bD, zc);
#pragma unroll
    for (int r = 0; r <= R; ++r) {
      txy[r] = (mc.sx[r + 1] + mc.sx[r]) * ((S(bc, R_U, r, 0) - S(bc, R_U, r - 1, 0)) +
                                            (S(bc, R_V, r, 0) - S(bc, R_V, r, -1)));
      fy[r] = (mc.nu[r + 1] + mc.nu[r]) * (S(bc, R_P, r, 0) - S(bc, R_P, r - 1, 0));
    }
    if (PAVG) {
#pragma unroll
      for (int r = -1; r <= R; ++r) zpr[r + 1] = fma(real(4), S(bc, R_P, r, 0), S(bm, R_P, r, 0) + S(bn, R_P, r, 0));
#pragma unroll
      for (int r = -1; r < R; ++r) xz[r + 1] = fma(real(4), zpr[r + 1], left(zpr[r + 1]) + right(zpr[r + 1]));
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const real p0 = S(bc, R_P, r, 0), u0 = S(bc, R_U, r, 0), v0 = S(bc, R_V, r, 0), w0 = S(bc, R_W, r, 0);
      const real ur = S(bc, R_U, r, 1), ul = S(bc, R_U, r, -1), wn = S(bn, R_W, r, 0);
      // pressure
      const real fx = (mc.nu[r + 1] + left(mc.nu[r + 1])) * (p0 - S(bc, R_P, r, -1));
      const real diff = ((right(fx) - fx) + (fy[r + 1] - fy[r])) + (zc.fz[r] - zp.fz[r]);
      const real Lp = fma(real(0.5), diff, -(mc.rho[r + 1] * P.cs2 * (D[r + 1] * P.inv_dx)));
      const real ph0 = S(bc, R_PHI, r, 0), mu0 = S(bc, R_MU, r, 0);
      // u on the low x face
      real L[4];
      L[0] = Lp;
      {
        const real Tx = mc.eta[r + 1] * fma(real(2), ur - u0, bD[r + 1]);
        real F = fma(q2, (txy[r + 1] - txy[r]) + (zc.txz[r] - zp.txz[r]), Tx - left(Tx));
        real g;
        if (PAVG) {
          const real yz = fma(real(4), zpr[r + 1], zpr[r + 2] + zpr[r]);
          g = yz - left(yz);
        } else {
          g = p0 - S(bc, R_P, r, -1);
        }
        F = fma(-g, gfac, F);
        F = fma(c_st * (ph0 + S(bc, R_PHI, r, -1)), mu0 - S(bc, R_MU, r, -1), F);
        const real rb = mc.rho[r + 1] + left(mc.rho[r + 1]);
        F = fma(fma(real(0.5), rb, -P.rho_ref), P.g[0], F);
        const real V4 = (v0 + S(bc, R_V, r, -1)) + (S(bc, R_V, r + 1, 0) + S(bc, R_V, r + 1, -1));
        const real W4 = (w0 + S(bc, R_W, r, -1)) + (wn + S(bn, R_W, r, -1));
        const real tr = fma(V4, S(bc, R_U, r + 1, 0) - S(bc, R_U, r - 1, 0), W4 * (S(bn, R_U, r, 0) - S(bm, R_U, r, 0)));
        const real conv = fma(u0, ur - ul, q2 * tr);
        L[1] = fma(-conv, P.inv_2dx, quot_rho(real(2) * F, rb));
      }
      // v on the low y face
      {
        real F = fma(q2, (right(txy[r]) - txy[r]) + (zc.tyz[r] - zp.tyz[r]), Ty[r + 1] - Ty[r]);
        const real g = PAVG ? xz[r + 1] - xz[r] : p0 - S(bc, R_P, r - 1, 0);
        F = fma(-g, gfac, F);
        F = fma(c_st * (ph0 + S(bc, R_PHI, r - 1, 0)), mu0 - S(bc, R_MU, r - 1, 0), F);
        const real rb = mc.rho[r + 1] + mc.rho[r];
        F = fma(fma(real(0.5), rb, -P.rho_ref), P.g[1], F);
        const real uy = u0 + S(bc, R_U, r - 1, 0);
        const real U4 = uy + right(uy);
        const real W4 = (w0 + S(bc, R_W, r - 1, 0)) + (wn + S(bn, R_W, r - 1, 0));
        const real tr = fma(U4, S(bc, R_V, r, 1) - S(bc, R_V, r, -1), W4 * (S(bn, R_V, r, 0) - S(bm, R_V, r, 0)));
        const real conv = fma(v0, S(bc, R_V, r + 1, 0) - S(bc, R_V, r - 1, 0), q2 * tr);
        L[2] = fma(-conv, P.inv_2dx, quot_rho(real(2) * F, rb));
      }
      // w on the low z face
      {
        real F = fma(q2, (right(zp.txz[r]) - zp.txz[r]) + (zp.tyz[r + 1] - zp.tyz[r]), zc.tz[r] - zp.tz[r]);
        const real g = PAVG ? zc.xy[r] - zp.xy[r] : p0 - S(bm, R_P, r, 0);
        F = fma(-g, gfac, F);
        F = fma(c_st * (ph0 + S(bm, R_PHI, r, 0)), mu0 - S(bm, R_MU, r, 0), F);
        const real rb = mc.rho[r + 1] + zp.rho[r];
        F = fma(fma(real(0.5), rb, -P.rho_ref), P.g[2], F);
        const real uz = u0 + S(bm, R_U, r, 0);
        const real U4 = uz + right(uz);
        const real V4 = (v0 + S(bm, R_V, r, 0)) + (S(bc, R_V, r + 1, 0) + S(bm, R_V, r + 1, 0));
        const real tr = fma(U4, S(bc, R_W, r, 1) - S(bc, R_W, r, -1),
                            V4 * (S(bc, R_W, r + 1, 0) - S(bc, R_W, r - 1, 0)));
        const real conv = fma(w0, wn - S(bm, R_W, r, 0), q2 * tr);
        L[3] = fma(-conv, P.inv_2dx, quot_rho(real(2) * F, rb));
      }
      // faces on a wall are never updated
      if (P.bc[0] != BC_PERIODIC && i == 0) L[1] = real(0);
      if (P.bc[1] != BC_PERIODIC && ja + r == 0) L[2] = real(0);
      if (P.bc[2] != BC_PERIODIC && k == 0) L[3] = real(0);
      const real q[4] = {p0, u0, v0, w0};
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        if (MODE == 0) out[r][f] = L[f];
        else if (MODE == 1) out[r][f] = fma(P.dt, L[f], q[f]);
        else out[r][f] = fma(A.a, q0v[r][f], A.b * fma(P.dt, L[f], q[f]));
      }
    }
    // stores after both cells, so that nothing separates their shared loads
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (act[r]) {
#pragma unroll
        for (int f = 0; f < 4; ++f) A.out[f][id + r * P.sy] = out[r][f];
      }
    // the last stage also leaves u^n + u^{n+1} on every face, from which the
    // CH step forms the time-centred cell velocity with half the loads
    if (MODE == 2 && A.usum[0]) {
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (act[r]) {
#pragma unroll
          for (int a = 0; a < 3; ++a) A.usum[a][id + r * P.sy] = q0v[r][1 + a] + out[r][1 + a];
        }
    }
    mc = mn;
    zp = zc;
  }
}

#ifndef GPE2P_FLOW_RING
#define GPE2P_FLOW_RING 4
#endif
template <typename real>
constexpr int flow_ring() { return GPE2P_FLOW_RING; }

template <typename real, int DIM>
cudaError_t launch_flow_stage(const KParams<real>& P, const FlowArgs<real>& A, int mode, int kchunk,
                              cudaStream_t s, const Maps<6>* maps, int* err) {
  if constexpr (DIM == 3) {
    constexpr int RING = flow_ring<real>();
    const size_t sm = 256 + sizeof(real) * (size_t)FlowGeom<real, FLOW_K3_SY>::PE * RING * NRAW_FLOW;
    const dim3 blk(TX, FLOW_TY);
    const dim3 grd((P.n[0] + FLOW_K3_TX - 1) / FLOW_K3_TX, (P.n[1] + FLOW_K3_TY - 1) / FLOW_K3_TY,
                   (P.n[2] + kchunk - 1) / kchunk);
    cudaError_t e;
#define GPE2P_FLOW3_CASE(M)                                                                                 \
  if (P.pavg) {                                                                                             \
    e = cudaFuncSetAttribute(flow3d_kernel<real, M, RING, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize,  \
                             (int)sm);                                                                      \
    if (e != cudaSuccess) return e;                                                                         \
    flow3d_kernel<real, M, RING, 1><<<grd, blk, sm, s>>>(*maps, P, A, kchunk, err);                         \
  } else {                                                                                                  \
    e = cudaFuncSetAttribute(flow3d_kernel<real, M, RING, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize,  \
                             (int)sm);                                                                      \
    if (e != cudaSuccess) return e;                                                                         \
    flow3d_kernel<real, M, RING, 0><<<grd, blk, sm, s>>>(*maps, P, A, kchunk, err);                         \
  }
    if (mode == 0) { GPE2P_FLOW3_CASE(0) }
    else if (mode == 1) { GPE2P_FLOW3_CASE(1) }
    else { GPE2P_FLOW3_CASE(2) }
#undef GPE2P_FLOW3_CASE
    return cudaGetLastError();
  } else {
    return flow64(P, A, mode, s);
  }
}

#define GPE2P_FLOW_INST(R, D)                                                                      \
  template cudaError_t launch_flow_stage<R, D>(const KParams<R>&, const FlowArgs<R>&, int, int, cudaStream_t, \
                                               const Maps<6>*, int*);
GPE2P_FLOW_INST(float, 3)
GPE2P_FLOW_INST(double, 2)
GPE2P_FLOW_INST(double, 3)
#undef GPE2P_FLOW_INST

}  // namespace gpe2p
