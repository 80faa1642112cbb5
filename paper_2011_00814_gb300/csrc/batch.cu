// batch.cu -- many independent 2D problems of uneven sizes advanced together.
//
// Every instance has its own parameters (Sec. 2, Sec. 4) and its own state;
// all instances step together.  The tiles of all instances form one work
// table of (instance, tile) items.  A step is the sequence of the 2D sweeps
// of the method (three flow stages, Eq. tvd-rk3; the CH stages of
// Eq. tvd-rk2 with mu recomputed, Eq. chem-pot), each sweep covering every
// item, and it runs in one of two forms:
//   persistent: one cooperative launch per step; the blocks walk the work
//               table sweep by sweep and meet at a grid barrier between
//               sweeps (a bounded wait: after the limit the block records an
//               error and returns);
//   per sweep:  one launch per sweep over the whole table; in FP32 without
//               conservative instances the flow stages are one fused pass and the
//               CH stages with mu another (step2d.cuh).
// Both are captured into CUDA graphs.  The form, and the tile shape of the sweeps, are
// chosen by timing the candidates when the batch is created (the autotuner); the
// fused passes' tiles by the number of tiles (fused_tall).  The
// per-tile arithmetic is the same device code as the single-instance 2D
// kernels (flow_ops.cuh, ch_ops.cuh), so an instance of a batch follows the
// single-instance path bit for bit.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/gpe2p.h"
#include "batch.h"
#include "ch_ops.cuh"
#include "diag_ops.cuh"
#include "flow_ops.cuh"
#include "gpe2p_dev.cuh"
#include "gpe2p_launch.h"
#include "step2d.cuh"

namespace gpe2p {

// ---------------------------------------------------------------------------
// device side
// ---------------------------------------------------------------------------

template <typename real>
struct BInst {
  KParams<real> P;
  real* Q[3][3];   // (p, u, v) of the three stage sets
  // phi^{n+1/2} and its mu, by the parity of the step: the fused CH step goes
  // from one set to the other, the stages of the other form keep one set
  real* phi[2];
  real* mu[2];
  real* phis;      // CH stage state
  real* mus;       // mu of the stage state
  real* uh[2];     // time-centred cell velocity
  real* z[Z_N];    // FP64: the terms frozen over the flow stages (fill_insts)
  real* us[2];     // u^n + u^{n+1} per face (advective form), left by the last flow stage
  int conservative;
};

struct BItem {
  int inst, i0, j0;
};

struct BarrierState {
  unsigned count;
  unsigned gen;
};

enum {
  SW_FLOW1 = 0, SW_FLOW2, SW_FLOW3, SW_UH, SW_CH1, SW_MU1, SW_CH2, SW_MU2, SW_N
};

// the centre velocity of the tile's cells for the conservative form (no halo)
template <typename real, int TXv, int TYv>
__device__ __forceinline__ void uh2d_tile(const KParams<real>& P, const real* u0, const real* v0, const real* u1,
                                          const real* v1, real* uh0, real* uh1, int i0, int j0) {
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int i = i0 + tid % TXv, j = j0 + 2 * (tid / TXv) + r;
    if (i < P.n[0] && j < P.n[1]) {
      const long long id = lin(P, i, j, 0);
      uh0[id] =
          real(0.25) * ((u0[id] + face_next<0>(u0, P, i, j, 0, id)) + (u1[id] + face_next<0>(u1, P, i, j, 0, id)));
      uh1[id] =
          real(0.25) * ((v0[id] + face_next<1>(v0, P, i, j, 0, id)) + (v1[id] + face_next<1>(v1, P, i, j, 0, id)));
    }
  }
}

template <typename real, int TXv, int TYv>
__device__ __forceinline__ void do_sweep(int sw, const BInst<real>& b, const BItem& it, int cur, real* sm) {
  const int s1 = 1 - cur, s2 = 2;
  if (sw <= SW_FLOW3) {
    FlowArgs<real> A;
    const int qin = sw == SW_FLOW1 ? cur : (sw == SW_FLOW2 ? s1 : s2);
    const int qout = sw == SW_FLOW2 ? s2 : s1;
    for (int f = 0; f < 3; ++f) {
      A.q0[f] = b.Q[cur][f];
      A.q[f] = b.Q[qin][f];
      A.out[f] = b.Q[qout][f];
    }
    A.q0[3] = A.q[3] = nullptr;
    A.out[3] = nullptr;
    A.phi = b.phi[cur];
    A.mu = b.mu[cur];
    const bool sums = sw == SW_FLOW3 && !b.conservative;
    A.usum[0] = sums ? b.us[0] : nullptr;
    A.usum[1] = sums ? b.us[1] : nullptr;
    A.usum[2] = nullptr;
    for (int k = 0; k < Z_N; ++k) A.z[k] = b.z[k];
    if (sw == SW_FLOW1) {
      A.a = real(0);
      A.b = real(1);
      if constexpr (sizeof(real) == 8) flow2d_tile64<1, TXv, TYv, TXv * TYv / 2, false>(b.P, A, it.i0, it.j0, sm);
    } else {
      A.a = sw == SW_FLOW2 ? real(0.75) : real(1.0 / 3.0);
      A.b = sw == SW_FLOW2 ? real(0.25) : real(2.0 / 3.0);
      if constexpr (sizeof(real) == 8) flow2d_tile64<2, TXv, TYv, TXv * TYv / 2, false>(b.P, A, it.i0, it.j0, sm);
    }
    return;
  }
  if (sw == SW_UH) {
    if (b.conservative)
      uh2d_tile<real, TXv, TYv>(b.P, b.Q[cur][1], b.Q[cur][2], b.Q[s1][1], b.Q[s1][2], b.uh[0], b.uh[1], it.i0,
                                it.j0);
    return;
  }
  if (sw == SW_MU1 || sw == SW_MU2) {
    if (sw == SW_MU1) mu2d_tile<real, TXv, TYv>(b.P, b.phis, b.mus, it.i0, it.j0, sm);
    else mu2d_tile<real, TXv, TYv>(b.P, b.phi[cur], b.mu[cur], it.i0, it.j0, sm);
    return;
  }
  CHArgs<real> C;
  C.uh[0] = b.uh[0];
  C.uh[1] = b.uh[1];
  C.uh[2] = nullptr;
  C.u0[0] = b.Q[cur][1];
  C.u0[1] = b.Q[cur][2];
  C.u1[0] = b.Q[s1][1];
  C.u1[1] = b.Q[s1][2];
  C.u0[2] = C.u1[2] = nullptr;
  C.scheme = 2;
  C.conservative = b.conservative;
  C.acc = nullptr;
  C.phin = b.phi[cur];
  C.usum[0] = b.conservative ? nullptr : b.us[0];
  C.usum[1] = b.conservative ? nullptr : b.us[1];
  C.usum[2] = nullptr;
  C.phi_lo = nullptr;
  if (sw == SW_CH1) {
    C.stage = 1;
    C.phis = b.phi[cur];
    C.mus = b.mu[cur];
    C.out = b.phis;
    C.compute_uh = !b.conservative;
  } else {
    C.stage = 2;
    C.phis = b.phis;
    C.mus = b.mus;
    C.out = b.phi[cur];
    C.compute_uh = 0;
  }
  ch2d_tile<real, TXv, TYv>(b.P, C, it.i0, it.j0, sm);
}

// the fused passes of an FP32 instance (step2d.cuh)
template <int NW, int R, bool AXI>
__device__ __forceinline__ void do_flow_fused(const BInst<float>& b, const BItem& it, int cur, float* sm) {
  FlowStepArgs<float> A;
  for (int f = 0; f < 3; ++f) {
    A.q[f] = b.Q[cur][f];
    A.out[f] = b.Q[1 - cur][f];
  }
  A.phi = b.phi[cur];
  A.mu = b.mu[cur];
  A.usum[0] = b.conservative ? nullptr : b.us[0];
  A.usum[1] = b.conservative ? nullptr : b.us[1];
  flow2d_fused_tile<float, NW, R, AXI>(b.P, A, it.i0, it.j0, sm);
}

template <int NW, int R>
__device__ __forceinline__ void do_ch_fused(const BInst<float>& b, const BItem& it, int cur, float* sm) {
  CHStepArgs<float> A;
  A.phi = b.phi[cur];
  A.mu = b.mu[cur];
  A.usum[0] = b.us[0];
  A.usum[1] = b.us[1];
  A.phi_out = b.phi[1 - cur];
  A.mu_out = b.mu[1 - cur];
  A.lo = nullptr;
  A.lo_out = nullptr;
  ch2d_fused_tile<float, NW, R>(b.P, A, it.i0, it.j0, sm);
}

// the work tables of a batch: the fused passes' tiles (FP32: flow of every
// instance, CH of the advective ones) and the tiles of the per-stage sweeps
// (FP64: every instance; FP32: the CH sweeps of the conservative instances)
struct BTables {
  const BItem *flow, *ch, *tiles;
  int nflow, nch, ntiles;
};

// all blocks of a cooperative launch meet here; false (block-uniform) if the
// wait ran past its limit.  With skip set the block does not arrive (a
// host-side fault injection used by the tests) and waits like the others.
__device__ __forceinline__ bool grid_barrier(BarrierState* bs, unsigned nblocks, long long limit, bool skip) {
  __syncthreads();
  int ok = 1;
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    volatile unsigned* gen = &bs->gen;
    const unsigned g = *gen;
    __threadfence();
    bool last = false;
    if (!skip) last = atomicAdd(&bs->count, 1u) + 1u == nblocks;
    if (last) {
      bs->count = 0u;
      __threadfence();
      atomicAdd(&bs->gen, 1u);
    } else {
      const long long t0 = clock64();
      while (*gen == g) {
        if (clock64() - t0 > limit) {
          ok = 0;
          break;
        }
        __nanosleep(64);
      }
    }
    __threadfence();
  }
  return __syncthreads_and(ok) != 0;
}

constexpr int ERR_BARRIER_TIMEOUT = 2;

// rows per thread of the fused passes in the persistent form's blocks of four
// warps: with four, their tiles are those of the short per-pass form
constexpr int PERSISTENT_R = 4;
static_assert(4 * PERSISTENT_R == FUSED_NW * FUSED_R, "the persistent form walks the short tiles' tables");

template <typename real, int TXv, int TYv>
__global__ void __launch_bounds__(TXv* TYv / 2) batch_persistent_kernel(const BInst<real>* __restrict__ insts,
                                                                     const BTables T, int cur, int any_cons,
                                                                     BarrierState* bs, long long limit, int skip_block,
                                                                     int* err) {
  extern __shared__ __align__(16) unsigned char smraw[];
  real* sm = reinterpret_cast<real*>(smraw);
  constexpr bool FUSED = sizeof(real) == 4;
  static_assert(TXv * TYv / 2 == 128, "four warps");
  auto meet = [&]() -> bool {
    if (grid_barrier(bs, gridDim.x, limit, (int)blockIdx.x == skip_block)) return true;
    if (threadIdx.x == 0 && threadIdx.y == 0) atomicExch(err, ERR_BARRIER_TIMEOUT);
    return false;
  };
  if constexpr (FUSED) {
    for (int w = blockIdx.x; w < T.nflow; w += gridDim.x) {
      const BItem it = T.flow[w];
      if (insts[it.inst].P.axisym) do_flow_fused<4, PERSISTENT_R, true>(insts[it.inst], it, cur, sm);
      else do_flow_fused<4, PERSISTENT_R, false>(insts[it.inst], it, cur, sm);
      __syncthreads();
    }
    if (!meet()) return;
    for (int w = blockIdx.x; w < T.nch; w += gridDim.x) {
      const BItem it = T.ch[w];
      do_ch_fused<4, PERSISTENT_R>(insts[it.inst], it, cur, sm);
      __syncthreads();
    }
  }
  for (int sw = FUSED ? (int)SW_UH : 0; sw < SW_N; ++sw) {
    if (FUSED && !any_cons) break;
    if (sw == SW_UH && !any_cons) continue;
    for (int w = blockIdx.x; w < T.ntiles; w += gridDim.x) {
      const BItem it = T.tiles[w];
      do_sweep<real, TXv, TYv>(sw, insts[it.inst], it, cur, sm);
    }
    if (sw < SW_N - 1 && !meet()) return;
  }
}

// one fused pass over its work table, a tile per block
template <int NW, int R, bool AXI>
__global__ void __launch_bounds__(32 * NW, flow_blocks(NW, R)) batch_flow_fused_kernel(const BInst<float>* __restrict__ insts,
                                                                            const BItem* __restrict__ items, int cur) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const BItem it = items[blockIdx.x];
  do_flow_fused<NW, R, AXI>(insts[it.inst], it, cur, reinterpret_cast<float*>(smraw));
}
template <int NW, int R>
__global__ void __launch_bounds__(32 * NW, ch_blocks(NW, R)) batch_ch_fused_kernel(
    const BInst<float>* __restrict__ insts, const BItem* __restrict__ items, int cur) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const BItem it = items[blockIdx.x];
  do_ch_fused<NW, R>(insts[it.inst], it, cur, reinterpret_cast<float*>(smraw));
}

// The diagnostics of instances k0 .. k0 + gridDim.x / nb - 1, nb blocks each: DIAG_NB
// (a constant: with it as an argument the 96 instances of the batch workload take
// 403 us in place of 393), or as many as give every SM eight blocks where the
// instances are few and have 256 cells for each.  The reduction is bound by the
// FP64 operations of the SMs that take part: one 512 x 512 instance of the 96 takes
// 64 us with 32 blocks and 50 so, 4096 x 4096 alone in its batch 4454 and 543 us.
constexpr int DIAG_NB = 32, DIAG_FILL = 152 * 8;
static int diag_blocks(long long count, long long cells) {
  const long long fill = std::min((DIAG_FILL + count - 1) / count, (cells + DIAG_THREADS - 1) / DIAG_THREADS);
  return (int)std::max<long long>(DIAG_NB, fill);
}
template <typename real, bool FEW>
__global__ void __launch_bounds__(DIAG_THREADS) batch_diag_kernel(const BInst<real>* __restrict__ insts, int k0, int few_nb,
                                                                 int cur, double* part) {
  const int nb = FEW ? few_nb : DIAG_NB;
  const int k = k0 + blockIdx.x / nb;
  const BInst<real>& b = insts[k];
  diag_block<real, 2>(b.P, b.Q[cur][0], b.Q[cur][1], b.Q[cur][2], nullptr, b.phi[cur], nullptr, blockIdx.x % nb, nb,
                      part + 4 * (size_t)blockIdx.x);
}
template <typename real>
__global__ void __launch_bounds__(DIAG_THREADS) batch_diag_final_kernel(const BInst<real>* __restrict__ insts, int k0,
                                                                       int nb, const double* part, double* out) {
  const double dx = 1.0 / (double)insts[k0 + blockIdx.x].P.inv_dx;
  diag_sum(part + 4 * (size_t)blockIdx.x * nb, nb, dx * dx, out + 4 * (size_t)blockIdx.x);
}

// one sweep SW over the work table, a tile per block: the sweep is a template
// parameter, so that each sweep's kernel has the registers of its own tile
// code (the flow stages need the most) and the others keep their occupancy
template <typename real, int TXv, int TYv, int SW>
__global__ void __launch_bounds__(TXv* TYv / 2) batch_sweep_kernel(const BInst<real>* __restrict__ insts,
                                                                const BItem* __restrict__ items, int cur) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const BItem it = items[blockIdx.x];
  do_sweep<real, TXv, TYv>(SW, insts[it.inst], it, cur, reinterpret_cast<real*>(smraw));
}

template <typename real, int TXv, int TYv>
constexpr size_t batch_smem() {
  // the largest staged set: the FP64 flow stage; in FP32 (conservative instances) the CH stage
  return sizeof(real) == 8 ? flow64_smem<TXv, TYv>(0) : sizeof(real) * (size_t)C_N * (TXv + 2) * (TYv + 2);
}
template <typename real, int TXv, int TYv>
constexpr size_t persistent_smem() {
  const size_t a = batch_smem<real, TXv, TYv>(), b = flow_fused_smem<float>(4 * PERSISTENT_R);
  return sizeof(real) == 4 && b > a ? b : a;
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

namespace {

struct Shape {
  int tx, ty;
};
const Shape kShapes[] = {{32, 8}, {64, 4}, {16, 16}};
constexpr int kNumShapes = 3;

long long pitch_of(int nx) { return ((long long)nx + 31) / 32 * 32; }

template <typename real>
KParams<real> kp2(const gpe2p_params& p) {
  KParams<real> P{};
  P.n[0] = p.nx;
  P.n[1] = p.ny;
  P.n[2] = 1;
  P.bc[0] = p.bc[0];
  P.bc[1] = p.bc[1];
  P.bc[2] = BC_PERIODIC;
  P.sy = pitch_of(p.nx);
  P.sz = pitch_of(p.nx) * p.ny;
  P.dt = (real)p.dt;
  P.inv_dx = (real)(1.0 / p.dx);
  P.inv_dx2 = (real)(1.0 / (p.dx * p.dx));
  P.inv_2dx = (real)(1.0 / (2.0 * p.dx));
  P.cs2 = (real)(p.cs * p.cs);
  P.rhoL = (real)p.rhoL;
  P.rhoG = (real)p.rhoG;
  P.etaL = (real)p.etaL;
  P.etaG = (real)p.etaG;
  P.rho_m = (real)(0.5 * (p.rhoL + p.rhoG));
  P.rho_d = (real)(0.5 * (p.rhoL - p.rhoG));
  P.eta_m = (real)(0.5 * (p.etaL + p.etaG));
  P.eta_d = (real)(0.5 * (p.etaL - p.etaG));
  P.rho_ref = (real)p.rho_ref;
  P.sigma = (real)p.sigma;
  P.M = (real)p.M;
  P.a4 = (real)(4.0 * (3.0 / (4.0 * p.W)));
  P.kappa = (real)(3.0 * p.W / 8.0);
  for (int c = 0; c < 3; ++c) P.g[c] = (real)p.g[c];
  P.bulk = p.bulk_visc;
  P.pavg = p.p_average;
  P.axisym = p.axisym;
  P.w1 = (real)(1.0 / 9.0);
  P.w2 = (real)(1.0 / 36.0);
  P.w3 = real(0);
  P.lap_c = (real)(6.0 / (p.dx * p.dx));
  P.grad_c = (real)(3.0 / p.dx);
  return P;
}

}  // namespace

struct BatchCtx {
  int n = 0;
  int esize = 4;
  int dev = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  std::vector<gpe2p_params> prm;
  std::vector<long long> ncell;        // cells per instance
  std::vector<size_t> field_off;       // byte offset of each instance's first field
  size_t field_bytes_max = 0;
  char* base = nullptr;
  void* insts_dev = nullptr;           // BInst<real>[n]
  std::vector<char> insts_host;        // the same, on the host
  BItem* items_dev[kNumShapes] = {};   // work tables of the per-stage sweeps per tile shape
  int nitems[kNumShapes] = {};
  // FP32: work tables of the fused passes, [0] short and [1] tall tiles
  BItem* flow_dev[2] = {};
  BItem* ch_dev[2] = {};
  int nflow[2] = {}, nch[2] = {};
  int naxi[2] = {};                    // flow tiles of axisymmetric instances, at the table's end
  int tall = 0;                        // the per-pass form's tiles
  BarrierState* bar = nullptr;
  int* err = nullptr;
  double* d_stage = nullptr;
  double* d_part = nullptr;
  double* d_out = nullptr;
  double* h_out = nullptr;
  int any_cons = 0;
  int cur = 0;
  long long step = 0;
  bool initialized = false;
  // autotuned configuration
  int shape = 0;
  int persistent = 0;
  int grid_persistent[kNumShapes] = {};
  bool persistent_ok = true;
  double tuned_ms = 0.0;
  double cand_ms[kNumShapes][2] = {};
  cudaGraphExec_t gexec[2] = {nullptr, nullptr};
  long long wait_limit = WAIT_LIMIT_DEFAULT;
  int skip_block = -1;
  std::string err_text;
};

// field roles inside an instance block
enum { BF_Q = 0, BF_PHI = 9, BF_MU = 10, BF_PHIS = 11, BF_MUS = 12, BF_UH = 13, BF_US = 15, BF_N = 17 };

template <typename real>
static void fill_insts(BatchCtx* b) {
  b->insts_host.assign(sizeof(BInst<real>) * b->n, 0);
  BInst<real>* I = reinterpret_cast<BInst<real>*>(b->insts_host.data());
  for (int k = 0; k < b->n; ++k) {
    const gpe2p_params& p = b->prm[k];
    const size_t fb = ((size_t)pitch_of(p.nx) * p.ny * b->esize + 255) / 256 * 256;
    char* c = b->base + b->field_off[k];
    auto fld = [&](int r) { return (real*)(c + (size_t)r * fb); };
    I[k].P = kp2<real>(p);
    for (int s = 0; s < 3; ++s)
      for (int f = 0; f < 3; ++f) I[k].Q[s][f] = fld(BF_Q + 3 * s + f);
    const bool fused = sizeof(real) == 4 && !p.ch_advection;
    I[k].phi[0] = fld(BF_PHI);
    I[k].mu[0] = fld(BF_MU);
    I[k].phi[1] = fld(fused ? BF_PHIS : BF_PHI);
    I[k].mu[1] = fld(fused ? BF_MUS : BF_MU);
    I[k].phis = fld(BF_PHIS);
    I[k].mus = fld(BF_MUS);
    // FP64: the frozen terms lie in the fields that the flow stages leave free.  The
    // face sums are written by the last stage, at a face by the thread that has
    // just read that face's frozen force, and the force alone may lie there.  No
    // field is left for the corner viscosities: the stages form them anew.
    static_assert(Z_N == 7, "every frozen term has its place");
    for (int z = 0; z < Z_N; ++z) I[k].z[z] = nullptr;
    if (sizeof(real) == 8) {
      I[k].z[Z_NX] = fld(BF_PHIS);
      I[k].z[Z_NY] = fld(BF_MUS);
      I[k].z[Z_RX] = fld(BF_UH);
      I[k].z[Z_RY] = fld(BF_UH + 1);
      I[k].z[Z_FX] = fld(BF_US);
      I[k].z[Z_FY] = fld(BF_US + 1);
    }
    I[k].uh[0] = fld(BF_UH);
    I[k].uh[1] = fld(BF_UH + 1);
    I[k].us[0] = fld(BF_US);
    I[k].us[1] = fld(BF_US + 1);
    I[k].conservative = p.ch_advection;
  }
}

template <int NW, int R>
static void launch_fused(BatchCtx* b, int t, int cur) {
  const BInst<float>* insts = (const BInst<float>*)b->insts_dev;
  const size_t sm = flow_fused_smem<float>(NW * R);
  const int planar = b->nflow[t] - b->naxi[t];  // the table's first items
  if (planar) batch_flow_fused_kernel<NW, R, false><<<planar, 32 * NW, sm, b->stream>>>(insts, b->flow_dev[t], cur);
  if (b->naxi[t])
    batch_flow_fused_kernel<NW, R, true><<<b->naxi[t], 32 * NW, sm, b->stream>>>(insts, b->flow_dev[t] + planar, cur);
  if (b->nch[t])
    batch_ch_fused_kernel<NW, R><<<b->nch[t], 32 * NW, ch_fused_smem<float>(NW * R), b->stream>>>(insts, b->ch_dev[t],
                                                                                                 cur);
}

template <typename real, int TXv, int TYv>
static cudaError_t enqueue_batch_shape(BatchCtx* b, int si, int persistent, int cur) {
  const BInst<real>* insts = (const BInst<real>*)b->insts_dev;
  cudaError_t e;
  if (persistent) {
    e = cudaMemsetAsync(b->bar, 0, sizeof(BarrierState), b->stream);
    if (e != cudaSuccess) return e;
    BTables T = {b->flow_dev[0], b->ch_dev[0], b->items_dev[si], b->nflow[0], b->nch[0], b->nitems[si]};
    int anyc = b->any_cons;
    long long lim = b->wait_limit;
    int skip = b->skip_block;
    void* args[] = {(void*)&insts,  (void*)&T,   (void*)&cur,  (void*)&anyc,
                    (void*)&b->bar, (void*)&lim, (void*)&skip, (void*)&b->err};
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(b->grid_persistent[si]);
    cfg.blockDim = dim3(TXv * TYv / 2);
    cfg.dynamicSmemBytes = persistent_smem<real, TXv, TYv>();
    cfg.stream = b->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelExC(&cfg, (const void*)batch_persistent_kernel<real, TXv, TYv>, args);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
  }
  const size_t smem = batch_smem<real, TXv, TYv>();
  const unsigned grid = (unsigned)b->nitems[si], nt = TXv * TYv / 2;
  const BItem* items = b->items_dev[si];
  cudaStream_t st = b->stream;
  if constexpr (sizeof(real) == 4) {
    if (b->tall) launch_fused<FUSED_NW_TALL, FUSED_R_TALL>(b, 1, cur);
    else launch_fused<FUSED_NW, FUSED_R>(b, 0, cur);
    if (!b->any_cons) return cudaGetLastError();
  } else {
    batch_sweep_kernel<real, TXv, TYv, SW_FLOW1><<<grid, nt, smem, st>>>(insts, items, cur);
    batch_sweep_kernel<real, TXv, TYv, SW_FLOW2><<<grid, nt, smem, st>>>(insts, items, cur);
    batch_sweep_kernel<real, TXv, TYv, SW_FLOW3><<<grid, nt, smem, st>>>(insts, items, cur);
  }
  if (b->any_cons) batch_sweep_kernel<real, TXv, TYv, SW_UH><<<grid, nt, smem, st>>>(insts, items, cur);
  batch_sweep_kernel<real, TXv, TYv, SW_CH1><<<grid, nt, smem, st>>>(insts, items, cur);
  batch_sweep_kernel<real, TXv, TYv, SW_MU1><<<grid, nt, smem, st>>>(insts, items, cur);
  batch_sweep_kernel<real, TXv, TYv, SW_CH2><<<grid, nt, smem, st>>>(insts, items, cur);
  batch_sweep_kernel<real, TXv, TYv, SW_MU2><<<grid, nt, smem, st>>>(insts, items, cur);
  static_assert(SW_N == 8, "the per-sweep form launches every sweep above, in order");
  return cudaGetLastError();
}

template <typename real>
static cudaError_t enqueue_batch(BatchCtx* b, int si, int persistent, int cur) {
  switch (si) {
    case 0: return enqueue_batch_shape<real, 32, 8>(b, si, persistent, cur);
    case 1: return enqueue_batch_shape<real, 64, 4>(b, si, persistent, cur);
    default: return enqueue_batch_shape<real, 16, 16>(b, si, persistent, cur);
  }
}

static cudaError_t enqueue_any(BatchCtx* b, int si, int persistent, int cur) {
  return b->esize == 4 ? enqueue_batch<float>(b, si, persistent, cur) : enqueue_batch<double>(b, si, persistent, cur);
}

// the tiles of tx x ty cells of the instances that take(k) selects, in order, on the device
// (planar instances first; naxi: the tiles of the axisymmetric ones)
template <typename Take>
static cudaError_t make_table(BatchCtx* b, int tx, int ty, Take take, BItem** dev, int* count, int* naxi = nullptr) {
  std::vector<BItem> items;
  for (int axi = 0; axi < 2; ++axi) {
    const size_t before = items.size();
    for (int k = 0; k < b->n; ++k) {
      if (!take(k) || b->prm[k].axisym != axi) continue;
      for (int j0 = 0; j0 < b->prm[k].ny; j0 += ty)
        for (int i0 = 0; i0 < b->prm[k].nx; i0 += tx) items.push_back({k, i0, j0});
    }
    if (axi && naxi) *naxi = (int)(items.size() - before);
  }
  *count = (int)items.size();
  if (items.empty()) return cudaSuccess;
  cudaError_t e = cudaMalloc((void**)dev, items.size() * sizeof(BItem));
  if (e != cudaSuccess) return e;
  return cudaMemcpy(*dev, items.data(), items.size() * sizeof(BItem), cudaMemcpyHostToDevice);
}

template <typename real, int TXv, int TYv>
static cudaError_t prepare_shape(BatchCtx* b, int si) {
  const size_t smem = batch_smem<real, TXv, TYv>(), psmem = persistent_smem<real, TXv, TYv>();
  cudaError_t e = cudaFuncSetAttribute(batch_persistent_kernel<real, TXv, TYv>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)psmem);
  if (e != cudaSuccess) return e;
  const void* sweeps[] = {(const void*)batch_sweep_kernel<real, TXv, TYv, SW_UH>,
                          (const void*)batch_sweep_kernel<real, TXv, TYv, SW_CH1>,
                          (const void*)batch_sweep_kernel<real, TXv, TYv, SW_MU1>,
                          (const void*)batch_sweep_kernel<real, TXv, TYv, SW_CH2>,
                          (const void*)batch_sweep_kernel<real, TXv, TYv, SW_MU2>};
  for (const void* k : sweeps)
    if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
  if constexpr (sizeof(real) == 8) {
    const void* flows[] = {(const void*)batch_sweep_kernel<real, TXv, TYv, SW_FLOW1>,
                           (const void*)batch_sweep_kernel<real, TXv, TYv, SW_FLOW2>,
                           (const void*)batch_sweep_kernel<real, TXv, TYv, SW_FLOW3>};
    for (const void* k : flows)
      if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
  }
  // FP32: the per-stage sweeps serve the conservative instances only
  e = make_table(b, TXv, TYv, [&](int k) { return sizeof(real) == 8 || b->prm[k].ch_advection; }, &b->items_dev[si],
                 &b->nitems[si]);
  if (e != cudaSuccess) return e;
  // the persistent grid: as many blocks as can be resident at once
  int per_sm = 0, nsm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_persistent_kernel<real, TXv, TYv>, TXv * TYv / 2,
                                                    psmem);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, b->dev);
  if (e != cudaSuccess) return e;
  long long g = (long long)per_sm * nsm, most = b->nitems[si];
  if (b->nflow[0] > most) most = b->nflow[0];
  if (b->nch[0] > most) most = b->nch[0];
  if (g > most) g = most;
  if (g < 1) g = 1;
  b->grid_persistent[si] = (int)g;
  return cudaSuccess;
}

// FP32: the work tables of the fused passes
static cudaError_t prepare_fused(BatchCtx* b) {
  auto any = [](int) { return true; };
  auto advective = [&](int k) { return !b->prm[k].ch_advection; };
  cudaError_t e;
  for (int t = 0; t < 2; ++t) {
    const int rows = t ? FUSED_NW_TALL * FUSED_R_TALL : FUSED_NW * FUSED_R;
    if ((e = make_table(b, FUSED_X, flow_rows(rows), any, &b->flow_dev[t], &b->nflow[t], &b->naxi[t])) != cudaSuccess) return e;
    if ((e = make_table(b, FUSED_X, ch_rows(rows), advective, &b->ch_dev[t], &b->nch[t])) != cudaSuccess) return e;
  }
  b->tall = b->nflow[1] >= 2 * 152;  // as for one problem
  return cudaSuccess;
}

template <typename real>
static cudaError_t prepare_all(BatchCtx* b) {
  cudaError_t e;
  if (sizeof(real) == 4 && (e = prepare_fused(b)) != cudaSuccess) return e;
  if ((e = prepare_shape<real, 32, 8>(b, 0)) != cudaSuccess) return e;
  if ((e = prepare_shape<real, 64, 4>(b, 1)) != cudaSuccess) return e;
  return prepare_shape<real, 16, 16>(b, 2);
}

static cudaError_t build_graphs_batch(BatchCtx* b) {
  for (int c = 0; c < 2; ++c) {
    if (b->gexec[c]) {
      cudaGraphExecDestroy(b->gexec[c]);
      b->gexec[c] = nullptr;
    }
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeRelaxed);
    if (e != cudaSuccess) return e;
    cudaError_t e1 = enqueue_any(b, b->shape, b->persistent, c);
    cudaError_t e2 = cudaStreamEndCapture(b->stream, &g);
    if (e1 != cudaSuccess || e2 != cudaSuccess) {
      if (g) cudaGraphDestroy(g);
      return e1 != cudaSuccess ? e1 : e2;
    }
    e = cudaGraphInstantiate(&b->gexec[c], g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// time every candidate on the (zero) state, keep the fastest, zero the state again
static cudaError_t autotune(BatchCtx* b, size_t state_bytes) {
  cudaEvent_t e0, e1;
  cudaError_t e = cudaEventCreate(&e0);
  if (e != cudaSuccess) return e;
  e = cudaEventCreate(&e1);
  if (e != cudaSuccess) return e;
  double best = 1e30;
  // without conservative instances no FP32 pass depends on the tile shape
  const int nshape = b->esize == 4 && !b->any_cons ? 1 : kNumShapes;
  for (int si = 0; si < nshape; ++si) {
    for (int pers = 0; pers < 2; ++pers) {
      b->cand_ms[si][pers] = -1.0;
      if (pers && !b->persistent_ok) continue;
      b->shape = si;
      b->persistent = pers;
      e = build_graphs_batch(b);
      if (e != cudaSuccess) {
        cudaGetLastError();
        if (pers) b->persistent_ok = false;
        continue;
      }
      const int reps = 4;
      for (int r = 0; r < 1 + reps; ++r) {
        if (r == 1) cudaEventRecord(e0, b->stream);
        if ((e = cudaGraphLaunch(b->gexec[r & 1], b->stream)) != cudaSuccess) break;
      }
      if (e == cudaSuccess) e = cudaEventRecord(e1, b->stream);
      if (e == cudaSuccess) e = cudaEventSynchronize(e1);
      if (e != cudaSuccess) return e;
      int errw = 0;
      cudaMemcpy(&errw, b->err, sizeof(int), cudaMemcpyDeviceToHost);
      if (errw != 0) {  // a barrier that timed out: the persistent form is not usable here
        cudaMemset(b->err, 0, sizeof(int));
        b->persistent_ok = false;
        continue;
      }
      float ms = 0.f;
      cudaEventElapsedTime(&ms, e0, e1);
      b->cand_ms[si][pers] = ms / reps;
      if (ms / reps < best) {
        best = ms / reps;
        b->tuned_ms = best;
      }
    }
  }
  // pick the best recorded candidate
  int bs = 0, bp = 0;
  double bm = 1e30;
  for (int si = 0; si < kNumShapes; ++si)
    for (int pers = 0; pers < 2; ++pers)
      if (b->cand_ms[si][pers] > 0.0 && b->cand_ms[si][pers] < bm) {
        bm = b->cand_ms[si][pers];
        bs = si;
        bp = pers;
      }
  b->shape = bs;
  b->persistent = bp;
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if ((e = cudaMemsetAsync(b->base, 0, state_bytes, b->stream)) != cudaSuccess) return e;
  if ((e = build_graphs_batch(b)) != cudaSuccess) return e;
  return cudaStreamSynchronize(b->stream);
}

int batch_create(const gpe2p_params* p, int n, void* stream, BatchCtx** out, std::string& why) {
  *out = nullptr;
  if (n < 1 || n > 65536) { why = "n must lie in [1, 65536]"; return GPE2P_EINVAL; }
  for (int k = 0; k < n; ++k) {
    if (p[k].dim != 2) { why = "batched instances must be 2D"; return GPE2P_EINVAL; }
    if (p[k].precision != p[0].precision) { why = "all instances must share one precision"; return GPE2P_EINVAL; }
    if (p[k].ch_scheme != 2) { why = "batched instances use TVD-RK2 for the CH step (ch_scheme = 2)"; return GPE2P_EINVAL; }
  }
  BatchCtx* b = new BatchCtx();
  b->n = n;
  b->esize = p[0].precision == 32 ? 4 : 8;
  b->prm.assign(p, p + n);
  cudaError_t e = cudaGetDevice(&b->dev);
  if (e == cudaSuccess && stream) b->stream = (cudaStream_t)stream;
  else if (e == cudaSuccess) {
    e = cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking);
    b->own_stream = true;
  }
  if (e != cudaSuccess) {
    why = std::string("CUDA set-up: ") + cudaGetErrorString(e);
    batch_destroy(b);
    return GPE2P_ECUDA;
  }
  // memory: BF_N fields per instance, then the staging, reduction, barrier
  size_t off = 0;
  long long maxcell = 0;
  for (int k = 0; k < n; ++k) {
    if (p[k].ch_advection) b->any_cons = 1;
    const size_t fb = ((size_t)pitch_of(p[k].nx) * p[k].ny * b->esize + 255) / 256 * 256;
    b->field_off.push_back(off);
    off += fb * BF_N;
    b->ncell.push_back((long long)p[k].nx * p[k].ny);
    if (b->ncell.back() > maxcell) maxcell = b->ncell.back();
  }
  const size_t state_bytes = off;
  const size_t stage_b = ((size_t)maxcell * sizeof(double) + 255) / 256 * 256;
  const size_t part_n = (size_t)n * DIAG_NB + DIAG_FILL + n;  // of any count up to n
  const size_t part_b = (part_n * 4 * sizeof(double) + 255) / 256 * 256;
  const size_t out_b = (((size_t)4 * n + 1) * sizeof(double) + 255) / 256 * 256;
  const size_t total = state_bytes + stage_b + part_b + out_b + 256;
  e = cudaMalloc((void**)&b->base, total);
  if (e != cudaSuccess) {
    why = std::string("device allocation: ") + cudaGetErrorString(e);
    batch_destroy(b);
    return GPE2P_ENOMEM;
  }
  b->d_stage = (double*)(b->base + state_bytes);
  b->d_part = (double*)(b->base + state_bytes + stage_b);
  // the error word and after it the results, so that one copy of their length brings both
  b->err = (int*)(b->base + state_bytes + stage_b + part_b);
  b->d_out = (double*)b->err + 1;
  b->bar = (BarrierState*)(b->base + state_bytes + stage_b + part_b + out_b);
  if (b->esize == 4) fill_insts<float>(b);
  else fill_insts<double>(b);
  e = cudaMalloc(&b->insts_dev, b->insts_host.size());
  if (e == cudaSuccess)
    e = cudaMemcpy(b->insts_dev, b->insts_host.data(), b->insts_host.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(b->base, 0, total);
  if (e == cudaSuccess) e = cudaMallocHost((void**)&b->h_out, (4 * (size_t)n + 1) * sizeof(double));
  if (e == cudaSuccess) e = b->esize == 4 ? prepare_all<float>(b) : prepare_all<double>(b);
  if (e == cudaSuccess) e = autotune(b, state_bytes);
  if (e != cudaSuccess) {
    why = std::string("batch set-up: ") + cudaGetErrorString(e);
    batch_destroy(b);
    return GPE2P_ECUDA;
  }
  *out = b;
  return GPE2P_OK;
}

void batch_destroy(BatchCtx* b) {
  if (!b) return;
  cudaSetDevice(b->dev);
  if (b->stream) cudaStreamSynchronize(b->stream);
  for (int c = 0; c < 2; ++c)
    if (b->gexec[c]) cudaGraphExecDestroy(b->gexec[c]);
  for (int s = 0; s < kNumShapes; ++s)
    if (b->items_dev[s]) cudaFree(b->items_dev[s]);
  for (int t = 0; t < 2; ++t) {
    if (b->flow_dev[t]) cudaFree(b->flow_dev[t]);
    if (b->ch_dev[t]) cudaFree(b->ch_dev[t]);
  }
  if (b->insts_dev) cudaFree(b->insts_dev);
  if (b->base) cudaFree(b->base);
  if (b->h_out) cudaFreeHost(b->h_out);
  if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
  delete b;
}

template <typename real>
static cudaError_t batch_init_impl(BatchCtx* b, int k, const double* const src[4]) {
  const BInst<real>* I = reinterpret_cast<const BInst<real>*>(b->insts_host.data());
  const KParams<real>& P = I[k].P;
  real* dst[4] = {I[k].Q[b->cur][0], I[k].Q[b->cur][1], I[k].Q[b->cur][2], I[k].phi[b->cur]};
  const int comp[4] = {-1, 0, 1, -1};
  cudaError_t e;
  for (int f = 0; f < 4; ++f) {
    e = cudaMemcpyAsync(b->d_stage, src[f], (size_t)b->ncell[k] * sizeof(double), cudaMemcpyHostToDevice,
                        b->stream);
    if (e != cudaSuccess) return e;
    if ((e = launch_from_double<real>(P, b->d_stage, dst[f], comp[f], b->ncell[k], b->stream)) != cudaSuccess)
      return e;
  }
  if ((e = launch_mu<real, 2>(P, I[k].phi[b->cur], I[k].mu[b->cur], 9, 1, b->stream, nullptr, b->err)) != cudaSuccess) return e;
  return cudaStreamSynchronize(b->stream);
}

int batch_init(BatchCtx* b, int k, const double* phi, const double* u, const double* v, const double* p,
               std::string& why) {
  if (k < 0 || k >= b->n) { why = "instance index out of range"; return GPE2P_EINVAL; }
  if (!phi || !u || !v || !p) { why = "a required field is NULL"; return GPE2P_EINVAL; }
  cudaSetDevice(b->dev);
  const double* src[4] = {p, u, v, phi};
  cudaError_t e = b->esize == 4 ? batch_init_impl<float>(b, k, src) : batch_init_impl<double>(b, k, src);
  if (e != cudaSuccess) { why = std::string("init: ") + cudaGetErrorString(e); return GPE2P_ECUDA; }
  b->initialized = true;
  b->step = 0;
  return GPE2P_OK;
}

template <typename real>
static cudaError_t batch_read_impl(BatchCtx* b, int k, double* const dst[5]) {
  const BInst<real>* I = reinterpret_cast<const BInst<real>*>(b->insts_host.data());
  const KParams<real>& P = I[k].P;
  const int c = b->cur;
  const real* src[5] = {I[k].Q[c][0], I[k].Q[c][1], I[k].Q[c][2], I[k].phi[c], I[k].mu[c]};
  cudaError_t e;
  for (int f = 0; f < 5; ++f) {
    if (!dst[f]) continue;
    if ((e = launch_to_double<real>(P, src[f], b->d_stage, b->ncell[k], b->stream)) != cudaSuccess) return e;
    e = cudaMemcpyAsync(dst[f], b->d_stage, (size_t)b->ncell[k] * sizeof(double), cudaMemcpyDeviceToHost,
                        b->stream);
    if (e != cudaSuccess) return e;
  }
  return cudaStreamSynchronize(b->stream);
}

int batch_read(BatchCtx* b, int k, double* phi, double* u, double* v, double* p, double* mu, std::string& why) {
  if (k < 0 || k >= b->n) { why = "instance index out of range"; return GPE2P_EINVAL; }
  cudaSetDevice(b->dev);
  double* dst[5] = {p, u, v, phi, mu};
  cudaError_t e = b->esize == 4 ? batch_read_impl<float>(b, k, dst) : batch_read_impl<double>(b, k, dst);
  if (e != cudaSuccess) { why = std::string("read: ") + cudaGetErrorString(e); return GPE2P_ECUDA; }
  return GPE2P_OK;
}

int batch_step(BatchCtx* b, std::string& why) {
  if (!b->initialized) { why = "step before any instance was initialised"; return GPE2P_ESTATE; }
  cudaSetDevice(b->dev);
  cudaError_t e = cudaGraphLaunch(b->gexec[b->cur], b->stream);
  if (e != cudaSuccess) { why = std::string("graph launch: ") + cudaGetErrorString(e); return GPE2P_ECUDA; }
  b->cur = 1 - b->cur;
  b->step += 1;
  return GPE2P_OK;
}

template <typename real>
static cudaError_t batch_diag_impl(BatchCtx* b, int k0, int count, int nb) {
  const BInst<real>* insts = (const BInst<real>*)b->insts_dev;
  auto kernel = nb == DIAG_NB ? batch_diag_kernel<real, false> : batch_diag_kernel<real, true>;
  kernel<<<(unsigned)count * nb, DIAG_THREADS, 0, b->stream>>>(insts, k0, nb, b->cur, b->d_part);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  batch_diag_final_kernel<real><<<(unsigned)count, DIAG_THREADS, 0, b->stream>>>(insts, k0, nb, b->d_part, b->d_out);
  return cudaGetLastError();
}

// All instances asked for are reduced by one launch, read back by one copy.
// (An instance at a time, with a wait for each, took 1.9 ms of the 10.7 ms of
// eight steps of 96 instances.)
int batch_diag(BatchCtx* b, int k, gpe2p_diag* d, std::string& why) {
  cudaSetDevice(b->dev);
  gpe2p_diag acc{};
  const int k0 = k < 0 ? 0 : k, count = k < 0 ? b->n : 1;
  if (k >= b->n) { why = "instance index out of range"; return GPE2P_EINVAL; }
  const int nb = diag_blocks(count, k < 0 ? *std::max_element(b->ncell.begin(), b->ncell.end()) : b->ncell[k]);
  cudaError_t e = b->esize == 4 ? batch_diag_impl<float>(b, k0, count, nb) : batch_diag_impl<double>(b, k0, count, nb);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(b->h_out, b->err, (1 + (size_t)4 * count) * sizeof(double), cudaMemcpyDeviceToHost, b->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  if (e != cudaSuccess) { why = std::string("diagnostics: ") + cudaGetErrorString(e); return GPE2P_ECUDA; }
  int errw = 0;
  std::memcpy(&errw, b->h_out, sizeof(int));
  if (errw != 0) {
    why = "a grid barrier or device-side copy did not complete within its bounded wait";
    return GPE2P_ETIMEOUT;
  }
  for (int q = 0; q < count; ++q) {
    const double* o = b->h_out + 1 + 4 * (size_t)q;
    acc.int_phi += o[0];
    acc.kinetic += o[1];
    acc.umax = o[2] > acc.umax ? o[2] : acc.umax;
    if (o[3] != 0.0 || !std::isfinite(o[0]) || !std::isfinite(o[1])) acc.nan_flag = 1;
  }
  acc.step = b->step;
  acc.t = (double)b->step * b->prm[k0].dt;
  *d = acc;
  return GPE2P_OK;
}

int batch_config(BatchCtx* b, int* tile_x, int* tile_y, int* persistent, double* ms) {
  // without conservative instances an FP32 step is the fused passes alone: the flow pass's tile
  const bool fused = b->esize == 4 && !b->any_cons;
  const int rows = b->tall && !b->persistent ? FUSED_NW_TALL * FUSED_R_TALL : FUSED_NW * FUSED_R;
  if (tile_x) *tile_x = fused ? FUSED_X : kShapes[b->shape].tx;
  if (tile_y) *tile_y = fused ? flow_rows(rows) : kShapes[b->shape].ty;
  if (persistent) *persistent = b->persistent;
  if (ms) *ms = b->tuned_ms;
  return GPE2P_OK;
}

int batch_fault(BatchCtx* b, int what, long long value, std::string& why) {
  cudaSetDevice(b->dev);
  if (what == GPE2P_FAULT_SKIP_BARRIER) {
    b->skip_block = (int)value;
  } else if (what == GPE2P_FAULT_WAIT_LIMIT) {
    if (value <= 0) { why = "wait limit must be positive"; return GPE2P_EINVAL; }
    b->wait_limit = value;
  } else if (what == GPE2P_FAULT_FORCE_PERSISTENT) {
    if (!b->persistent_ok) { why = "the persistent form is not available on this device"; return GPE2P_EINVAL; }
    b->persistent = value ? 1 : 0;
  } else if (what == GPE2P_FAULT_CLEAR) {
    b->skip_block = -1;
    b->wait_limit = WAIT_LIMIT_DEFAULT;
    if (cudaMemsetAsync(b->err, 0, sizeof(int), b->stream) != cudaSuccess ||
        cudaStreamSynchronize(b->stream) != cudaSuccess) {
      why = "clearing the error word failed";
      return GPE2P_ECUDA;
    }
  } else {
    why = "unknown fault-injection switch";
    return GPE2P_EINVAL;
  }
  cudaError_t e = build_graphs_batch(b);
  if (e != cudaSuccess) { why = std::string("graph rebuild: ") + cudaGetErrorString(e); return GPE2P_ECUDA; }
  return GPE2P_OK;
}

template <typename real>
int batch_instance(BatchCtx* b, int k, KParams<real>* P, real* f[5], int* iso) {
  if (k < 0 || k >= b->n || (int)sizeof(real) != b->esize) return GPE2P_EINVAL;
  const BInst<real>* I = reinterpret_cast<const BInst<real>*>(b->insts_host.data());
  const int c = b->cur;
  *P = I[k].P;
  f[0] = I[k].phi[c];
  f[1] = I[k].Q[c][1];
  f[2] = I[k].Q[c][2];
  f[3] = I[k].Q[c][0];
  f[4] = I[k].mu[c];
  *iso = b->prm[k].iso;
  return GPE2P_OK;
}
template int batch_instance<float>(BatchCtx*, int, KParams<float>*, float* [5], int*);
template int batch_instance<double>(BatchCtx*, int, KParams<double>*, double* [5], int*);

void batch_mark_initialized(BatchCtx* b) { b->initialized = true; }
int* batch_err(BatchCtx* b) { return b->err; }
int batch_dev(const BatchCtx* b) { return b->dev; }
int batch_esize(const BatchCtx* b) { return b->esize; }

cudaStream_t batch_stream(const BatchCtx* b) { return b->stream; }

long long batch_cells(const BatchCtx* b) {
  long long s = 0;
  for (long long c : b->ncell) s += c;
  return s;
}

int batch_size(const BatchCtx* b) { return b->n; }
int batch_dim(const BatchCtx*) { return 2; }

}  // namespace gpe2p
