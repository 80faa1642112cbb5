// ring3d.cuh -- the z-marching plane pipeline shared by the 3D stencil kernels.
//
// A block owns a TX x TY column of cells and a range of z-planes.  Each plane
// of every input field, with a one-cell halo in x and y, arrives in shared
// memory by one TMA copy per field (a box of BX x SY elements starting at
// x = i0 - A so that the start is 16-byte aligned); RING slots let several
// planes be in flight while the block computes plane k from planes k-1, k and
// k+1.  Cells of the staged region that lie outside the domain (the halo of
// boundary tiles, and the ghost planes k = -1 and k = nz, which are not copied)
// are then overwritten by the threads with the boundary rules of
// gpe2p_dev.cuh.
#pragma once

#include "gpe2p_dev.cuh"
#include "tma.cuh"

namespace gpe2p {

// kinds of staged fields, for the ghost rules
enum { K_CEN = 0, K_FACE0 = 1, K_FACE1 = 2, K_FACE2 = 3, K_CVEC0 = 4, K_CVEC1 = 5, K_CVEC2 = 6 };

template <typename real>
__device__ __forceinline__ real ld_kind(int kind, const real* __restrict__ f, const KParams<real>& P, int i,
                                        int j, int k) {
  switch (kind) {
    case K_FACE0: return ld_face<0>(f, P, i, j, k);
    case K_FACE1: return ld_face<1>(f, P, i, j, k);
    case K_FACE2: return ld_face<2>(f, P, i, j, k);
    case K_CVEC0: return ld_cvec<0>(f, P, i, j, k);
    case K_CVEC1: return ld_cvec<1>(f, P, i, j, k);
    case K_CVEC2: return ld_cvec<2>(f, P, i, j, k);
    default: return ld_cen(f, P, i, j, k);
  }
}

// SYv: rows of a staged plane (the tile's rows plus the two halo rows)
template <typename real, int SYv = SY>
struct RingGeom {
  static constexpr int A = 16 / (int)sizeof(real);     // alignment of the box start, elements
  static constexpr int BX = TX + 2 * A;                // box width
  static constexpr int ROWS = SYv;
  static constexpr int PE = ((BX * SYv * (int)sizeof(real) + 127) / 128) * 128 / (int)sizeof(real);
  static constexpr uint32_t BOX_BYTES = BX * SYv * sizeof(real);
  // element (lx, ly) of the staged region (lx, ly in [0, SX) x [0, SYv)): global
  // cell (i0 - 1 + lx, j0 - 1 + ly)
  __device__ __forceinline__ static int at(int lx, int ly) { return ly * BX + lx + A - 1; }
  __device__ __forceinline__ static int start(int i0) { return i0 - A; }
};

// The flow stage's staged region: 32 columns, the block's 30 and one on each side,
// one per lane.  The box starts on the 16-byte boundary at or below the first;
// element (lx, ly) lies at at(lx, ly) + shift(i0).
template <typename real, int SYv>
struct FlowGeom {
  static constexpr int A = 16 / (int)sizeof(real);
  static constexpr int BX = 32 + A;
  static constexpr int PE = ((BX * SYv * (int)sizeof(real) + 127) / 128) * 128 / (int)sizeof(real);
  static constexpr uint32_t BOX_BYTES = BX * SYv * sizeof(real);
  __device__ __forceinline__ static int at(int lx, int ly) { return ly * BX + lx; }
  __device__ __forceinline__ static int start(int i0) { return (i0 - 1) & ~(A - 1); }
  __device__ __forceinline__ static int shift(int i0) { return (i0 - 1) & (A - 1); }
};

template <int NMAP>
struct Maps {
  CUtensorMap m[NMAP];
};

// The pipeline state of one block.  NRAW fields are staged per plane; lane 0 of
// each of the first NISS warps issues its share of a plane's copies.  (A single
// issuing thread spends about a hundred instructions a plane on six copies,
// which the block's other warps wait out at the next barrier: shared, a step of
// 256 x 256 x 512 takes 1.2 % less.)
template <typename real, int NRAW, int RING, int SYv = SY, typename Geom = RingGeom<real, SYv>, int NISS = 1>
struct Ring {
  static_assert(RING >= 4 && RING <= 8, "slots of a ring (its barriers take 64 bytes)");
  using G = Geom;
  uint64_t* bar;  // RING barriers
  real* raw;      // RING x NRAW x PE
  int first, last;  // planes kbeg-1 .. kend (inclusive)
  int i0, j0;
  int x0;           // first staged column (16-byte aligned)
  int issued;       // last plane issued
  bool lose_first;  // test switch: report the wait for the first plane as timed out
  __device__ __forceinline__ int slot(int kk) const { return (int)((unsigned)(kk - first) % RING); }
  __device__ __forceinline__ uint32_t parity(int kk) const { return ((unsigned)(kk - first) / RING) & 1u; }
  __device__ __forceinline__ real* plane(int kk, int f) const { return raw + ((size_t)slot(kk) * NRAW + f) * G::PE; }

  // an issuing thread: start its copies of plane kk (or, for a ghost plane, just arrive)
  __device__ __forceinline__ void issue(const KParams<real>& P, const CUtensorMap* maps, int kk) {
    uint64_t* b = &bar[slot(kk)];
    const int me = threadIdx.y;
    if (kk >= 0 && kk < P.n[2] && (NISS == 1 || me < NRAW)) {
      const int mine = NISS == 1 ? NRAW : (NRAW - 1 - me) / NISS + 1;
      mbar_arrive_expect_tx(b, mine * G::BOX_BYTES);
#pragma unroll
      for (int f = 0; f < NRAW; f += NISS)
        if (NISS == 1 || f + me < NRAW) tma_load_3d(plane(kk, f + me), &maps[f + me], x0, j0 - 1, kk, b);
    } else {
      mbar_arrive(b);
    }
    issued = kk;
  }
  __device__ __forceinline__ bool issuer() const { return threadIdx.x == 0 && threadIdx.y < NISS; }

  // lose: the test switch of the timeout path (the wait for the first plane
  // still completes, so no copy is left in flight, and then reports a timeout)
  __device__ __forceinline__ void start(const KParams<real>& P, const CUtensorMap* maps, int kbeg, int kend,
                                        int i0_, int j0_, bool lose = false) {
    lose_first = lose;
    first = kbeg - 1;
    last = kend;
    i0 = i0_;
    j0 = j0_;
    x0 = G::start(i0_);
    issued = first - 1;
    if (threadIdx.x == 0 && threadIdx.y == 0) {
      for (int s = 0; s < RING; ++s) mbar_init(&bar[s], NISS);
      fence_mbar_init();
    }
    __syncthreads();
    if (issuer()) {
      const int upto = min(last, first + RING - 1);
      for (int kk = first; kk <= upto; ++kk) issue(P, maps, kk);
    }
    issued = min(last, first + RING - 1);
  }

  // all threads: wait for plane kk; false (block-uniform) on timeout
  __device__ __forceinline__ bool wait(int kk) {
    const bool ok = mbar_wait_bounded(&bar[slot(kk)], parity(kk), WAIT_CYCLES) && !(lose_first && kk == first);
    return !__syncthreads_or(!ok);
  }

  // all threads, after the wait for plane kk (every thread is then done with
  // plane kk - 3): start plane kk - 3 + RING in the freed slot
  __device__ __forceinline__ void refill(const KParams<real>& P, const CUtensorMap* maps, int kk) {
    const int nk = kk - 3 + RING;
    if (issuer() && nk <= last && nk > issued) issue(P, maps, nk);
  }

  // after a timeout: record it, let this block's copies in flight land, return
  __device__ __forceinline__ void fail(int* err, int from) {
    if (threadIdx.x == 0 && threadIdx.y == 0) {
      atomicExch(err, ERR_TMA_TIMEOUT);
      for (int kk = from; kk <= issued; ++kk) mbar_wait_bounded(&bar[slot(kk)], parity(kk), WAIT_CYCLES / 2);
    }
  }
};

// The ghost cells of a staged plane inside the domain: the columns at -1 and nx and
// the rows at -1 and ny of a tile that reaches them (staged cells further out are
// read by no cell of the domain).  Candidate q < ghost_count<SYv>() of the tile
// at (i0, j0): its staged position, or false if the tile does not have it.
template <int SYv, int SXv = SX>
constexpr int ghost_count() { return 2 * SYv + 2 * SXv; }
template <int SYv, int SXv = SX, typename real>
__device__ __forceinline__ bool ghost_cell(const KParams<real>& P, int i0, int j0, int q, int& lx, int& ly) {
  if (q < 2 * SYv) {
    ly = q >> 1;
    lx = (q & 1) ? P.n[0] - i0 + 1 : 0;
    return ((q & 1) ? lx < SXv : i0 == 0) && j0 - 1 + ly <= P.n[1];
  }
  q -= 2 * SYv;
  lx = q >> 1;
  ly = (q & 1) ? P.n[1] - j0 + 1 : 0;
  return ((q & 1) ? ly < SYv : j0 == 0) && i0 - 1 + lx <= P.n[0];
}

// The value of a ghost cell (gi, gj) of plane kk.  Across a wall it mirrors a cell
// that the same plane holds in shared memory (pl: the staged field): a copy there
// costs a tile at the boundary nothing, while the global loads of ld_kind cost
// it their latency in every plane.  Across a periodic side the other end
// of the domain is read.
template <typename G, typename real>
__device__ __forceinline__ real ghost_value(int kind, const real* pl, const real* __restrict__ f,
                                            const KParams<real>& P, int i0, int j0, int gi, int gj, int kk) {
  // out of the domain across a wall, and across a periodic side
  const bool ax = gi < 0 || gi >= P.n[0], ay = gj < 0 || gj >= P.n[1];
  const bool px = ax && P.bc[0] == BC_PERIODIC, py = ay && P.bc[1] == BC_PERIODIC;
  const bool ox = ax && !px, oy = ay && !py;
  int x = px ? wrap1(gi, P.n[0]) : clampi(gi, 0, P.n[0] - 1), y = py ? wrap1(gj, P.n[1]) : clampi(gj, 0, P.n[1] - 1);
  bool neg = false;
  if (kind == K_FACE0 || kind == K_FACE1) {
    // odd about a wall face along the component's axis, zero on it
    const bool along_x = kind == K_FACE0;
    if (along_x ? ox : oy) {
      const int g = along_x ? gi : gj, n = P.n[along_x ? 0 : 1];
      if (g >= n || n < 2) return real(0);
      if (along_x) x = 1;
      else y = 1;
      neg = true;
    }
    if ((along_x ? oy : ox) && P.bc[along_x ? 1 : 0] == BC_NOSLIP) neg = !neg;
  } else if (kind == K_FACE2) {
    if (ox && P.bc[0] == BC_NOSLIP) neg = !neg;
    if (oy && P.bc[1] == BC_NOSLIP) neg = !neg;
  } else if (kind == K_CVEC0) {
    neg = ox;
  } else if (kind == K_CVEC1) {
    neg = oy;
  }
  const real v = px || py ? f[lin(P, x, y, kk)] : pl[G::at(x - i0 + 1, y - j0 + 1)];
  return neg ? -v : v;
}

// The plane beyond a z wall, field by field: dst from src, the plane next to the
// wall with its own ghosts in place.  (The w face outside is read by no
// updated face; on the high wall, w = 0.)
template <int KIND, typename real>
__device__ __forceinline__ real zwall_value(const KParams<real>& P, real v) {
  if (KIND == K_FACE2) return real(0);
  if (KIND == K_CVEC2) return -v;
  if (KIND == K_FACE0 || KIND == K_FACE1) return P.bc[2] == BC_NOSLIP ? -v : v;
  return v;
}

// shared-memory bytes of a kernel with NRAW staged and NDER derived fields
// (derived fields keep four planes, indexed by the plane number mod 4):
// 128 bytes of slack to align the base, 128 for the barriers, then the planes
template <typename real, int NRAW, int NDER, int RING, int SYv = SY>
constexpr size_t ring_smem_bytes() {
  return 256 + sizeof(real) * (size_t)RingGeom<real, SYv>::PE * (RING * NRAW + 4 * NDER);
}

// the 128-byte aligned start of the dynamic shared memory
__device__ __forceinline__ unsigned char* smem_base128(unsigned char* p) {
  const uint32_t off = smem_u32(p);
  return p + ((128u - (off & 127u)) & 127u);
}

}  // namespace gpe2p
