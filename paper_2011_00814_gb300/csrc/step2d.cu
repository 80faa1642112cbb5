// step2d.cu -- the single-problem launches of the fused 2D FP32 step and of its
// rates (step2d.cuh).
#include "step2d.cuh"

namespace gpe2p {

template <int NW, int R, bool AXI, bool RATES>
__global__ void __launch_bounds__(32 * NW, flow_blocks(NW, R))
    flow2d_fused_kernel(const __grid_constant__ KParams<float> P, const FlowStepArgs<float> A) {
  extern __shared__ __align__(16) unsigned char smraw[];
  after_previous_kernel();
  flow2d_fused_tile<float, NW, R, AXI, RATES>(P, A, blockIdx.x * FUSED_X, blockIdx.y * flow_rows(NW * R),
                                              reinterpret_cast<float*>(smraw));
}

template <int NW, int R, bool RATES>
__global__ void __launch_bounds__(32 * NW, ch_blocks(NW, R))
    ch2d_fused_kernel(const __grid_constant__ KParams<float> P, const CHStepArgs<float> A) {
  extern __shared__ __align__(16) unsigned char smraw[];
  after_previous_kernel();
  ch2d_fused_tile<float, NW, R, RATES>(P, A, blockIdx.x * FUSED_X, blockIdx.y * ch_rows(NW * R),
                                       reinterpret_cast<float*>(smraw));
}

template <int NW, int R, bool RATES>
static cudaError_t flow_go(const KParams<float>& P, const FlowStepArgs<float>& A, cudaStream_t s) {
  constexpr size_t sm = flow_fused_smem<float>(NW * R);
  static_assert(sm <= 48 * 1024, "no opt-in shared memory");
  constexpr int TYf = flow_rows(NW * R);
  const dim3 grd((P.n[0] + FUSED_X - 1) / FUSED_X, (P.n[1] + TYf - 1) / TYf);
  return launch_step(P.axisym ? flow2d_fused_kernel<NW, R, true, RATES> : flow2d_fused_kernel<NW, R, false, RATES>, true,
                     grd, 32 * NW, sm, s, P, A);
}

template <int NW, int R, bool RATES>
static cudaError_t ch_go(const KParams<float>& P, const CHStepArgs<float>& A, cudaStream_t s) {
  constexpr size_t sm = ch_fused_smem<float>(NW * R);
  static_assert(sm <= 48 * 1024, "no opt-in shared memory");
  constexpr int TYc = ch_rows(NW * R);
  const dim3 grd((P.n[0] + FUSED_X - 1) / FUSED_X, (P.n[1] + TYc - 1) / TYc);
  return launch_step(ch2d_fused_kernel<NW, R, RATES>, true, grd, 32 * NW, sm, s, P, A);
}

cudaError_t launch_flow_fused(const KParams<float>& P, const FlowStepArgs<float>& A, bool rates, cudaStream_t s) {
  if (fused_tall(P.n[0], P.n[1]))
    return rates ? flow_go<FUSED_NW_TALL, FUSED_R_TALL, true>(P, A, s) : flow_go<FUSED_NW_TALL, FUSED_R_TALL, false>(P, A, s);
  return rates ? flow_go<FUSED_NW, FUSED_R, true>(P, A, s) : flow_go<FUSED_NW, FUSED_R, false>(P, A, s);
}

cudaError_t launch_ch_fused(const KParams<float>& P, const CHStepArgs<float>& A, bool rates, cudaStream_t s) {
  if (fused_tall(P.n[0], P.n[1]))
    return rates ? ch_go<FUSED_NW_TALL, FUSED_R_TALL, true>(P, A, s) : ch_go<FUSED_NW_TALL, FUSED_R_TALL, false>(P, A, s);
  return rates ? ch_go<FUSED_NW, FUSED_R, true>(P, A, s) : ch_go<FUSED_NW, FUSED_R, false>(P, A, s);
}

}  // namespace gpe2p
