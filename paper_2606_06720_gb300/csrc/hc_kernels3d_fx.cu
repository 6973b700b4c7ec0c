// fx64 instantiations of the 3D step kernels.
#define HC_FX_UNIT
#include "hc_kernels3d.cuh"

namespace hc {

template void z_grad<fx64, fx64>(const Geo<fx64>&, int, cx<fx64>*, const cx<fx64>*,
                                     cx<fx64>*, const cx<float>*, Tri<cx<fx64>*>, SolveState*,
                                     int, cudaStream_t);
template void axis_fft<fx64>(const Geo<fx64>&, int, int, int, Tri<cx<fx64>*>,
                               Tri<cx<fx64>*>, fx64, cudaStream_t);
template void z_fwd_project<fx64>(const Geo<fx64>&, const cx<fx64>*, cx<fx64>*, SolveState*,
                                    cudaStream_t);
template void z_div<fx64>(const Geo<fx64>&, int, Tri<cx<fx64>*>, const cx<fx64>*,
                            const cx<fx64>*, cx<fx64>*, cx<float>*, cx<float>*, SolveState*,
                            cudaStream_t);
template void row_apply3<fx64, fx64>(const Geo<fx64>&, Tri<cx<fx64>*>, Tri<const fx64*>,
                                         const fx64*, Tri<cx<fx64>*>, SolveState*,
                                         cudaStream_t);
template void row_apply3<fx64, float>(const Geo<fx64>&, Tri<cx<fx64>*>, Tri<const float*>,
                                        const float*, Tri<cx<fx64>*>, SolveState*,
                                        cudaStream_t);
template void row_split3<fx64>(const Geo<fx64>&, Tri<cx<fx64>*>, Tri<const fx64*>, const fx64*,
                                Tri<fx64*>, SplitCoef, SolveState*, cudaStream_t);
template void heat_axis<fx64>(const Geo<fx64>&, int, Tri<fx64*>, Tri<fx64*>, SolveState*,
                               cudaStream_t);
template void z_gradnorm<fx64>(const Geo<fx64>&, Tri<cx<fx64>*>, SolveState*, int, cudaStream_t);

void set_smem_limits_3d_fx(int refined) {
  if (!refined) {
    set_smem_limits_3d_t<fx64>();
    set_smem_limits_row3<fx64, fx64>();
    set_smem_limits_zgrad<fx64, fx64>();
    return;
  }
  allow_smem(k3_axis_fft<fx64, -1, 1>);
  allow_smem(k3_axis_fft<fx64, +1, 1>);
  allow_smem(k3_axis_fft<fx64, -1, 3>);
  allow_smem(k3_axis_fft<fx64, +1, 3>);
  allow_smem(k3_zfwd_project<fx64>);
  allow_smem(k3_zdiv<fx64, CD_DECIDE>);
  allow_smem(k3_row_apply<fx64, float, false>);
  set_smem_limits_zgrad<fx64, fx64>();
}

}  // namespace hc
