// fx64 instantiations of the 2D step kernels: FP64 contexts, and the refined
// modes' certifying residual.
#define HC_FX_UNIT
#include "hc_kernels.cuh"

namespace hc {

template void row_r2c<fx64>(const Geo<fx64>&, const fx64*, const fx64*, cx<fx64>*,
                              cx<fx64>*, cudaStream_t);
template void row_c2r<fx64>(const Geo<fx64>&, const cx<fx64>*, const cx<fx64>*, fx64*,
                              fx64*, SolveState*, int, cudaStream_t);
template void row_apply<fx64, fx64>(const Geo<fx64>&, const cx<fx64>*, const cx<fx64>*,
                                        const fx64*, const fx64*, const fx64*, cx<fx64>*,
                                        cx<fx64>*, SolveState*, cudaStream_t);
template void row_apply<fx64, float>(const Geo<fx64>&, const cx<fx64>*, const cx<fx64>*,
                                        const float*, const float*, const float*, cx<fx64>*,
                                        cx<fx64>*, SolveState*, cudaStream_t);
template void row_split<fx64>(const Geo<fx64>&, const cx<fx64>*, const cx<fx64>*, const fx64*,
                               const fx64*, const fx64*, cx<fx64>*, cx<fx64>*, SplitCoef, SolveState*,
                               cudaStream_t);
template void col_fwd<fx64>(const Geo<fx64>&, const cx<fx64>*, const cx<fx64>*, cx<fx64>*,
                              cx<fx64>*, int, int, SolveState*, cudaStream_t);
template void col_inv<fx64>(const Geo<fx64>&, const cx<fx64>*, cx<fx64>*, fx64,
                              cudaStream_t);
template void col_grad<fx64, fx64>(const Geo<fx64>&, int, cx<fx64>*, const cx<fx64>*,
                                       cx<fx64>*, const cx<float>*, cx<fx64>*, cx<fx64>*,
                                       SolveState*, int, cudaStream_t);
template void col_div<fx64>(const Geo<fx64>&, int, const cx<fx64>*, const cx<fx64>*,
                              const cx<fx64>*, const cx<fx64>*, cx<fx64>*, cx<float>*,
                              cx<float>*, SolveState*, cudaStream_t);
template void col_heat<fx64>(const Geo<fx64>&, cx<fx64>*, cx<fx64>*, SolveState*, cudaStream_t);
template void col_gradnorm<fx64>(const Geo<fx64>&, const cx<fx64>*, const cx<fx64>*, SolveState*, int,
                                 cudaStream_t);
template void row_adj_point<fx64>(const Geo<fx64>&, cx<fx64>*, cx<fx64>*, const cx<fx64>*, const cx<fx64>*,
                                const fx64*, const fx64*, fx64*, fx64*, SplitCoef, AdjState*, cudaStream_t);
template void row_adj_press<fx64>(const Geo<fx64>&, const cx<fx64>*, const cx<fx64>*, const cx<fx64>*,
                                const cx<fx64>*, const fx64*, const fx64*, const fx64*, const fx64*, fx64*,
                                fx64*, double*, cudaStream_t);
template void col_lap_dot<fx64>(const Geo<fx64>&, const cx<fx64>*, const cx<fx64>*, double, AdjState*,
                              cudaStream_t);

// FP64 residual S - A p of a certification (lagged certification): the
// pressure p and the m it was solved with are the caller's; the state sc
// skips it when nothing awaits certification (sc->done) and receives
// ||S - A p||^2 in sc->cert_r2.  Non-persistent passes, nothing else written.
void cert_resid(const Geo<double>& gd, const cx<double>* p, const float* mx, const float* my,
                const float* r, const cx<double>* b, cx<double>* G, SolveState* sc, cudaStream_t s) {
  const Geo<fx64> g = as_fx(gd);
  const int nb = g.H >> g.ltc, nt = col_threads(g);
  cx<fx64>* Gx = fxp(G);
  cx<fx64>* Gy = Gx + (size_t)g.ny * g.H;
  k_col_grad<fx64, fx64, CG_PLAIN><<<nb, nt, col_smem(g, 1), s>>>(
      g, fxp(const_cast<cx<double>*>(p)), nullptr, nullptr, nullptr, Gx, Gy, sc, 1);
  const size_t sm = row_smem(g) + (size_t)3 * g.rpc * g.nx * sizeof(float);
  k_row_apply<fx64, float, false, 1><<<g.ny >> g.lrpc, row_threads(g), sm, s>>>(g, Gx, Gy, mx, my, r,
                                                                               Gx, Gy, sc);
  k_col_div<fx64, CD_CERT><<<nb, nt, col_smem(g, 2), s>>>(g, Gx, Gy, nullptr, fxp(b), nullptr, nullptr,
                                                          nullptr, sc);
}

// A refined context launches only the residuals and p's transforms.
void set_smem_limits_fx(int refined) {
  if (!refined) {
    set_smem_limits_t<fx64>();
    set_smem_limits_grad<fx64, fx64>();
    return;
  }
  allow_smem(k_row_r2c<fx64>);
  allow_smem(k_col_fwd<fx64, 1>);
  allow_smem(k_col_inv<fx64>);
  allow_smem(k_row_c2r<fx64>);
  set_smem_limits_grad<fx64, fx64>();
  allow_smem(k_row_apply<fx64, float, false, 1>);
  allow_smem(k_col_div<fx64, CD_CERT>);
  allow_smem(k_col_div<fx64, CD_DECIDE>);
}

}  // namespace hc
