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

__global__ void __launch_bounds__(256) k_pinv_table(Geo<double> g, const SolveState* st) {
  const Pc<double> pc = pc_of<double>(st);
  const size_t total = (size_t)g.ny * g.H;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (size_t)gridDim.x * blockDim.x)
    g.pinv[i] = pinv_sym(g, (int)(i & (size_t)(g.H - 1)), (int)(i >> g.lH), pc);
}
void pinv_table(const Geo<double>& g, const SolveState* st, cudaStream_t s) {
  k_pinv_table<<<upd_blocks((size_t)g.ny * g.H), 256, 0, s>>>(g, st);
}

__global__ void __launch_bounds__(cta_bound<fx64>(512)) k_col_div_upd(
    Geo<fx64> g, const cx<fx64>* __restrict__ Qx, const cx<fx64>* __restrict__ Qy,
    const cx<double>* __restrict__ d, cx<double>* __restrict__ x, cx<double>* __restrict__ r,
    SolveState* st) {
  if (st->done) {
    if (st->graph_mode && blockIdx.x == 0 && threadIdx.x == 0)
      cudaGraphSetConditional(st->h_cur, 0u);
    return;
  }
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<fx64>* sm = reinterpret_cast<cx<fx64>*>(smem_raw);
  const ColIdx c = col_idx(g);
  const int H = g.H, se = slab_elems(g);
  cx<fx64>* const sl1[1] = {sm + c.b};
  cx<fx64>* const pk = sm + se + c.b;
  const double rho = st->rho, n = (double)g.nx * (double)g.ny;
  const double share = dots_share(g.dots, g.ny >> g.lrpc);
#pragma unroll 1
  for (int q = 0; q < 2; ++q) {
    const cx<fx64>* const Q = (q == 0 ? Qx : Qy) + c.kx;
    cx<fx64> v[1][8];
#pragma unroll
    for (int s = 0; s < 8; ++s) v[0][s] = Q[(unsigned)(c.j + s * c.NY8) * (unsigned)H];
    fft_canon<-1, 1>(v, sl1, 1 << g.ltc, c.j, g.lny, g.twy);
    const fx64 ax = g.kxd[c.kx];
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const int ky = c.j + s * c.NY8;
      cx<fx64>& t = pk[padk(ky) << g.ltc];
      if (q == 0) {
        t = cscale(v[0][s], ax);
      } else {
        const fx64 ay = g.kyd[ky];
        t = cmk<fx64>(t.x + ay * v[0][s].x, t.y + ay * v[0][s].y);
      }
    }
  }
  const double gkg = dots_total(share), dq = gkg * n;
  const bool ok = dq > 0 && isfinite(dq);
  const double alpha = ok ? rho / dq : 0.0;
  const double w = c.kx == 0 ? 1.0 : 2.0;
  double acc[2] = {0.0, 0.0};
  if (ok) {
#pragma unroll 4
    for (int s = 0; s < 8; ++s) {
      const int ky = c.j + s * c.NY8;
      const size_t i = (size_t)ky * H + c.kx;
      const cx<fx64> t = pk[padk(ky) << g.ltc];  // A d = (t.y, -t.x)
      const cx<double> dv = d[i], xv = x[i];
      cx<double> rv = r[i];
      x[i] = cmk<double>(xv.x + alpha * dv.x, xv.y + alpha * dv.y);
      rv = cmk<double>(rv.x - alpha * t.y.v, rv.y + alpha * t.x.v);
      r[i] = rv;
      const double r2 = rv.x * rv.x + rv.y * rv.y;
      acc[0] += r2;
      acc[1] += r2 * g.pinv[i];
    }
    acc[0] *= w;
    acc[1] *= w;
  }
  double tot[2];
  if (last_cta_sum<2>(acc, g.partials, &st->ticket[TK_UPDATE], tot) && threadIdx.x == 0)
    cg_fused_finish(st, gkg, n, tot[0], tot[1]);
}
void col_div_upd(const Geo<double>& gd, const cx<double>* Qx, const cx<double>* Qy, const cx<double>* d,
                 cx<double>* x, cx<double>* r, SolveState* st, cudaStream_t s) {
  const Geo<fx64> g = as_fx(gd);
  k_col_div_upd<<<g.H >> g.ltc, col_threads(g), col_smem(g, 2), s>>>(g, fxp(Qx), fxp(Qy), d, x, r, st);
}

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
    allow_smem(k_col_div_upd);
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
