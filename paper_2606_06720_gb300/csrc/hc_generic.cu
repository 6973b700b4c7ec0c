// hc_generic.cu -- the step on 2D grids whose sizes are not powers of two:
// N = 2^a 3^b 5^c per axis, among them the paper's N = 50 2^k grids of its
// grid-convergence study (Section 4, Tables 1-3).  FP64 throughout.
//
// Transforms are mixed-radix Stockham FFTs (radix 2, 3, 4, 5 passes) of one row,
// or of a column's two fields together, held in a CTA's shared memory, with the
// CTA's threads sharing each pass's butterflies.  Their arithmetic is the 64-bit
// block fixed point of hc_fixed.cuh, because the FP64 pipe is narrow: with FP64
// passes one transform at a time the four CG kernels of 400 x 400 took 108 us,
// now 44.  Passes divide by 2: from an L2 norm of 2^61 the largest
// growth up to 4096 points, 5^5, leaves every input of a pass below 2^61.7 and,
// with a factor of at most sqrt(5) inside it, every value below 2^62.9.
// The spectral state is the unpacked half spectrum:
// ny rows of Hh = nx/2 + 1 values (kx = 0 .. nx/2), row-major, unnormalised
// DFTs.  A step makes the same passes as the power-of-two path, each fused
// with the same pointwise work:
//   column gradient   d = M^-1 r + beta d (CG) or p, times i xi / n, inverse along y
//   row apply         inverse along x, q = (m.g) m + r g, <d, A d> by parts, forward along x
//   column divergence forward along y, -i xi . q^ (CG output or the residual S - A p)
//                     (CG: with x += alpha d, r -= alpha A d, the two dot products)
//   split step        gradient, row pass with activation + relaxation, column
//                     pass with the heat factor exp(-D^2 |xi|^2 dt), row back-transform
// and the same one-thread solve bookkeeping (SolveState), so CG, its stopping
// rule, kappa / Kbar and the diagnostics of Section 2.5 are shared code.
#include "hc_kernels.cuh"

namespace hc {

namespace {

// ------------------------------------------------------------------ small DFTs
// t c for a constant 0 < c < 1 with 2^62 c = 2^32 H + L, L signed; |t| <= 2^62.5.
// The dropped product of the low limbs is L/2^31 on average: it joins the
// rounding constant.
template <int H, int L>
__device__ __forceinline__ long long fmul_const(long long t) {
  const int th = (int)(t >> 32);
  long long cross;
  asm("mad.wide.u32 %0, %1, %2, %3;"
      : "=l"(cross)
      : "r"((unsigned)t), "r"((unsigned)H), "l"(0x20000000LL + L / 2));
  cross = mad32(th, L, cross);
  return (mul32(th, H) << 2) + (cross >> 30);
}
// v w / 2 (fmul without half of its shift) and v / 2, rounded as fmul rounds.
__device__ __forceinline__ fxc fmul2(fxc v, const FxW& w) {
  const int vxl = (int)v.x, vyl = (int)v.y;
  const unsigned bx = (unsigned)vxl >> 31, by = (unsigned)vyl >> 31;
  const int vxh = (int)(v.x >> 32) + (int)bx;
  const int vyh = (int)(v.y >> 32) + (int)by;
  const long long cr = mad32(vyl, w.nh, mad32(vyh, w.nl, mad32(vxl, w.xh, mul32(vxh, w.xl))));
  const long long ci = mad32(vyl, w.xh, mad32(vyh, w.xl, mad32(vxl, w.ph, mul32(vxh, w.pl))));
  fxc r;
  r.x = (mad32(vyh, w.nh, mul32(vxh, w.xh)) << 1) + ((cr + (long long)(0x3fffffffu + bx)) >> 31);
  r.y = (mad32(vyh, w.xh, mul32(vxh, w.ph)) << 1) + ((ci + (long long)(0x3fffffffu + by)) >> 31);
  return r;
}
__device__ __forceinline__ long long fhalf1(long long v) {
  return (v + (long long)((unsigned)v >> 31)) >> 1;
}

// Kernel exp(S 2 pi i j k / R), natural order in and out.  Radix 3: cos(2 pi/3) =
// -1/2, sin(2 pi/3) = sqrt(3)/2.  Radix 5: with c1, c2 = cos(2 pi/5), cos(4 pi/5),
// c1 + c2 = -1/2 and c1 - c2 = sqrt(5)/2; s1, s2 = sin(2 pi/5), sin(4 pi/5) =
// sqrt(10 +- 2 sqrt 5)/4, and s1 b1 + s2 b2, s2 b1 - s1 b2 share s2 (b1 + b2).
template <int S>
__device__ __forceinline__ void gdft3(fxc* v) {
  const fxc a = fadd(v[1], v[2]), b = fsub(v[1], v[2]);
  const fxc t = fxc{v[0].x - fhalf1(a.x), v[0].y - fhalf1(a.y)};
  const fxc u = fmul_si<S>(fxc{fmul_const<929887697, -1332128537>(b.x),
                               fmul_const<929887697, -1332128537>(b.y)});  // sqrt(3)/2
  v[0] = fadd(v[0], a);
  v[1] = fadd(t, u);
  v[2] = fsub(t, u);
}

template <int S>
__device__ __forceinline__ void gdft5(fxc* v) {
  const fxc a1 = fadd(v[1], v[4]), b1 = fsub(v[1], v[4]);
  const fxc a2 = fadd(v[2], v[3]), b2 = fsub(v[2], v[3]);
  const fxc a = fadd(a1, a2), d = fsub(a1, a2), e = fadd(b1, b2);
  const fxc t = fxc{v[0].x - fquarter1(a.x), v[0].y - fquarter1(a.y)};
  const fxc m = fxc{fmul_const<600239927, 803819395>(d.x), fmul_const<600239927, 803819395>(d.y)};  // sqrt(5)/4
  const fxc p = fxc{fmul_const<631129609, -357254181>(e.x), fmul_const<631129609, -357254181>(e.y)};    // s2
  const fxc q1 = fxc{fmul_const<390059550, -1644870943>(b1.x), fmul_const<390059550, -1644870943>(b1.y)};  // s1 - s2
  const fxc q2 = fxc{b2.x + fmul_const<578576943, 1935587992>(b2.x), b2.y + fmul_const<578576943, 1935587992>(b2.y)};  // s1 + s2
  const fxc u1 = fmul_si<S>(fadd(p, q1)), u2 = fmul_si<S>(fsub(p, q2));
  const fxc t1 = fadd(t, m), t2 = fsub(t, m);
  v[0] = fadd(v[0], a);
  v[1] = fadd(t1, u1);
  v[4] = fsub(t1, u1);
  v[2] = fadd(t2, u2);
  v[3] = fsub(t2, u2);
}

// One radix-R pass of NB length-N Stockham FFTs, by all threads of the CTA:
// butterfly j < N/R takes src[j + r N/R], r < R, twiddles element r by
// w^(r k), k = j mod Ns, w = exp(S 2 pi i / (Ns R)) (a table entry
// tw[m] = exp(-2 pi i m / N), conjugated for S = +1), and writes
// dst[(j / Ns) Ns R + k + r Ns].
template <int S, int R, int NB>
__device__ __forceinline__ void gpass(const fxc* __restrict__ src, fxc* __restrict__ dst, int N, int Ns,
                                      const FxTw* __restrict__ tw) {
  const int nb = N / R, step = nb / Ns;
  const float inv = 1.0f / (float)Ns;
  for (int i = threadIdx.x; i < NB * nb; i += blockDim.x) {
    const int o = (NB > 1 && i >= nb) ? N : 0, j = o ? i - nb : i;
    const int k = j - Ns * (int)(((float)j + 0.5f) * inv);  // j mod Ns
    fxc v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = src[o + j + r * nb];
    if (Ns > 1) {
      v[0] = fxc{fhalf1(v[0].x), fhalf1(v[0].y)};
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = fmul2(v[r], fx_w<S>(tw, r * k * step));
    }
    if constexpr (R == 2) {
      const fxc t = v[0];
      v[0] = fadd(t, v[1]);
      v[1] = fsub(t, v[1]);
    }
    if constexpr (R == 3) gdft3<S>(v);
    if constexpr (R == 4) fdft4<S>(v[0], v[1], v[2], v[3]);
    if constexpr (R == 5) gdft5<S>(v);
    const int base = o + (j - k) * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) dst[base + r * Ns] = v[r];
  }
}

// NB length-N transforms of the values at a, a + N (scratch b, as long), S = -1
// forward, +1 inverse (unnormalised).  The caller synchronises after filling a;
// returns the buffer that holds the results, synchronised.
template <int S, int NB = 1>
__device__ cx<double>* gfft(cx<double>* ad, cx<double>* bd, int N, const int* rad, int np,
                            const FxTw* __restrict__ tw) {
  // scales (fx_scales): per warp first, relative to the warp's largest exponent
  __shared__ int2 s_part[8 * NB];
  FxScale sc[NB];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int t = 0; t < NB; ++t) {
    const cx<double>* x = ad + t * N;
    int e = 0;
    for (int k = threadIdx.x; k < N; k += blockDim.x)
      e = max(e, max(__double2hiint(x[k].x) & 0x7fffffff, __double2hiint(x[k].y) & 0x7fffffff));
    e = __reduce_max_sync(0xffffffffu, e);
    const int off20 = ((e >> 20) - 127) << 20;
    float f2 = 0.0f;
    for (int k = threadIdx.x; k < N; k += blockDim.x) {
      f2 = fx_sumsq(f2, x[k].x, off20);
      f2 = fx_sumsq(f2, x[k].y, off20);
    }
    for (int off = 16; off > 0; off >>= 1) f2 += __shfl_xor_sync(0xffffffffu, f2, off);
    if (lane == 0) s_part[t * 8 + warp] = make_int2(e, __float_as_int(f2));
  }
  __syncthreads();
#pragma unroll
  for (int t = 0; t < NB; ++t) {
    int em = 0;
    float f2 = 0.0f;
    for (int w = 0; w < nw; ++w) fx_merge(em, f2, s_part[t * 8 + w]);
    sc[t] = fx_scale_of(em, f2);
  }
  fxc *a = reinterpret_cast<fxc*>(ad), *b = reinterpret_cast<fxc*>(bd);
#pragma unroll
  for (int t = 0; t < NB; ++t) {
    const int b20 = ((1024 + sc[t].e) << 20) + 0xfffff;  // 2^61
    const double up = sc[t].small ? 0x1p512 : 1.0;
    for (int k = t * N + threadIdx.x; k < (t + 1) * N; k += blockDim.x) {
      const cx<double> v = ad[k];
      if (sc[t].small) a[k] = fxc{fx_from(v.x * up, b20), fx_from(v.y * up, b20)};
      else a[k] = fxc{fx_from(v.x, b20), fx_from(v.y, b20)};
    }
  }
  __syncthreads();
  int Ns = 1;
  for (int p = 0; p < np; ++p) {
    const int R = rad[p];
    if (R == 2)
      gpass<S, 2, NB>(a, b, N, Ns, tw);
    else if (R == 3)
      gpass<S, 3, NB>(a, b, N, Ns, tw);
    else if (R == 4)
      gpass<S, 4, NB>(a, b, N, Ns, tw);
    else
      gpass<S, 5, NB>(a, b, N, Ns, tw);
    __syncthreads();
    fxc* t = a;
    a = b;
    b = t;
    Ns *= R;
  }
  cx<double>* rd = reinterpret_cast<cx<double>*>(a);
#pragma unroll
  for (int t = 0; t < NB; ++t) {
    const FxOut o = fx_out_at(sc[t], 1024 + sc[t].e + np - 1);
    for (int k = t * N + threadIdx.x; k < (t + 1) * N; k += blockDim.x) {
      const fxc v = a[k];
      cx<double> d = cmk<double>(fx_to(v.x, o.eb), fx_to(v.y, o.eb));
      if (!o.plain) d = cmk<double>(d.x * o.f1 * o.f2, d.y * o.f1 * o.f2);
      rd[k] = d;
    }
  }
  __syncthreads();
  return rd;
}

// Parseval weight of half-spectrum column kx: 1 for kx = 0 and (even nx) the
// Nyquist column, 2 for the others, whose mirror columns are not stored.
__device__ __forceinline__ double gweight(const GenGeo& g, int kx) {
  return (kx == 0 || 2 * kx == g.nx) ? 1.0 : 2.0;
}
// Null modes of the operator (reading R2): every index 0 or a Nyquist index.
__device__ __forceinline__ bool gnull(const GenGeo& g, int kx, int ky) {
  return (kx == 0 || 2 * kx == g.nx) && (ky == 0 || 2 * ky == g.ny);
}

// Full-length row z = A + i B of two real fields from their half spectra
// (the mirror half by conjugate symmetry); B may be null.
__device__ __forceinline__ void gload_pair(const GenGeo& g, const cx<double>* A, const cx<double>* B,
                                           cx<double>* z) {
  const int N = g.nx, H = g.Hh;
  for (int k = threadIdx.x; k < N; k += blockDim.x) {
    const int kk = k < H ? k : N - k;
    const cx<double> a = A[kk], b = B ? B[kk] : czero<double>();
    z[k] = k < H ? cmk<double>(a.x - b.y, a.y + b.x) : cmk<double>(a.x + b.y, b.x - a.y);
  }
}
// Half spectra of a and b from the spectrum Z of the row a + i b.
__device__ __forceinline__ void gstore_pair(const GenGeo& g, const cx<double>* Z, cx<double>* A,
                                            cx<double>* B) {
  const int N = g.nx, H = g.Hh;
  for (int k = threadIdx.x; k < H; k += blockDim.x) {
    const cx<double> z = Z[k], zc = Z[k == 0 ? 0 : N - k];
    A[k] = cmk<double>(0.5 * (z.x + zc.x), 0.5 * (z.y - zc.y));
    if (B) B[k] = cmk<double>(0.5 * (z.y + zc.y), -0.5 * (z.x - zc.x));
  }
}

}  // namespace

// ------------------------------------------------------------------ column gradient
// NB = 2: both fields' transforms together; 1: one after the other (columns too
// long for four buffers in shared memory).
template <int MODE, int NB>
__global__ void __launch_bounds__(256) gk_col_grad(GenGeo g, const cx<double>* __restrict__ in,
                                                   const cx<double>* __restrict__ rvec,
                                                   cx<double>* dio, cx<double>* __restrict__ Gx,
                                                   cx<double>* __restrict__ Gy, SolveState* st,
                                                   int check_done) {
  if (check_done && st->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int ny = g.ny, H = g.Hh, kx = blockIdx.x;
  cx<double>* A = reinterpret_cast<cx<double>*>(smem_raw);
  cx<double>* B = A + NB * ny;
  const double invn = 1.0 / ((double)g.nx * (double)ny);
  const double kxv = g.kxd[kx];
  bool first = false;
  double beta = 0;
  Pc<double> pc{};
  if (MODE == CG_DUPDATE) {
    first = st->first != 0;
    beta = st->beta;
    pc = pc_of<double>(st);
  }
  for (int q = 0; q < 2; q += NB) {
    for (int ky = threadIdx.x; ky < ny; ky += blockDim.x) {
      const size_t idx = (size_t)ky * H + kx;
      const double kyv = g.kyd[ky];
      cx<double> v;
      if (MODE != CG_DUPDATE) {
        v = in[idx];
      } else if (q > 0) {  // updated by this thread
        v = dio[idx];
      } else {
        const cx<double> z = cscale(rvec[idx], g.pinv[idx]);
        v = first ? z : cadd(z, cscale(dio[idx], beta));
        dio[idx] = v;
      }
      const double a = kxv * invn, b = kyv * invn;
      const cx<double> vx = cmk<double>(-a * v.y, a * v.x), vy = cmk<double>(-b * v.y, b * v.x);
      A[ky] = q == 0 ? vx : vy;  // i (xi / n) P
      if (NB > 1) A[ny + ky] = vy;
    }
    __syncthreads();
    const cx<double>* R = gfft<+1, NB>(A, B, ny, g.ry, g.nry, g.qy);
    for (int ky = threadIdx.x; ky < ny; ky += blockDim.x) {
      (q == 0 ? Gx : Gy)[(size_t)ky * H + kx] = R[ky];
      if (NB > 1) Gy[(size_t)ky * H + kx] = R[ny + ky];
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ row apply
// DOT: the CG variant; <d, A d> = n sum g . K g (summation by parts), as in the
// power-of-two row pass, one partial per row.
template <bool DOT>
__global__ void __launch_bounds__(256) gk_row_apply(GenGeo g, const cx<double>* Gx,
                                                    const cx<double>* Gy,
                                                    const double* __restrict__ mx,
                                                    const double* __restrict__ my,
                                                    const double* __restrict__ rr, cx<double>* Qx,
                                                    cx<double>* Qy, SolveState* st) {
  if (DOT && st->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int N = g.nx, H = g.Hh, y = blockIdx.x;
  cx<double>* A = reinterpret_cast<cx<double>*>(smem_raw);
  cx<double>* B = A + N;
  gload_pair(g, Gx + (size_t)y * H, Gy + (size_t)y * H, A);
  __syncthreads();
  cx<double>* R = gfft<+1>(A, B, N, g.rx, g.nrx, g.qx);
  double gkg = 0.0;
  const size_t ro = (size_t)y * N;
  for (int x = threadIdx.x; x < N; x += blockDim.x) {
    const double gx = R[x].x, gy = R[x].y;
    const double ax = mx[ro + x], ay = my[ro + x], r = rr[ro + x];
    const double mg = ax * gx + ay * gy;
    if (DOT) gkg += mg * mg + r * (gx * gx + gy * gy);
    R[x] = cmk<double>(ax * mg + r * gx, ay * mg + r * gy);
  }
  __syncthreads();
  cx<double>* R2 = gfft<-1>(R, R == A ? B : A, N, g.rx, g.nrx, g.qx);
  gstore_pair(g, R2, Qx + (size_t)y * H, Qy + (size_t)y * H);
  if (DOT) {
    double a1[1] = {gkg};  // the CTA's partial: gk_col_div_upd forms alpha
    block_sum<1>(a1);
    if (threadIdx.x == 0) g.dots[blockIdx.x] = a1[0];
  }
}

// ------------------------------------------------------------------ column divergence
// The forward transforms along y of a column's two fields, in shared memory.
template <int NB>
__device__ __forceinline__ void gdiv_fields(const GenGeo& g, const cx<double>* __restrict__ Qx,
                                            const cx<double>* __restrict__ Qy, const cx<double>*& Rx,
                                            const cx<double>*& Ry) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int ny = g.ny, H = g.Hh, kx = blockIdx.x;
  cx<double>* A = reinterpret_cast<cx<double>*>(smem_raw);
  cx<double>* B = A + NB * ny;
  for (int q = 0; q < 2; q += NB) {
    for (int ky = threadIdx.x; ky < ny; ky += blockDim.x) {
      const size_t idx = (size_t)ky * H + kx;
      A[ky] = (q == 0 ? Qx : Qy)[idx];
      if (NB > 1) A[ny + ky] = Qy[idx];
    }
    __syncthreads();
    const cx<double>* R = gfft<-1, NB>(A, B, ny, g.ry, g.nry, g.qy);
    if (NB > 1) {
      Rx = R;
      Ry = R + ny;
    } else if (q == 0) {  // waits in a third buffer
      cx<double>* T = B + ny;
      for (int ky = threadIdx.x; ky < ny; ky += blockDim.x) T[ky] = R[ky];
      Rx = T;
      __syncthreads();
    } else {
      Ry = R;
    }
  }
}

// -i (xi_x Qx^ + xi_y Qy^) after those.  CD_PLAIN: written to out; CD_RESID: out =
// b - A p and the CG start.
template <int MODE, int NB>
__global__ void __launch_bounds__(256) gk_col_div(GenGeo g, const cx<double>* __restrict__ Qx,
                                                  const cx<double>* __restrict__ Qy,
                                                  const cx<double>* __restrict__ bvec,
                                                  cx<double>* __restrict__ out, SolveState* st) {
  const int ny = g.ny, H = g.Hh, kx = blockIdx.x;
  const double kxv = g.kxd[kx];
  const cx<double>*Rx, *R;
  gdiv_fields<NB>(g, Qx, Qy, Rx, R);
  const double w = gweight(g, kx);
  double acc[2] = {0.0, 0.0};
  Pc<double> pc{};
  if (MODE == CD_RESID) pc = pc_of<double>(st);
  for (int ky = threadIdx.x; ky < ny; ky += blockDim.x) {
    const size_t idx = (size_t)ky * H + kx;
    const double b = g.kyd[ky];
    const cx<double> t = cmk<double>(kxv * Rx[ky].x + b * R[ky].x, kxv * Rx[ky].y + b * R[ky].y);
    const cx<double> q = cmk<double>(t.y, -t.x);
    if constexpr (MODE == CD_RESID) {
      const cx<double> rv = csub(bvec[idx], q);
      out[idx] = rv;
      const double r2 = rv.x * rv.x + rv.y * rv.y;
      acc[0] += w * r2;
      acc[1] += w * r2 * pinv_ab(kxv, b, pc);
    } else {
      out[idx] = q;
    }
  }
  if constexpr (MODE == CD_RESID) {
    double t2[2];
    if (last_cta_sum<2>(acc, g.partials, &st->ticket[TK_RESID], t2) && threadIdx.x == 0)
      resid_init(st, t2[0], t2[1]);
  }
}

// ------------------------------------------------------------------ CG update
// The preconditioner symbol of the running step (k_pinv_table).
__global__ void __launch_bounds__(256) gk_pinv_table(GenGeo g, const SolveState* st) {
  const Pc<double> pc = pc_of<double>(st);
  const size_t total = (size_t)g.ny * g.Hh;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (size_t)gridDim.x * blockDim.x)
    g.pinv[i] = pinv_ab(g.kxd[i % (size_t)g.Hh], g.kyd[i / (size_t)g.Hh], pc);
}

// Divergence pass and CG update in one (k_col_div_upd): with alpha from the row
// pass's partials, x += alpha d, r -= alpha A d and the sums for beta.
template <int NB>
__global__ void __launch_bounds__(256) gk_col_div_upd(GenGeo g, const cx<double>* __restrict__ Qx,
                                                      const cx<double>* __restrict__ Qy,
                                                      const cx<double>* __restrict__ d,
                                                      cx<double>* __restrict__ x,
                                                      cx<double>* __restrict__ r, SolveState* st) {
  if (st->done) {
    if (st->graph_mode && blockIdx.x == 0 && threadIdx.x == 0)
      cudaGraphSetConditional(st->h_cur, 0u);
    return;
  }
  const double rho = st->rho, n = (double)g.nx * (double)g.ny;
  const double share = dots_share(g.dots, g.ny);
  const cx<double>*Rx, *Ry;
  gdiv_fields<NB>(g, Qx, Qy, Rx, Ry);
  const double gkg = dots_total(share), dq = gkg * n;
  const bool ok = dq > 0 && isfinite(dq);
  const double alpha = ok ? rho / dq : 0.0;
  const int H = g.Hh, kx = blockIdx.x;
  const double w = gweight(g, kx), kxv = g.kxd[kx];
  double acc[2] = {0.0, 0.0};
  if (ok)
    for (int ky = threadIdx.x; ky < g.ny; ky += blockDim.x) {
      const size_t i = (size_t)ky * H + kx;
      const double b = g.kyd[ky];
      // A d = (t.y, -t.x)
      const cx<double> t = cmk<double>(kxv * Rx[ky].x + b * Ry[ky].x, kxv * Rx[ky].y + b * Ry[ky].y);
      const cx<double> dv = d[i], xv = x[i];
      cx<double> rv = r[i];
      x[i] = cmk<double>(xv.x + alpha * dv.x, xv.y + alpha * dv.y);
      rv = cmk<double>(rv.x - alpha * t.y, rv.y + alpha * t.x);
      r[i] = rv;
      const double r2 = rv.x * rv.x + rv.y * rv.y;
      acc[0] += r2;
      acc[1] += r2 * g.pinv[i];
    }
  acc[0] *= w;
  acc[1] *= w;
  double tot[2];
  if (last_cta_sum<2>(acc, g.partials, &st->ticket[TK_UPDATE], tot) && threadIdx.x == 0)
    cg_fused_finish(st, gkg, n, tot[0], tot[1]);
}

// ------------------------------------------------------------------ split step
// Row pass: grad p^{k+1} (from the column pass), activation and relaxation per
// point (split_point, as the power-of-two row pass), the energy's pointwise
// sums of m^k with diagnostics on, then the forward transform along x of the
// new m into Mx, My (the gradient's buffers).
__global__ void __launch_bounds__(256) gk_row_split(GenGeo g, cx<double>* Gx, cx<double>* Gy,
                                                    const double* __restrict__ mx,
                                                    const double* __restrict__ my,
                                                    const double* __restrict__ rr, SplitCoef cf,
                                                    SolveState* st) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int N = g.nx, H = g.Hh, y = blockIdx.x;
  cx<double>* A = reinterpret_cast<cx<double>*>(smem_raw);
  cx<double>* B = A + N;
  gload_pair(g, Gx + (size_t)y * H, Gy + (size_t)y * H, A);
  __syncthreads();
  cx<double>* R = gfft<+1>(A, B, N, g.rx, g.nrx, g.qx);
  const size_t ro = (size_t)y * N;
  const bool diag = st->diag != 0;
  bool finite = true;
  EnergyAcc<double> en;
  for (int x = threadIdx.x; x < N; x += blockDim.x) {
    const double gx = R[x].x, gy = R[x].y;
    double ax = mx[ro + x], ay = my[ro + x];
    if (diag) en.add(rr[ro + x], gx * gx + gy * gy, ax * gx + ay * gy, ax * ax + ay * ay, cf.gamma);
    split_point<double>(ax, ay, gx, gy, cf.c2dt, cf);
    finite = finite && isfinite(ax) && isfinite(ay);
    R[x] = cmk<double>(ax, ay);
  }
  if (!finite) st->nonfinite = 1;
  if (diag) en.finish(g.partials, st);
  __syncthreads();
  cx<double>* R2 = gfft<-1>(R, R == A ? B : A, N, g.rx, g.nrx, g.qx);
  gstore_pair(g, R2, Gx + (size_t)y * H, Gy + (size_t)y * H);
}

// Column pass of the diffusion, in place: forward along y, times
// exp(-D^2 |xi|^2 dt) / n (eq. diffusion_space_discrete), inverse along y.
// With diagnostics, sum |grad m_new|^2 = n sum w |xi~|^2 |v|^2 (v = F(m_new)/n).
template <int NB>
__global__ void __launch_bounds__(256) gk_col_heat(GenGeo g, cx<double>* Mx, cx<double>* My,
                                                   SolveState* st) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int ny = g.ny, H = g.Hh, kx = blockIdx.x;
  cx<double>* A = reinterpret_cast<cx<double>*>(smem_raw);
  cx<double>* B = A + NB * ny;
  const double invn = 1.0 / ((double)g.nx * (double)ny);
  const double w = gweight(g, kx), a = g.kxd[kx];
  double gm = 0.0;
  for (int f = 0; f < 2; f += NB) {
    for (int t = 0; t < NB; ++t)
      for (int ky = threadIdx.x; ky < ny; ky += blockDim.x)
        A[t * ny + ky] = (f + t == 0 ? Mx : My)[(size_t)ky * H + kx];
    __syncthreads();
    cx<double>* R = gfft<-1, NB>(A, B, ny, g.ry, g.nry, g.qy);
    for (int t = 0; t < NB; ++t)
      for (int ky = threadIdx.x; ky < ny; ky += blockDim.x) {
        const cx<double> v = cscale(R[t * ny + ky], g.hx[kx] * g.hy[ky] * invn);
        R[t * ny + ky] = v;
        const double b = g.kyd[ky];
        gm += w * (a * a + b * b) * (v.x * v.x + v.y * v.y);
      }
    __syncthreads();
    cx<double>* R2 = gfft<+1, NB>(R, R == A ? B : A, ny, g.ry, g.nry, g.qy);
    for (int t = 0; t < NB; ++t)
      for (int ky = threadIdx.x; ky < ny; ky += blockDim.x)
        (f + t == 0 ? Mx : My)[(size_t)ky * H + kx] = R2[t * ny + ky];
    __syncthreads();
  }
  if (st && st->diag) gradnorm_finish(gm, (double)g.nx * (double)ny, g.partials, st, 1);
}

// Row back-transform of two fields: half spectra A, B -> physical a, b (B, b
// may be null).  With kappa_update: the sums of m_a m_b for the next
// preconditioner, the non-finite check, and with diagnostics sum |new - old|^2.
__global__ void __launch_bounds__(256) gk_row_c2r(GenGeo g, const cx<double>* A, const cx<double>* B,
                                                  double* a, double* b, SolveState* st,
                                                  int kappa_update) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int N = g.nx, H = g.Hh, y = blockIdx.x;
  cx<double>* Z = reinterpret_cast<cx<double>*>(smem_raw);
  cx<double>* W = Z + N;
  gload_pair(g, A + (size_t)y * H, B ? B + (size_t)y * H : nullptr, Z);
  __syncthreads();
  cx<double>* R = gfft<+1>(Z, W, N, g.rx, g.nrx, g.qx);
  const size_t ro = (size_t)y * N;
  const bool diag = kappa_update && st->diag;
  double mxx = 0, myy = 0, mxy = 0, d2 = 0;
  bool finite = true;
  for (int x = threadIdx.x; x < N; x += blockDim.x) {
    const double u = R[x].x, v = R[x].y;
    if (diag) {
      const double du = u - a[ro + x], dv = v - b[ro + x];
      d2 += du * du + dv * dv;
    }
    a[ro + x] = u;
    if (b) b[ro + x] = v;
    if (kappa_update) {
      mxx += u * u;
      myy += v * v;
      mxy += u * v;
      finite = finite && isfinite(u) && isfinite(v);
    }
  }
  if (kappa_update) {
    if (!finite) st->nonfinite = 1;
    double acc[4] = {mxx, myy, mxy, d2}, tot[4];
    if (last_cta_sum<4>(acc, g.partials, &st->ticket[TK_MSUM], tot) && threadIdx.x == 0) {
      set_mm2(st, tot[0], tot[1], tot[2]);
      if (diag) st->dm2 = tot[3];
    }
  }
}

// ------------------------------------------------------------------ plain transforms
// Forward transform along x of the real rows a (+ i b): half spectra A (, B).
__global__ void __launch_bounds__(256) gk_row_fwd(GenGeo g, const double* __restrict__ a,
                                                  const double* __restrict__ b, cx<double>* A,
                                                  cx<double>* B) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int N = g.nx, H = g.Hh, y = blockIdx.x;
  cx<double>* Z = reinterpret_cast<cx<double>*>(smem_raw);
  cx<double>* W = Z + N;
  const size_t ro = (size_t)y * N;
  for (int x = threadIdx.x; x < N; x += blockDim.x)
    Z[x] = cmk<double>(a[ro + x], b ? b[ro + x] : 0.0);
  __syncthreads();
  cx<double>* R = gfft<-1>(Z, W, N, g.rx, g.nrx, g.qx);
  gstore_pair(g, R, A + (size_t)y * H, B ? B + (size_t)y * H : nullptr);
}

// Forward transform along y of one or two half-spectrum fields.  project:
// the null modes of field 0 are zeroed (the solvability condition, reading
// R2) and, with st, sum w |F|^2 of field 0 goes to st->outer_b2.  gradnorm:
// instead, sum w |xi~|^2 |F|^2 / n over both fields (|grad m|^2 of the
// physical fields) goes to st->gm2 (the outputs may then be null).
__global__ void __launch_bounds__(256) gk_col_fwd(GenGeo g, const cx<double>* in0,
                                                  const cx<double>* in1, cx<double>* out0,
                                                  cx<double>* out1, int project, int gradnorm,
                                                  SolveState* st) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int ny = g.ny, H = g.Hh, kx = blockIdx.x;
  cx<double>* A = reinterpret_cast<cx<double>*>(smem_raw);
  cx<double>* B = A + ny;
  const double w = gweight(g, kx), a = g.kxd[kx];
  double acc = 0.0;
  for (int f = 0; f < (in1 ? 2 : 1); ++f) {
    const cx<double>* in = f == 0 ? in0 : in1;
    cx<double>* out = f == 0 ? out0 : out1;
    for (int ky = threadIdx.x; ky < ny; ky += blockDim.x) A[ky] = in[(size_t)ky * H + kx];
    __syncthreads();
    cx<double>* R = gfft<-1>(A, B, ny, g.ry, g.nry, g.qy);
    for (int ky = threadIdx.x; ky < ny; ky += blockDim.x) {
      cx<double> v = R[ky];
      if (project && f == 0 && gnull(g, kx, ky)) v = czero<double>();
      if (out) out[(size_t)ky * H + kx] = v;
      const double n2 = v.x * v.x + v.y * v.y;
      if (gradnorm) {
        const double b = g.kyd[ky];
        acc += w * (a * a + b * b) * n2;
      } else if (f == 0) {
        acc += w * n2;
      }
    }
    __syncthreads();
  }
  if (gradnorm && st) {
    gradnorm_finish(acc, 1.0 / ((double)g.nx * (double)ny), g.partials, st, 0);
  } else if (project && st) {
    double a1[1] = {acc}, t1[1];
    if (last_cta_sum<1>(a1, g.partials, &st->ticket[TK_PROJ], t1) && threadIdx.x == 0)
      st->outer_b2 = t1[0];
  }
}

// Inverse transform along y of one half-spectrum field, times scale.
__global__ void __launch_bounds__(256) gk_col_inv(GenGeo g, const cx<double>* in, cx<double>* out,
                                                  double scale) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int ny = g.ny, H = g.Hh, kx = blockIdx.x;
  cx<double>* A = reinterpret_cast<cx<double>*>(smem_raw);
  cx<double>* B = A + ny;
  for (int ky = threadIdx.x; ky < ny; ky += blockDim.x) A[ky] = in[(size_t)ky * H + kx];
  __syncthreads();
  cx<double>* R = gfft<+1>(A, B, ny, g.ry, g.nry, g.qy);
  for (int ky = threadIdx.x; ky < ny; ky += blockDim.x)
    out[(size_t)ky * H + kx] = cscale(R[ky], scale);
}

// ------------------------------------------------------------------ launchers
namespace {
constexpr int kGenThreads = 256;
size_t gcol_smem(const GenGeo& g, int bufs) { return (size_t)bufs * g.ny * sizeof(cx<double>); }
size_t grow_smem(const GenGeo& g) { return (size_t)2 * g.nx * sizeof(cx<double>); }
// Columns whose two fields fit shared memory together (two buffers each).
bool gpair(const GenGeo& g) { return g.ny <= 3000; }
// Threads for `points` of a CTA's transforms: two points each (the passes of a
// radix-4 butterfly leave half of them idle, but the conversions and pointwise
// loops are longer: 400^2 row pass 30 us at four points a thread, 22 at two).
int gthreads(int points) {
  const int t = (points / 2 + 31) / 32 * 32;
  return t < 64 ? 64 : (t > kGenThreads ? kGenThreads : t);
}
int gupd_blocks(const GenGeo& g) {
  const size_t b = ((size_t)g.ny * g.Hh + kGenThreads - 1) / kGenThreads;
  return (int)(b < 608 ? b : 608);
}
}  // namespace

void gen_col_grad(const GenGeo& g, int mode, const cx<double>* in, const cx<double>* rvec,
                  cx<double>* dio, cx<double>* Gx, cx<double>* Gy, SolveState* st, int check_done,
                  cudaStream_t s) {
  const auto k = mode == CG_DUPDATE
                     ? (gpair(g) ? gk_col_grad<CG_DUPDATE, 2> : gk_col_grad<CG_DUPDATE, 1>)
                     : (gpair(g) ? gk_col_grad<CG_PLAIN, 2> : gk_col_grad<CG_PLAIN, 1>);
  k<<<g.Hh, gthreads(2 * g.ny), gcol_smem(g, gpair(g) ? 4 : 2), s>>>(g, in, rvec, dio, Gx, Gy, st,
                                                                     check_done);
}
void gen_row_apply(const GenGeo& g, const cx<double>* Gx, const cx<double>* Gy, const double* mx,
                   const double* my, const double* r, cx<double>* Qx, cx<double>* Qy,
                   SolveState* st, cudaStream_t s) {
  if (st)
    gk_row_apply<true><<<g.ny, gthreads(g.nx), grow_smem(g), s>>>(g, Gx, Gy, mx, my, r, Qx, Qy, st);
  else
    gk_row_apply<false><<<g.ny, gthreads(g.nx), grow_smem(g), s>>>(g, Gx, Gy, mx, my, r, Qx, Qy, st);
}
void gen_col_div(const GenGeo& g, int mode, const cx<double>* Qx, const cx<double>* Qy,
                 const cx<double>* b, cx<double>* out, SolveState* st, cudaStream_t s) {
  const auto k = mode == CD_RESID ? (gpair(g) ? gk_col_div<CD_RESID, 2> : gk_col_div<CD_RESID, 1>)
                                  : (gpair(g) ? gk_col_div<CD_PLAIN, 2> : gk_col_div<CD_PLAIN, 1>);
  k<<<g.Hh, gthreads(2 * g.ny), gcol_smem(g, gpair(g) ? 4 : 3), s>>>(g, Qx, Qy, b, out, st);
}
void gen_pinv_table(const GenGeo& g, const SolveState* st, cudaStream_t s) {
  gk_pinv_table<<<gupd_blocks(g), kGenThreads, 0, s>>>(g, st);
}
void gen_col_div_upd(const GenGeo& g, const cx<double>* Qx, const cx<double>* Qy, const cx<double>* d,
                     cx<double>* x, cx<double>* r, SolveState* st, cudaStream_t s) {
  const auto k = gpair(g) ? gk_col_div_upd<2> : gk_col_div_upd<1>;
  k<<<g.Hh, gthreads(2 * g.ny), gcol_smem(g, gpair(g) ? 4 : 3), s>>>(g, Qx, Qy, d, x, r, st);
}
void gen_row_split(const GenGeo& g, cx<double>* Gx, cx<double>* Gy, const double* mx,
                   const double* my, const double* r, SplitCoef cf, SolveState* st,
                   cudaStream_t s) {
  gk_row_split<<<g.ny, gthreads(g.nx), grow_smem(g), s>>>(g, Gx, Gy, mx, my, r, cf, st);
}
void gen_col_heat(const GenGeo& g, cx<double>* Mx, cx<double>* My, SolveState* st, cudaStream_t s) {
  const auto k = gpair(g) ? gk_col_heat<2> : gk_col_heat<1>;
  k<<<g.Hh, gthreads(2 * g.ny), gcol_smem(g, gpair(g) ? 4 : 2), s>>>(g, Mx, My, st);
}
void gen_row_c2r(const GenGeo& g, const cx<double>* A, const cx<double>* B, double* a, double* b,
                 SolveState* st, int kappa_update, cudaStream_t s) {
  gk_row_c2r<<<g.ny, gthreads(g.nx), grow_smem(g), s>>>(g, A, B, a, b, st, kappa_update);
}
void gen_row_fwd(const GenGeo& g, const double* a, const double* b, cx<double>* A, cx<double>* B,
                 cudaStream_t s) {
  gk_row_fwd<<<g.ny, gthreads(g.nx), grow_smem(g), s>>>(g, a, b, A, B);
}
void gen_col_fwd(const GenGeo& g, const cx<double>* in0, const cx<double>* in1, cx<double>* out0,
                 cx<double>* out1, int project, int gradnorm, SolveState* st, cudaStream_t s) {
  gk_col_fwd<<<g.Hh, gthreads(g.ny), gcol_smem(g, 2), s>>>(g, in0, in1, out0, out1, project, gradnorm,
                                                        st);
}
void gen_col_inv(const GenGeo& g, const cx<double>* in, cx<double>* out, double scale,
                 cudaStream_t s) {
  gk_col_inv<<<g.Hh, gthreads(g.ny), gcol_smem(g, 2), s>>>(g, in, out, scale);
}

void set_smem_limits_gen() {
  allow_smem(gk_col_grad<CG_PLAIN, 1>);
  allow_smem(gk_col_grad<CG_PLAIN, 2>);
  allow_smem(gk_col_grad<CG_DUPDATE, 1>);
  allow_smem(gk_col_grad<CG_DUPDATE, 2>);
  allow_smem(gk_row_apply<true>);
  allow_smem(gk_row_apply<false>);
  allow_smem(gk_col_div<CD_PLAIN, 1>);
  allow_smem(gk_col_div<CD_PLAIN, 2>);
  allow_smem(gk_col_div_upd<1>);
  allow_smem(gk_col_div_upd<2>);
  allow_smem(gk_col_div<CD_RESID, 1>);
  allow_smem(gk_col_div<CD_RESID, 2>);
  allow_smem(gk_row_split);
  allow_smem(gk_col_heat<1>);
  allow_smem(gk_col_heat<2>);
  allow_smem(gk_row_c2r);
  allow_smem(gk_row_fwd);
  allow_smem(gk_col_fwd);
  allow_smem(gk_col_inv);
}

}  // namespace hc
