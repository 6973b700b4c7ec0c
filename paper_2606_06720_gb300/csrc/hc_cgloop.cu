// hc_cgloop.cu -- the CG loop of a 2D solve as one cooperative kernel.
//
// On grids up to about 10^6 points an iteration's launches (three or four kernels and the
// loop node's turn) cost as much as their work: at 512^2 an iteration took 40 us, of which
// the kernels ran 29, each of them mostly the latency of its start, its loads and its last
// CTA's sums.  Here one launch runs the whole loop.  Every CTA keeps the same column tile
// and the same rows throughout, so x, r and d never leave it (registers and shared memory),
// m and r of the coefficient are staged once, and only the transposed fields Gx, Gy and
// three sums an iteration pass between CTAs, across three grid barriers.  Each CTA forms
// alpha, beta and the stop test from the CTAs' partial sums, all in the same order, so all
// leave the loop together and none waits for a last CTA.
//
// Measured (us an iteration, separate kernels -> loop; several hundred iterations): FP32 512^2
// 40 -> 20; FP64 32^2 60 -> 40, 64^2 58 -> 33, 256^2 76 -> 43, 512^2 82 -> 62, 1024x512 (512
// threads at 128 registers) 108 -> 108, so FP64 stops at 256 threads.  What is left: FP32, the
// three barriers and the L2 latency of Gx and Gy around them; FP64, a warp's own instructions.
// Beyond 512 threads a CTA (2^20 points) x, r and d no longer fit on the chip.
#include "hc_kernels.cuh"

namespace hc {

// Loops of several callers on one device (threads, streams, the chains of a batch).  Two loops
// whose CTAs each hold SMs that the other's missing ones wait for would both stand still, so the
// CTAs that wait at a time must all fit.  They are counted on the device, solve by solve: a
// one-thread kernel before the loop claims its room or, where there is none, refuses the launch,
// which then returns at once and is tried again.  (A lock held by the host call, the rule before,
// kept callers apart for all steps of a call: eight solvers of 64^2 FP64 on eight threads 28 ms for
// four steps, sixteen in a batch 55, now 10 and 8; with separate kernels, FP64 passes 24 and 23.
// The claim inside the loop kernel saved its launch but changed the code of the FP64 loop: 64^2
// 30.1 -> 31.5 us an iteration.)
//
// What fits: a CTA of a kernel of which `per` fit an SM takes 1/per of every resource at most,
// counted in sixteenths, u = 16 / per (per rounded down to a power of two, 16 at most).  An SM has
// room for it unless more than 16 - u sixteenths are taken, and with u_min the smallest u about
// that means 16 - u + u_min at least.  So each of the CTAs has an SM to go to if all of them
// together are no more than the SMs, or take no more than SMs * (16 - u_max + u_min) sixteenths.
// (An SM's free registers may lie in pieces; a barrier whose CTA finds no place is then given up
// and the launch repeated.  In the crowds of the tests none was.)
// g_loop_room holds the CTAs per u = 1, 2, 4, 8, 16 in fields of 12 bits (2432 CTAs at most), and
// in bit 60 that a solve has waited for long (kLoopTurnNs): then only such solves enter, so that
// one that needs the whole device gets it.
constexpr int kRoomBits = 12;
constexpr unsigned long long kRoomTurn = 1ull << 60, kLoopTurnNs = 2000000ull;
constexpr unsigned kLoopPauseNs = 4000;  // after a refusal, before the next try
__device__ unsigned long long g_loop_room;

__host__ __device__ inline bool room_ok(unsigned long long room, int sms) {
  int ctas = 0, units = 0, lo = 0, hi = 0;
  for (int k = 0; k < 5; ++k) {
    const int n = (int)(room >> (k * kRoomBits)) & ((1 << kRoomBits) - 1);
    if (!n) continue;
    if (!ctas) lo = 1 << k;
    hi = 1 << k;
    ctas += n;
    units += n << k;
  }
  return ctas <= sms || units <= sms * (16 - hi + lo);
}

// The grid barriers of one launch.  The launch is cooperative, so every CTA is resident and
// arrives; a wait is bounded all the same (st->loop_polls polls), because another stream's
// kernel may hold an SM that a CTA waits for.  A barrier completes for every CTA or for none: one
// that gives up marks the word with a compare-and-swap that fails once the count is complete, and
// whoever sees the mark gives up too.  A CTA still polling an earlier barrier leaves as well, and
// no later one completes without it.  x is stored after the last barrier, so a launch that is
// given up has changed nothing and can simply be repeated (loop_leave).
// Arrivals count in twos (the count may wrap); the mark is bit 0, and 2^30 more, so that one
// comparison ends a poll either way.
struct LoopBar {
  unsigned* word;
  unsigned polls;
  unsigned target = 0;
  // What any CTA wrote before it is visible to every thread after it.  False in every thread
  // once the launch is given up.
  // (One counter, polled with acquires: a word per CTA that a warp polls took 2.4 us more a
  // barrier at 128 CTAs, relaxed polls and one fence 0.3 us more; polls one at a time, ten steps
  // of 64^2 FP64 13.84 ms, unrolled by four 13.79.)
  __device__ __forceinline__ bool wait() {
    __shared__ int s_ok;
    target += 2 * gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned v = target - 1u;
      if (polls == 0)  // no wait at all: marked in place of arriving
        asm volatile("red.release.gpu.global.or.b32 [%0], 1;" ::"l"(word) : "memory");
      else
        asm volatile("red.release.gpu.global.add.u32 [%0], 2;" ::"l"(word) : "memory");
#pragma unroll 4
      for (unsigned i = 0; i < polls && !past(v); ++i)
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(word) : "memory");
      if (!past(v)) v = give_up();
      s_ok = !(v & 1u);
    }
    __syncthreads();
    return s_ok != 0;
  }
  __device__ __forceinline__ bool past(unsigned v) const { return (int)(v - target) >= 0; }
  // The word after this CTA's mark, or as it is where it is marked or complete already.  Each
  // failed swap is an arrival, or another CTA's mark: at most one round per CTA.
  __device__ __noinline__ unsigned give_up() {
    unsigned v, old;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(word) : "memory");
    for (unsigned i = 0; i <= gridDim.x; ++i) {
      if ((v & 1u) || past(v)) return v;
      asm volatile("atom.acq_rel.gpu.global.cas.b32 %0, [%1], %2, %3;"
                   : "=r"(old)
                   : "l"(word), "r"(v), "r"((v + 0x40000000u) | 1u)
                   : "memory");
      if (old == v) break;
      v = old;
    }
    return 1u;
  }
};

// The scalars of a solve, kept by every thread alike.
struct LoopCg {
  double rho, rnorm2, alpha, beta;
  int it, done, status;
};

// After the row pass: the step length, as cg_alpha_from.
__device__ __forceinline__ bool loop_alpha(LoopCg& k, double gkg, double n, int refined,
                                           double thresh2) {
  const double dq = gkg * n;
  if (dq > 0 && isfinite(dq)) {
    k.alpha = k.rho / dq;
    return true;
  }
  k.alpha = 0.0;
  k.done = 1;
  if (!isfinite(dq)) k.status = HC_ENONFINITE;
  else if (!refined && k.rnorm2 > thresh2) k.status = HC_ENOCONV;
  return false;
}
// After the update: beta and the stop test, as cg_step_finish.
__device__ __forceinline__ void loop_beta(LoopCg& k, double rr, double rz, double thresh2,
                                          int maxit) {
  k.rnorm2 = rr;
  k.beta = k.rho > 0 ? rz / k.rho : 0.0;
  k.rho = rz;
  k.it += 1;
  if (!isfinite(rr)) {
    k.status = HC_ENONFINITE;
    k.done = 1;
  } else if (rr <= thresh2) {
    k.done = 1;
  } else if (k.it >= maxit) {
    k.done = 1;
    k.status = HC_ENOCONV;
  }
}
// The end of the loop, one thread of the grid: the solve state as the kernels of an
// iteration would have left it.
__device__ __forceinline__ void loop_finish(SolveState* st, const LoopCg& k, int its) {
  st->rnorm2 = k.rnorm2;
  st->alpha = k.alpha;
  st->alpha_f = (float)k.alpha;
  st->beta = k.beta;
  st->beta_f = (float)k.beta;
  st->rho = k.rho;
  st->it = k.it;
  st->total_it += its;
  st->loop_count[1] += its;
  if (k.status) st->status = k.status;
  st->first = 0;
  st->done = 1;
  predict_residual(st);
  if (st->graph_mode) cudaGraphSetConditional(st->h_cur, 0u);
}
// A solve of a call in which an earlier one was given up for good ends here.
__device__ __forceinline__ bool loop_gave_up(SolveState* st) {
  if (!st->loop_timeout) return false;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st->done = 1;
    if (st->graph_mode) cudaGraphSetConditional(st->h_cur, 0u);
  }
  return true;
}
// A launch that was refused (2) or given up (3): one thread.  The solve is as it was, so it runs
// again (the WHILE node's next turn, or the host's next launch), until st->loop_patience ns after
// the first such launch.
__device__ __forceinline__ void loop_lost(SolveState* st, int how) {
  st->loop_count[how] += 1;
  unsigned long long now;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
  if (!st->loop_since) st->loop_since = now;
  if (now - st->loop_since >= st->loop_patience) {
    st->loop_since = 0ull;
    st->loop_turn = 0;
    st->loop_timeout = 1;
    st->done = 1;
    if (st->graph_mode) cudaGraphSetConditional(st->h_cur, 0u);
  } else if (now - st->loop_since >= kLoopTurnNs) {
    st->loop_turn = 1;
  }
}
// The last CTA to leave re-arms the barriers and gives the launch's room back.
__device__ __forceinline__ void loop_leave(SolveState* st, const LoopRoom& room, bool live) {
  if (threadIdx.x != 0) return;
  unsigned t;
  asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(t) : "l"(&st->loop_exit) : "memory");
  if (t != gridDim.x - 1) return;
  st->loop_exit = 0u;
  st->loop_bar = 0u;
  if (room.need) atomicAdd(&g_loop_room, 0ull - room.need);
  if (live) {
    st->loop_since = 0ull;
    st->loop_turn = 0;
    st->loop_count[0] += 1;
  } else {
    loop_lost(st, 3);
  }
}

// One thread, before a loop kernel: room for it, or a refusal.  The swap assumes an idle device at
// first; each failed one is another solve's.
__global__ void k_loop_claim(SolveState* st, LoopRoom room) {
  if (st->done || st->loop_timeout) return;
  const bool turn = st->loop_turn != 0;
  unsigned long long cur = 0ull;
  for (int i = 0; i < 256; ++i) {
    const unsigned long long next = (turn ? cur & ~kRoomTurn : cur) + room.need;
    const bool fits = room_ok(next & ~kRoomTurn, room.sms) && (turn || !(cur & kRoomTurn));
    if (!fits && i > 0) break;
    const unsigned long long old = atomicCAS(&g_loop_room, cur, fits ? next : cur);
    if (old == cur && fits) {
      st->loop_refused = 0;
      return;
    }
    cur = old;
  }
  st->loop_refused = 1;
  loop_lost(st, 2);
  if (st->loop_turn) atomicOr(&g_loop_room, kRoomTurn);
  __nanosleep(kLoopPauseNs);
}

// Sum over the CTAs of K values (K doubles each at p[cta * stride]), in every thread.
template <int K>
__device__ __forceinline__ void grid_total(const double* p, int stride, double (&tot)[K]) {
  __shared__ double s_tot[K];
  double w[K];
#pragma unroll
  for (int k = 0; k < K; ++k) w[k] = 0.0;
  for (unsigned c = threadIdx.x; c < gridDim.x; c += blockDim.x)
#pragma unroll
    for (int k = 0; k < K; ++k) w[k] += __ldcg(&p[c * stride + k]);
  block_sum<K>(w);
  if (threadIdx.x == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) s_tot[k] = w[k];
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) tot[k] = s_tot[k];
}

// FP32 inner solve (x, r column-major).  g's tile (tc, rpc) is the loop's: blockDim.x threads
// carry two fields of 8 values of a column, or 8 values of two rows.  The arithmetic is the
// separate kernels' to the bit, roundings written out; only the order of the sums differs.
// row_sums: a row's share of <d, A d> is summed by itself, as where those kernels put one row
// on a thread.
// MAXT: 512 threads at 128 registers (some spills), or 256 without.
template <int MAXT>
__global__ void __launch_bounds__(MAXT, 1) k_cg_loop_f32(Geo<float> g, cx<float>* x,
                                                        const cx<float>* r, cx<float>* Gx,
                                                        cx<float>* Gy, const float* mx,
                                                        const float* my, const float* rf,
                                                        SolveState* st, LoopRoom room, int row_sums) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (st->done) return;  // nothing writes it before every CTA has passed a barrier
  if (loop_gave_up(st) || st->loop_refused) return;
  using C = cx<float>;
  C* sm = reinterpret_cast<C*>(smem_raw);
  const int nt = blockDim.x, t = threadIdx.x, H = g.H;
  const ColIdx c = col_idx(g);
  const int se = slab_elems(g);
  C* const csl[2] = {sm + c.b, sm + se + c.b};
  // rows
  const int l8 = g.lnx - 3, N = g.nx, N8 = 1 << l8;
  const int rj = t & (N8 - 1), r0 = (t >> l8) * 2, y0 = (blockIdx.x << g.lrpc) + r0;
  C* const rsl[2] = {sm + (size_t)r0 * N, sm + (size_t)(r0 + 1) * N};
  C* const Ra[2] = {Gx + (size_t)y0 * H, Gx + (size_t)(y0 + 1) * H};
  C* const Rb[2] = {Gy + (size_t)y0 * H, Gy + (size_t)(y0 + 1) * H};
  // behind the slabs: this CTA's rows of mx, my, r, then x (slot s of thread t at s nt + t)
  float* sf = reinterpret_cast<float*>(sm + 18 * nt);
  C* xs = reinterpret_cast<C*>(sf + 3 * (size_t)g.rpc * N) + t;
  {
    const size_t row0 = ((size_t)blockIdx.x << g.lrpc) * N;
    const int per = (int)(((size_t)g.rpc * N * sizeof(float)) >> 4);
    const float* const src[3] = {mx + row0, my + row0, rf + row0};
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      char* dst = reinterpret_cast<char*>(sf + (size_t)q * g.rpc * N);
      const char* from = reinterpret_cast<const char*>(src[q]);
      for (int i = t; i < per; i += nt) cp_async16(dst + 16 * i, from + 16 * i);
    }
    cp_async_commit();
  }
  const double n = (double)g.nx * (double)g.ny, thresh2 = st->thresh2;
  const int maxit = st->maxit;
  const Pc<float> pc = pc_of<float>(st);
  LoopCg k{st->rho, st->rnorm2, 0.0, 0.0, st->it, 0, 0};
  const int it0 = k.it;
  LoopBar bar{&st->loop_bar, st->loop_polls};
  const float invn = exp2_neg<float>(g.lnx + g.lny), kx = g.kxd[c.kx];
  const float ax = kx * invn;
  const float wt = c.kx == 0 ? 1.0f : 2.0f;  // Parseval weight of a packed column
  float pv[8];  // the preconditioner symbol
  C rv[8], dv[8];
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const int ky = c.j + s * c.NY8;
    const float b = g.kyd[ky];
    const float xa = __fmul_rn(pc.xx, kx), xb = __fmul_rn(__fmul_rn(2.0f, pc.xy), kx);
    const float yb = __fmul_rn(pc.yy, b);
    const float s2 = __fmaf_rn(yb, b, __fmaf_rn(xa, kx, __fmul_rn(xb, b)));
    pv[s] = s2 > 0.0f ? 1.0f / s2 : 0.0f;
    const size_t i = cmi(g, ky, c.kx);
    rv[s] = r[i];
    dv[s] = czero<float>();
    xs[(size_t)s * nt] = x[i];
  }
  cp_async_wait_all();
  bool live = true;  // the launch has not been given up
  while (true) {
    // gradient of d = M^-1 r + beta d
    const bool first = k.it == it0;
    const float beta = (float)k.beta;
    C v[2][8];
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const C z = cmk<float>(__fmul_rn(rv[s].x, pv[s]), __fmul_rn(rv[s].y, pv[s]));
      const C P = first ? z : cmk<float>(__fmaf_rn(dv[s].x, beta, z.x), __fmaf_rn(dv[s].y, beta, z.y));
      dv[s] = P;
      const float ay = g.kyd[c.j + s * c.NY8] * invn;
      v[0][s] = cmk<float>(__fmul_rn(-ax, P.y), __fmul_rn(ax, P.x));
      v[1][s] = cmk<float>(__fmul_rn(-ay, P.y), __fmul_rn(ay, P.x));
    }
    fft_canon<+1, 2>(v, csl, g.tc, c.j, g.lny, g.twy);
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const size_t idx = (size_t)(c.j + s * c.NY8) * H + c.kx;
      Gx[idx] = v[0][s];
      Gy[idx] = v[1][s];
    }
    live = bar.wait();
    if (!live) break;
    // (m m + r I) grad d along the rows, in place
    load_rows_c2r<2>(v, (const C* const*)Ra, (const C* const*)Rb, rj, N8);
    fft_canon<+1, 2, true>(v, rsl, 1, rj, g.lnx, g.twx);
    float gk = 0.0f, gk0 = 0.0f;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const float* smx = sf + (size_t)(r0 + q) * N;
      const float* smy = smx + (size_t)g.rpc * N;
      const float* srr = smy + (size_t)g.rpc * N;
      if (q == 1 && row_sums) {
        gk0 = gk;
        gk = 0.0f;
      }
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        const int xp = rj + s * N8;
        const float gx = v[q][s].x, gy = v[q][s].y;
        const float a = smx[xp], b = smy[xp], rr = srr[xp];
        const float mg = __fmaf_rn(a, gx, __fmul_rn(b, gy));
        const float g2 = __fmaf_rn(gx, gx, __fmul_rn(gy, gy));
        gk = __fadd_rn(gk, __fmaf_rn(rr, g2, __fmul_rn(mg, mg)));
        v[q][s] = cmk<float>(__fmaf_rn(rr, gx, __fmul_rn(a, mg)), __fmaf_rn(rr, gy, __fmul_rn(b, mg)));
      }
    }
    fft_rows_r2c<2>(v, rsl, rj, g.lnx, g.twx, Ra, Rb);
    {
      float h[1] = {gk}, l[1] = {0.0f};
      pair_add(h[0], l[0], gk0, 0.0f);
      double p[1];
      cta_pair_sums<1>(h, l, p);
      if (t == 0) g.dots[blockIdx.x] = p[0];
    }
    live = bar.wait();
    if (!live) break;
    // A d = -div; x += alpha d, r -= alpha A d
    const double share = t < (int)gridDim.x ? __ldcg(&g.dots[t]) : 0.0;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const size_t idx = (size_t)(c.j + s * c.NY8) * H + c.kx;
      v[0][s] = Gx[idx];
      v[1][s] = Gy[idx];
    }
    fft_canon<-1, 2>(v, csl, g.tc, c.j, g.lny, g.twy);
    double w = share;
    for (int i = t + nt; i < (int)gridDim.x; i += nt) w += __ldcg(&g.dots[i]);
    const double gkg = dots_total(w);
    if (!loop_alpha(k, gkg, n, 1, thresh2)) break;
    const float alpha = (float)k.alpha;
    DotAcc<float> rr, rz;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const float ay = g.kyd[c.j + s * c.NY8];
      const C q = cmk<float>(__fmaf_rn(kx, v[0][s].y, __fmul_rn(ay, v[1][s].y)),
                             -__fmaf_rn(kx, v[0][s].x, __fmul_rn(ay, v[1][s].x)));
      const C xv = xs[(size_t)s * nt];
      xs[(size_t)s * nt] = cmk<float>(__fmaf_rn(alpha, dv[s].x, xv.x), __fmaf_rn(alpha, dv[s].y, xv.y));
      rv[s] = cmk<float>(__fmaf_rn(-alpha, q.x, rv[s].x), __fmaf_rn(-alpha, q.y, rv[s].y));
      rr.add_prod(wt * rv[s].x, rv[s].x);
      rr.add_prod(wt * rv[s].y, rv[s].y);
      const float wp = wt * pv[s];
      rz.add_prod(wp * rv[s].x, rv[s].x);
      rz.add_prod(wp * rv[s].y, rv[s].y);
    }
    {
      float h[2] = {rr.hi, rz.hi}, l[2] = {rr.lo, rz.lo};
      double p[2];
      cta_pair_sums<2>(h, l, p);
      if (t == 0) {
        g.partials[(size_t)blockIdx.x * kPartialStride] = p[0];
        g.partials[(size_t)blockIdx.x * kPartialStride + 1] = p[1];
      }
    }
    live = bar.wait();
    if (!live) break;
    double tot[2];
    grid_total<2>(g.partials, kPartialStride, tot);
    loop_beta(k, tot[0], tot[1], thresh2, maxit);
    if (k.done) break;
  }
  if (live) {
#pragma unroll
    for (int s = 0; s < 8; ++s) x[cmi(g, c.j + s * c.NY8, c.kx)] = xs[(size_t)s * nt];
  }
  if (live && blockIdx.x == 0 && t == 0) loop_finish(st, k, k.it - it0);
  loop_leave(st, room, live);
}

// Plain FP64 solve (fx64 transforms, row-major x and r).  A warp's instructions are what
// bounds a small grid here (64^2: one warp on each of 16 SMs, 8400 instructions an iteration),
// a third of their time the fetch of code that a lone warp runs through once.  So a thread
// carries one transform of 8 values at a time, and the iteration's four transforms are four
// turns of a loop around one copy of the code: forward ones all, an inverse one with real and
// imaginary parts exchanged before and after.  The two halves of the CTA take the two fields
// of the same columns, and share out the columns' values for everything else (half h owns
// slots 4 h .. 4 h + 3), which cross between them through ex.
__global__ void __launch_bounds__(256, 1) k_cg_loop_fx(Geo<fx64> g, cx<double>* x,
                                                        const cx<double>* r, cx<fx64>* Gx,
                                                        cx<fx64>* Gy, const fx64* mx,
                                                        const fx64* my, const fx64* rf,
                                                        SolveState* st, LoopRoom room) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (st->done) return;  // nothing writes it before every CTA has passed a barrier
  if (loop_gave_up(st) || st->loop_refused) return;
  using C = cx<fx64>;
  C* sm = reinterpret_cast<C*>(smem_raw);
  const int nt = blockDim.x, hn = nt >> 1, t = threadIdx.x, H = g.H;
  const int f = t >= hn ? 1 : 0, u = t - f * hn;  // field, thread within the half
  const int b = u & (g.tc - 1), j = u >> g.ltc, col = (blockIdx.x << g.ltc) + b;
  const int NY8 = 1 << (g.lny - 3), se = slab_elems(g);
  C* const cslab = sm + f * se + b;
  C* const G = f == 0 ? Gx : Gy;
  const int l8 = g.lnx - 3, N = g.nx, N8 = 1 << l8;
  const int rj = t & (N8 - 1), r0 = t >> l8;
  const size_t y0 = ((size_t)blockIdx.x << g.lrpc) + r0;
  C* const rslab = sm + (size_t)r0 * (N + N8);
  C* const Ra[1] = {Gx + y0 * H};
  C* const Rb[1] = {Gy + y0 * H};
  // behind the slabs (9 nt values): ex (slot s of thread u at s hn + u), then this CTA's rows
  // of mx, my, r
  C* const ex = sm + 9 * nt + u;
  fx64* sf = reinterpret_cast<fx64*>(sm + 13 * nt);
  {
    const size_t row0 = ((size_t)blockIdx.x << g.lrpc) * N;
    const int per = (int)(((size_t)g.rpc * N * sizeof(fx64)) >> 4);
    const fx64* const src[3] = {mx + row0, my + row0, rf + row0};
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      char* dst = reinterpret_cast<char*>(sf + (size_t)q * g.rpc * N);
      const char* from = reinterpret_cast<const char*>(src[q]);
      for (int i = t; i < per; i += nt) cp_async16(dst + 16 * i, from + 16 * i);
    }
    cp_async_commit();
  }
  const double n = (double)g.nx * (double)g.ny, invn = 1.0 / n, thresh2 = st->thresh2;
  const int maxit = st->maxit;
  LoopCg k{st->rho, st->rnorm2, 0.0, 0.0, st->it, 0, 0};
  const int it0 = k.it;
  LoopBar bar{&st->loop_bar, st->loop_polls};
  const double kx = g.kxd[col].v;
  const double w = col == 0 ? 1.0 : 2.0;  // Parseval weight of a packed column
  cx<double> xv[4], rv[4], dv[4];
  double pv[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const size_t e = (size_t)(j + (4 * f + i) * NY8) * H + col;
    xv[i] = x[e];
    rv[i] = r[e];
    dv[i] = cmk<double>(0.0, 0.0);
    pv[i] = g.pinv[e];
  }
  cp_async_wait_all();
  bool live = true;  // the launch has not been given up
  C v[1][8];
  int phase = 0;  // columns inverse, rows inverse, rows forward, columns forward
#pragma unroll 1
  while (true) {
    if (phase == 0) {
      // gradient of d = M^-1 r + beta d
      const bool first = k.it == it0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const cx<double> z = cmk<double>(rv[i].x * pv[i], rv[i].y * pv[i]);
        dv[i] = first ? z : cmk<double>(z.x + k.beta * dv[i].x, z.y + k.beta * dv[i].y);
        ex[(4 * f + i) * hn] = cmk<fx64>(dv[i].x, dv[i].y);
      }
      __syncthreads();
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        const C P = ex[s * hn];
        const fx64 a = (f == 0 ? kx : g.kyd[j + s * NY8].v) * invn;
        v[0][s] = cmk<fx64>(a * P.x, -a * P.y);  // i (k/n) P, exchanged
      }
    } else if (phase == 1) {
      load_rows_c2r<1>(v, (const C* const*)Ra, (const C* const*)Rb, rj, N8);
#pragma unroll
      for (int s = 0; s < 8; ++s) v[0][s] = cmk<fx64>(v[0][s].y, v[0][s].x);
    } else if (phase == 3) {
#pragma unroll
      for (int s = 0; s < 8; ++s) v[0][s] = G[(size_t)(j + s * NY8) * H + col];
    }
    const bool cols = phase == 0 || phase == 3;
    C* const sl[1] = {cols ? cslab : rslab};
    const int ks = cols ? 1 << g.ltc : 1, jt = cols ? j : rj, lN = cols ? g.lny : g.lnx;
    const C* const tw = cols ? g.twy : g.twx;
    const double share = phase == 3 ? dots_share(g.dots, gridDim.x) : 0.0;
    fxc fi[1][8];
    FxScale sc[1];
    if (lN >= kFxMinLog) {
      fx_run<-1, 1, false>(v, fi, sl, ks, jt, lN, tw, sc);
      if (phase != 2) {
        const FxOut o = fx_out(sc[0], lN, 0);
#pragma unroll
        for (int s = 0; s < 8; ++s) v[0][s] = cmk<fx64>(fx_to(fi[0][s].x, o.eb), fx_to(fi[0][s].y, o.eb));
        if (!o.plain) {
#pragma unroll
          for (int s = 0; s < 8; ++s)
            v[0][s] = cmk<fx64>(v[0][s].x.v * o.f1 * o.f2, v[0][s].y.v * o.f1 * o.f2);
        }
      }
    } else {
      fft_rt<-1, 1, false>(v, sl, ks, jt, lN, tw);
    }
    if (phase == 0) {
#pragma unroll
      for (int s = 0; s < 8; ++s)
        G[(size_t)(j + s * NY8) * H + col] = cmk<fx64>(v[0][s].y, v[0][s].x);
      live = bar.wait();
      if (!live) break;
      phase = 1;
    } else if (phase == 1) {
      // (m m + r I) grad d along the rows
      double gkg = 0.0;
      const fx64* smx = sf + (size_t)r0 * N;
      const fx64* smy = smx + (size_t)g.rpc * N;
      const fx64* srr = smy + (size_t)g.rpc * N;
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        const int xp = rj + s * N8;
        const fx64 gx = v[0][s].y, gy = v[0][s].x;
        const fx64 ax = smx[xp], ay = smy[xp], rr = srr[xp];
        const fx64 mg = ax * gx + ay * gy;
        gkg += (mg * mg + rr * (gx * gx + gy * gy)).v;
        v[0][s] = cmk<fx64>(ax * mg + rr * gx, ay * mg + rr * gy);
      }
      double a1[1] = {gkg};
      block_sum<1>(a1);
      if (t == 0) g.dots[blockIdx.x] = a1[0];
      phase = 2;
    } else if (phase == 2) {
      if (lN >= kFxMinLog) fx_store_r2c<1>(fi, sc, sl, rj, lN, Ra, Rb);
      else store_rows_r2c<1>(v, sl, rj, N, H, Ra, Rb);
      live = bar.wait();
      if (!live) break;
      phase = 3;
    } else {
      // A d = -div; x += alpha d, r -= alpha A d
#pragma unroll
      for (int s = 0; s < 8; ++s) {  // the other half's slots go to it
        const fx64 a = f == 0 ? kx : g.kyd[j + s * NY8].v;
        v[0][s] = cscale(v[0][s], a);
        if ((s >= 4) != (f == 1)) ex[s * hn] = v[0][s];
      }
      const double gkg = dots_total(share);  // its barriers also order ex
      if (!loop_alpha(k, gkg, n, 0, thresh2)) break;
      double acc[2] = {0.0, 0.0};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const C o = ex[(4 * f + i) * hn];
        const C own = f == 0 ? v[0][i] : v[0][4 + i];
        const double tx = own.x.v + o.x.v, ty = own.y.v + o.y.v;  // A d = (ty, -tx)
        xv[i] = cmk<double>(xv[i].x + k.alpha * dv[i].x, xv[i].y + k.alpha * dv[i].y);
        rv[i] = cmk<double>(rv[i].x - k.alpha * ty, rv[i].y + k.alpha * tx);
        const double r2 = rv[i].x * rv[i].x + rv[i].y * rv[i].y;
        acc[0] += r2;
        acc[1] += r2 * pv[i];
      }
      acc[0] *= w;
      acc[1] *= w;
      block_sum<2>(acc);
      if (t == 0) {
        g.partials[(size_t)blockIdx.x * kPartialStride] = acc[0];
        g.partials[(size_t)blockIdx.x * kPartialStride + 1] = acc[1];
      }
      live = bar.wait();
      if (!live) break;
      double tot[2];
      grid_total<2>(g.partials, kPartialStride, tot);
      loop_beta(k, tot[0], tot[1], thresh2, maxit);
      if (k.done) break;
      phase = 0;
    }
  }
  if (live) {
#pragma unroll
    for (int i = 0; i < 4; ++i) x[(size_t)(j + (4 * f + i) * NY8) * H + col] = xv[i];
  }
  if (live && blockIdx.x == 0 && t == 0) loop_finish(st, k, k.it - it0);
  loop_leave(st, room, live);
}

static inline size_t loop_smem(int nt, int rpc, int nx) {
  return (size_t)18 * nt * sizeof(cx<float>) + (size_t)3 * rpc * nx * sizeof(float) +
         (size_t)8 * nt * sizeof(cx<float>);
}

static inline size_t loop_smem_fx(int nt) {
  return (size_t)13 * nt * sizeof(cx<fx64>) + (size_t)24 * nt * sizeof(fx64);
}

// Threads of a CTA: `per` values each in either pass (FP32: 16, two fields or two rows; fx64:
// 8), enough of them for a column and for a row group, at most 128 CTAs, so that all are
// resident at one a SM.
static int loop_threads(int nx, int ny, int per) {
  const long long n = (long long)nx * ny;
  int nt = 32;
  while (nt < 2 * ny / per || nt < nx / 8 || n / (per * nt) > 128) nt *= 2;
  if (nt > 512 || n < (long long)per * nt) return 0;
  const int tc = per * nt / (2 * ny);
  return tc > 32 || tc > nx / 2 ? 0 : nt;
}

// The shape of a loop of `grid` CTAs, or none where this device cannot hold them all.
template <typename K>
static LoopShape loop_shape(K kernel, int nt, size_t smem, long long grid) {
  allow_smem(kernel);
  int dev = 0, sms = 0, coop = 0, per = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, nt, smem) != cudaSuccess) {
    cudaGetLastError();
    return LoopShape{};
  }
  if (!coop || per < 1) return LoopShape{};
  int k = 4;  // a CTA takes 2^k sixteenths of an SM
  while (k > 0 && per >= 2 << (4 - k)) --k;
  // a single CTA waits for nobody
  const LoopRoom room{grid > 1 ? (unsigned long long)grid << (k * kRoomBits) : 0ull, sms};
  return room_ok(room.need, sms) ? LoopShape{nt, room} : LoopShape{};
}

// Geometry of the loop's passes: per values a thread.
template <typename T>
static Geo<T> loop_geo(const Geo<T>& g0, int nt, int per) {
  Geo<T> g = g0;
  g.tc = per * nt / (2 * g.ny);
  g.rpc = per * nt / g.nx;
  for (g.ltc = 0; (1 << g.ltc) < g.tc;) ++g.ltc;
  for (g.lrpc = 0; (1 << g.lrpc) < g.rpc;) ++g.lrpc;
  return g;
}

bool cg_loop_shares(const LoopShape& sh) { return room_ok(2 * sh.room.need, sh.room.sms); }

LoopShape cg_loop_shape_f32(int nx, int ny) {
  const int nt = loop_threads(nx, ny, 16);
  if (!nt) return LoopShape{};
  const long long grid = (long long)nx * ny / (16 * nt);
  return loop_shape(nt <= 256 ? k_cg_loop_f32<256> : k_cg_loop_f32<512>, nt,
                    loop_smem(nt, 16 * nt / nx, nx), grid);
}
LoopShape cg_loop_shape_fx(int nx, int ny) {
  const int nt = loop_threads(nx, ny, 8);
  // 512 threads would have to fit 128 registers: 1024x512 108 us an iteration either way,
  // 32x2048 (16 CTAs) 110 -> 129
  if (!nt || nt > 256) return LoopShape{};
  return loop_shape(k_cg_loop_fx, nt, loop_smem_fx(nt), (long long)nx * ny / (8 * nt));
}

void cg_loop_f32(const Geo<float>& g0, const LoopShape& sh, cx<float>* x, const cx<float>* r,
                 cx<float>* Gx, cx<float>* Gy, const float* mx, const float* my, const float* rf,
                 SolveState* st, cudaStream_t s) {
  const int nt = sh.nt;
  Geo<float> g = loop_geo(g0, nt, 16);
  LoopRoom room = sh.room;
  int row_sums = g0.rpc < 2;
  void* args[] = {&g, &x, &r, &Gx, &Gy, &mx, &my, &rf, &st, &room, &row_sums};
  if (room.need) k_loop_claim<<<1, 1, 0, s>>>(st, room);
  cudaLaunchCooperativeKernel((const void*)(nt <= 256 ? k_cg_loop_f32<256> : k_cg_loop_f32<512>),
                              dim3(g.H >> g.ltc), dim3(nt), args, loop_smem(nt, g.rpc, g.nx), s);
}
void cg_loop_fx(const Geo<double>& g0, const LoopShape& sh, cx<double>* x, const cx<double>* r,
                cx<double>* Gx, cx<double>* Gy, const double* mx, const double* my,
                const double* rf, SolveState* st, cudaStream_t s) {
  Geo<fx64> g = loop_geo(as_fx(g0), sh.nt, 8);
  LoopRoom room = sh.room;
  void* args[] = {&g, &x, &r, &Gx, &Gy, &mx, &my, &rf, &st, &room};
  if (room.need) k_loop_claim<<<1, 1, 0, s>>>(st, room);
  cudaLaunchCooperativeKernel((const void*)k_cg_loop_fx, dim3(g.H >> g.ltc), dim3(sh.nt), args,
                              loop_smem_fx(sh.nt), s);
}

}  // namespace hc
