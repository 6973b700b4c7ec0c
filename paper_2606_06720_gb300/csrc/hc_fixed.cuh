// hc_fixed.cuh -- the FP64 transforms' arithmetic on the integer pipes (fx64).
//
// Why.  GB300 issues FP64 at 1/64 of its FP32 rate (measured: 1.5-1.8 lanes per
// clock and SM for an FMA or a conversion), while 32-bit additions run at 128 and
// 32 x 32 + 64-bit multiply-adds at 64 lanes.  So a transform of FP64 data is
// computed in 64-bit block fixed point: find the L2 norm of the transform's
// input, scale it to 2^61, run the Stockham passes on 64-bit integers, convert
// back to FP64.  Per point and pass that is about 70 integer instructions where
// the FP64 transform had 9 FP64 ones.
//
// Range.  A radix-8 pass multiplies the vector's L2 norm by sqrt(8) and every
// twiddled pass begins by dividing by 4, so with ||input||_2 <= 2^61 no modulus
// exceeds 2^62.5 (sqrt(8) 2^61 after the first pass, less after the others; the
// partial sums inside a butterfly obey the same Cauchy-Schwarz bound) and no
// component overflows 63 bits.
//
// Accuracy.  A pass rounds to about one unit, and the outputs' root mean square
// is 2^54 units or more, so the passes add a few 2^-55 to the relative L2 error;
// the rounding to FP64 at the end (2^-54) dominates.  Measured against long
// double over 64 .. 4096 points, white, smooth, sparse and 10^15-range inputs: a
// 2D transform is off by 0.5-1.4e-16 where the FP64 passes were off by
// 1.1-2.9e-16, and no output is further off than before.  As an FP64 transform's,
// the error is relative to the transform's norm, not to each element.
//
// Measured (GB300, us per launch, FP64 passes -> these): residual of 2048^2,
// gradient 309 -> 113, row pass 672 -> 187, divergence 367 -> 178; 256^3, z
// gradient 1339 -> 374, y 1258 -> 327, row pairs 3040 -> 1077, z divergence
// 1576 -> 526; plain FP64 CG iteration of 1024^2, 417 -> 214.  What bounds them
// now is instruction issue at 24 warps per SM (1.6-1.9 of 4 per clock) and, in
// the row and divergence passes, the FP64 pipe (half busy with the pointwise
// part).
#pragma once

#include "hc_internal.cuh"

namespace hc {

struct alignas(16) fxc {
  long long x, y;
};

__device__ __forceinline__ fxc fadd(fxc a, fxc b) { return fxc{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ fxc fsub(fxc a, fxc b) { return fxc{a.x - b.x, a.y - b.y}; }
template <int S>
__device__ __forceinline__ fxc fmul_si(fxc a) {  // a * (S i)
  return S > 0 ? fxc{-a.y, a.x} : fxc{a.y, -a.x};
}
// a b (+ c), one multiply-add.
__device__ __forceinline__ long long mul32(int a, int b) {
  long long d;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ long long mad32(int a, int b, long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}
// acc + (cr + k) / 2^32: the carry out of cr's low word rounds.
__device__ __forceinline__ long long add_upper(long long acc, long long cr, unsigned k) {
  unsigned lo, hi, drop;
  const int ch = (int)(cr >> 32);
  asm("{\n\tadd.cc.u32 %2, %3, %4;\n\taddc.cc.u32 %0, %5, %6;\n\taddc.u32 %1, %7, %8;\n\t}"
      : "=r"(lo), "=r"(hi), "=r"(drop)
      : "r"((unsigned)cr), "r"(k), "r"((unsigned)acc), "r"(ch), "r"((unsigned)(acc >> 32)),
        "r"(ch >> 31));
  return (long long)(((unsigned long long)hi << 32) | lo);
}

// v w / 4 for a twiddle w (Q62): the high-limb products and the upper half of
// the cross products, rounded; the dropped low-limb product is below one unit.
struct FxW {  // w with the signs that a direction needs: re = x wx + y ny, im = x py + y wx
  int xh, xl, ph, pl, nh, nl;
};
template <int S>
__device__ __forceinline__ FxW fx_w(const FxTw* __restrict__ tw, int m) {
  const int4 t = __ldg(reinterpret_cast<const int4*>(tw + m));
  FxW w;
  w.xh = t.x;
  w.xl = t.y;
  if (S < 0) {
    w.ph = t.z;
    w.pl = t.w;
    w.nh = -t.z;
    w.nl = -t.w;
  } else {
    w.ph = -t.z;
    w.pl = -t.w;
    w.nh = t.z;
    w.nl = t.w;
  }
  return w;
}
// The rounding constant is 2^31 or one less by a bit of the data: with w = 1 the
// quotients v / 4 end in .5 a quarter of the time, and always rounding them up
// would add up over the terms of a zero-frequency output.
__device__ __forceinline__ fxc fmul(fxc v, const FxW& w) {
  const int vxl = (int)v.x, vyl = (int)v.y;
  const unsigned bx = (unsigned)vxl >> 31, by = (unsigned)vyl >> 31;
  const int vxh = (int)(v.x >> 32) + (int)bx;
  const int vyh = (int)(v.y >> 32) + (int)by;
  const long long cr =
      mad32(vyl, w.nh, mad32(vyh, w.nl, mad32(vxl, w.xh, mul32(vxh, w.xl))));
  const long long ci =
      mad32(vyl, w.xh, mad32(vyh, w.xl, mad32(vxl, w.ph, mul32(vxh, w.pl))));
  fxc r;
  r.x = add_upper(mad32(vyh, w.nh, mul32(vxh, w.xh)), cr, 0x7fffffffu + bx);
  r.y = add_upper(mad32(vyh, w.xh, mul32(vxh, w.ph)), ci, 0x7fffffffu + by);
  return r;
}
__device__ __forceinline__ long long fquarter1(long long v) {
  return (v + (long long)(1u + ((unsigned)v >> 31))) >> 2;
}
__device__ __forceinline__ fxc fquarter(fxc v) { return fxc{fquarter1(v.x), fquarter1(v.y)}; }

// t / sqrt(2): 2^63 / sqrt(2) = 2^32 * 0x5A82799A - 0x0310CDBE; the rounding
// constant holds the mean of the dropped low product as well.
__device__ __forceinline__ long long fhalf_sqrt(long long t) {
  const int th = (int)(t >> 32);
  const unsigned tl = (unsigned)t;
  long long cross;
  asm("mad.wide.u32 %0, %1, %2, %3;"
      : "=l"(cross)
      : "r"(tl), "r"(0x5A82799Au), "l"(0x40000000LL - 0x018866DF));
  cross = mad32(th, -0x0310CDBE, cross);
  return (mul32(th, 0x5A82799A) << 1) + (cross >> 31);
}

template <int S>
__device__ __forceinline__ void fdft4(fxc& a0, fxc& a1, fxc& a2, fxc& a3) {
  const fxc t0 = fadd(a0, a2), t1 = fsub(a0, a2), t2 = fadd(a1, a3);
  const fxc t3 = fmul_si<S>(fsub(a1, a3));
  a0 = fadd(t0, t2);
  a2 = fsub(t0, t2);
  a1 = fadd(t1, t3);
  a3 = fsub(t1, t3);
}
template <int S>
__device__ __forceinline__ void fdft8(fxc* v) {
  fxc e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
  fxc o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  fdft4<S>(e0, e1, e2, e3);
  fdft4<S>(o0, o1, o2, o3);
  if constexpr (S < 0) {
    o1 = fxc{fhalf_sqrt(o1.x + o1.y), fhalf_sqrt(o1.y - o1.x)};
    o3 = fxc{fhalf_sqrt(o3.y - o3.x), -fhalf_sqrt(o3.x + o3.y)};
  } else {
    o1 = fxc{fhalf_sqrt(o1.x - o1.y), fhalf_sqrt(o1.y + o1.x)};
    o3 = fxc{-fhalf_sqrt(o3.x + o3.y), fhalf_sqrt(o3.x - o3.y)};
  }
  o2 = fmul_si<S>(o2);
  v[0] = fadd(e0, o0);
  v[4] = fsub(e0, o0);
  v[1] = fadd(e1, o1);
  v[5] = fsub(e1, o1);
  v[2] = fadd(e2, o2);
  v[6] = fsub(e2, o2);
  v[3] = fadd(e3, o3);
  v[7] = fsub(e3, o3);
}

// ------------------------------------------------------------------ conversions
// Scale of one transform: the input's integers are x 2^(61 - e), e the least
// integer (or one more) with ||x||_2 <= 2^e.
struct FxScale {
  int e;
  bool bad;    // the input holds an infinity or a NaN: so does every output
  bool small;  // the input's exponents are near the bottom of FP64: x 2^512 is transformed
};

// A finite double as an integer, truncated: x 2^(61 - e); b20 = (1024 + e) 2^20 +
// 2^20 - 1, from which subtracting the exponent and mantissa bits leaves the
// shift in the upper bits.
__device__ __forceinline__ long long fx_from(double x, int b20) {
  const int h = __double2hiint(x);
  const unsigned l = (unsigned)__double2loint(x);
  const int rs = min((b20 - (h & 0x7fffffff)) >> 20, 63);
  const unsigned mh = ((unsigned)h & 0xfffffu) | 0x100000u;
  const unsigned long long m =
      (((unsigned long long)__funnelshift_l(l, mh, 10) << 32) | (l << 10)) >> rs;
  return h < 0 ? -(long long)m : (long long)m;
}

// v 2^(eb - 1085) rounded to FP64; eb in [64, 2046].  The leading zeros come
// from the exponent of the upper word as a float (64 lanes per clock against
// 16 for a count); only a value below 2^32 needs the count.
__device__ __forceinline__ double fx_to(long long v, int eb) {
  const int s = (int)(v >> 32);
  unsigned long long a = (unsigned long long)(v < 0 ? -v : v);
  unsigned ah = (unsigned)(a >> 32);
  if (ah == 0) {
    if (a == 0) return 0.0;
    const int up = __clz((int)(unsigned)a) + 31;  // bring the top bit to 62
    a <<= up;
    ah = (unsigned)(a >> 32);
    eb -= up;
  }
  const int f = __float_as_int(__uint2float_rz(ah)) >> 23;  // 127 + position of the top bit
  const int n1 = 157 - f;                                   // leading zeros of a, less one
  const unsigned long long m = ((a << n1) + 0x200ULL) >> 10;  // 2^52 .. 2^53
  const int hi = (int)(m >> 32) + ((f + eb - 158) << 20);
  return __hiloint2double(hi | (s & (int)0x80000000), (int)(unsigned)m);
}

// acc + (x 2^(1023 - E))^2 with off20 = (E - 127) 2^20, |x| 2^(1023 - E) < 2.
__device__ __forceinline__ float fx_sumsq(float acc, double x, int off20) {
  const int t = max((__double2hiint(x) & 0x7fffffff) - off20, 0);
  const float f = __uint_as_float(__funnelshift_l((unsigned)__double2loint(x), (unsigned)t, 3));
  return fmaf(f, f, acc);
}
// Merge a partial (largest upper word, sum of squares relative to its exponent).
__device__ __forceinline__ void fx_merge(int& em, float& a, int2 p) {
  const int d = (em >> 20) - (p.x >> 20);  // bring both sums to the larger exponent
  const float f = __int_as_float(max(127 - 2 * abs(d), 0) << 23);
  a = d < 0 ? a * f + __int_as_float(p.y) : a + __int_as_float(p.y) * f;
  em = max(em, p.x);
}
// S < 2^(k+1), k its exponent, so ||x|| < 2^(E - 1023 + (k + 2) / 2); the factor
// covers the float sum's rounding.
__device__ __forceinline__ FxScale fx_scale_of(int em, float a) {
  const int k = (__float_as_int(a * 1.001f) >> 23) - 127, e = em >> 20;
  FxScale sc;
  sc.bad = e == 2047;
  sc.small = e < 160;
  sc.e = em == 0 ? 0 : e - 1023 + ((k + 2) >> 1) + (sc.small ? 512 : 0);
  return sc;
}

// The scales of NV transforms: one per lane group.  Lanes of a transform are
// `ks` apart within a warp, min(32 / ks, N/8) of them, and its warps follow one
// another; the warps' partial maxima and sums meet in the transform's slab.
template <int NV>
__device__ __forceinline__ void fx_scales(const cx<fx64> (&v)[NV][8], cx<fx64>* const* sl,
                                          int ks, int j, int lN, FxScale (&sc)[NV]) {
  const int N8 = 1 << (lN - 3);
  const unsigned mask = blockDim.x >= 32 ? 0xffffffffu : (1u << blockDim.x) - 1u;
  const int top = min(32, N8 * ks);  // lane offsets ks .. top/2
  const int nw = (N8 * ks) >> 5;     // warps of a transform (0, 1: a single one)
  int E[NV];
  float S[NV];
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    int e = 0;
#pragma unroll
    for (int s = 0; s < 8; ++s)
      e = max(e, max(__double2hiint(v[q][s].x.v) & 0x7fffffff, __double2hiint(v[q][s].y.v) & 0x7fffffff));
    for (int off = ks; off < top; off <<= 1) e = max(e, __shfl_xor_sync(mask, e, off));
    E[q] = e;
    const int off20 = ((e >> 20) - 127) << 20;
    float a = 0.0f;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      a = fx_sumsq(a, v[q][s].x.v, off20);
      a = fx_sumsq(a, v[q][s].y.v, off20);
    }
    for (int off = ks; off < top; off <<= 1) a += __shfl_xor_sync(mask, a, off);
    S[q] = a;
  }
  if (nw > 1) {  // uniform: every transform of a CTA has the same length
    const int w = (j * ks) >> 5;
    __syncthreads();
    if (((j * ks) & 31) == 0) {
#pragma unroll
      for (int q = 0; q < NV; ++q) {
        int2* p = reinterpret_cast<int2*>(sl[q] + (size_t)w * ks);
        *p = make_int2(E[q], __float_as_int(S[q]));
      }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      int em = 0;
      float a = 0.0f;
      for (int i = 0; i < nw; ++i)
        fx_merge(em, a, *reinterpret_cast<const int2*>(sl[q] + (size_t)i * ks));
      E[q] = em;
      S[q] = a;
    }
  }
#pragma unroll
  for (int q = 0; q < NV; ++q) sc[q] = fx_scale_of(E[q], S[q]);
}

// ------------------------------------------------------------------ the passes
// As fft_rt, on integers; every twiddled pass divides by 4.
template <int S, int NV, bool SWZ>
__device__ __forceinline__ void fx_passes(fxc (&v)[NV][8], fxc* const* sl, int ks, int j, int lN,
                                          const FxTw* __restrict__ tw) {
  const int N8 = 1 << (lN - 3);
  const int jslot = slot_base<fx64, SWZ>(j, ks);
  int lNs = 0, rem = lN;
#pragma unroll 1
  while (rem >= 3) {
    const int k = j & ((1 << lNs) - 1);
    if (lNs > 0) {
      const int step = k << (lN - 3 - lNs);
#pragma unroll
      for (int q = 0; q < NV; ++q) v[q][0] = fquarter(v[q][0]);
#pragma unroll
      for (int r = 1; r < 8; ++r) {
        const FxW w = fx_w<S>(tw, r * step);
#pragma unroll
        for (int q = 0; q < NV; ++q) v[q][r] = fmul(v[q][r], w);
      }
    }
#pragma unroll
    for (int q = 0; q < NV; ++q) fdft8<S>(v[q]);
    if (rem == 3) return;
    const int bslot = slot_base<fx64, SWZ>(((j >> lNs) << (lNs + 3)) + k, ks);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int e = slot_plus<fx64, SWZ>(bslot, r << lNs, ks);
#pragma unroll
      for (int q = 0; q < NV; ++q) sl[q][e] = v[q][r];
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const int e = slot_plus<fx64, SWZ>(jslot, s * N8, ks);
#pragma unroll
      for (int q = 0; q < NV; ++q) v[q][s] = sl[q][e];
    }
    lNs += 3;
    rem -= 3;
  }
  if (rem == 2) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int step = ((j + u * N8) & ((1 << lNs) - 1)) << (lN - 2 - lNs);
#pragma unroll
      for (int q = 0; q < NV; ++q) v[q][u] = fquarter(v[q][u]);
#pragma unroll
      for (int r = 1; r < 4; ++r) {
        const FxW w = fx_w<S>(tw, r * step);
#pragma unroll
        for (int q = 0; q < NV; ++q) v[q][u + 2 * r] = fmul(v[q][u + 2 * r], w);
      }
#pragma unroll
      for (int q = 0; q < NV; ++q) fdft4<S>(v[q][u], v[q][u + 2], v[q][u + 4], v[q][u + 6]);
    }
  } else {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int k = (j + u * N8) & ((1 << lNs) - 1);
      const FxW w = fx_w<S>(tw, k << (lN - 1 - lNs));
#pragma unroll
      for (int q = 0; q < NV; ++q) {
        const fxc a = fquarter(v[q][u]), b = fmul(v[q][u + 4], w);
        v[q][u] = fadd(a, b);
        v[q][u + 4] = fsub(a, b);
      }
    }
  }
}

// Inputs to integers (v is consumed) and the passes; sc receives the scales.
template <int S, int NV, bool SWZ>
__device__ __forceinline__ void fx_run(cx<fx64> (&v)[NV][8], fxc (&f)[NV][8],
                                           cx<fx64>* const* sl, int ks, int j, int lN,
                                           const cx<fx64>* __restrict__ tw, FxScale (&sc)[NV]) {
  fx_scales<NV>(v, sl, ks, j, lN, sc);
  fxc* fs[NV];
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    fs[q] = reinterpret_cast<fxc*>(sl[q]);
    if (sc[q].small) {
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        v[q][s].x *= fx64(0x1p512);
        v[q][s].y *= fx64(0x1p512);
      }
    }
    const int b20 = ((1024 + sc[q].e) << 20) + 0xfffff;
#pragma unroll
    for (int s = 0; s < 8; ++s) f[q][s] = fxc{fx_from(v[q][s].x.v, b20), fx_from(v[q][s].y.v, b20)};
  }
  fx_passes<S, NV, SWZ>(f, fs, ks, j, lN, reinterpret_cast<const FxTw*>(tw));
}

// How a transform's integers go back to FP64, times 2^-half: by fx_to at eb
// alone, or (inputs at the ends of FP64's range or not finite) by two factors more.
struct FxOut {
  int eb;
  bool plain;
  double f1, f2;
};
__device__ __forceinline__ double fx_pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }
// Integers v stand for v 2^(eb - 1085).
__device__ __forceinline__ FxOut fx_out_at(const FxScale& sc, int eb) {
  FxOut o;
  o.eb = eb;
  o.plain = !sc.bad && !sc.small && o.eb <= 2045;
  o.f1 = o.f2 = 1.0;
  if (!o.plain) {
    const int ex = o.eb - 1085 - (sc.small ? 512 : 0);
    o.eb = 1085;
    o.f1 = sc.bad ? __longlong_as_double(0x7ff8000000000000LL) : fx_pow2(ex / 2);
    o.f2 = fx_pow2(ex - ex / 2);
  }
  return o;
}
__device__ __forceinline__ FxOut fx_out(const FxScale& sc, int lN, int half) {
  return fx_out_at(sc, 1024 + sc.e + 2 * (lN > 9 ? 3 : (lN > 6 ? 2 : 1)) - half);
}

// fft_canon for FP64 data of length 2^lN, lN >= kFxMinLog.
template <int S, int NV, bool SWZ>
__device__ __forceinline__ void fft_fixed(cx<fx64> (&v)[NV][8], cx<fx64>* const* sl, int ks,
                                          int j, int lN, const cx<fx64>* __restrict__ tw) {
  FxScale sc[NV];
  fxc f[NV][8];
  fx_run<S, NV, SWZ>(v, f, sl, ks, j, lN, tw, sc);
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    const FxOut o = fx_out(sc[q], lN, 0);
#pragma unroll
    for (int s = 0; s < 8; ++s)
      v[q][s] = cmk<fx64>(fx_to(f[q][s].x, o.eb), fx_to(f[q][s].y, o.eb));
    if (!o.plain) {
#pragma unroll
      for (int s = 0; s < 8; ++s)
        v[q][s] = cmk<fx64>(v[q][s].x.v * o.f1 * o.f2, v[q][s].y.v * o.f1 * o.f2);
    }
  }
}

// Forward transform of NV rows a + i b and their packed half spectra
// (store_rows_r2c), the separation on the integers: halving is a change of
// exponent and the sums stay off the FP64 pipe.  (Two outputs of one transform
// have a joint modulus within the vector's norm, so their sum fits as well.)
template <int NV>
__device__ __forceinline__ void fx_store_r2c(const fxc (&f)[NV][8], const FxScale (&sc)[NV],
                                             cx<fx64>* const* sl, int j, int lN, cx<fx64>* const* A,
                                             cx<fx64>* const* B) {
  const int N = 1 << lN, N8 = N >> 3, H = N >> 1;
  __syncthreads();
#pragma unroll
  for (int s = 0; s < 8; ++s)
#pragma unroll
    for (int q = 0; q < NV; ++q)
      reinterpret_cast<fxc*>(sl[q])[rswz<fx64>(j + s * N8)] = f[q][s];
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    const fxc* slab = reinterpret_cast<const fxc*>(sl[q]);
    const FxOut o = fx_out(sc[q], lN, 1);
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      const int k = j + s * N8;  // k < H
      const fxc z = slab[rswz<fx64>(k)], zc = slab[rswz<fx64>(k == 0 ? H : N - k)];
      fxc a = fxc{z.x + zc.x, z.y - zc.y}, b = fxc{z.y + zc.y, zc.x - z.x};
      int eb = o.eb;
      if (k == 0) {  // the two real columns: no sums, not halved
        a = fxc{z.x, zc.x};
        b = fxc{z.y, zc.y};
        ++eb;
      }
      cx<fx64> ad = cmk<fx64>(fx_to(a.x, eb), fx_to(a.y, eb));
      cx<fx64> bd = cmk<fx64>(fx_to(b.x, eb), fx_to(b.y, eb));
      if (!o.plain) {
        ad = cmk<fx64>(ad.x.v * o.f1 * o.f2, ad.y.v * o.f1 * o.f2);
        bd = cmk<fx64>(bd.x.v * o.f1 * o.f2, bd.y.v * o.f1 * o.f2);
      }
      A[q][k] = ad;
      if (B[q]) B[q][k] = bd;
    }
  }
}
template <int NV>
__device__ __forceinline__ void fft_fixed_r2c(cx<fx64> (&v)[NV][8], cx<fx64>* const* sl, int j,
                                              int lN, const cx<fx64>* __restrict__ tw,
                                              cx<fx64>* const* A, cx<fx64>* const* B) {
  FxScale sc[NV];
  fxc f[NV][8];
  fx_run<-1, NV, true>(v, f, sl, 1, j, lN, tw, sc);
  fx_store_r2c<NV>(f, sc, sl, j, lN, A, B);
}

}  // namespace hc
