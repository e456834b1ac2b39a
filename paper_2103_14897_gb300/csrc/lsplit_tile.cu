// Deterministic compact-kernel steps on two-dimensional tiles.
//
// In the interaction frame (state psi~ = K(-t) psi) a layer factor with a
// compact kernel only adds, to every element, a few neighbours along one axis:
//   y_m = x_m + sum_{0 < |d| <= BV} c_d e^{2 pi i t (kappa(m) - kappa(m - d))} x_{m-d}.
// So several consecutive factors of a call, of both layers, act on a 2D tile
// of the lifted array that is loaded once with a halo: BV columns per layer-1
// factor and BV rows per layer-2 factor on each side.  A pass reads one array
// and writes another (tiles overlap in their halos), and the passes of a call
// alternate between the caller's array and a second one.
//
// Wrapped halo elements keep the frame of their true index j mod q.  The phase
// of a pair factorises over the tile, kappa(m, n) = A m^2 + X m n + C n^2:
//   t (kappa(m) - kappa(m')) = t A (m^2 - m'^2)  +  t X n (m - m'),
// a table U_d over the axis (with the tap c_d) times V_n^d over the other
// axis, both small tables per tile and factor; where the pair straddles the
// end of the box, m - m' = d - q w and the neighbour carries V_n^{-q w} too.
//
// What it is for.  complex64: boxes whose in-place passes are bound by their
// launches; a pass of 3 or 4 factors on 32 x 32 tiles takes about 5 us, where
// each factor's launch takes 3 to 5 us (401 x 129, 50 Lie steps: 430 -> 170 us;
// 20 Strang steps against in place: 257 x 257 113 / 172 us, 513 x 513 191 / 238 us).  complex128: every box (2049 x
// 2049, 4 Strang steps: 6.56 -> 1.62 ms, at 67 % issue, about 670 instructions
// per element of a tile's extent and factor; 65 x 65, 100 steps: 20.8 -> 1.30 ms,
// on 16 x 16 tiles so that the box spreads over the SMs).
//
// Sweep: a thread owns one line (row for layer 1, column for layer 2; lanes
// take adjacent lines, the odd row pitch makes both free of bank conflicts)
// and SEG consecutive elements of it, walked with a sliding window of 2 BV + 1
// old values in registers: 1 + 2 BV / SEG shared loads and one store per
// element instead of 2 BV + 1 loads, in place, two barriers per factor.
//
// complex64: 16 FMAs per tap pair and element, no phase evaluation in the
// sweep; a thread takes two lines in the two lanes of paired FP32 operations
// (real and imaginary parts in separate planes, the table entries doubled), so
// that the FMA pipe and not the issue slots bounds it.  complex128: the FP64 pipe
// of sm_103a runs at 1/64 of the FP32 rate, so only x + correction is formed in
// FP64 (two additions per component, the rounding of the plain form); the
// correction, at most 2^-7 of its neighbours, is formed in pairs of floats (about
// 2^-46 relative, 2^-53 and less of the neighbours) on the FP32 pipe, the taps
// |d| >= 3 (at most 2^-30) in single floats.  The pairs are scaled by the tile's
// largest exponent, so the whole FP64 range is taken; neighbours below 2^-143 of
// the largest count as zero.  The kinetic phases turn the taps from factor to
// factor, so that their rounding does not add up: 33 x 25, Strang, error against
// 80-bit arithmetic with the same kinetic phases, in place in FP64 and here: 100
// steps 1.1e-14 and 1.3e-15, 1000 steps 1.1e-13 and 4.2e-15, 20000 steps 2.1e-12
// and 3.7e-14 (tau max v = 3.4e-3; 2.5e-12 and 1.3e-12 at 1e-3).
#include "lsplit_kernels.cuh"
#include "lsplit_pair.cuh"

namespace lsk {
namespace {

// ---------------------------------------------------------------- pairs of floats
struct CDF { DF x, y; };

// a b + c d (SUB: a b - c d)
template <bool SUB> __device__ __forceinline__ DF dot2(DF a, DF b, DF c, DF d) {
  const float ch = SUB ? -c.h : c.h, cl = SUB ? -c.l : c.l;
  const float p = __fmul_rn(a.h, b.h), q = __fmul_rn(ch, d.h);
  float e = __fadd_rn(fmaf(a.h, b.h, -p), fmaf(ch, d.h, -q));
  e = fmaf(a.h, b.l, e);
  e = fmaf(a.l, b.h, e);
  e = fmaf(ch, d.l, e);
  e = fmaf(cl, d.h, e);
  float s, r;
  two_sum(p, q, s, r);
  return quick(s, __fadd_rn(r, e));
}
__device__ __forceinline__ CDF mul(CDF a, CDF b) {
  return CDF{dot2<true>(a.x, b.x, a.y, b.y), dot2<false>(a.x, b.y, a.y, b.x)};
}
__device__ __forceinline__ CDF conj(CDF a) { return CDF{a.x, DF{-a.y.h, -a.y.l}}; }
// acc += a b (acc as an unnormalised high and low part)
__device__ __forceinline__ void mac1(DF& acc, DF a, DF b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, e);
  e = fmaf(a.l, b.h, e);
  float r;
  two_sum(acc.h, p, acc.h, r);
  acc.l = __fadd_rn(acc.l, __fadd_rn(r, e));
}
__device__ __forceinline__ void mac(CDF& acc, CDF a, CDF b) {
  mac1(acc.x, a.x, b.x);
  mac1(acc.x, DF{-a.y.h, -a.y.l}, b.y);
  mac1(acc.y, a.x, b.y);
  mac1(acc.y, a.y, b.x);
}
__device__ __forceinline__ CDF as_cdf(float4 v) { return CDF{DF{v.x, v.y}, DF{v.z, v.w}}; }
__device__ __forceinline__ float4 as_f4(CDF v) { return make_float4(v.x.h, v.x.l, v.y.h, v.y.l); }

// exp(2 pi i t / 2^64) as pairs of floats, about 2^-46: the nearest of 256
// directions from a table, the rest (|a| <= 2 pi / 512, exact integer split
// into 24 + 32 bits) by the Taylor series of sine and cosine.
__device__ __forceinline__ CDF cis_df(uint64_t t, const float4* __restrict__ tab) {
  const uint32_t j = (uint32_t)((t + (1ull << 55)) >> 56);
  const int64_t r = (int64_t)(t - ((uint64_t)j << 56));
  const float rh = (float)(int32_t)(r >> 32), rl = (float)(uint32_t)r * 0x1p-32f;
  // a = (rh + rl) 2 pi / 2^32, the constant as a pair
  constexpr float ph = 6.28318530717958647692f, pl = (float)(6.28318530717958647692 - (double)ph);
  const float a0 = __fmul_rn(rh, ph);
  float e = fmaf(rh, ph, -a0);
  e = fmaf(rh, pl, e);
  e = fmaf(rl, ph, e);
  DF a = quick(a0, e);
  a.h *= 0x1p-32f;
  a.l *= 0x1p-32f;
  const float q = __fmul_rn(a.h, a.h);
  const float qe = fmaf(2.0f * a.h, a.l, fmaf(a.h, a.h, -q));
  // sin a = a - a^3 / 6 + a^5 / 120, cos a = 1 - a^2 / 2 + a^4 / 24 - a^6 / 720
  const float s3 = __fmul_rn(__fmul_rn(a.h, q), fmaf(q, 1.0f / 120.0f, -1.0f / 6.0f));
  const DF sn = quick(a.h, __fadd_rn(a.l, s3));
  const float c4 = __fmul_rn(__fmul_rn(q, q), fmaf(q, -1.0f / 720.0f, 1.0f / 24.0f));
  const float hq = -0.5f * q;
  const float c0 = __fadd_rn(1.0f, hq);
  const float ce = __fsub_rn(hq, __fsub_rn(c0, 1.0f));
  const DF cs = quick(c0, __fadd_rn(ce, fmaf(-0.5f, qe, c4)));
  return mul(as_cdf(tab[j & 255]), CDF{cs, sn});
}

// exp(2 pi i t / 2^64) in FP64: the nearest of 1024 directions from a table,
// the rest (|a| <= pi / 1024) by the Taylor series (terms beyond a^5 and a^4
// are below 2e-18); 12 FP64 operations.
__device__ __forceinline__ double2 cis_d(uint64_t t, const double2* __restrict__ tab) {
  const uint32_t j = (uint32_t)((t + (1ull << 53)) >> 54);
  const int64_t r = (int64_t)(t - ((uint64_t)j << 54));
  const double a = (double)r * (6.28318530717958647692 * 0x1p-64);
  const double q = a * a;
  const double s = a * fma(q, fma(q, 1.0 / 120.0, -1.0 / 6.0), 1.0);
  const double c = fma(q, fma(q, 1.0 / 24.0, -0.5), 1.0);
  const double2 w = tab[j & 1023];
  return make_double2(fma(w.x, c, -w.y * s), fma(w.x, s, w.y * c));
}

// ---------------------------------------------------------------- arithmetic per type
template <typename Real, int BV> struct Ar;

template <int BV> struct Ar<double, BV> {
  using E = double2;
  using W = CDF;
  using V = CDF;
  static constexpr int kTabF4 = 4 + (BV > 2 ? BV - 2 : 0);
  struct Scale {
    int off;        // (largest exponent field - 167) << 20
    bool bad;       // the tile holds an infinity or a NaN
  };
  // float pair of a double, scaled by 2^(167 - 127 - largest exponent): the
  // top 24 bits of the significand and the next 23; elements below 2^-143 of
  // the largest are zero.  Integer operations only.
  static __device__ __forceinline__ DF split(double x, const Scale& sc) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const int h = (int)(hi & 0x7fffffffu) - sc.off;
    const uint32_t sg = hi & 0x80000000u;
    const bool ok = h >= (24 << 20);
    const uint32_t f = __funnelshift_l(lo, (uint32_t)h, 3);
    const uint32_t base = (f & 0x7f800000u) - (23u << 23);
    const float g = __fsub_rn(__uint_as_float(base | ((lo & 0x1fffffffu) >> 6)), __uint_as_float(base));
    DF r;
    r.h = __uint_as_float(ok ? (f | sg) : 0u);
    r.l = __uint_as_float(ok ? (__float_as_uint(g) ^ sg) : 0u);
    if (sc.bad && (hi & 0x7ff00000u) == 0x7ff00000u) r.h = __uint_as_float(0x7fc00000u);
    return r;
  }
  static __device__ __forceinline__ double widen(float f, const Scale& sc) {
    const uint32_t b = __float_as_uint(f), m = b & 0x7fffffffu;
    const int h = (int)(m >> 3) + sc.off;
    const bool ok = m >= 0x00800000u && h >= (1 << 20);
    return __hiloint2double(ok ? (int)((uint32_t)h | (b & 0x80000000u)) : 0, ok ? (int)(b << 29) : 0);
  }
  static __device__ __forceinline__ W load(const E& e, const Scale& sc) { return CDF{split(e.x, sc), split(e.y, sc)}; }
  static __device__ __forceinline__ V cis(uint64_t t, const float4* tab) { return cis_df(t, tab); }
  static __device__ __forceinline__ V conj_(V v) { return conj(v); }
  static __device__ __forceinline__ V mul_(V a, V b) { return mul(a, b); }
  static __device__ __forceinline__ W turn(W x, V v) { return mul(x, v); }
  static __device__ __forceinline__ void put(float4* u, int stride, int d, V p, V m, const float4* taps) {
    const CDF a = mul(as_cdf(taps[kTileMaxB + d]), p), b = mul(as_cdf(taps[kTileMaxB - d]), m);
    if (d <= 2) {
      u[(2 * d - 2) * stride] = as_f4(a);
      u[(2 * d - 1) * stride] = as_f4(b);
    } else {
      u[(d + 1) * stride] = make_float4(a.x.h, a.y.h, b.x.h, b.y.h);
    }
  }
  struct Lines {
    CDF v1, v2;
    float2 w[BV > 2 ? BV - 2 : 1];        // V^3 .. in single floats
  };
  static __device__ __forceinline__ void lines(Lines& L, V v) {
    L.v1 = v;
    L.v2 = mul(v, v);
    if constexpr (BV > 2) {
      float2 p = make_float2(L.v2.x.h, L.v2.y.h);
      const float2 q = make_float2(v.x.h, v.y.h);
#pragma unroll
      for (int d = 3; d <= BV; ++d) L.w[d - 3] = p = cmul(p, q);
    }
  }
  struct Acc {
    CDF a;
    float2 s;
  };
  static __device__ __forceinline__ void zero(Acc& a) {
    a.a = CDF{DF{0.f, 0.f}, DF{0.f, 0.f}};
    a.s = make_float2(0.f, 0.f);
  }
  template <int d>
  static __device__ __forceinline__ void tap(Acc& s, const float4* u, int stride, const Lines& L, W xm, W xp) {
    if constexpr (d <= 2) {
      const CDF v = d == 1 ? L.v1 : L.v2;
      mac(s.a, mul(as_cdf(u[(2 * d - 2) * stride]), v), xm);
      mac(s.a, mul(as_cdf(u[(2 * d - 1) * stride]), conj(v)), xp);
    } else {
      const float4 c = u[(d + 1) * stride];
      const float2 v = L.w[d - 3];
      const float wx = fmaf(c.x, v.x, -c.y * v.y), wy = fmaf(c.x, v.y, c.y * v.x);
      const float zx = fmaf(c.z, v.x, c.w * v.y), zy = fmaf(c.w, v.x, -c.z * v.y);
      s.s.x = fmaf(wx, xm.x.h, fmaf(-wy, xm.y.h, fmaf(zx, xp.x.h, fmaf(-zy, xp.y.h, s.s.x))));
      s.s.y = fmaf(wx, xm.y.h, fmaf(wy, xm.x.h, fmaf(zx, xp.y.h, fmaf(zy, xp.x.h, s.s.y))));
    }
  }
  static __device__ __forceinline__ double add(double x, DF c, float s, const Scale& sc) {
    const DF r = quick(c.h, __fadd_rn(c.l, s));
    const double y = x + (widen(r.h, sc) + widen(r.l, sc));
    return sc.bad && isnan(r.h) ? __hiloint2double(0x7ff80000, 0) : y;
  }
  static __device__ __forceinline__ E finish(const E& x, const W&, const Acc& s, const Scale& sc) {
    return make_double2(add(x.x, s.a.x, s.s.x, sc), add(x.y, s.a.y, s.s.y, sc));
  }
};

template <int BV> struct TapLoop {
  template <class A>
  static __device__ __forceinline__ void run(typename A::Acc& s, const float4* u, int stride,
                                             const typename A::Lines& L, const typename A::W* win) {
    // the smallest taps first
    if constexpr (BV >= 5) A::template tap<5>(s, u, stride, L, win[BV - 5], win[BV + 5]);
    if constexpr (BV >= 4) A::template tap<4>(s, u, stride, L, win[BV - 4], win[BV + 4]);
    if constexpr (BV >= 3) A::template tap<3>(s, u, stride, L, win[BV - 3], win[BV + 3]);
    if constexpr (BV >= 2) A::template tap<2>(s, u, stride, L, win[BV - 2], win[BV + 2]);
    A::template tap<1>(s, u, stride, L, win[BV - 1], win[BV + 1]);
  }
};

// wrap count floor(a / q); tile extents reach past a box end by a few turns at most
__device__ __forceinline__ int wraps(int a, int q) {
  int w = 0;
  while (a < 0) {
    a += q;
    --w;
  }
  while (a >= q) {
    a -= q;
    ++w;
  }
  return w;
}

// The tile of this CTA: result rows [r0, r0 + vr) and columns
// [c0, c0 + vc), extents re x ce with the halos.
struct TileGeo {
  const TileInst* in;
  int M1, M2, hr, hc, r0, c0, vr, vc, re, ce;
  __device__ __forceinline__ explicit TileGeo(const TileArgs& a) {
    in = &a.one;
    const int tile = blockIdx.x;
    M1 = in->M1;
    M2 = in->M2;
    hr = a.hr;
    hc = a.hc;
    const int ntc = (M1 + a.tc - 1) / a.tc;
    r0 = (tile / ntc) * a.tr;
    c0 = (tile % ntc) * a.tc;
    vr = min(a.tr, M2 - r0);
    vc = min(a.tc, M1 - c0);
    re = vr + 2 * hr;
    ce = vc + 2 * hc;
  }
};

// What one factor needs of the tile: own axis (na positions from oa, length
// qa, first signed index la), other axis likewise, t A and t X.
struct FactorGeo {
  bool l1;
  int na, nb, oa, ob, qa, qb, la, lb;
  uint64_t tA, tX;
  const float4* taps;
  __device__ __forceinline__ FactorGeo(const TileArgs& a, const TileGeo& g, int f) {
    l1 = a.layer[f] == 1;
    const TileInst& in = *g.in;
    const uint64_t t = (uint64_t)a.t[f];
    tA = t * (l1 ? in.A1 : in.A2);
    tX = t * in.X;
    na = l1 ? g.ce : g.re;
    nb = l1 ? g.re : g.ce;
    oa = l1 ? g.c0 - g.hc : g.r0 - g.hr;
    ob = l1 ? g.r0 - g.hr : g.c0 - g.hc;
    qa = l1 ? g.M1 : g.M2;
    qb = l1 ? g.M2 : g.M1;
    la = l1 ? in.lo1 : in.lo2;
    lb = l1 ? in.lo2 : in.lo1;
    taps = in.taps[l1 ? 0 : 1];
  }
  // true signed indices of extent positions
  __device__ __forceinline__ int64_t own(int k) const { return (int64_t)la + (oa + k - wraps(oa + k, qa) * qa); }
  __device__ __forceinline__ int64_t other(int k) const { return (int64_t)lb + (ob + k - wraps(ob + k, qb) * qb); }
};

// Shared-memory layout of a tile: BV spare rows and columns on every side (the
// sweeps run over the whole extent; what they read there only reaches elements
// outside the tile's result), an odd row pitch.
template <int BV, int RE, int CE> struct TileShape {
  static constexpr int kPitch = (CE + 2 * BV) | 1;
  static constexpr int kElems = (RE + 2 * BV) * kPitch;
  static constexpr int kAxis = RE > CE ? RE : CE;   // table stride
};

// One factor along an axis: `sp` is the thread's first element, `step` the
// distance of neighbours, `u` the table at that element.
template <class A, int BV, int SEG, int STRIDE>
__device__ __forceinline__ void sweep(typename A::E* sp, int step, const float4* u, typename A::V v, bool active,
                                      bool seam, const signed char* om, typename A::V vq,
                                      const typename A::Scale& sc) {
  typename A::W win[2 * BV + 1];
  typename A::E rb[BV];
  if (active) {
#pragma unroll
    for (int k = 0; k < 2 * BV; ++k) win[k] = A::load(sp[(k - BV) * step], sc);
#pragma unroll
    for (int k = 0; k < BV; ++k) rb[k] = sp[(SEG + k) * step];
  }
  __syncthreads();
  if (active) {
    typename A::Lines L;
    A::lines(L, v);
    if (!seam) {
      // (not unrolled: the body is some 600 instructions)
#pragma unroll 1
      for (int i = 0; i < SEG; ++i) {
        typename A::E nx = sp[(i + BV) * step];
        if (i + BV >= SEG) {   // the next thread's segment
          nx = rb[SEG < BV ? BV - SEG : 0];
#pragma unroll
          for (int k = 0; k + 1 < BV; ++k) rb[k] = rb[k + 1];
        }
        win[2 * BV] = A::load(nx, sc);
        typename A::Acc s;
        A::zero(s);
        TapLoop<BV>::template run<A>(s, u + i, STRIDE, L, win);
        sp[i * step] = A::finish(sp[i * step], win[BV], s, sc);
#pragma unroll
        for (int k = 0; k < 2 * BV; ++k) win[k] = win[k + 1];
      }
    } else {
      // pairs that straddle the end of the box: the neighbour times V_n^{-q w}
      const typename A::V vc = A::conj_(vq);
#pragma unroll 1
      for (int i = 0; i < SEG; ++i) {
        typename A::E nx = sp[(i + BV) * step];
        if (i + BV >= SEG) {   // the next thread's segment
          nx = rb[SEG < BV ? BV - SEG : 0];
#pragma unroll
          for (int k = 0; k + 1 < BV; ++k) rb[k] = rb[k + 1];
        }
        win[2 * BV] = A::load(nx, sc);
        typename A::W t[2 * BV + 1];
        const int o = om[i];
#pragma unroll
        for (int k = 0; k <= 2 * BV; ++k) {
          const int w = o - om[i + k - BV];
          t[k] = win[k];
          if (w != 0) t[k] = A::turn(win[k], w > 0 ? vc : vq);
        }
        typename A::Acc s;
        A::zero(s);
        TapLoop<BV>::template run<A>(s, u + i, STRIDE, L, t);
        sp[i * step] = A::finish(sp[i * step], win[BV], s, sc);
#pragma unroll
        for (int k = 0; k < 2 * BV; ++k) win[k] = win[k + 1];
      }
    }
  }
  __syncthreads();
}

// ---------------------------------------------------------------- complex128
template <int BV, int RE, int CE, int SEG, int MINB>
__global__ void __launch_bounds__(RE * CE / SEG, MINB) tile_f64_kernel(const __grid_constant__ TileArgs a) {
  using A = Ar<double, BV>;
  using Sh = TileShape<BV, RE, CE>;
  constexpr int NT = RE * CE / SEG, NW = NT / 32, P = Sh::kPitch, AX = Sh::kAxis;
  static_assert(NT % 32 == 0 && CE % 16 == 0 && CE % SEG == 0 && RE % SEG == 0, "tile shape");
  extern __shared__ __align__(16) unsigned char smraw[];
  double2* x = reinterpret_cast<double2*>(smraw);
  float4* tu = reinterpret_cast<float4*>(x + Sh::kElems);
  float4* tv = tu + a.nf * A::kTabF4 * AX;
  __shared__ signed char s_om[2][AX + 2 * BV];
  __shared__ int s_red[NW];
  __shared__ float4 s_e[kTileMaxF][BV];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const TileGeo g(a);
  const TileInst& in = *g.in;
  const double2* src = reinterpret_cast<const double2*>(a.flip ? in.alt : in.psi);
  double2* dst = reinterpret_cast<double2*>(a.flip ? in.psi : in.alt);
  double2* xt = x + BV * P + BV;   // element (row 0, column 0) of the tile
  pass_begin();
  // ---- wrap counts of both axes, U and V tables of every factor
  for (int i = tid; i < 2 * (AX + 2 * BV); i += NT) {
    const int ax = i >= AX + 2 * BV ? 1 : 0, k = i - ax * (AX + 2 * BV) - BV;
    s_om[ax][k + BV] = (signed char)(ax ? wraps(g.r0 - g.hr + k, g.M2) : wraps(g.c0 - g.hc + k, g.M1));
  }
  if (tid < a.nf * BV) {
    const int f = tid / BV, d = tid % BV + 1;
    const uint64_t tA = (uint64_t)a.t[f] * (a.layer[f] == 1 ? in.A1 : in.A2);
    s_e[f][d - 1] = as_f4(cis_df((uint64_t)0 - tA * (uint64_t)(d * d), a.ctab));
  }
  __syncthreads();
  for (int i = tid; i < a.nf * 2 * AX; i += NT) {
    const int f = i / (2 * AX), k = i % AX;
    const FactorGeo q(a, g, f);
    if (i % (2 * AX) >= AX) {
      if (k < q.nb) tv[f * AX + k] = as_f4(cis_df(q.tX * (uint64_t)q.other(k), a.ctab));
    } else if (k < q.na) {
      // U_d = c_d e^{2 pi i t A (m^2 - m'^2)}: powers of w = e^{2 pi i t 2 A m}
      // where m - m' = d
      float4* u = tu + f * A::kTabF4 * AX + k;
      const signed char* om = &s_om[q.l1 ? 0 : 1][BV + k];
      const int64_t m = q.own(k);
      const CDF w = cis_df(2 * q.tA * (uint64_t)m, a.ctab);
      CDF p = w;
#pragma unroll
      for (int d = 1; d <= BV; ++d) {
        const CDF e = as_cdf(s_e[f][d - 1]);
        CDF up = mul(e, p), um = mul(e, conj(p));
        if (om[0] != om[-d]) {
          const int64_t mm = q.own(k - d);
          up = cis_df(q.tA * (uint64_t)(m * m - mm * mm), a.ctab);
        }
        if (om[0] != om[d]) {
          const int64_t mp = q.own(k + d);
          um = cis_df(q.tA * (uint64_t)(m * m - mp * mp), a.ctab);
        }
        A::put(u, AX, d, up, um, q.taps);
        if (d < BV) p = mul(p, w);
      }
    }
  }
  // ---- load, wrapping both indices
  pass_wait();
  {
    constexpr int LW = CE < 32 ? CE : 32, NC = CE / LW;   // lanes along a row
    const int lc = tid % LW;
    int col[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      const int mu = g.c0 - g.hc + lc + LW * k;
      col[k] = mu - wraps(mu, g.M1) * g.M1;
    }
    for (int r = tid / LW; r < g.re; r += NT / LW) {
      const int nu = g.r0 - g.hr + r;
      const double2* gp = src + (int64_t)(nu - wraps(nu, g.M2) * g.M2) * in.pitch;
#pragma unroll
      for (int k = 0; k < NC; ++k)
        if (lc + LW * k < g.ce) cp_async16(xt + r * P + lc + LW * k, gp + col[k]);
    }
  }
  cp_async_wait_all();
  __syncthreads();
  // largest finite exponent of the tile, and whether anything is not finite
  typename A::Scale sc;
  {
    int mx = 0;
    bool bad = false;
    for (int i = tid; i < RE * CE; i += NT)
      if (i / CE < g.re && i % CE < g.ce) {
        const double2 v = xt[(i / CE) * P + i % CE];
        const int e1 = (__double2hiint(v.x) >> 20) & 0x7ff, e2 = (__double2hiint(v.y) >> 20) & 0x7ff;
        bad |= e1 == 0x7ff || e2 == 0x7ff;
        mx = max(mx, max(e1 == 0x7ff ? 0 : e1, e2 == 0x7ff ? 0 : e2));
      }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) s_red[warp] = mx;
    sc.bad = __syncthreads_or(bad);
#pragma unroll
    for (int w = 0; w < NW; ++w) mx = max(mx, s_red[w]);
    sc.off = (mx - 167) * (1 << 20);
  }
  // ---- factors: lanes along the other axis, SEG elements of this axis per thread
  for (int f = 0; f < a.nf; ++f) {
    const FactorGeo q(a, g, f);
    const int lines = q.l1 ? RE : CE;
    const int line = tid % lines, e0 = (tid / lines) * SEG;
    const bool active = line < q.nb && e0 < q.na;
    const signed char* om = &s_om[q.l1 ? 0 : 1][BV + e0];
    const bool seam = om[-BV] != om[SEG - 1 + BV];
    const int ln = min(line, q.nb - 1);
    const CDF v = as_cdf(tv[f * AX + ln]);
    CDF vq = v;
    if (active && seam) vq = cis_df(q.tX * (uint64_t)(q.other(ln) * q.qa), a.ctab);
    double2* sp = q.l1 ? xt + line * P + e0 : xt + e0 * P + line;
    sweep<A, BV, SEG, AX>(sp, q.l1 ? 1 : P, tu + f * A::kTabF4 * AX + e0, v, active, seam, om, vq, sc);
  }
  // ---- store the tile's result; the call's last pass applies Lambda K(T)
  for (int r = warp; r < g.vr; r += NW) {
    double2* gp = dst + (int64_t)(g.r0 + r) * in.pitch + g.c0;
    const double2* s = xt + (r + g.hr) * P + g.hc;
    const uint64_t n = (uint64_t)(int64_t)(in.lo2 + g.r0 + r);
    const uint64_t qx = in.X * n, qn = in.A2 * (n * n);
    for (int k = lane; k < g.vc; k += 32) {
      double2 y = s[k];
      if (a.last) {
        const uint64_t m = (uint64_t)(int64_t)(in.lo1 + g.c0 + k);
        double2 w = cis_d(in.lam_turns - (uint64_t)a.T * ((in.A1 * m + qx) * m + qn), a.ptab);
        w.x -= w.x * in.lam_def;
        w.y -= w.y * in.lam_def;
        y = cmul(y, w);
      }
      gp[k] = y;
    }
  }
}

// ---------------------------------------------------------------- complex64
// Two lines per thread, A and B = A + lines / 2, in the lanes of paired FP32
// operations.  Per factor and index of the axis the table holds, for each d,
// U_d and U_-d with every component doubled.
template <int BV> struct LinesF {
  float2 x[BV], y[BV], ny[BV];     // (re, re), (im, im), -(im, im) of V^d on lines A and B
};
template <int BV>
__device__ __forceinline__ void tapsum_f(const float4* u, int stride, const LinesF<BV>& L, const float2* wr,
                                         const float2* wi, float2& cr, float2& ci) {
  float2 a = make_float2(0.f, 0.f), b = a, c = a;
#pragma unroll
  for (int d = BV; d >= 1; --d) {
    const float4 p = u[(2 * d - 2) * stride], m = u[(2 * d - 1) * stride];
    const float2 px = make_float2(p.x, p.y), py = make_float2(p.z, p.w);
    const float2 mx = make_float2(m.x, m.y), my = make_float2(m.z, m.w);
    const float2 vx = L.x[d - 1], vy = L.y[d - 1], vn = L.ny[d - 1];
    const float2 Wx = __ffma2_rn(py, vn, __fmul2_rn(px, vx)), Wy = __ffma2_rn(px, vy, __fmul2_rn(py, vx));
    const float2 Zx = __ffma2_rn(my, vy, __fmul2_rn(mx, vx)), Zy = __ffma2_rn(mx, vn, __fmul2_rn(my, vx));
    a = __ffma2_rn(Wx, wr[BV - d], a);
    b = __ffma2_rn(Wy, wi[BV - d], b);
    c = __ffma2_rn(Wx, wi[BV - d], c);
    c = __ffma2_rn(Wy, wr[BV - d], c);
    a = __ffma2_rn(Zx, wr[BV + d], a);
    b = __ffma2_rn(Zy, wi[BV + d], b);
    c = __ffma2_rn(Zx, wi[BV + d], c);
    c = __ffma2_rn(Zy, wr[BV + d], c);
  }
  cr = __ffma2_rn(b, make_float2(-1.f, -1.f), a);
  ci = c;
}

template <int BV, int SEG, int STRIDE>
__device__ __forceinline__ void sweep_f(float* __restrict__ re, float* __restrict__ im, int step, int ofs,
                                        const float4* __restrict__ u, float2 va, float2 vb, bool active, bool seam,
                                        const signed char* om, float2 qa, float2 qb) {
  // U elements per block: their BV-th right neighbours are loaded together,
  // and the window of a block needs no shifting inside it
  constexpr int U = SEG < 4 ? SEG : 4;
  static_assert(SEG % U == 0, "blocks");
  float2 wr[2 * BV + U], wi[2 * BV + U], rr[BV], ri[BV];
  if (active) {
#pragma unroll
    for (int k = 0; k < 2 * BV; ++k) {
      const int o = (k - BV) * step;
      wr[k] = make_float2(re[o], re[o + ofs]);
      wi[k] = make_float2(im[o], im[o + ofs]);
    }
#pragma unroll
    for (int k = 0; k < BV; ++k) {
      const int o = (SEG + k) * step;
      rr[k] = make_float2(re[o], re[o + ofs]);
      ri[k] = make_float2(im[o], im[o + ofs]);
    }
  }
  __syncthreads();
  if (active) {
    LinesF<BV> L;
    {
      float2 pa = va, pb = vb;
#pragma unroll
      for (int d = 0; d < BV; ++d) {
        L.x[d] = make_float2(pa.x, pb.x);
        L.y[d] = make_float2(pa.y, pb.y);
        L.ny[d] = make_float2(-pa.y, -pb.y);
        if (d + 1 < BV) {
          pa = cmul(pa, va);
          pb = cmul(pb, vb);
        }
      }
    }
    auto put = [&](int o, int k, float2 cr, float2 ci) {
      const float2 yr = __fadd2_rn(wr[BV + k], cr), yi = __fadd2_rn(wi[BV + k], ci);
      re[o] = yr.x;
      re[o + ofs] = yr.y;
      im[o] = yi.x;
      im[o + ofs] = yi.y;
    };
    if (!seam) {
#pragma unroll 1
      for (int i = 0; i < SEG; i += U) {
#pragma unroll
        for (int k = 0; k < U; ++k) {
          const int o = (BV + k) * step;
          wr[2 * BV + k] = make_float2(re[o], re[o + ofs]);
          wi[2 * BV + k] = make_float2(im[o], im[o + ofs]);
        }
        if (i + U >= SEG) {
          // the last block reaches into the next thread's segment
#pragma unroll
          for (int k = 0; k < U; ++k)
            if (k + BV >= U) {
              wr[2 * BV + k] = rr[k + BV - U];
              wi[2 * BV + k] = ri[k + BV - U];
            }
        }
#pragma unroll
        for (int k = 0; k < U; ++k) {
          float2 cr, ci;
          tapsum_f<BV>(u + k, STRIDE, L, wr + k, wi + k, cr, ci);
          put(k * step, k, cr, ci);
        }
#pragma unroll
        for (int k = 0; k < 2 * BV; ++k) {
          wr[k] = wr[k + U];
          wi[k] = wi[k + U];
        }
        re += U * step;
        im += U * step;
        u += U;
      }
    } else {
      // pairs that straddle the end of the box: the neighbour times V_n^{-q w}
#pragma unroll 1
      for (int i = 0; i < SEG; ++i) {
        const int o = BV * step;
        wr[2 * BV] = make_float2(re[o], re[o + ofs]);
        wi[2 * BV] = make_float2(im[o], im[o + ofs]);
        if (i + BV >= SEG) {
          wr[2 * BV] = rr[SEG < BV ? BV - SEG : 0];
          wi[2 * BV] = ri[SEG < BV ? BV - SEG : 0];
#pragma unroll
          for (int k = 0; k + 1 < BV; ++k) {
            rr[k] = rr[k + 1];
            ri[k] = ri[k + 1];
          }
        }
        float2 tr[2 * BV + 1], ti[2 * BV + 1];
#pragma unroll
        for (int j = 0; j <= 2 * BV; ++j) {
          const int w = om[0] - om[j - BV];
          tr[j] = wr[j];
          ti[j] = wi[j];
          if (w != 0) {
            const float sg = w > 0 ? -1.f : 1.f;
            const float2 ta = cmul(make_float2(wr[j].x, wi[j].x), make_float2(qa.x, sg * qa.y));
            const float2 tb = cmul(make_float2(wr[j].y, wi[j].y), make_float2(qb.x, sg * qb.y));
            tr[j] = make_float2(ta.x, tb.x);
            ti[j] = make_float2(ta.y, tb.y);
          }
        }
        float2 cr, ci;
        tapsum_f<BV>(u, STRIDE, L, tr, ti, cr, ci);
        put(0, 0, cr, ci);
#pragma unroll
        for (int k = 0; k < 2 * BV; ++k) {
          wr[k] = wr[k + 1];
          wi[k] = wi[k + 1];
        }
        re += step;
        im += step;
        ++u;
        ++om;
      }
    }
  }
  __syncthreads();
}

// U table of one factor at axis position k (hardware sine and cosine: the
// phases only multiply the correction, taps of size s |v|)
template <int BV, int AX>
__device__ __forceinline__ void table_u(const FactorGeo& q, const signed char* om, int k, float4* u) {
  const int64_t m = q.own(k);
  const float2 w = cis_fast(2 * q.tA * (uint64_t)m);
  float2 p = w;
#pragma unroll
  for (int d = 1; d <= BV; ++d) {
    const float2 e = cis_fast((uint64_t)0 - q.tA * (uint64_t)(d * d));
    float2 up = cmul(e, p), um = cmulconj(e, p);
    if (om[0] != om[-d]) {
      const int64_t mm = q.own(k - d);
      up = cis_fast(q.tA * (uint64_t)(m * m - mm * mm));
    }
    if (om[0] != om[d]) {
      const int64_t mp = q.own(k + d);
      um = cis_fast(q.tA * (uint64_t)(m * m - mp * mp));
    }
    const float4 cp = q.taps[kTileMaxB + d], cm = q.taps[kTileMaxB - d];
    up = cmul(up, make_float2(cp.x, cp.z));
    um = cmul(um, make_float2(cm.x, cm.z));
    u[(2 * d - 2) * AX] = make_float4(up.x, up.x, up.y, up.y);
    u[(2 * d - 1) * AX] = make_float4(um.x, um.x, um.y, um.y);
    if (d < BV) p = cmul(p, w);
  }
}

template <int BV, int RE, int CE, int SEG, int MINB>
__global__ void __launch_bounds__(RE * CE / (2 * SEG), MINB) tile_f32_kernel(const __grid_constant__ TileArgs a) {
  using Sh = TileShape<BV, RE, CE>;
  constexpr int NT = RE * CE / (2 * SEG), NW = NT / 32, P = Sh::kPitch, AX = Sh::kAxis;
  static_assert(NT % 32 == 0 && RE % 32 == 0 && CE % 32 == 0 && CE % SEG == 0 && RE % SEG == 0, "tile shape");
  extern __shared__ __align__(16) unsigned char smraw[];
  float4* tu = reinterpret_cast<float4*>(smraw);                   // [nf][2 BV][AX]
  float2* tv = reinterpret_cast<float2*>(tu + a.nf * 2 * BV * AX);  // [nf][AX]
  float* xr = reinterpret_cast<float*>(tv + a.nf * AX);
  float* xi = xr + Sh::kElems;
  __shared__ signed char s_om[2][AX + 2 * BV];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const TileGeo g(a);
  const TileInst& in = *g.in;
  const float2* src = reinterpret_cast<const float2*>(a.flip ? in.alt : in.psi);
  float2* dst = reinterpret_cast<float2*>(a.flip ? in.psi : in.alt);
  constexpr int O = BV * P + BV;   // element (row 0, column 0) of the tile
  pass_begin();
  constexpr int NR = RE / NW, NC = CE / 32;
  static_assert(RE % NW == 0, "rows per warp");
  float2 v[NR][NC];
  auto load = [&]() {   // all loads of the tile in flight, wrapping both indices
    pass_wait();
    int col[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      const int mu = g.c0 - g.hc + lane + 32 * k;
      col[k] = lane + 32 * k < g.ce ? mu - wraps(mu, g.M1) * g.M1 : -1;
    }
#pragma unroll
    for (int j = 0; j < NR; ++j) {
      const int nu = g.r0 - g.hr + warp + j * NW;
      const float2* gp = src + (int64_t)(nu - wraps(nu, g.M2) * g.M2) * in.pitch;
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        v[j][k] = make_float2(0.f, 0.f);
        if (warp + j * NW < g.re && col[k] >= 0) v[j][k] = __ldcg(gp + col[k]);
      }
    }
  };
  // ---- wrap counts of both axes, then the tables of every factor (while the
  // previous pass drains)
  for (int i = tid; i < 2 * (AX + 2 * BV); i += NT) {
    const int ax = i >= AX + 2 * BV ? 1 : 0, k = i - ax * (AX + 2 * BV) - BV;
    s_om[ax][k + BV] = (signed char)(ax ? wraps(g.r0 - g.hr + k, g.M2) : wraps(g.c0 - g.hc + k, g.M1));
  }
  __syncthreads();
  for (int i = tid; i < a.nf * 2 * AX; i += NT) {
    const int f = i / (2 * AX), k = i % AX;
    const FactorGeo q(a, g, f);
    if (i % (2 * AX) >= AX) {
      if (k < q.nb) tv[f * AX + k] = cis_fast(q.tX * (uint64_t)q.other(k));
    } else if (k < q.na) {
      table_u<BV, AX>(q, &s_om[q.l1 ? 0 : 1][BV + k], k, tu + f * 2 * BV * AX + k);
    }
  }
  load();
#pragma unroll
  for (int j = 0; j < NR; ++j)
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      xr[O + (warp + j * NW) * P + lane + 32 * k] = v[j][k].x;
      xi[O + (warp + j * NW) * P + lane + 32 * k] = v[j][k].y;
    }
  __syncthreads();
  // ---- factors
  for (int f = 0; f < a.nf; ++f) {
    const bool l1 = a.layer[f] == 1;
    const int half = (l1 ? RE : CE) / 2;
    const int line = tid % half, e0 = (tid / half) * SEG;
    const int na = l1 ? g.ce : g.re, nb = l1 ? g.re : g.ce;
    const bool active = line < nb && e0 < na;
    const signed char* om = &s_om[l1 ? 0 : 1][BV + e0];
    const bool seam = om[-BV] != om[SEG - 1 + BV];
    const float2* vt = tv + f * AX;
    const int lna = min(line, nb - 1), lnb = min(line + half, nb - 1);
    float2 qa = make_float2(1.f, 0.f), qb = qa;
    if (active && seam) {
      const FactorGeo q(a, g, f);
      qa = cis_fast(q.tX * (uint64_t)(q.other(lna) * q.qa));
      qb = cis_fast(q.tX * (uint64_t)(q.other(lnb) * q.qa));
    }
    const int o = O + (l1 ? line * P + e0 : e0 * P + line);
    sweep_f<BV, SEG, AX>(xr + o, xi + o, l1 ? 1 : P, l1 ? half * P : half, tu + f * 2 * BV * AX + e0, vt[lna], vt[lnb],
                         active, seam, om, qa, qb);
  }
  // ---- store the tile's result; the call's last pass applies Lambda K(T)
#pragma unroll 2
  for (int r = warp; r < g.vr; r += NW) {
    float2* gp = dst + (int64_t)(g.r0 + r) * in.pitch + g.c0;
    const int so = O + (r + g.hr) * P + g.hc;
    if (!a.last) {
#pragma unroll
      for (int j = 0; j < NC; ++j) {
        const int k = lane + 32 * j;
        if (k < g.vc) gp[k] = make_float2(xr[so + k], xi[so + k]);
      }
    } else {
      const uint64_t n = (uint64_t)(int64_t)(in.lo2 + g.r0 + r);
      const uint64_t qx = in.X * n, qn = in.A2 * (n * n);
      for (int k = lane; k < g.vc; k += 32) {
        const uint64_t m = (uint64_t)(int64_t)(in.lo1 + g.c0 + k);
        Phase<float> ph = phase_of<float>(in.lam_turns - (uint64_t)a.T * ((in.A1 * m + qx) * m + qn));
        ph.half_e += (float)in.lam_def;
        gp[k] = apply_phase<float>(make_float2(xr[so + k], xi[so + k]), ph);
      }
    }
  }
}

// Raise a kernel's shared-memory limit to the device's (the attribute belongs to
// the process, so nothing may lower it again).
template <int BV, int RE, int CE, int SEG, int MINB>
cudaError_t launch_f32(const TileArgs* a, int64_t ntiles, size_t max_block, cudaStream_t st) {
  using Sh = TileShape<BV, RE, CE>;
  const auto k = tile_f32_kernel<BV, RE, CE, SEG, MINB>;
  if (!a) return allow_smem(k, max_block);
  const size_t smem = (size_t)2 * Sh::kElems * sizeof(float) +
                      (size_t)a->nf * Sh::kAxis * (2 * BV * sizeof(float4) + sizeof(float2));
  return launch_pdl(k, (unsigned)ntiles, RE * CE / (2 * SEG), smem, st, *a);
}
template <int BV, int RE, int CE, int SEG, int MINB>
cudaError_t launch_f64(const TileArgs* a, int64_t ntiles, size_t max_block, cudaStream_t st) {
  using Sh = TileShape<BV, RE, CE>;
  const auto k = tile_f64_kernel<BV, RE, CE, SEG, MINB>;
  if (!a) return allow_smem(k, max_block);
  const size_t smem = (size_t)Sh::kElems * sizeof(double2) +
                      (size_t)a->nf * Sh::kAxis * (Ar<double, BV>::kTabF4 + 1) * sizeof(float4);
  return launch_pdl(k, (unsigned)ntiles, RE * CE / SEG, smem, st, *a);
}

// The instance for bv and ext: launch it with *a, or (a NULL) prepare it.
template <typename Real>
cudaError_t tile_kernel(const TileArgs* a, int bv, int ext, int64_t ntiles, size_t max_block, cudaStream_t st) {
#define LS_TILE(F, B, E, ...) \
  if (bv == B && ext == E) return F<B, E, E, __VA_ARGS__>(a, ntiles, max_block, st);
  if constexpr (sizeof(Real) == 4) {
    LS_TILE(launch_f32, 2, 32, 2, 2)
    LS_TILE(launch_f32, 3, 32, 2, 2)
  } else {
    LS_TILE(launch_f64, 3, 16, 1, 2)
    LS_TILE(launch_f64, 3, 32, 2, 1)
    LS_TILE(launch_f64, 3, 64, 16, 2)
    LS_TILE(launch_f64, 4, 16, 1, 2)
    LS_TILE(launch_f64, 4, 32, 2, 1)
    LS_TILE(launch_f64, 4, 64, 16, 2)
    LS_TILE(launch_f64, 5, 32, 2, 1)
    LS_TILE(launch_f64, 5, 64, 16, 2)
  }
#undef LS_TILE
  return cudaErrorInvalidValue;
}

}  // namespace

template <typename Real> cudaError_t launch_tile(const TileArgs& a, int bv, int ext, int64_t ntiles, cudaStream_t st) {
  if (ntiles <= 0) return cudaSuccess;
  if (a.nf < 1 || a.nf > kTileMaxF || ntiles > 0x7fffffff || a.tr + 2 * a.hr > ext || a.tc + 2 * a.hc > ext ||
      a.tr < 1 || a.tc < 1)
    return cudaErrorInvalidValue;
  return tile_kernel<Real>(&a, bv, ext, ntiles, 0, st);
}
template <typename Real> cudaError_t tile_prepare(int bv, int ext, size_t max_block) {
  return tile_kernel<Real>(nullptr, bv, ext, 0, max_block, nullptr);
}
template cudaError_t launch_tile<float>(const TileArgs&, int, int, int64_t, cudaStream_t);
template cudaError_t launch_tile<double>(const TileArgs&, int, int, int64_t, cudaStream_t);
template cudaError_t tile_prepare<float>(int, int, size_t);
template cudaError_t tile_prepare<double>(int, int, size_t);

}  // namespace lsk
