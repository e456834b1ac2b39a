// Observables of a 1D box in one pass over the state: norm, kinetic energy,
// mean wavevector, overlap and both potential energies (Eq. (2.4)-(2.5)).
//
// The potential energy needs no transform: with the real potential
// v(x) = w_0 + 2 Re sum_{h > 0} w_h e^{2 pi i h x / L} on the layer's grid,
//   (1/q) sum_p v(x_p) |psi(x_p)|^2 = w_0 sum_m |x_m|^2
//                                   + 2 Re sum_{h > 0} w_h sum_m x_m conj(x_{(m + h) mod q})
// for every slice, a correlation with the neighbours |h| <= 8 (along the row
// for layer 1, along the column for layer 2).  The transform form took two
// Bluestein passes (254 + 207 us on 2049 x 2049 complex64) and its FP32
// transforms left 1e-7; the correlation is exact to the accumulation.
//
// FP64 accumulation of every product would be bound by the FP64 pipe (128 us
// for the norm and the kinetic terms alone): complex64 products are exact in
// pairs of floats and accumulate there (2^-48 per addition), per warp item of
// up to 512 elements of a row; items are added in FP64.  The kinetic terms use
// k = B1 (m - m0) + (B1 m0 + B2 n), m0 the row's index of smallest |k|, so
// that only integer moments of |x|^2 are summed per element.
//
// 2049 x 2049 complex64 with an overlap: 740 -> 138 us per call, 20 us of it
// the launches and the read-back.  In the kernel (95 us) the FP64 pipe is 76 %
// busy with the conversions and sums at the end of each item and with items
// outside the pairs' range; about 330 instructions per element, 43 % issue.
#include "lsplit_kernels.cuh"
#include "lsplit_pair.cuh"

namespace lsk {
namespace {

constexpr int kObsChunk = 512;   // elements of a row per warp item

// Accumulators of one sum per type
template <typename Real> struct Sum;
template <> struct Sum<float> {
  DF a{0.f, 0.f};
  float c = 0.f;   // rounding of the low part (sums of one sign, where it would show)
  __device__ __forceinline__ void mac(float x, float y) { pair_mac(a, x, y); }
  __device__ __forceinline__ void add(float p, float e) {
    float r, t;
    two_sum(a.h, p, a.h, r);
    two_sum(a.l, __fadd_rn(r, e), a.l, t);
    c = __fadd_rn(c, t);
  }
  __device__ __forceinline__ double get() const { return (double)a.h + ((double)a.l + (double)c); }
};
template <> struct Sum<double> {
  double a = 0.0;
  __device__ __forceinline__ void mac(double x, double y) { a = fma(x, y, a); }
  __device__ __forceinline__ double get() const { return a; }
};

// moments |x|^2, m' |x|^2, m'^2 |x|^2
template <typename C> __device__ __forceinline__ void moments(Sum<float>* s, C v, int mi) {
  const float m = (float)mi;   // |m'| below the box length: exact
  const float p = __fmul_rn(v.x, v.x), q = __fmul_rn(v.y, v.y);
  float h, r;
  two_sum(p, q, h, r);
  const float l = __fadd_rn(r, __fadd_rn(fmaf(v.x, v.x, -p), fmaf(v.y, v.y, -q)));
  s[0].add(h, l);
  const float h1 = __fmul_rn(h, m), l1 = fmaf(l, m, fmaf(h, m, -h1));
  s[1].add(h1, l1);
  const float h2 = __fmul_rn(h1, m), l2 = fmaf(l1, m, fmaf(h1, m, -h2));
  s[2].add(h2, l2);
}
template <typename C> __device__ __forceinline__ void moments(Sum<double>* s, C v, int mi) {
  const double x = v.x, y = v.y, m = (double)mi;
  const double a2 = fma(x, x, y * y), t = m * a2;
  s[0].a += a2;
  s[1].a += t;
  s[2].a = fma(m, t, s[2].a);
}

// largest magnitude of a component, as bits (NaN above everything)
__device__ __forceinline__ uint32_t mag(float2 v) {
  return max(__float_as_uint(v.x) & 0x7fffffffu, __float_as_uint(v.y) & 0x7fffffffu);
}
// Components between which the sums of an item fit pairs of floats: up to 2^36
// the second moment, at most 2 2^72 m'^2 per element and 16 elements per lane,
// stays finite for |m'| < 2^24; from 2^-40 on what a product below 2^-102 loses
// of its low part (2^-149 each, 2^11 of them) is 2^-58 of the item's norm.
constexpr uint32_t kLow = (127u - 40u) << 23, kHigh = (127u + 36u) << 23;
// Overlap products: below this the lost low parts would show (2^-138 of 2^-90)
constexpr uint32_t kLowProd = (127u - 90u) << 23;

// <chi, psi> over the elements [c0, c1) of a row
template <typename Acc, typename C>
__device__ __forceinline__ void overlap(const C* x, const C* y, int c0, int c1, double* ov) {
  Acc re, im;
#pragma unroll 4
  for (int m = c0 + (threadIdx.x & 31); m < c1; m += 32) {
    const C v = x[m], c = y[m];
    re.mac(c.x, v.x);
    re.mac(c.y, v.y);
    im.mac(c.x, v.y);
    im.mac(-c.y, v.x);
  }
  ov[0] = re.get();
  ov[1] = im.get();
}

// One item: elements [c0, c1) of a row; Acc the accumulators' type.  Returns
// false if a neighbour left the range of the pairs (nothing is added then).
template <typename Acc, typename C>
__device__ __forceinline__ bool item(const ObsArgs& a, const C* psi, const C* chi, int row, int c0, int c1,
                                     double* acc) {
  constexpr bool pairs = std::is_same<Acc, Sum<float>>::value;
  const int lane = threadIdx.x & 31, M1 = a.M1, M2 = a.M2;
  const C* x = psi + (int64_t)row * a.pitch;
  const double kn = a.b2 * (double)(a.lo2 + row);
  // row's index of smallest |k| (inside the box, so |m'| < M1)
  const double mz = a.b1 != 0.0 ? -kn / a.b1 : 0.0;
  const int m0 = (int)fmin(fmax(rint(mz), (double)a.lo1), (double)(a.lo1 + M1 - 1));
  const double dk = fma(a.b1, (double)m0, kn);
  Acc s[3];
#pragma unroll 4
  for (int m = c0 + lane; m < c1; m += 32) moments(s, x[m], a.lo1 + m - m0);
  const double s0 = s[0].get(), s1 = s[1].get(), s2 = s[2].get();
  double ov[2] = {0.0, 0.0}, ep[2] = {a.w0[0] * s0, a.w0[1] * s0};
  uint32_t mx = 0;
  if (chi) {
    const C* y = chi + (int64_t)row * a.pitch;
    uint32_t pm = 0, cm = 0;   // largest product and chi
    if constexpr (pairs) {
#pragma unroll 4
      for (int m = c0 + lane; m < c1; m += 32) {
        const uint32_t q = mag(y[m]);
        cm = max(cm, q);
        pm = max(pm, __float_as_uint(__fmul_rn(__uint_as_float(q), __uint_as_float(mag(x[m])))));
      }
      mx = cm;
      pm = __reduce_max_sync(0xffffffffu, pm);
      cm = __reduce_max_sync(0xffffffffu, cm);
    }
    if (!pairs || (cm != 0 && pm < kLowProd)) overlap<Sum<double>>(x, y, c0, c1, ov);
    else overlap<Acc>(x, y, c0, c1, ov);
  }
  // sum_m x_m conj(x_{m + h}) for the harmonics of both layers
#pragma unroll 1
  for (int L = 0; L < 2; ++L) {
#pragma unroll 1
    for (int k = 0; k < a.nh[L]; ++k) {
      const int h = a.h[L][k];
      const C* y = x + h;
      if (L == 1) y = psi + (int64_t)(row + h >= M2 ? row + h - M2 : row + h) * a.pitch;
      Acc re, im;
#pragma unroll 4
      for (int m = c0 + lane; m < c1; m += 32) {
        const C v = x[m], w = y[L == 0 && m + h >= M1 ? m - M1 : m];
        if constexpr (pairs) mx = max(mx, mag(w));
        re.mac(v.x, w.x);
        re.mac(v.y, w.y);
        im.mac(v.y, w.x);
        im.mac(-v.x, w.y);
      }
      ep[L] += 2.0 * (a.wr[L][k] * re.get() - a.wi[L][k] * im.get());
    }
  }
  if (pairs && __any_sync(0xffffffffu, mx >= kHigh)) return false;
  acc[0] += s0;
  acc[1] += 0.5 * (a.b1 * a.b1 * s2 + 2.0 * a.b1 * dk * s1 + dk * dk * s0);
  acc[2] += a.b1 * s1 + dk * s0;
  acc[4] += ov[0];
  acc[5] += ov[1];
  acc[6] += ep[0];
  acc[7] += ep[1];
  return true;
}

template <typename Real> __global__ void __launch_bounds__(256) obs1d_kernel(const ObsArgs a, double* partials) {
  using C = typename CT<Real>::C;
  const C* psi = reinterpret_cast<const C*>(a.psi);
  const C* chi = reinterpret_cast<const C*>(a.chi);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nch = (a.M1 + kObsChunk - 1) / kObsChunk;
  const int64_t items = (int64_t)a.M2 * nch;
  double acc[kObsQ];
#pragma unroll
  for (int q = 0; q < kObsQ; ++q) acc[q] = 0.0;
  for (int64_t it = (int64_t)blockIdx.x * 8 + warp; it < items; it += (int64_t)gridDim.x * 8) {
    const int row = (int)(it / nch), c0 = (int)(it - (int64_t)row * nch) * kObsChunk;
    const int c1 = min(a.M1, c0 + kObsChunk);
    if constexpr (sizeof(Real) == 4) {
      // pairs of floats while the item's largest component is between kLow and
      // kHigh (chi and neighbours: below kHigh); else FP64
      uint32_t mx = 0;
#pragma unroll 4
      for (int m = c0 + lane; m < c1; m += 32) mx = max(mx, mag(psi[(int64_t)row * a.pitch + m]));
      mx = __reduce_max_sync(0xffffffffu, mx);
      if (mx >= kLow && mx < kHigh && item<Sum<float>>(a, psi, chi, row, c0, c1, acc)) continue;
      if (mx == 0 && !chi) continue;
    }
    item<Sum<double>>(a, psi, chi, row, c0, c1, acc);
  }
  __shared__ double red[8][kObsQ];
#pragma unroll
  for (int q = 0; q < kObsQ; ++q) {
    double v = acc[q];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) red[warp][q] = v;
  }
  __syncthreads();
  if (threadIdx.x < kObsQ) {
    double v = 0.0;
    for (int w = 0; w < 8; ++w) v += red[w][threadIdx.x];
    partials[blockIdx.x * kObsQ + threadIdx.x] = v;
  }
}

}  // namespace

template <typename Real> cudaError_t launch_obs1d(const ObsArgs& a, double* partials, int nblocks, cudaStream_t st) {
  obs1d_kernel<Real><<<nblocks, 256, 0, st>>>(a, partials);
  return cudaGetLastError();
}
template cudaError_t launch_obs1d<float>(const ObsArgs&, double*, int, cudaStream_t);
template cudaError_t launch_obs1d<double>(const ObsArgs&, double*, int, cudaStream_t);

}  // namespace lsk
