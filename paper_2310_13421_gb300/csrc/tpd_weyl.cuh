// The d-point DFT of one class of a Weyl-basis level in IEEE arithmetic, and
// its constants (see tpd_weyl.cu), shared by the complex128 and complex64
// kernels.
#pragma once

#include <cuda_runtime.h>

#include <cmath>

namespace tpd {

template <class T>
struct Cx {
  T re, im;
};

template <class T>
__device__ __forceinline__ Cx<T> cadd(Cx<T> a, Cx<T> b) { return {a.re + b.re, a.im + b.im}; }
template <class T>
__device__ __forceinline__ Cx<T> csub(Cx<T> a, Cx<T> b) { return {a.re - b.re, a.im - b.im}; }
// a * (wr + i wi), written without contraction into fused multiply-adds
template <class T>
__device__ __forceinline__ Cx<T> cmul(Cx<T> a, T wr, T wi) {
  if constexpr (sizeof(T) == 8)
    return {__dsub_rn(__dmul_rn(a.re, wr), __dmul_rn(a.im, wi)), __dadd_rn(__dmul_rn(a.re, wi), __dmul_rn(a.im, wr))};
  else
    return {__fsub_rn(__fmul_rn(a.re, wr), __fmul_rn(a.im, wi)), __fadd_rn(__fmul_rn(a.re, wi), __fmul_rn(a.im, wr))};
}

template <class T>
struct Twiddles {
  T re[8], im[8];     // omega^k, k < d
  T h;                // sqrt(3) / 2 (d = 3)
  T scale;            // factor applied to every output of this launch
};

// The d-point DFT of one class in the arithmetic T (y_b = sum_c omega^-bc x_c
// for the decomposition, omega^+bc for the composition).
template <class T, int D, bool kDec>
__device__ __forceinline__ void dft_ieee(const Cx<T> (&x)[D], Cx<T> (&y)[D], const Twiddles<T>& tw) {
  if constexpr (D == 3) {
    const Cx<T> sm = cadd(x[1], x[2]), u = csub(x[1], x[2]);
    const Cx<T> m = csub(x[0], Cx<T>{sm.re * T(0.5), sm.im * T(0.5)});
    const Cx<T> hu = {u.re * tw.h, u.im * tw.h};
    y[0] = cadd(x[0], sm);
    // -i h u = (h u.im, -h u.re); the composition takes +i h u for y1
    const Cx<T> mihu = {hu.im, -hu.re};
    y[1] = kDec ? cadd(m, mihu) : csub(m, mihu);
    y[2] = kDec ? csub(m, mihu) : cadd(m, mihu);
  } else {
#pragma unroll
    for (int b = 0; b < D; ++b) {
      Cx<T> acc = x[0];
#pragma unroll
      for (int c = 1; c < D; ++c) {
        const int k = kDec ? (D - (b * c) % D) % D : (b * c) % D;
        acc = cadd(acc, cmul(x[c], tw.re[k], tw.im[k]));
      }
      y[b] = acc;
    }
  }
}

// One block of a level, y from x: decomposition, x_c = A_{c+a, c} ->
// Omega_{a,b} at (b, a+b); composition, Omega_{a,b} at (b, a+b) -> A_{c+a, c}.
// S: double2 / float2.
template <class T, int D, bool kDec, class S>
__device__ __forceinline__ void weyl_block_ieee(const S (&x)[D][D], S (&y)[D][D], const Twiddles<T>& tw) {
#pragma unroll
  for (int a = 0; a < D; ++a) {
    Cx<T> u[D], v[D];
#pragma unroll
    for (int c = 0; c < D; ++c) {
      const S e = kDec ? x[(c + a) % D][c] : x[c][(a + c) % D];
      u[c] = {e.x, e.y};
    }
    dft_ieee<T, D, kDec>(u, v, tw);
#pragma unroll
    for (int b = 0; b < D; ++b) {
      S& o = kDec ? y[b][(a + b) % D] : y[(b + a) % D][b];
      o.x = v[b].re * tw.scale;
      o.y = v[b].im * tw.scale;
    }
  }
}

// A cosine or sine within a few ulps of 0, +-1/2 or +-1 is that value
// exactly, so quarter and sixth turns carry no rounding.
inline double exact_if_near_half_integer(double v) {
  const double h = std::nearbyint(2.0 * v) * 0.5;
  return std::fabs(v - h) <= 4e-16 ? h : v;
}

template <class T>
inline Twiddles<T> twiddles(int d, double scale) {
  Twiddles<T> t{};
  const double pi = 3.14159265358979323846;
  for (int k = 0; k < d; ++k) {
    t.re[k] = (T)exact_if_near_half_integer(std::cos(2.0 * pi * k / d));
    t.im[k] = (T)exact_if_near_half_integer(std::sin(2.0 * pi * k / d));
  }
  t.h = (T)(std::sqrt(3.0) * 0.5);
  t.scale = (T)scale;
  return t;
}

// n levels on complex64, several per pass (tpd_weyl_c64.cu)
cudaError_t weyl_c64(bool dec, const float2* src, float2* mat, int n, int d, double last_scale, cudaStream_t st);

// n levels on complex128 in block fixed point, d = 2, 3, 4 (tpd_weyl_fixed.cu)
cudaError_t weyl_fixed(bool dec, const double2* src, double2* mat, int n, int d, double last_scale, cudaStream_t st);

}  // namespace tpd
