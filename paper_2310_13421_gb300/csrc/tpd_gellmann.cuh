// One qudit level of the generalized Gell-Mann basis on one d x d block, and
// its constants (see tpd_gellmann.cu), shared by the complex128 and complex64
// kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>

namespace tpd {

constexpr int kGmMaxD = 5;

template <class T> struct GmVec;
template <> struct GmVec<double> { using t = double2; };
template <> struct GmVec<float> { using t = float2; };

// single roundings, never contracted into an fma
__device__ __forceinline__ double gadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double gsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double gmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float gadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float gsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float gmul(float a, float b) { return __fmul_rn(a, b); }

// x / 2 and 2 x.  For complex128 with integer instructions, bit for bit the
// fp64 product for every input (normal: the exponent field moves by one;
// zero and subnormal: the magnitude bits halved to nearest even, or doubled;
// 2 x beyond the largest double: Inf; Inf and NaN pass unchanged), so the
// fp64 pipe -- which bounds these kernels on GB300 -- only carries the adds,
// subtractions and the irrational diagonal factors.  complex64: the fp32
// multiply (not the bound there).
__device__ __forceinline__ double ghalf(double x) {
  const long long b = __double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7FF);
  const long long sgn = b & (long long)0x8000000000000000ull, v = b & 0x7FFFFFFFFFFFFFFFll;
  const long long sub = sgn | ((v >> 1) + ((v & (v >> 1)) & 1));         // e <= 1: v / 2, ties to even
  return __longlong_as_double(e >= 2 && e < 0x7FF ? b - (1ll << 52) : (e < 2 ? sub : b));
}
__device__ __forceinline__ double gtwice(double x) {
  const long long b = __double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7FF);
  const long long sgn = b & (long long)0x8000000000000000ull, v = b & 0x7FFFFFFFFFFFFFFFll;
  return __longlong_as_double(e == 0 ? (sgn | (v << 1))
                                     : e < 0x7FE ? b + (1ll << 52) : (e == 0x7FE ? (sgn | 0x7FF0000000000000ll) : b));
}
__device__ __forceinline__ float ghalf(float x) { return __fmul_rn(x, 0.5f); }
__device__ __forceinline__ float gtwice(float x) { return __fmul_rn(x, 2.0f); }

template <class T>
struct GmConst {
  T hc[kGmMaxD];   // c_l / 2: the decomposition's diagonal factors (l >= 1)
  T c[kGmMaxD];    // c_l: the composition's diagonal factors
  T lc[kGmMaxD];   // l c_l
  T l[kGmMaxD];    // l (as T)
  T inv_d;         // 1 / d (the identity's coefficient)
  T scale;         // factor on every output of this launch (the composition's last level)
  int scaled;      // scale != 1
};

// The two parts of a level, on registers: an off-diagonal pair (a = x_jk,
// b = x_kj, j < k) and the diagonal, each in place.
template <bool kDec, class S>
__device__ __forceinline__ void gm_pair(S& a, S& b) {
  const S x = a, z = b;
  if constexpr (kDec) {
    a = {ghalf(gadd(x.x, z.x)), ghalf(gadd(x.y, z.y))};
    const auto tr = ghalf(gsub(x.x, z.x)), ti = ghalf(gsub(x.y, z.y));
    b = {-ti, tr};                                             // i (x - z) / 2
  } else {
    a = {gadd(x.x, z.y), gsub(x.y, z.x)};                      // x - i z
    b = {gsub(x.x, z.y), gadd(x.y, z.x)};                      // x + i z
  }
}

template <class T, int D, bool kDec, class S>
__device__ __forceinline__ void gm_diag(S (&x)[D], const GmConst<T>& k) {
  if constexpr (kDec) {
    S P = x[0];                                                // running sum_{m<l} x_mm
#pragma unroll
    for (int l = 1; l < D; ++l) {
      const S xl = x[l];
      S lx = xl;                                               // l x_ll
      if (l == 2) lx = S{gtwice(xl.x), gtwice(xl.y)};
      if (l >= 3) lx = S{gmul(k.l[l], xl.x), gmul(k.l[l], xl.y)};
      if (l == 1)                                              // c_1 / 2 = 1/2 exactly
        x[l] = {ghalf(gsub(P.x, lx.x)), ghalf(gsub(P.y, lx.y))};
      else
        x[l] = {gmul(k.hc[l], gsub(P.x, lx.x)), gmul(k.hc[l], gsub(P.y, lx.y))};
      P = {gadd(P.x, xl.x), gadd(P.y, xl.y)};
    }
    if constexpr (D == 2) x[0] = {ghalf(P.x), ghalf(P.y)};
    else x[0] = {gmul(P.x, k.inv_d), gmul(P.y, k.inv_d)};
  } else {
    const S y0 = x[0];
    S Q = {T(0), T(0)};                                        // running sum_{l>m} c_l y_ll
#pragma unroll
    for (int m = D - 1; m >= 1; --m) {
      const S ym = x[m];
      // c_1 = 1 and 1 c_1 = 1 exactly: no multiply for m = 1
      const S cy = m == 1 ? ym : S{gmul(k.c[m], ym.x), gmul(k.c[m], ym.y)};
      const S lcy = m == 1 ? ym : S{gmul(k.lc[m], ym.x), gmul(k.lc[m], ym.y)};
      x[m] = {gadd(y0.x, gsub(Q.x, lcy.x)), gadd(y0.y, gsub(Q.y, lcy.y))};
      Q = {gadd(Q.x, cy.x), gadd(Q.y, cy.y)};
    }
    x[0] = {gadd(y0.x, Q.x), gadd(y0.y, Q.y)};
  }
}

// A whole block of a level, in place.
template <class T, int D, bool kDec, class S>
__device__ __forceinline__ void gm_block(S (&x)[D][D], const GmConst<T>& k) {
#pragma unroll
  for (int j = 0; j < D; ++j)
#pragma unroll
    for (int i = j + 1; i < D; ++i) gm_pair<kDec>(x[j][i], x[i][j]);
  S g[D];
#pragma unroll
  for (int m = 0; m < D; ++m) g[m] = x[m][m];
  gm_diag<T, D, kDec>(g, k);
#pragma unroll
  for (int m = 0; m < D; ++m) x[m][m] = g[m];
  if (k.scaled) {
#pragma unroll
    for (int r = 0; r < D; ++r)
#pragma unroll
      for (int c = 0; c < D; ++c) x[r][c] = {gmul(x[r][c].x, k.scale), gmul(x[r][c].y, k.scale)};
  }
}

template <class T>
inline GmConst<T> gm_const(int d, double scale) {
  GmConst<T> k{};
  for (int l = 1; l < d; ++l) {
    const double c = std::sqrt(2.0 / ((double)l * (double)(l + 1)));
    k.c[l] = (T)c;
    k.hc[l] = (T)(0.5 * c);
    k.lc[l] = (T)((double)l * c);
    k.l[l] = (T)l;
  }
  k.inv_d = (T)(1.0 / d);
  k.scale = (T)scale;
  k.scaled = scale != 1.0;
  return k;
}

// n levels on complex64, several per pass (tpd_gellmann_c64.cu)
cudaError_t gellmann_c64(bool dec, const float2* src, float2* mat, int n, int d, double last_scale, cudaStream_t st);

}  // namespace tpd
