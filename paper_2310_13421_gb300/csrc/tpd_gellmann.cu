// Decomposition in the generalized Gell-Mann basis of n qudits of dimension
// d: the other tensorized basis Sec. V names as a natural candidate for the
// method.  For one qudit the d^2 Hermitian elements carry a label (r, c) of
// the d x d grid: the identity at (0, 0); the diagonal
// D_l = sqrt(2 / (l (l+1))) (sum_{m<l} E_mm - l E_ll) at (l, l), l >= 1;
// the symmetric S_jk = E_jk + E_kj at (j, k) and the antisymmetric
// A_jk = -i E_jk + i E_kj at (k, j), j < k.  Their squares have trace d
// (identity) or 2 (every other element), and they are orthogonal.  For
// n qudits an element is the tensor product over the digit pairs of its
// label, with N_(r,c) the product of those traces, and
//     A = sum g_(r,c) G_(r,c),     g_(r,c) = tr(G_(r,c) A) / N_(r,c).
// For d = 2 the elements are I, X, Y, Z at the positions where Eq. 4 puts
// their weights: the Pauli decomposition itself.
//
// The recursion of Eqs. 3-5 carries over: tr((G (x) G') A) contracts qudit 1
// with G and the rest with G', so the coefficients are d x d blocks of
// cumulative weights computed level by level, one qudit at a time, in any
// order.  One level maps each d x d block x (the qudit's row and column
// digits, all other digits fixed) in place to
//     (j, k), j < k:  (x_jk + x_kj) / 2           (symmetric)
//     (k, j), j < k:  i (x_jk - x_kj) / 2         (antisymmetric)
//     (l, l), l >= 1: c_l / 2 (sum_{m<l} x_mm - l x_ll),   c_l = sqrt(2 / (l (l+1)))
//     (0, 0):         (1 / d) sum_m x_mm
// (for d = 2 exactly Eq. 4), and the composition inverts it:
//     x_jk = y_jk - i y_kj,  x_kj = y_jk + i y_kj,
//     x_mm = y_00 + sum_{l>m} c_l y_ll - m c_m y_mm.
// On the GPU every level is applied to all blocks at once.  complex128: one
// launch per qudit, each thread one block of d^2 elements held in registers,
// a grid-stride loop (bound by the fp64 pipe, so fusing levels would not help).
// complex64: several levels per pass (tpd_gellmann_c64.cu).  Arithmetic: IEEE
// fp64 (complex128) or fp32 (complex64), rounded every level, without
// contraction into fused multiply-adds, so real and imaginary parts see the
// same operations: conjugate blocks of a Hermitian input stay exact conjugates
// level by level, and its coefficients come out exactly real.
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>

#include "tpd.h"
#include "tpd_gellmann.cuh"

namespace tpd {
namespace {

// One qudit level on every d x d block: digit stride s (d^k), N = d^n,
// nblk = (N / D)^2 blocks (< 2^30 for N <= 65536).
// src: the level's input, mat itself but for the first level of an
// out-of-place call.
template <int D, bool kDec>
__global__ void __launch_bounds__(256) k_gellmann_level(const double2* src, double2* mat, uint32_t N, uint32_t s,
                                                        uint32_t nblk, const GmConst<double> k) {
  const uint32_t M = N / D;                      // combinations of the other digits per row / column
  for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < nblk; q += gridDim.x * blockDim.x) {
    const uint32_t qr = q / M, qc = q - qr * M;
    const uint32_t R = (qr / s) * s * D + qr % s;      // row with this qudit's digit 0
    const uint32_t C = (qc / s) * s * D + qc % s;      // column likewise
    const long long base = (long long)R * N + C, rs = (long long)s * N;
    double2 x[D][D];
#pragma unroll
    for (int r = 0; r < D; ++r)
#pragma unroll
      for (int c = 0; c < D; ++c) x[r][c] = src[base + r * rs + (long long)c * s];
    gm_block<double, D, kDec>(x, k);
#pragma unroll
    for (int r = 0; r < D; ++r)
#pragma unroll
      for (int c = 0; c < D; ++c) mat[base + r * rs + (long long)c * s] = x[r][c];
  }
}

template <bool kDec>
cudaError_t gm_levels(const double2* src, double2* m, int n, int d, double last_scale, cudaStream_t st) {
  uint32_t N = 1;
  for (int k = 0; k < n; ++k) N *= (uint32_t)d;
  const uint32_t nblk = (N / d) * (N / d);
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  long long grid = ((long long)nblk + 255) / 256;
  if (grid > 16ll * nsm) grid = 16ll * nsm;
  if (grid < 1) grid = 1;
  uint32_t s = 1;
  for (int k = 0; k < n; ++k, s *= (uint32_t)d) {
    const GmConst<double> kc = gm_const<double>(d, !kDec && k == n - 1 ? last_scale : 1.0);
    switch (d) {
      case 2: k_gellmann_level<2, kDec><<<(unsigned)grid, 256, 0, st>>>(src, m, N, s, nblk, kc); break;
      case 3: k_gellmann_level<3, kDec><<<(unsigned)grid, 256, 0, st>>>(src, m, N, s, nblk, kc); break;
      case 4: k_gellmann_level<4, kDec><<<(unsigned)grid, 256, 0, st>>>(src, m, N, s, nblk, kc); break;
      default: k_gellmann_level<5, kDec><<<(unsigned)grid, 256, 0, st>>>(src, m, N, s, nblk, kc); break;
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    src = m;
  }
  return cudaSuccess;
}

tpd_status gellmann_run(bool dec, const void* src, void* A, int n, int d, int dtype, double scale, const tpd_options* opt,
                        void* stream) {
  if (src == nullptr || A == nullptr || d < 2 || d > kGmMaxD || n < 1 || (dtype != TPD_C128 && dtype != TPD_C64))
    return TPD_ERR_INVALID_ARG;
  const int prec = opt ? opt->precision : TPD_PREC_DEFAULT;
  if (prec != TPD_PREC_DEFAULT && prec != TPD_PREC_PLAIN) return TPD_ERR_INVALID_ARG;
  long long N = 1;
  for (int k = 0; k < n; ++k) {
    N *= d;
    if (N > 65536) return TPD_ERR_INVALID_ARG;
  }
  if (!dec && (!std::isfinite(scale) || scale == 0.0)) return TPD_ERR_INVALID_ARG;
  const size_t align = dtype == TPD_C128 ? 16 : 8;
  const uintptr_t m = reinterpret_cast<uintptr_t>(A), sp = reinterpret_cast<uintptr_t>(src);
  if (m % align || sp % align) return TPD_ERR_MISALIGNED;
  const size_t bytes = align * (size_t)(N * N);
  if (m != sp && m < sp + bytes && sp < m + bytes) return TPD_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaError_t e;
  if (dtype == TPD_C128) {
    const double2* in = static_cast<const double2*>(src);
    double2* out = static_cast<double2*>(A);
    e = dec ? gm_levels<true>(in, out, n, d, 1.0, st) : gm_levels<false>(in, out, n, d, scale, st);
  } else {
    e = gellmann_c64(dec, static_cast<const float2*>(src), static_cast<float2*>(A), n, d, dec ? 1.0 : scale, st);
  }
  return e == cudaSuccess ? TPD_OK : TPD_ERR_CUDA;
}

}  // namespace
}  // namespace tpd

extern "C" {

tpd_status tpd_gellmann_decompose(void* A, int n, int d, int dtype, const tpd_options* opt, void* stream) {
  return tpd::gellmann_run(true, A, A, n, d, dtype, 1.0, opt, stream);
}

tpd_status tpd_gellmann_compose(void* C, int n, int d, int dtype, double scale, const tpd_options* opt,
                                void* stream) {
  return tpd::gellmann_run(false, C, C, n, d, dtype, scale, opt, stream);
}

tpd_status tpd_gellmann_decompose_to(const void* A, void* G, int n, int d, int dtype, const tpd_options* opt,
                                     void* stream) {
  return tpd::gellmann_run(true, A, G, n, d, dtype, 1.0, opt, stream);
}

tpd_status tpd_gellmann_compose_to(const void* C, void* A, int n, int d, int dtype, double scale,
                                   const tpd_options* opt, void* stream) {
  return tpd::gellmann_run(false, C, A, n, d, dtype, scale, opt, stream);
}

}  // extern "C"
