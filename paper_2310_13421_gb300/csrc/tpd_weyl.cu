// Decomposition in the Weyl (clock-and-shift) basis of n qudits of dimension
// d: the tensorized basis Sec. V names as the natural next candidate for the
// method.  With omega = exp(2 pi i / d), X|j> = |j+1 mod d>, Z|j> = omega^j |j>
// and W_{a,b} = X^a Z^b (tensor products over the qudits), the weights of
// A in Mat(d^n) are c_{a,b} = d^-n tr(W_{a,b}^* A).
//
// The same recursion as Eqs. 3-5: partitioning A into d x d blocks A_{rc}
// (qudit 1's digits), A = sum_{a,b} W_{a,b} (x) Omega_{a,b} with the
// cumulative matrix weights
//     Omega_{a,b} = d^-1 sum_c omega^(-b c) A_{c+a, c}
// (the d x d analogue of Eq. 4: for each shift a, a length-d DFT along the
// block's a-th cyclic diagonal), and the levels commute.  On the GPU every
// level is applied to all d x d blocks at once, in place: several levels per
// pass over the matrix in complex64 and in the block fixed point, one launch
// per qudit, each thread one block of d^2 elements in registers, in IEEE
// fp64.  Omega_{a,b}
// goes to the block position (row digit b, column digit a + b mod d), which
// for d = 2 is where the Pauli decomposition puts I, X, Y, Z (with
// W_{1,1} = XZ = -iY).  The composition inverts each level:
// A_{c+a, c} = sum_b omega^(b c) Omega_{a,b}.
//
// Arithmetic.  complex64: IEEE fp32, rounded every level (tpd_weyl_c64.cu).
// complex128: by default (d = 2, 3, 4) a block fixed point, as for the Pauli
// basis (tpd_weyl_fixed.cu); d = 5 and TPD_PREC_PLAIN run IEEE fp64 rounded
// every level (the paper's arithmetic carried over), here.  The fp64 pipe of
// GB300 issues ~2 operations per clock per SM, far below what a level at HBM
// speed needs; integer instructions are not.  d = 3 uses the 3-point DFT
// written out (4 real additions-or-multiplications per element and level
// instead of 12): with s = x1 + x2, u = x1 - x2, m = x0 - s/2, h = sqrt(3)/2,
//     y0 = x0 + s,   y1 = m - i h u,   y2 = m + i h u     (omega^-bc)
// and the conjugate signs for the composition.
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>

#include "tpd.h"
#include "tpd_weyl.cuh"

namespace tpd {
namespace {

// One qudit level on every d x d block in IEEE fp64: digit stride s (d^k for
// qudit n - k), N = d^n, nblk = (N / D)^2 blocks; src: the level's input, mat
// itself but for the first level of an out-of-place call.
template <int D, bool kDec>
__global__ void __launch_bounds__(256) k_weyl_level(const double2* src, double2* mat, long long N, long long s,
                                                    long long nblk, const Twiddles<double> tw) {
  const long long M = N / D;                 // other-digit combinations per row / column
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < nblk;
       q += (long long)gridDim.x * blockDim.x) {
    const long long qr = q / M, qc = q - qr * M;
    const long long R = (qr / s) * s * D + qr % s;   // digit k of the row set to 0
    const long long Cc = (qc / s) * s * D + qc % s;  // and of the column
    const long long base = R * N + Cc, rs = s * N;
    double2 in[D][D], out[D][D];
#pragma unroll
    for (int r = 0; r < D; ++r)
#pragma unroll
      for (int c = 0; c < D; ++c) in[r][c] = src[base + r * rs + c * s];
    weyl_block_ieee<double, D, kDec>(in, out, tw);
#pragma unroll
    for (int r = 0; r < D; ++r)
#pragma unroll
      for (int c = 0; c < D; ++c) mat[base + r * rs + c * s] = out[r][c];
  }
}

template <bool kDec>
cudaError_t launch_levels(const double2* src, double2* m, int n, int d, double last_scale, cudaStream_t st) {
  long long N = 1;
  for (int k = 0; k < n; ++k) N *= d;
  const long long nblk = (N / d) * (N / d);   // < 2^30: N <= 65536
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  long long grid = (nblk + 255) / 256;
  if (grid > 16ll * nsm) grid = 16ll * nsm;
  if (grid < 1) grid = 1;
  const unsigned g = (unsigned)grid;
  long long s = 1;
  for (int k = 0; k < n; ++k, s *= d) {
    // the decomposition's 1/d per level; the composition's scale on its last level
    const double sc = kDec ? 1.0 / d : (k == n - 1 ? last_scale : 1.0);
    const Twiddles<double> tw = twiddles<double>(d, sc);
    switch (d) {
      case 2: k_weyl_level<2, kDec><<<g, 256, 0, st>>>(src, m, N, s, nblk, tw); break;
      case 3: k_weyl_level<3, kDec><<<g, 256, 0, st>>>(src, m, N, s, nblk, tw); break;
      case 4: k_weyl_level<4, kDec><<<g, 256, 0, st>>>(src, m, N, s, nblk, tw); break;
      default: k_weyl_level<5, kDec><<<g, 256, 0, st>>>(src, m, N, s, nblk, tw); break;
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    src = m;
  }
  return cudaSuccess;
}

tpd_status weyl_run(bool dec, const void* src, void* A, int n, int d, int dtype, double scale, const tpd_options* opt,
                    void* stream) {
  if (src == nullptr || A == nullptr || d < 2 || d > 5 || n < 1 || (dtype != TPD_C128 && dtype != TPD_C64)) return TPD_ERR_INVALID_ARG;
  // arithmetic: complex128 block fixed point (d <= 4) unless PLAIN is asked
  // for; complex64 fp32; FIXED for d = 5 or complex64 and COMPENSATED are
  // not offered
  const int prec = opt ? opt->precision : TPD_PREC_DEFAULT;
  if (prec != TPD_PREC_DEFAULT && prec != TPD_PREC_PLAIN && prec != TPD_PREC_FIXED) return TPD_ERR_INVALID_ARG;
  if (prec == TPD_PREC_FIXED && (dtype != TPD_C128 || d > 4)) return TPD_ERR_INVALID_ARG;
  const bool fixed = dtype == TPD_C128 && d <= 4 && prec != TPD_PREC_PLAIN;
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
    if (fixed) e = weyl_fixed(dec, in, out, n, d, scale, st);
    else e = dec ? launch_levels<true>(in, out, n, d, 1.0, st) : launch_levels<false>(in, out, n, d, scale, st);
  } else {
    e = weyl_c64(dec, static_cast<const float2*>(src), static_cast<float2*>(A), n, d, scale, st);
  }
  return e == cudaSuccess ? TPD_OK : TPD_ERR_CUDA;
}

}  // namespace
}  // namespace tpd

extern "C" {

tpd_status tpd_weyl_decompose(void* A, int n, int d, int dtype, const tpd_options* opt, void* stream) {
  return tpd::weyl_run(true, A, A, n, d, dtype, 1.0, opt, stream);
}

tpd_status tpd_weyl_compose(void* C, int n, int d, int dtype, double scale, const tpd_options* opt,
                            void* stream) {
  return tpd::weyl_run(false, C, C, n, d, dtype, scale, opt, stream);
}

tpd_status tpd_weyl_decompose_to(const void* A, void* C, int n, int d, int dtype, const tpd_options* opt,
                                 void* stream) {
  return tpd::weyl_run(true, A, C, n, d, dtype, 1.0, opt, stream);
}

tpd_status tpd_weyl_compose_to(const void* C, void* A, int n, int d, int dtype, double scale, const tpd_options* opt,
                               void* stream) {
  return tpd::weyl_run(false, C, A, n, d, dtype, scale, opt, stream);
}

}  // extern "C"
