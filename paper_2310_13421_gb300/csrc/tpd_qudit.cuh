// Several qudit levels of a complex64 Weyl-basis decomposition (or composition)
// in one pass over the matrix (tpd_weyl_c64.cu), and the levels per pass
// that the other qudit kernels share.
//
// A level acts on every d x d block of one qudit's row and column digits,
// all other digits fixed, and the levels of different qudits commute.  A pass
// of K levels (digit strides s, s d, ..., s d^(K-1)) works on tiles of
// d^K x d^K digit values times P others, held in shared memory: the tile is
// copied in (cp.async, one element each), each level but the last updates it
// in place block by block -- one thread a block, d^2 elements in registers --
// and the last level stores its outputs to global memory.  Every level
// applies the operations, and the roundings, that it applies alone.
//
// Why: a level on its own reads and writes the whole matrix, and complex64
// levels are bound by that traffic, so the passes, not the levels, set the
// time: d = 3, n = 9 decomposition 9.63 ms in nine levels, 5.07 ms in three
// passes of three (3.7 TB/s; a capture of the same tiles with the Gell-Mann map
// had shared-memory wavefronts 60-73 % busy and 77 instructions an element).
//
// Tile layout.  k0 > 0 (s >= P): P = d^LP0 consecutive columns share the other
// digits; an element is at ((i B + j) P + p), B = d^K.  The runs of P
// elements start anywhere (d^n is rarely even), so consecutive CTAs take
// consecutive runs and meet their neighbours' half sectors in L2.  k0 = 0
// (s = 1): the levels' columns are contiguous themselves; PM = d^LPM adjacent
// column groups make the tile, an element is at ((i PM + g) B + j).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace tpd {

// defined in tpd_kernels_c128.cu (see tpd_kernels_impl.cuh)
cudaError_t ensure_smem_limit(const void* fn, size_t bytes);

__host__ __device__ constexpr uint32_t ipow(uint32_t d, int k) { return k <= 0 ? 1u : d * ipow(d, k - 1); }

constexpr int kQuditThreads = 256;

struct QuditPass {
  const float2* src;         // only read; may be mat
  float2* mat;
  uint32_t N;                // d^n
  uint32_t s;                // digit stride of the pass's first level
  uint32_t col_tiles;        // tiles per row group
};

// Op: the level's map on a block, Op::block<D>(x, y, c, last): y from x.
// CTAs per SM: 4 (64 registers) while a block's inputs and outputs fit.
template <class Op, int D, int K, int LP0, int LPM>
__global__ void __launch_bounds__(kQuditThreads, D <= 3 ? 4 : 2)
    k_qudit_pass(const QuditPass a, const typename Op::Const c) {
  static_assert(LP0 == 0 || LPM == 0, "passenger columns or column groups");
  constexpr uint32_t B = ipow(D, K), P = ipow(D, LP0), W = B * P * ipow(D, LPM), T = B * W;
  extern __shared__ __align__(16) unsigned char smem[];
  float2* const t = reinterpret_cast<float2*>(smem);
  const uint32_t rg = blockIdx.x / a.col_tiles, ct = blockIdx.x - rg * a.col_tiles;
  // first row and column of the tile, and the row stride of digit value i
  uint32_t row0, col0;
  if constexpr (LP0 > 0) {
    const uint32_t hr = rg / a.s, lr = rg - hr * a.s;
    const uint32_t per = a.s / P, hc = ct / per, lc = ct - hc * per;
    row0 = hr * a.s * B + lr;
    col0 = hc * a.s * B + lc * P;
  } else {
    row0 = rg * B;                                       // s = 1
    col0 = ct * W;
  }
  const uint32_t base = row0 * a.N + col0;               // element indices: N <= 65536, so below 2^32
  const uint32_t rs = LP0 > 0 ? a.s * a.N : a.N;
  for (uint32_t e = threadIdx.x; e < T; e += blockDim.x) {
    const uint32_t i = e / W, x = e - i * W;
    uint32_t off = x;
    if constexpr (LP0 > 0) {
      const uint32_t j = x / P;
      off = j * a.s + (x - j * P);
    }
    const unsigned dst = (unsigned)__cvta_generic_to_shared(t + e);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(a.src + (uint32_t)(base + i * rs + off))
                 : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
#pragma unroll
  for (int l = 0; l < K; ++l) {
    // the block's other digits: lo below the column digit, mid between the
    // two, hi above the row digit
    const uint32_t cs = P * ipow(D, l), bs = W * ipow(D, l);   // strides of the column and row digit
    const uint32_t nlo = cs, nmid = bs / (cs * D);
    for (uint32_t q = threadIdx.x; q < T / (D * D); q += blockDim.x) {
      const uint32_t q1 = q / nlo, lo = q - q1 * nlo;
      const uint32_t hi = q1 / nmid, mid = q1 - hi * nmid;
      float2 x[D][D], y[D][D];
      const float2* const in = t + (lo + mid * (cs * D) + hi * (bs * D));
#pragma unroll
      for (int r = 0; r < D; ++r)
#pragma unroll
        for (int k = 0; k < D; ++k) x[r][k] = in[r * bs + k * cs];
      Op::template block<D>(x, y, c, l + 1 == K);
      if (l + 1 < K) {
        float2* const o = t + (lo + mid * (cs * D) + hi * (bs * D));
#pragma unroll
        for (int r = 0; r < D; ++r)
#pragma unroll
          for (int k = 0; k < D; ++k) o[r * bs + k * cs] = y[r][k];
      } else {
        // the last level: column lo + k cs (+ its group), row mid' + r B / D
        uint32_t off, crow, ccol;
        if constexpr (LP0 > 0) {
          const uint32_t j = lo / P;                     // mid: the row's lower digits
          off = mid * rs + j * a.s + (lo - j * P);
          ccol = (B / D) * a.s;
        } else {
          const uint32_t i = mid / ipow(D, LPM), g = mid - i * ipow(D, LPM);
          off = i * rs + g * B + lo;
          ccol = B / D;
        }
        crow = (B / D) * rs;
#pragma unroll
        for (int r = 0; r < D; ++r)
#pragma unroll
          for (int k = 0; k < D; ++k) a.mat[(uint32_t)(base + off + r * crow + k * ccol)] = y[r][k];
      }
    }
    if (l + 1 < K) __syncthreads();
  }
}

template <class Op>
struct QuditKernel {
  void (*fn)(const QuditPass, const typename Op::Const);
  uint32_t per_tile_cols;    // columns of a tile: B P PM
  uint32_t tile;             // elements
};

template <class Op, int D, int K, int LP0, int LPM>
QuditKernel<Op> qudit_kernel() {
  return {k_qudit_pass<Op, D, K, LP0, LPM>, ipow(D, K + LP0 + LPM), ipow(D, 2 * K + LP0 + LPM)};
}

// Levels per pass at most: tiles of up to 52 KB (d = 3: 27 x 27 x 9) with the
// longest runs that leave four CTAs an SM.  (The complex64 Gell-Mann passes
// follow it; the block fixed point has fixed_max_levels, tpd_weyl_fixed.cu.)
constexpr int qudit_max_levels(int d) { return d == 2 ? 4 : (d == 3 ? 3 : 2); }

// The kernel of a pass of K levels from level k0 of n: the most columns
// beside the levels' own that the matrix has there, up to tiles of 2^11 to
// 3^8 elements (the passes of fewer levels take more columns).
template <class Op>
QuditKernel<Op> pick_qudit(int d, int K, int k0, int n) {
  const int up = n - K;
  if (k0 == 0) {
    switch (d * 8 + K) {
      case 2 * 8 + 4: return up >= 3 ? qudit_kernel<Op, 2, 4, 0, 3>() : qudit_kernel<Op, 2, 4, 0, 0>();
      case 2 * 8 + 3:
        return up >= 5 ? qudit_kernel<Op, 2, 3, 0, 5>()
                       : (up >= 2 ? qudit_kernel<Op, 2, 3, 0, 2>() : qudit_kernel<Op, 2, 3, 0, 0>());
      case 2 * 8 + 2: return qudit_kernel<Op, 2, 2, 0, 0>();
      case 2 * 8 + 1: return qudit_kernel<Op, 2, 1, 0, 0>();
      case 3 * 8 + 3: return up >= 2 ? qudit_kernel<Op, 3, 3, 0, 2>() : qudit_kernel<Op, 3, 3, 0, 0>();
      case 3 * 8 + 2: return up >= 2 ? qudit_kernel<Op, 3, 2, 0, 2>() : qudit_kernel<Op, 3, 2, 0, 0>();
      case 3 * 8 + 1: return qudit_kernel<Op, 3, 1, 0, 0>();
      case 4 * 8 + 2: return up >= 2 ? qudit_kernel<Op, 4, 2, 0, 2>() : qudit_kernel<Op, 4, 2, 0, 0>();
      case 4 * 8 + 1: return qudit_kernel<Op, 4, 1, 0, 0>();
      case 5 * 8 + 2: return up >= 1 ? qudit_kernel<Op, 5, 2, 0, 1>() : qudit_kernel<Op, 5, 2, 0, 0>();
      default: return qudit_kernel<Op, 5, 1, 0, 0>();
    }
  }
  switch (d * 8 + K) {
    case 2 * 8 + 4: return qudit_kernel<Op, 2, 4, 4, 0>();
    case 2 * 8 + 3: return k0 >= 6 ? qudit_kernel<Op, 2, 3, 6, 0>() : qudit_kernel<Op, 2, 3, 3, 0>();
    case 2 * 8 + 2: return qudit_kernel<Op, 2, 2, 3, 0>();
    case 3 * 8 + 3: return qudit_kernel<Op, 3, 3, 2, 0>();
    case 3 * 8 + 2: return k0 >= 3 ? qudit_kernel<Op, 3, 2, 3, 0>() : qudit_kernel<Op, 3, 2, 2, 0>();
    case 4 * 8 + 2: return qudit_kernel<Op, 4, 2, 2, 0>();
    case 4 * 8 + 1: return k0 >= 4 ? qudit_kernel<Op, 4, 1, 4, 0>() : qudit_kernel<Op, 4, 1, 2, 0>();
    case 5 * 8 + 2: return qudit_kernel<Op, 5, 2, 1, 0>();
    default: return k0 >= 3 ? qudit_kernel<Op, 5, 1, 3, 0>() : qudit_kernel<Op, 5, 1, 2, 0>();
  }
}

// All n levels, level 0 first: as few passes as the tiles allow, of sizes as
// equal as can be, the larger first.  src may be mat; only the first pass
// reads it.  consts(last): the level constants of a pass (last: the pass that
// applies a composition's scale).
template <class Op, class Consts>
cudaError_t run_qudit(const float2* src, float2* mat, int n, int d, Consts consts, cudaStream_t st) {
  const uint32_t N = ipow((uint32_t)d, n);
  const int most = qudit_max_levels(d), passes = (n + most - 1) / most;
  int k0 = 0;
  for (int p = 0; p < passes; ++p) {
    const int K = n / passes + (p < n % passes ? 1 : 0);
    const QuditKernel<Op> k = pick_qudit<Op>(d, K, k0, n);
    QuditPass a;
    a.src = p == 0 ? src : mat;
    a.mat = mat;
    a.N = N;
    a.s = ipow((uint32_t)d, k0);
    a.col_tiles = N / k.per_tile_cols;
    const unsigned long long tiles = (unsigned long long)(N / ipow((uint32_t)d, K)) * a.col_tiles;
    const size_t bytes = (size_t)k.tile * sizeof(float2);
    cudaError_t e = ensure_smem_limit((const void*)k.fn, bytes);
    if (e != cudaSuccess) return e;
    const uint32_t blocks = k.tile / (uint32_t)(d * d);
    const uint32_t threads = blocks >= (uint32_t)kQuditThreads ? (uint32_t)kQuditThreads : (blocks + 31) / 32 * 32;
    k.fn<<<(unsigned)tiles, threads, bytes, st>>>(a, consts(p + 1 == passes));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k0 += K;
  }
  return cudaSuccess;
}

}  // namespace tpd
