// complex64 levels of the generalized Gell-Mann basis, several per pass over
// the matrix.
//
// A level only combines x_jk with x_kj, and the diagonal x_mm among
// themselves, and leaves the results at the same positions.  So the d^2
// digit values of one qudit fall into closed sets -- d (d-1) / 2 pairs and the
// diagonal -- and those of K qudits into the products of K such sets, of 2^K to
// d^K elements (d = 3, K = 3: 64 sets of 8 to 27 elements).  A thread takes a
// closed set: it loads the elements, applies the K levels in registers, in
// the order and with the roundings of single levels, and stores them where they were; no
// two threads touch the same element, so nothing is exchanged or waited for.
// A level on its own reads and writes the whole matrix, which is what bounds
// it (d = 3, n = 9: 1.06 ms a level, 5.86 TB/s): the passes set the time.
//
// Lanes.  The passes after the first (digit stride s > 1): consecutive lanes
// take consecutive settings of the other digits, i.e. consecutive columns, and
// all of a warp's lanes the same set, so the pattern (pair or diagonal per
// digit) is uniform.  The first pass (s = 1), whose own digits are the
// contiguous columns, copies a tile of d^K rows by PM d^K columns into shared
// memory and back in full lines, and lanes take the PM column groups and the
// sets of one pattern.
//
// Measured (GB300, d = 3, n = 9, 6.2 GB moved a pass): first pass 1.25 ms
// (4.9 TB/s: issue and the barriers between its copy and its sets), s = 27
// 1.15 ms, s = 729 1.01 ms (6.2 TB/s); the decomposition 10.5 -> 3.41 ms against
// single levels after a copy, and 5.13 ms with the three levels of a tile
// exchanged block by block through shared memory (bank conflicts and index
// arithmetic: 77 instructions an element against 27).  Three CTAs of 256 threads an SM (80
// registers; the 27-element set spills 100 bytes): two 1.19 / 1.10, four 1.15 /
// 1.01, five 1.25 / 1.11 ms for the later passes; the first pass at four 1.43
// ms, and 1.42-1.96 ms with a third of the columns in a tile.
#include "tpd_gellmann.cuh"
#include "tpd_qudit.cuh"

namespace tpd {
namespace {

constexpr int kGmThreads = 256;
constexpr int kGmWarps = kGmThreads / 32;

// pair p of d digits: (0,1), (0,2), (1,2), (0,3), (1,3), (2,3), (0,4), ...
// (3 bits a pair: the ten of d = 5 fit a word)
__device__ __forceinline__ uint32_t pair_lo(uint32_t p) { return (0x1a211040u >> (3 * p)) & 7u; }
__device__ __forceinline__ uint32_t pair_hi(uint32_t p) { return (0x2491b691u >> (3 * p)) & 7u; }

// Pattern Pat (bit m set: digit m's set is the diagonal): the set's elements
// per value of digit M, and the digit's values.
template <int D, int Pat, int M>
struct SetShape {
  static constexpr int kDigits = ((Pat >> M) & 1) ? D : 2;
  static constexpr int kStride = SetShape<D, Pat, M - 1>::kStride * SetShape<D, Pat, M - 1>::kDigits;
};
template <int D, int Pat>
struct SetShape<D, Pat, 0> {
  static constexpr int kDigits = (Pat & 1) ? D : 2;
  static constexpr int kStride = 1;
};

// offsets of a digit's set elements: pairs (j,k) at o0 and (k,j) at o1, the
// diagonal's v at v * o0
struct SetDigit {
  uint32_t o0, o1;
};

// offset of element e of a set
template <int D, int Pat, int M, int K>
__device__ __forceinline__ uint32_t set_offset(int e, const SetDigit (&dg)[K]) {
  if constexpr (M == K) {
    return 0u;
  } else {
    using Sh = SetShape<D, Pat, M>;
    const int v = (e / Sh::kStride) % Sh::kDigits;
    uint32_t o;
    if constexpr (((Pat >> M) & 1) != 0) o = (uint32_t)v * dg[M].o0;
    else o = v ? dg[M].o1 : dg[M].o0;
    return o + set_offset<D, Pat, M + 1, K>(e, dg);
  }
}

// levels M, M + 1, ... on a set in registers
template <int D, int Pat, int M, int K, bool kDec, int S>
__device__ __forceinline__ void set_levels(float2 (&x)[S], const GmConst<float>& c) {
  if constexpr (M < K) {
    constexpr int st = SetShape<D, Pat, M>::kStride, nd = SetShape<D, Pat, M>::kDigits;
#pragma unroll
    for (int hi = 0; hi < S / (st * nd); ++hi)
#pragma unroll
      for (int lo = 0; lo < st; ++lo) {
        const int e = hi * (st * nd) + lo;
        if constexpr (((Pat >> M) & 1) != 0) {
          float2 g[D];
#pragma unroll
          for (int v = 0; v < D; ++v) g[v] = x[e + v * st];
          gm_diag<float, D, kDec>(g, c);
#pragma unroll
          for (int v = 0; v < D; ++v) x[e + v * st] = g[v];
        } else {
          gm_pair<kDec>(x[e], x[e + st]);
        }
      }
    set_levels<D, Pat, M + 1, K, kDec, S>(x, c);
  }
}

// The K levels on the closed set with these digits, from `in` to `out` (element `base` on).
template <int D, int K, int Pat, bool kDec>
__device__ __forceinline__ void gm_set(const float2* in, float2* out, uint32_t base, const SetDigit (&dg)[K],
                                       const GmConst<float>& c, bool last) {
  constexpr int S = SetShape<D, Pat, K - 1>::kStride * SetShape<D, Pat, K - 1>::kDigits;
  float2 x[S];
#pragma unroll
  for (int e = 0; e < S; ++e) x[e] = in[base + set_offset<D, Pat, 0, K>(e, dg)];
  set_levels<D, Pat, 0, K, kDec, S>(x, c);
  if (last && c.scaled) {
#pragma unroll
    for (int e = 0; e < S; ++e) x[e] = {gmul(x[e].x, c.scale), gmul(x[e].y, c.scale)};
  }
#pragma unroll
  for (int e = 0; e < S; ++e) out[base + set_offset<D, Pat, 0, K>(e, dg)] = x[e];
}

// gm_set for a run-time pattern
template <int D, int K, bool kDec, int Pat = 0>
__device__ __forceinline__ void gm_set_of(int pat, const float2* in, float2* out, uint32_t base,
                                          const SetDigit (&dg)[K], const GmConst<float>& c, bool last) {
  if constexpr (Pat + 1 < (1 << K)) {
    if (pat != Pat) {
      gm_set_of<D, K, kDec, Pat + 1>(pat, in, out, base, dg, c, last);
      return;
    }
  }
  gm_set<D, K, Pat, kDec>(in, out, base, dg, c, last);
}

// A pass after the first.  CTA: 32 settings of the other digits (one a lane);
// its warps take the sets in turn.  M = N / d^K, nq = M^2.
template <int D, int K, bool kDec>
__global__ void __launch_bounds__(kGmThreads, 3)
    k_gm_pass(const float2* src, float2* mat, uint32_t N, uint32_t s, uint32_t M, uint32_t nq, const GmConst<float> c,
              int last) {
  constexpr uint32_t B = ipow(D, K), NP = D * (D - 1) / 2, NT = ipow(NP + 1, K);
  const uint32_t q = blockIdx.x * 32 + (threadIdx.x & 31);
  if (q >= nq) return;
  const uint32_t qr = q / M, qc = q - qr * M;
  const uint32_t hr = qr / s, hc = qc / s;
  const uint32_t base = (hr * s * B + (qr - hr * s)) * N + hc * s * B + (qc - hc * s);
  for (uint32_t t = threadIdx.x >> 5; t < NT; t += kGmWarps) {
    SetDigit dg[K];
    int pat = 0;
    uint32_t u = t, w = s;
#pragma unroll
    for (int m = 0; m < K; ++m, w *= D) {
      const uint32_t p = u % (NP + 1);
      u /= NP + 1;
      if (p == NP) {
        pat |= 1 << m;
        dg[m] = {w * (N + 1), 0u};
      } else {
        dg[m] = {w * (pair_lo(p) * N + pair_hi(p)), w * (pair_hi(p) * N + pair_lo(p))};
      }
    }
    gm_set_of<D, K, kDec>(pat, src, mat, base, dg, c, last != 0);
  }
}

// The sets of pattern Pat (and the patterns after it) of a tile in shared
// memory, rows of W elements, PM column groups.  Each pattern's items start
// at the warp after the last pattern's, so that no warp gets all the short ones.
template <int D, int K, bool kDec, int PM, int Pat = 0>
__device__ __forceinline__ void gm_tile_sets(float2* t, uint32_t warp0, const GmConst<float>& c, bool last) {
  if constexpr (Pat < (1 << K)) {
    constexpr uint32_t W = PM * ipow(D, K), NP = D * (D - 1) / 2;
    uint32_t n = PM;
#pragma unroll
    for (int m = 0; m < K; ++m)
      if (!((Pat >> m) & 1)) n *= NP;
    const uint32_t nw = blockDim.x / 32;
    const uint32_t warp = threadIdx.x / 32 >= warp0 ? threadIdx.x / 32 - warp0 : threadIdx.x / 32 + nw - warp0;
    for (uint32_t it = warp * 32 + (threadIdx.x & 31); it < n; it += blockDim.x) {
      uint32_t u = it / PM, w = 1;
      const uint32_t g = it - u * PM;
      SetDigit dg[K];
#pragma unroll
      for (int m = 0; m < K; ++m, w *= D) {
        if ((Pat >> m) & 1) {
          dg[m] = {w * (W + 1), 0u};
        } else {
          const uint32_t p = u % NP;
          u /= NP;
          dg[m] = {w * (pair_lo(p) * W + pair_hi(p)), w * (pair_hi(p) * W + pair_lo(p))};
        }
      }
      gm_set<D, K, Pat, kDec>(t, t, g * ipow(D, K), dg, c, last);
    }
    gm_tile_sets<D, K, kDec, PM, Pat + 1>(t, (warp0 + (n + 31) / 32) % nw, c, last);
  }
}

// The first pass (s = 1).  CTA: one group of d^K rows, PM groups of d^K columns.
template <int D, int K, int LPM, bool kDec>
__global__ void __launch_bounds__(kGmThreads, 3)
    k_gm_first(const float2* src, float2* mat, uint32_t N, uint32_t col_tiles, const GmConst<float> c, int last) {
  constexpr uint32_t B = ipow(D, K), PM = ipow(D, LPM), W = PM * B;
  extern __shared__ __align__(16) unsigned char smem[];
  float2* const t = reinterpret_cast<float2*>(smem);
  const uint32_t rg = blockIdx.x / col_tiles, ct = blockIdx.x - rg * col_tiles;
  // thread: column x of every kRows-th row of the tile (W <= 256)
  static_assert(W <= (uint32_t)kGmThreads, "a row is copied by one thread per column");
  constexpr uint32_t kRows = kGmThreads / W;
  const uint32_t i0 = threadIdx.x / W, x = threadIdx.x - i0 * W;
  const uint32_t base = rg * B * N + ct * W + i0 * N + x;
  const bool copies = i0 < kRows;
  if (copies) {
    unsigned dst = (unsigned)__cvta_generic_to_shared(t + (i0 * W + x));
    uint32_t g = base;
#pragma unroll 9
    for (uint32_t i = i0; i < B; i += kRows, g += kRows * N, dst += kRows * W * 8)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src + g) : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  gm_tile_sets<D, K, kDec, (int)PM>(t, 0u, c, last != 0);
  __syncthreads();
  if (copies) {
    uint32_t g = base;
#pragma unroll 9
    for (uint32_t i = i0; i < B; i += kRows, g += kRows * N) mat[g] = t[i * W + x];
  }
}

using FirstKernel = void (*)(const float2*, float2*, uint32_t, uint32_t, const GmConst<float>, int);
using PassKernelGm = void (*)(const float2*, float2*, uint32_t, uint32_t, uint32_t, uint32_t, const GmConst<float>,
                              int);

struct First {
  FirstKernel fn;
  uint32_t cols, tile;
};
template <int D, int K, int LPM, bool kDec>
First first() {
  return {k_gm_first<D, K, LPM, kDec>, ipow(D, K + LPM), ipow(D, 2 * K + LPM)};
}

// The first pass's kernel: as many column groups as the matrix has (up = n - K
// digits above), up to 52 KB tiles (three CTAs an SM, as for the later passes).
template <bool kDec>
First pick_first(int d, int K, int up) {
  switch (d * 8 + K) {
    case 2 * 8 + 4: return up >= 3 ? first<2, 4, 3, kDec>() : first<2, 4, 0, kDec>();
    case 2 * 8 + 3:
      return up >= 5 ? first<2, 3, 5, kDec>() : (up >= 2 ? first<2, 3, 2, kDec>() : first<2, 3, 0, kDec>());
    case 2 * 8 + 2: return first<2, 2, 0, kDec>();
    case 2 * 8 + 1: return first<2, 1, 0, kDec>();
    case 3 * 8 + 3: return up >= 2 ? first<3, 3, 2, kDec>() : first<3, 3, 0, kDec>();
    case 3 * 8 + 2: return up >= 2 ? first<3, 2, 2, kDec>() : first<3, 2, 0, kDec>();
    case 3 * 8 + 1: return first<3, 1, 0, kDec>();
    case 4 * 8 + 2: return up >= 2 ? first<4, 2, 2, kDec>() : first<4, 2, 0, kDec>();
    case 4 * 8 + 1: return first<4, 1, 0, kDec>();
    case 5 * 8 + 2: return up >= 1 ? first<5, 2, 1, kDec>() : first<5, 2, 0, kDec>();
    default: return first<5, 1, 0, kDec>();
  }
}

template <bool kDec>
PassKernelGm pick_pass(int d, int K) {
  switch (d * 8 + K) {
    case 2 * 8 + 4: return k_gm_pass<2, 4, kDec>;
    case 2 * 8 + 3: return k_gm_pass<2, 3, kDec>;
    case 2 * 8 + 2: return k_gm_pass<2, 2, kDec>;
    case 3 * 8 + 3: return k_gm_pass<3, 3, kDec>;
    case 3 * 8 + 2: return k_gm_pass<3, 2, kDec>;
    case 4 * 8 + 2: return k_gm_pass<4, 2, kDec>;
    case 4 * 8 + 1: return k_gm_pass<4, 1, kDec>;
    case 5 * 8 + 2: return k_gm_pass<5, 2, kDec>;
    default: return k_gm_pass<5, 1, kDec>;
  }
}

// All n levels, level 0 first: as few passes as possible, of sizes as equal as
// can be, the larger first (a pass of one level after the first: d = 4, 5 only).
template <bool kDec>
cudaError_t run(const float2* src, float2* mat, int n, int d, double last_scale, cudaStream_t st) {
  const uint32_t N = ipow((uint32_t)d, n);
  const int most = qudit_max_levels(d), passes = (n + most - 1) / most;
  int k0 = 0;
  for (int p = 0; p < passes; ++p) {
    const int K = n / passes + (p < n % passes ? 1 : 0), last = p + 1 == passes;
    const GmConst<float> c = gm_const<float>(d, last ? last_scale : 1.0);
    cudaError_t e;
    if (p == 0) {
      const First f = pick_first<kDec>(d, K, n - K);
      const size_t bytes = (size_t)f.tile * sizeof(float2);
      if ((e = ensure_smem_limit((const void*)f.fn, bytes)) != cudaSuccess) return e;
      const uint32_t col_tiles = N / f.cols;
      f.fn<<<N / ipow((uint32_t)d, K) * col_tiles, kGmThreads, bytes, st>>>(src, mat, N, col_tiles, c, last);
    } else {
      const uint32_t M = N / ipow((uint32_t)d, K), nq = M * M;
      pick_pass<kDec>(d, K)<<<(nq + 31) / 32, kGmThreads, 0, st>>>(mat, mat, N, ipow((uint32_t)d, k0), M, nq, c, last);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k0 += K;
  }
  return cudaSuccess;
}

}  // namespace

cudaError_t gellmann_c64(bool dec, const float2* src, float2* mat, int n, int d, double last_scale,
                         cudaStream_t st) {
  return dec ? run<true>(src, mat, n, d, last_scale, st) : run<false>(src, mat, n, d, last_scale, st);
}

}  // namespace tpd
