// complex128 levels of the Weyl basis in block fixed point (d = 2, 3, 4),
// several per pass over the matrix.
//
// The K levels of a pass combine only elements whose row digits exceed their
// column digits by the same a = (a_1..a_K) mod d: a *class*, d^K elements
// (c + a, c), whose weights Omega_{a,b} go to (b, a + b).  A thread takes one
// class: it loads the elements, puts them on one binary point in int64 (set by
// the largest exponent among their components, with headroom for the sums),
// applies the K levels of d-point DFTs in registers and rounds each output to
// double once (RNE).  d = 2, 4: the DFTs are exact (twiddles +-1, +-i) and the
// 1/d a power of two.  d = 3: with s = x1 + x2, u = x1 - x2,
//     y0 = x0 + s,   y1,2 = (x0 - s/2) -+ i (sqrt(3)/2) u   (decomposition),
// s/2 toward zero and (sqrt(3)/2) u to the nearest integer; the class's largest
// component lands in [2^56, 2^57) for K = 3, so a level loses a unit of 2^-57 of
// it, less than the rounding to double it replaces; 1/3^n is applied once, on the
// last pass (the passes before take a power of two instead), as a 62-bit
// fraction before the rounding.  Every step is an odd function that keeps zero, so
// zero sums stay zero, conjugate inputs stay conjugate and -A gives the negated
// weights.  Classes that meet Inf or NaN run IEEE fp64, level by level, with the
// same factor a pass (a later class may take elements from both).
//
// Why: one level a launch converts every element to int64 and back each time
// and reads and writes the whole matrix (d = 3, n = 9: 2.46 ms a level); a
// pass of three levels converts once.  Measured there: 8.9 ms (passes of 3.08,
// 2.71 and 3.04 ms, 4.0-4.6 TB/s: 138 integer instructions an element at
// twelve warps an SM, the shift / logic pipe 57 % busy) against 22.1 ms for nine
// levels and a copy of 1.8 ms before them.
//
// The outputs of class a go where class -a was read, so the two exchange
// places: a CTA holds both, one a warp, with a barrier between its loads and
// its stores (a = -a keeps to itself).  Lanes take consecutive settings of
// the other digits, i.e. consecutive columns.  The first pass (digit stride 1),
// whose own digits are the contiguous columns, stages a tile of d^K rows and
// G d^K columns in shared memory and moves it in full lines.
#include <cuda_runtime.h>
#include <stdint.h>

#include "tpd_arith.cuh"
#include "tpd_qudit.cuh"
#include "tpd_weyl.cuh"

namespace tpd {
namespace {

// round(sqrt(3) / 2 * 2^62)
constexpr unsigned long long kHalfSqrt3 = 3993837246235628775ull;

// The integer nearest to u c, c = C / 2^62 < 1, |u| < 2^62.7: an odd function
// that keeps 0 (a tie needs u C = 2^61 mod 2^62, for odd C u = +-2^61 alone).
// With u = 2^32 uh + ul, C = 2^32 ch + cl, the products by the low word of C
// that are signed take it as cl - 2^32 where cl >= 2^31 (and ch + 1), so that
// every factor is one 32-bit multiply; the discarded low half of ul cl cannot
// move the rounding.
__device__ __forceinline__ long long mul_frac(long long u, unsigned long long C) {
  const int uh = (int)(u >> 32);
  const uint32_t ul = (uint32_t)u, ch = (uint32_t)(C >> 32), cl = (uint32_t)C;
  long long t = (long long)((unsigned long long)ul * ch + __umulhi(ul, cl));
  t += (long long)uh * (int)cl + (1ll << 29);
  const long long h = (long long)uh * (int)(ch + (cl >> 31)) + (t >> 32);
  return (long long)(((unsigned long long)h << 2) | ((uint32_t)t >> 30));
}

// s / 2 toward zero
__device__ __forceinline__ long long half_tz(long long s) {
  return (s + (long long)((unsigned long long)s >> 63)) >> 1;
}

// headroom bits of K levels, the components below 2^(62 - G): d = 2, 4, sums
// of d^K components below 2^62; d = 3, of 3^K sqrt(2) times a component at
// most, below 2^62.7.
__host__ __device__ constexpr int weyl_headroom(int d, int K) {
  return d == 2 ? K : (d == 4 ? 2 * K : (K == 1 ? 2 : (K == 2 ? 3 : 5)));
}
// |v| < 2^63 times 2^-T in the normal range, also after rounding up
__device__ __forceinline__ bool weyl_fast_range(int T) { return T <= 1022 && T >= -960; }

struct WeylScale {
  int pow2;            // outputs times 2^pow2 ...
  unsigned long long frac;   // ... times frac / 2^62 (0: 1) before the rounding ...
  double mul;          // ... and times this after it (1 normally)
  double ieee[4];      // the IEEE path's factor of each level of the pass: together the pass's
  double h;            // sqrt(3) / 2
};

// Class pairs a CTA of a later pass: 128 threads, three CTAs an SM.  Warps that
// start together share the instruction cache (a class of 27 is ~4,000
// straight-line instructions): d = 3, n = 9 passes 2.77 / 3.11, 2.71 / 3.04,
// 2.78 / 3.38, 3.29 / 3.76 ms with 1, 2, 3, 6 (the barrier spans them all).
constexpr int kPairs = 2;

// classes in pairs (a, -a), two self-paired ones together; 255: none
struct ClassTab {
  uint8_t a[32];
  int units;
};

// levels of a pass on one class in IEEE arithmetic (Inf / NaN), out of line
template <int D, int K, bool kDec>
__device__ __noinline__ void weyl_class_ieee(double2* x, const WeylScale& sc) {
  constexpr int B = (int)ipow(D, K);
  Twiddles<double> tw;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    // exact for d = 2, 4; d = 3 uses h alone
    tw.re[k] = D == 2 ? (k ? -1.0 : 1.0) : (k == 0 ? 1.0 : (k == 2 ? -1.0 : 0.0));
    tw.im[k] = D == 2 ? 0.0 : (k == 1 ? 1.0 : (k == 3 ? -1.0 : 0.0));
  }
  tw.h = sc.h;
  for (int m = 0, st = 1; m < K; ++m, st *= D)
    for (int g = 0; g < B / D; ++g) {
      const int e = (g / st) * (st * D) + g % st;
      Cx<double> u[D], v[D];
#pragma unroll
      for (int c = 0; c < D; ++c) u[c] = {x[e + c * st].x, x[e + c * st].y};
      dft_ieee<double, D, kDec>(u, v, tw);
#pragma unroll
      for (int b = 0; b < D; ++b) x[e + b * st] = make_double2(v[b].re * sc.ieee[m], v[b].im * sc.ieee[m]);
    }
}

// outputs outside the normal range, out of line: int64 sums to the doubles' bits
template <int B>
__device__ __noinline__ void weyl_class_rare(longlong2* t, int T) {
  for (int e = 0; e < B; ++e) {
    t[e].x = __double_as_longlong(FixedArith::to_double_int(t[e].x, T));
    t[e].y = __double_as_longlong(FixedArith::to_double_int(t[e].y, T));
  }
}

// one d-point DFT in int64
template <int D, bool kDec>
__device__ __forceinline__ void dft_int(long long (&r)[D], long long (&i)[D]) {
  if constexpr (D == 2) {
    const long long tr = r[0] - r[1], ti = i[0] - i[1];
    r[0] += r[1]; i[0] += i[1];
    r[1] = tr; i[1] = ti;
  } else if constexpr (D == 4) {
    const long long t0r = r[0] + r[2], t0i = i[0] + i[2], t1r = r[0] - r[2], t1i = i[0] - i[2];
    const long long t2r = r[1] + r[3], t2i = i[1] + i[3], t3r = r[1] - r[3], t3i = i[1] - i[3];
    r[0] = t0r + t2r; i[0] = t0i + t2i;
    r[2] = t0r - t2r; i[2] = t0i - t2i;
    // decomposition: y1 = t1 - i t3, y3 = t1 + i t3; composition: conjugate twiddles
    constexpr int p = kDec ? 1 : 3, m = kDec ? 3 : 1;
    r[p] = t1r + t3i; i[p] = t1i - t3r;
    r[m] = t1r - t3i; i[m] = t1i + t3r;
  } else {
    const long long sr = r[1] + r[2], si = i[1] + i[2];
    const long long hr = mul_frac(r[1] - r[2], kHalfSqrt3), hi = mul_frac(i[1] - i[2], kHalfSqrt3);
    const long long mr = r[0] - half_tz(sr), mi = i[0] - half_tz(si);
    r[0] += sr; i[0] += si;
    constexpr int p = kDec ? 1 : 2, m = kDec ? 2 : 1;     // p: m - i h u
    r[p] = mr + hi; i[p] = mi - hr;
    r[m] = mr - hi; i[m] = mi + hr;
  }
}

// digit M and above of the class's K levels
template <int D, int K, bool kDec, int M, int B>
__device__ __forceinline__ void class_levels(long long (&re)[B], long long (&im)[B]) {
  if constexpr (M < K) {
    constexpr int st = (int)ipow(D, M);
#pragma unroll
    for (int g = 0; g < B / D; ++g) {
      const int e = (g / st) * (st * D) + g % st;
      long long r[D], i[D];
#pragma unroll
      for (int c = 0; c < D; ++c) { r[c] = re[e + c * st]; i[c] = im[e + c * st]; }
      dft_int<D, kDec>(r, i);
#pragma unroll
      for (int c = 0; c < D; ++c) { re[e + c * st] = r[c]; im[e + c * st] = i[c]; }
    }
    class_levels<D, K, kDec, M + 1, B>(re, im);
  }
}

// Offsets of a class's elements, additive over the digits: element v of digit
// m is at row digit v + a_m, column digit v (kShift = true), or at row digit
// v, column digit a_m + v (false); row and column strides rs, cs of digit 0.
template <int D, int K>
struct ClassOffsets {
  uint32_t o[K][D];
  __device__ __forceinline__ ClassOffsets(uint32_t a, uint32_t rs, uint32_t cs, bool shift_row) {
#pragma unroll
    for (int m = 0; m < K; ++m, rs *= D, cs *= D) {
      const uint32_t am = a % D;
      a /= D;
#pragma unroll
      for (int v = 0; v < D; ++v) {
        const uint32_t w = v + am >= D ? v + am - D : v + am;
        o[m][v] = shift_row ? w * rs + v * cs : v * rs + w * cs;
      }
    }
  }
  __device__ __forceinline__ uint32_t at(int e) const {
    uint32_t s = 0;
    int x = e;
#pragma unroll
    for (int m = 0; m < K; ++m) {
      s += o[m][x % D];
      x /= D;
    }
    return s;
  }
};

// A class in registers: loaded doubles in x (bits), outputs' bits in x.
template <int D, int K, bool kDec>
__device__ __forceinline__ void weyl_class(double2 (&x)[ipow(D, K)], const WeylScale& sc) {
  constexpr int B = (int)ipow(D, K), G = weyl_headroom(D, K);
  uint32_t h = 0;
#pragma unroll
  for (int e = 0; e < B; ++e)
    h = max(h, max((uint32_t)__double2hiint(x[e].x) & 0x7fffffffu, (uint32_t)__double2hiint(x[e].y) & 0x7fffffffu));
  const int E = (int)(h >> 20);
  if (E == 2047) {
    double2 t[B];
#pragma unroll
    for (int e = 0; e < B; ++e) t[e] = x[e];
    weyl_class_ieee<D, K, kDec>(t, sc);
#pragma unroll
    for (int e = 0; e < B; ++e) x[e] = t[e];
    return;
  }
  // onto the class's binary point: x * 2^S, S = 1084 - G - max(E, 1)
  const int sb = 9 - G - max(E, 1);
  long long re[B], im[B];
#pragma unroll
  for (int e = 0; e < B; ++e) {
    re[e] = FixedArith::to_fixed(x[e].x, sb);
    im[e] = FixedArith::to_fixed(x[e].y, sb);
  }
  class_levels<D, K, kDec, 0, B>(re, im);
  if (sc.frac != 0) {
#pragma unroll
    for (int e = 0; e < B; ++e) {
      re[e] = mul_frac(re[e], sc.frac);
      im[e] = mul_frac(im[e], sc.frac);
    }
  }
  const int T = sb + 1075 - sc.pow2;                     // value = sum * 2^-T
  if (weyl_fast_range(T)) {
    // real parts through the fp64 conversion unit, imaginary parts through
    // integer instructions (identical roundings): the pipes share the work
#pragma unroll
    for (int e = 0; e < B; ++e)
      x[e] = make_double2(FixedArith::to_double_cvt_fast(re[e], T), FixedArith::to_double_fast(im[e], T));
  } else {
    longlong2 t[B];
#pragma unroll
    for (int e = 0; e < B; ++e) t[e] = make_longlong2(re[e], im[e]);
    weyl_class_rare<B>(t, T);
#pragma unroll
    for (int e = 0; e < B; ++e) x[e] = make_double2(__longlong_as_double(t[e].x), __longlong_as_double(t[e].y));
  }
  if (sc.mul != 1.0) {
#pragma unroll
    for (int e = 0; e < B; ++e) { x[e].x *= sc.mul; x[e].y *= sc.mul; }
  }
}

// A pass after the first: digit stride s, M = N / d^K, nq = M^2 settings of
// the other digits; blockIdx.y: a pair of classes.
template <int D, int K, bool kDec>
__global__ void __launch_bounds__(64 * kPairs, 6 / kPairs)
    k_weyl_class(double2* mat, uint32_t N, uint32_t s, uint32_t M, uint32_t nq, const __grid_constant__ ClassTab tab,
                 const __grid_constant__ WeylScale sc) {
  constexpr uint32_t B = ipow(D, K);
  const uint32_t a = tab.a[2 * blockIdx.y + ((threadIdx.x >> 5) & 1)];
  const uint32_t q = (blockIdx.x * kPairs + (threadIdx.x >> 6)) * 32 + (threadIdx.x & 31);
  const bool on = a < B && q < nq;
  const uint32_t qr = q / M, qc = q - qr * M;
  const uint32_t hr = qr / s, hc = qc / s;
  double2* const p = mat + (uint32_t)((hr * s * B + (qr - hr * s)) * N + hc * s * B + (qc - hc * s));
  double2 x[B];
  if (on) {
    const ClassOffsets<D, K> in(a, s * N, s, kDec);
#pragma unroll
    for (int e = 0; e < (int)B; ++e) x[e] = p[in.at(e)];
  }
  __syncthreads();                                       // class -a is loaded, too
  if (on) {
    weyl_class<D, K, kDec>(x, sc);
    const ClassOffsets<D, K> out(a, s * N, s, !kDec);
#pragma unroll
    for (int e = 0; e < (int)B; ++e) p[out.at(e)] = x[e];
  }
}

// The first pass (s = 1): one group of d^K rows, G groups of d^K columns
// (fewer in a row group's last tile), every class of them in the CTA.
template <int D, int K, int G, bool kDec>
__global__ void __launch_bounds__((ipow(D, K) * G + 31) / 32 * 32, ipow(D, K) * G > 160 ? 2 : 4)
    k_weyl_first(const double2* src, double2* mat, uint32_t N, uint32_t M, uint32_t col_tiles,
                 const __grid_constant__ WeylScale sc) {
  constexpr uint32_t B = ipow(D, K), W = B * G;
  extern __shared__ __align__(16) unsigned char smem[];
  double2* const t = reinterpret_cast<double2*>(smem);
  const uint32_t rg = blockIdx.x / col_tiles, ct = blockIdx.x - rg * col_tiles;
  const uint32_t groups = min((uint32_t)G, M - ct * G), x0 = threadIdx.x;
  const uint32_t base = rg * B * N + ct * W + x0;
  const bool copies = x0 < groups * B;                   // column x0 of the tile
  if (copies) {
    unsigned dst = (unsigned)__cvta_generic_to_shared(t + x0);
    uint32_t g = base;
#pragma unroll 9
    for (uint32_t i = 0; i < B; ++i, g += N, dst += W * 16)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src + g) : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  const uint32_t a = threadIdx.x / G, g = threadIdx.x - a * G;
  const bool on = a < B && g < groups;
  double2* const p = t + g * B;
  double2 x[B];
  if (on) {
    const ClassOffsets<D, K> in(a, W, 1, kDec);
#pragma unroll
    for (int e = 0; e < (int)B; ++e) x[e] = p[in.at(e)];
  }
  __syncthreads();                                       // every class is in registers
  if (on) {
    weyl_class<D, K, kDec>(x, sc);
    const ClassOffsets<D, K> out(a, W, 1, !kDec);
#pragma unroll
    for (int e = 0; e < (int)B; ++e) p[out.at(e)] = x[e];
  }
  __syncthreads();
  if (copies) {
    uint32_t o = base;
#pragma unroll 9
    for (uint32_t i = 0; i < B; ++i, o += N) mat[o] = t[i * W + x0];
  }
}

using FirstFn = void (*)(const double2*, double2*, uint32_t, uint32_t, uint32_t, const WeylScale);
using PassFn = void (*)(double2*, uint32_t, uint32_t, uint32_t, uint32_t, const ClassTab, const WeylScale);

struct First {
  FirstFn fn;
  uint32_t B, G;
};
template <int D, int K, int G, bool kDec>
First first() {
  return {k_weyl_first<D, K, G, kDec>, ipow(D, K), (uint32_t)G};
}

// Column groups of the first pass's tile: what keeps twelve warps an SM busy
// (d = 3, K = 3: two CTAs of 189 of 192 threads, 82 KB each; 27 elements of 16
// bytes a thread leave no room for more).
template <bool kDec>
First pick_first(int d, int K) {
  switch (d * 8 + K) {
    case 2 * 8 + 4: return first<2, 4, 8, kDec>();
    case 2 * 8 + 3: return first<2, 3, 16, kDec>();
    case 2 * 8 + 2: return first<2, 2, 8, kDec>();
    case 2 * 8 + 1: return first<2, 1, 16, kDec>();
    case 3 * 8 + 3: return first<3, 3, 7, kDec>();
    case 3 * 8 + 2: return first<3, 2, 14, kDec>();
    case 3 * 8 + 1: return first<3, 1, 10, kDec>();
    case 4 * 8 + 2: return first<4, 2, 8, kDec>();
    default: return first<4, 1, 8, kDec>();
  }
}

template <bool kDec>
PassFn pick_pass(int d, int K) {
  switch (d * 8 + K) {
    case 2 * 8 + 4: return k_weyl_class<2, 4, kDec>;
    case 2 * 8 + 3: return k_weyl_class<2, 3, kDec>;
    case 2 * 8 + 2: return k_weyl_class<2, 2, kDec>;
    case 3 * 8 + 3: return k_weyl_class<3, 3, kDec>;
    case 3 * 8 + 2: return k_weyl_class<3, 2, kDec>;
    case 4 * 8 + 2: return k_weyl_class<4, 2, kDec>;
    default: return k_weyl_class<4, 1, kDec>;
  }
}

ClassTab class_pairs(int d, int K) {
  ClassTab t;
  for (uint8_t& a : t.a) a = 255;
  const int B = (int)ipow((uint32_t)d, K);
  int at = 0, lone = 0;
  uint8_t self[32];
  for (int a = 0; a < B; ++a) {
    int na = 0, w = 1;
    for (int m = 0, x = a; m < K; ++m, x /= d, w *= d) na += (d - x % d) % d * w;
    if (a == na) self[lone++] = (uint8_t)a;
    else if (a < na) { t.a[at++] = (uint8_t)a; t.a[at++] = (uint8_t)na; }
  }
  for (int i = 0; i < lone; ++i) t.a[at + i] = self[i];
  t.units = (at + lone + 1) / 2;
  return t;
}

// exponent of an exact power of two, else 0 with *resid = v
int split_pow2(double v, double* resid) {
  int e = 0;
  const double m = std::frexp(v, &e);
  if (m == 0.5 || m == -0.5) {
    *resid = m < 0 ? -1.0 : 1.0;
    return e - 1;
  }
  *resid = v;
  return 0;
}

template <bool kDec>
cudaError_t run(const double2* src, double2* mat, int n, int d, double last_scale, cudaStream_t st) {
  const uint32_t N = ipow((uint32_t)d, n);
  const int most = qudit_max_levels(d), passes = (n + most - 1) / most;
  int k0 = 0, taken = 0;             // taken: powers of two applied by the passes so far (d = 3)
  for (int p = 0; p < passes; ++p) {
    const int K = n / passes + (p < n % passes ? 1 : 0);
    const bool last = p + 1 == passes;
    WeylScale sc;
    sc.pow2 = 0; sc.frac = 0; sc.mul = 1.0;
    sc.h = std::sqrt(3.0) * 0.5;
    double whole = 1.0;               // the factor of the pass, on either path (their classes meet in later passes)
    if (!kDec) {
      if (last) {
        whole = last_scale;
        sc.pow2 = split_pow2(last_scale, &sc.mul);
      }
    } else if (d != 3) {
      sc.pow2 = d == 2 ? -K : -2 * K;
      whole = std::ldexp(1.0, sc.pow2);
    } else if (!last) {
      // 3^K / 2^sc in [1/2, 1): the values never grow from pass to pass
      const int take = K == 1 ? 2 : (K == 2 ? 4 : 5);
      sc.pow2 = -take;
      whole = std::ldexp(1.0, -take);
      taken += take;
    } else {
      // 2^taken / 3^n = 2^pow2 frac / 2^62, the fraction in [1/2, 1)
      const unsigned long long t3 = ipow(3u, n);
      int e = 0;
      while ((1ull << e) < t3) ++e;                       // 2^(e-1) < 3^n < 2^e
      sc.frac = (unsigned long long)((((unsigned __int128)1 << (62 + e - 1)) + t3 / 2) / t3);
      sc.pow2 = taken - (e - 1);
      whole = std::ldexp(1.0, taken) / (double)t3;
    }
    // (a decomposition's levels before the last by 1/2 or 1/4, exactly: the values never grow)
    const double each = kDec ? (d == 2 ? 0.5 : 0.25) : 1.0;
    for (int m = 0; m < 4; ++m) sc.ieee[m] = each;
    for (int m = 0; m + 1 < K; ++m) whole /= each;
    sc.ieee[K - 1] = whole;
    cudaError_t e;
    if (p == 0) {
      const First f = pick_first<kDec>(d, K);
      const size_t bytes = (size_t)f.B * f.B * f.G * sizeof(double2);
      if ((e = ensure_smem_limit((const void*)f.fn, bytes)) != cudaSuccess) return e;
      const uint32_t M = N / f.B, col_tiles = (M + f.G - 1) / f.G;
      f.fn<<<M * col_tiles, (f.B * f.G + 31) / 32 * 32, bytes, st>>>(src, mat, N, M, col_tiles, sc);
    } else {
      const uint32_t M = N / ipow((uint32_t)d, K), nq = M * M;
      const ClassTab tab = class_pairs(d, K);
      pick_pass<kDec>(d, K)<<<dim3((nq + 32 * kPairs - 1) / (32 * kPairs), (unsigned)tab.units), 64 * kPairs, 0, st>>>(mat, N, ipow((uint32_t)d, k0), M,
                                                                                       nq, tab, sc);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k0 += K;
  }
  return cudaSuccess;
}

}  // namespace

cudaError_t weyl_fixed(bool dec, const double2* src, double2* mat, int n, int d, double last_scale, cudaStream_t st) {
  return dec ? run<true>(src, mat, n, d, 1.0, st) : run<false>(src, mat, n, d, last_scale, st);
}

}  // namespace tpd
