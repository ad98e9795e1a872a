// complex128 levels of the Weyl basis in block fixed point (d = 2, 3, 4),
// several per pass over the matrix.
//
// The K levels of a pass combine only elements whose row digits exceed their
// column digits by the same a = (a_1..a_K) mod d: a *class*, d^K elements
// (c + a, c), whose weights Omega_{a,b} go to (b, a + b).  A thread takes one
// class: it loads the elements, applies the K levels of d-point DFTs in
// registers in int64 and rounds each output to double once (RNE).  At every
// level the d elements that a DFT adds are on a binary point of their own, set by
// the largest among them with headroom for the sums -- from the doubles'
// exponents at the first level, from the leading bits of the sums at the
// later ones -- so elements that cancel at one level cost the small ones that
// meet the remainder at the next no bits.  d = 2, 4: the DFTs are exact (twiddles +-1,
// +-i) and the 1/d a power of two.  d = 3, doubled: with s = x1 + x2, u = x1 - x2,
//     2 y0 = 2 (x0 + s),   2 y1,2 = (2 x0 - s) -+ i sqrt(3) u   (decomposition),
// sqrt(3) u to the nearest integer; the largest component lands in [2^58, 2^59).
// 1/3^n is applied once, on the last pass (the passes before take a power of
// two instead), as a 62-bit fraction before the rounding.  Every step is an odd
// function that keeps zero, so zero sums stay zero, conjugate inputs stay
// conjugate and -A gives the negated weights.  A thread whose class meets Inf or
// NaN goes level by level, in doubles: the d elements of a DFT in IEEE fp64 if
// one of them is not finite, else as above, with the same factor a pass (a later
// class may take elements from both).
//
// Why: one level a launch converts every element to int64 and back each time
// and reads and writes the whole matrix (d = 3, n = 9: 2.46 ms a level, 22.1 ms
// and a copy of 1.8 ms before them); a pass of two converts once.  Measured there:
// 14.2 ms, passes of 2.8, 3.1, 2.9, 2.8 and (one level and 3^-n) 2.6 ms, bound by
// integer issue.  With one binary point for a whole class of 27 it was 10.0 ms in
// three passes, but elements that cancel then took the small ones' low bits along.
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

// round(sqrt(3) * 2^62)
constexpr unsigned long long kSqrt3 = 7987674492471257551ull;

// |v|, with the sign left in `sign` (bit 31)
__device__ __forceinline__ unsigned long long magnitude(long long v, int& sign) {
  sign = (int)(v >> 32);
  asm("{\n\t.reg .pred neg;\n\tsetp.lt.s32 neg, %1, 0;\n\t@neg neg.s64 %0, %0;\n\t}" : "+l"(v) : "r"(sign));
  return (unsigned long long)v;
}
// m 2^-right toward zero with that sign (PTX clamps the amount at 64)
__device__ __forceinline__ long long shifted_signed(unsigned long long m, int right, int sign) {
  asm("{\n\t.reg .pred neg;\n\tsetp.lt.s32 neg, %2, 0;\n\tshr.u64 %0, %0, %1;\n\t@neg neg.s64 %0, %0;\n\t}"
      : "+l"(m) : "r"(right), "r"(sign));
  return (long long)m;
}

// The integer nearest to u c, c = C / 2^62, for |u| <= 2^62 and c < 1 or |u| <=
// 2^60 and c < 2: an odd function that keeps 0 (ties aside, |u| = 2^61 for an odd
// C: one unit there, which no rounding to double sees for sqrt(3) or 3^-n).
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

// Headroom bits of one level: components below 2^(62 - G) give (d = 3: doubled)
// sums below 2^62.
template <int D>
constexpr int kHeadroom = D == 2 ? 1 : (D == 4 ? 2 : 3);

// The d elements that one DFT adds, element c in units of 2^-t[c], onto one
// binary point, the largest component's leading bit at bit 61 - G (shifted left
// to bit 62, then right toward zero); returns that point (zeros only: 0).
template <int D>
__device__ __forceinline__ int weyl_align(long long (&r)[D], long long (&i)[D], const int (&t)[D]) {
  constexpr int kZero = 1 << 20;                         // a zero element's place: beyond every other
  unsigned long long a[D], b[D];
  int sa[D], sb[D], q[D], lz[D], Q = kZero;
#pragma unroll
  for (int c = 0; c < D; ++c) {
    a[c] = magnitude(r[c], sa[c]);
    b[c] = magnitude(i[c], sb[c]);
    const unsigned long long m = a[c] | b[c];
    lz[c] = __clzll((long long)m);
    q[c] = m ? t[c] + lz[c] : kZero;
  }
#pragma unroll
  for (int c = 0; c < D; ++c) Q = min(Q, q[c]);
  const int T = Q - 2 - kHeadroom<D>;
#pragma unroll
  for (int c = 0; c < D; ++c) {
    asm("shl.b64 %0, %0, %1;" : "+l"(a[c]) : "r"(lz[c] - 1));
    asm("shl.b64 %0, %0, %1;" : "+l"(b[c]) : "r"(lz[c] - 1));
  }
#pragma unroll
  for (int c = 0; c < D; ++c) {
    r[c] = shifted_signed(a[c], q[c] - Q + 1 + kHeadroom<D>, sa[c]);
    i[c] = shifted_signed(b[c], q[c] - Q + 1 + kHeadroom<D>, sb[c]);
  }
  return Q == kZero ? 0 : T;
}

// The factor of a pass: 2^pow2 times frac / 2^62 (0: 1) before the rounding to
// double, and mul (1 normally) after it.
struct WeylScale {
  int pow2;
  unsigned long long frac;
  double mul;
  // level by level (Inf / NaN): levels before the last take 2^each, the last
  // the rest of pow2 and frac (rest: as one double)
  int each;
  double rest;
  double h;            // sqrt(3) / 2
};

// Class pairs a CTA of a later pass: 128 threads.  Warps that start together
// share the instruction cache (a class is thousands of straight-line
// instructions), but the barrier spans them all: d = 3, n = 9, two levels at
// digit stride 81 3.12, 2.88, 3.31, 3.28 ms with 1, 2, 3, 4.
constexpr int kPairs = 2;

// classes in pairs (a, -a), two self-paired ones together; 255: none
struct ClassTab {
  uint8_t a[32];
  int units;
};

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
    const long long hr = mul_frac(r[1] - r[2], kSqrt3), hi = mul_frac(i[1] - i[2], kSqrt3);
    const long long mr = 2 * r[0] - sr, mi = 2 * i[0] - si;
    r[0] = 2 * (r[0] + sr); i[0] = 2 * (i[0] + si);
    constexpr int p = kDec ? 1 : 2, m = kDec ? 2 : 1;     // p: m - i h u
    r[p] = mr + hi; i[p] = mi - hr;
    r[m] = mr - hi; i[m] = mi + hr;
  }
}

// levels 1 and above of the class; t[e]: the point of element e's sums, kept
// at the element with digit 0 of the level
template <int D, int K, bool kDec, int M, int B>
__device__ __forceinline__ void class_levels(long long (&re)[B], long long (&im)[B], int (&t)[B]) {
  if constexpr (M < K) {
    constexpr int st = (int)ipow(D, M), before = st / D;  // strides of this level's digit and the last one's
    int tn[B];
#pragma unroll
    for (int g = 0; g < B / D; ++g) {
      const int e = (g / st) * (st * D) + g % st;
      long long r[D], i[D];
      int tc[D];
#pragma unroll
      for (int c = 0; c < D; ++c) {
        const int x = e + c * st;
        r[c] = re[x]; i[c] = im[x];
        tc[c] = t[x - x / before % D * before];
      }
      tn[e] = weyl_align<D>(r, i, tc) + (D == 3 ? 1 : 0);
      dft_int<D, kDec>(r, i);
#pragma unroll
      for (int c = 0; c < D; ++c) { re[e + c * st] = r[c]; im[e + c * st] = i[c]; }
    }
#pragma unroll
    for (int g = 0; g < B / D; ++g) {
      const int e = (g / st) * (st * D) + g % st;
      t[e] = tn[e];
    }
    class_levels<D, K, kDec, M + 1, B>(re, im, t);
  }
}

__device__ __forceinline__ uint32_t exp_field(const double2& x) {
  return max((uint32_t)__double2hiint(x.x) & 0x7fffffffu, (uint32_t)__double2hiint(x.y) & 0x7fffffffu) >> 20;
}

// The elements of a DFT, of largest exponent field E, through the first level:
// onto their binary point, x 2^S with S = 1084 - G - max(E, 1).  Returns the sums' point.
template <int D, bool kDec>
__device__ __forceinline__ int first_level(const double2 (&x)[D], int E, long long (&r)[D], long long (&i)[D]) {
  const int sb = 9 - kHeadroom<D> - max(E, 1);
#pragma unroll
  for (int c = 0; c < D; ++c) {
    r[c] = FixedArith::to_fixed(x[c].x, sb);
    i[c] = FixedArith::to_fixed(x[c].y, sb);
  }
  dft_int<D, kDec>(r, i);
  return sb + 1075 + (D == 3 ? 1 : 0);
}

// The levels of a class one after another in doubles, out of line (Inf / NaN).
template <int D, int K, bool kDec>
__device__ __noinline__ void weyl_class_levels(double2* x, const WeylScale& sc) {
  constexpr int B = (int)ipow(D, K);
  Twiddles<double> tw;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    // exact for d = 2, 4; d = 3 uses h alone
    tw.re[k] = D == 2 ? (k ? -1.0 : 1.0) : (k == 0 ? 1.0 : (k == 2 ? -1.0 : 0.0));
    tw.im[k] = D == 2 ? 0.0 : (k == 1 ? 1.0 : (k == 3 ? -1.0 : 0.0));
  }
  tw.h = sc.h;
  const double each = sc.each == 0 ? 1.0 : (sc.each == -1 ? 0.5 : 0.25);
  for (int m = 0, st = 1; m < K; ++m, st *= D) {
    const bool end = m + 1 == K;
    for (int g = 0; g < B / D; ++g) {
      const int e = (g / st) * (st * D) + g % st;
      double2 in[D];
      uint32_t E = 0;
#pragma unroll
      for (int c = 0; c < D; ++c) {
        in[c] = x[e + c * st];
        E = max(E, exp_field(in[c]));
      }
      if (E == 2047) {
        Cx<double> u[D], v[D];
#pragma unroll
        for (int c = 0; c < D; ++c) u[c] = {in[c].x, in[c].y};
        dft_ieee<double, D, kDec>(u, v, tw);
        const double f = end ? sc.rest : each;
#pragma unroll
        for (int b = 0; b < D; ++b) x[e + b * st] = make_double2(v[b].re * f, v[b].im * f);
      } else {
        long long r[D], i[D];
        const int T = first_level<D, kDec>(in, (int)E, r, i) - (end ? sc.pow2 - (K - 1) * sc.each : sc.each);
#pragma unroll
        for (int b = 0; b < D; ++b) {
          if (end && sc.frac != 0) {
            r[b] = mul_frac(r[b], sc.frac);
            i[b] = mul_frac(i[b], sc.frac);
          }
          x[e + b * st] = make_double2(FixedArith::to_double_int(r[b], T) * (end ? sc.mul : 1.0),
                                       FixedArith::to_double_int(i[b], T) * (end ? sc.mul : 1.0));
        }
      }
    }
  }
}

// outputs outside the normal range, out of line: int64 sums to the doubles' bits
template <int B>
__device__ __noinline__ void weyl_class_rare(longlong2* v, const int* T) {
  for (int e = 0; e < B; ++e) {
    v[e].x = __double_as_longlong(FixedArith::to_double_int(v[e].x, T[e]));
    v[e].y = __double_as_longlong(FixedArith::to_double_int(v[e].y, T[e]));
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
  constexpr int B = (int)ipow(D, K), last = B / D;       // last: stride of the last level's digit
  uint32_t E[B / D], most = 0;
#pragma unroll
  for (int g = 0; g < B / D; ++g) {
    E[g] = 0;
#pragma unroll
    for (int c = 0; c < D; ++c) E[g] = max(E[g], exp_field(x[g * D + c]));
    most = max(most, E[g]);
  }
  if (most == 2047) {
    double2 t[B];
#pragma unroll
    for (int e = 0; e < B; ++e) t[e] = x[e];
    weyl_class_levels<D, K, kDec>(t, sc);
#pragma unroll
    for (int e = 0; e < B; ++e) x[e] = t[e];
    return;
  }
  long long re[B], im[B];
  int t[B];
#pragma unroll
  for (int g = 0; g < B / D; ++g) {
    double2 in[D];
    long long r[D], i[D];
#pragma unroll
    for (int c = 0; c < D; ++c) in[c] = x[g * D + c];
    t[g * D] = first_level<D, kDec>(in, (int)E[g], r, i);
#pragma unroll
    for (int c = 0; c < D; ++c) { re[g * D + c] = r[c]; im[g * D + c] = i[c]; }
  }
  class_levels<D, K, kDec, 1, B>(re, im, t);
  if (sc.frac != 0) {
#pragma unroll
    for (int e = 0; e < B; ++e) {
      re[e] = mul_frac(re[e], sc.frac);
      im[e] = mul_frac(im[e], sc.frac);
    }
  }
  bool fast = true;                                      // value = sum 2^-t
#pragma unroll
  for (int e = 0; e < last; ++e) {
    t[e] -= sc.pow2;
    fast &= FixedArith::fast_range(t[e]);
  }
  if (fast) {
    // real parts through the fp64 conversion unit, imaginary parts through
    // integer instructions (identical roundings): the pipes share the work
#pragma unroll
    for (int e = 0; e < B; ++e)
      x[e] = make_double2(FixedArith::to_double_cvt_fast(re[e], t[e % last]), FixedArith::to_double_fast(im[e], t[e % last]));
  } else {
    longlong2 v[B];
    int T[B];
#pragma unroll
    for (int e = 0; e < B; ++e) {
      v[e] = make_longlong2(re[e], im[e]);
      T[e] = t[e % last];
    }
    weyl_class_rare<B>(v, T);
#pragma unroll
    for (int e = 0; e < B; ++e) x[e] = make_double2(__longlong_as_double(v[e].x), __longlong_as_double(v[e].y));
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
__global__ void __launch_bounds__((ipow(D, K) * G + 31) / 32 * 32, ipow(D, K) >= 16 ? 3 : 4)
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

// Levels per pass at most: one level more adds an alignment and a DFT to every
// element, one pass more a conversion each way and the matrix's traffic.  d = 3,
// n = 9: two levels take 2.7-3.2 ms a pass (nine elements a thread, 95
// registers, twenty warps an SM), three 4.7-5.3 ms (27 elements, 168 registers
// and spills, twelve warps).
constexpr int fixed_max_levels(int d) { return d == 3 ? 2 : qudit_max_levels(d); }

// Column groups of the first pass's tile: up to 128 threads a CTA.
template <bool kDec>
First pick_first(int d, int K) {
  switch (d * 8 + K) {
    case 2 * 8 + 4: return first<2, 4, 8, kDec>();
    case 2 * 8 + 3: return first<2, 3, 16, kDec>();
    case 2 * 8 + 2: return first<2, 2, 8, kDec>();
    case 2 * 8 + 1: return first<2, 1, 16, kDec>();
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
    case 3 * 8 + 2: return k_weyl_class<3, 2, kDec>;
    case 3 * 8 + 1: return k_weyl_class<3, 1, kDec>;
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
  const int most = fixed_max_levels(d), passes = (n + most - 1) / most;
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
      // 3^levels / 2^taken in [1/2, 1): the values never grow beyond the input's, nor shrink much below
      sc.pow2 = taken;
      while ((1u << taken) < ipow(3u, k0 + K)) ++taken;
      sc.pow2 -= taken;
      whole = std::ldexp(1.0, sc.pow2);
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
    sc.each = kDec ? (d == 2 ? -1 : -2) : 0;
    sc.rest = std::ldexp(whole, -(K - 1) * sc.each);
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
      const dim3 grid((nq + 32 * kPairs - 1) / (32 * kPairs), (unsigned)tab.units);
      pick_pass<kDec>(d, K)<<<grid, 64 * kPairs, 0, st>>>(mat, N, ipow((uint32_t)d, k0), M, nq, tab, sc);
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
