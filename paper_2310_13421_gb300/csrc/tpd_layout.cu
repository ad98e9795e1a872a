// Output-layout conversion and sum-of-squares reduction (memory-bound helpers
// around the decomposition).
//
// Layouts.  RC: the weight of string t at flat index r*N + c with
// t_j = 2 r_{n-j} + c_{n-j} (where the butterfly leaves it).  STRING: at the
// base-4 index s = sum_j t_j 4^(n-j) (t_1 most significant), i.e. bit 2b+1 of
// s is row bit r_b and bit 2b is column bit c_b: s interleaves the bits of c
// and r.  A CTA converts one block of 2^k x 2^k (rows x columns) that shares
// all higher index bits: in RC it is 2^k runs of 2^k contiguous elements, in
// STRING one run of 4^k contiguous elements (its s-bits below 2k are the
// interleaved low bits).  Both sides are read and written in full 128-byte
// lines through a shared-memory transpose.
#include <cuda_runtime.h>
#include <stdint.h>

#include "tpd_launch.h"

namespace tpd {

namespace {

// spread the low 16 bits of x to the even bit positions
__device__ __forceinline__ uint32_t spread16(uint32_t x) {
  x &= 0xffffu;
  x = (x | (x << 8)) & 0x00ff00ffu;
  x = (x | (x << 4)) & 0x0f0f0f0fu;
  x = (x | (x << 2)) & 0x33333333u;
  x = (x | (x << 1)) & 0x55555555u;
  return x;
}

// gather the even bit positions of x into the low 16 bits
__device__ __forceinline__ uint32_t compact16(uint32_t x) {
  x &= 0x55555555u;
  x = (x | (x >> 1)) & 0x33333333u;
  x = (x | (x >> 2)) & 0x0f0f0f0fu;
  x = (x | (x >> 4)) & 0x00ff00ffu;
  x = (x | (x >> 8)) & 0x0000ffffu;
  return x;
}

// Whole matrices of n < 5: blockDim.x = 4^k threads, one element each.
template <class T>
__global__ void __launch_bounds__(256) k_layout(const T* __restrict__ src, T* __restrict__ dst, int n, int k,
                                                int to_string) {
  __shared__ T tile[256];
  const uint32_t K = 1u << k;
  const uint32_t tid = threadIdx.x;
  // higher bits of the block: rh, ch (n-k bits each), interleaved in STRING order
  const uint64_t b = blockIdx.x + (uint64_t)blockIdx.y * gridDim.x;
  const uint32_t ch = compact16((uint32_t)b) | (compact16((uint32_t)(b >> 32)) << 16);
  const uint32_t rh = compact16((uint32_t)(b >> 1)) | (compact16((uint32_t)(b >> 33)) << 16);
  const uint64_t N = 1ull << n;
  const uint64_t rc_base = ((uint64_t)rh << k) * N + ((uint64_t)ch << k);   // row rh*K, column ch*K
  const uint64_t s_base = b << (2 * k);
  // thread's element in RC order within the block: (r_low, c_low) = (tid / K, tid % K)
  const uint32_t rl = tid >> k, cl = tid & (K - 1);
  const uint32_t sl = spread16(cl) | (spread16(rl) << 1);   // its position in STRING order
  if (to_string) {
    tile[sl] = src[rc_base + (uint64_t)rl * N + cl];       // read RC rows
    __syncthreads();
    dst[s_base + tid] = tile[tid];                          // write the STRING run
  } else {
    tile[tid] = src[s_base + tid];                          // read the STRING run
    __syncthreads();
    dst[rc_base + (uint64_t)rl * N + cl] = tile[sl];        // write RC rows
  }
}

// k = 5 (n >= 5): 32 x 32 elements a CTA, four a thread: runs of 32 columns
// (512 bytes in complex128, 256 in complex64) on the RC side and four loads in
// flight a thread.  The shared index is swizzled so that neither side
// conflicts: the spread column bits 2 and 3 (string bits 4 and 6) also move
// the low bits 1 and 3.  n = 13 complex64: 0.149 ms (7.2 TB/s) against 0.275 ms
// for 16 x 16 elements, one a thread (128-byte runs).
constexpr int kLayoutPer = 4;

__device__ __forceinline__ uint32_t layout_swizzle(uint32_t i) { return i ^ ((i >> 3) & 10u); }

template <class T>
__global__ void __launch_bounds__(256) k_layout32(const T* __restrict__ src, T* __restrict__ dst, int n,
                                                  int to_string) {
  __shared__ T tile[1024];
  const uint32_t tid = threadIdx.x, cl = tid & 31u, r0 = tid >> 5;
  const uint64_t b = blockIdx.x + (uint64_t)blockIdx.y * gridDim.x;
  const uint32_t ch = compact16((uint32_t)b) | (compact16((uint32_t)(b >> 32)) << 16);
  const uint32_t rh = compact16((uint32_t)(b >> 1)) | (compact16((uint32_t)(b >> 33)) << 16);
  const uint64_t rc = (((uint64_t)rh * 32 + r0) << n) + (uint64_t)ch * 32 + cl, s0 = b << 10;
  const uint32_t sc = spread16(cl);
  T x[kLayoutPer];
  if (to_string) {
#pragma unroll
    for (int i = 0; i < kLayoutPer; ++i) x[i] = src[rc + ((uint64_t)(8 * i) << n)];
#pragma unroll
    for (int i = 0; i < kLayoutPer; ++i) tile[layout_swizzle(sc | (spread16(r0 + 8 * i) << 1))] = x[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kLayoutPer; ++i) dst[s0 + tid + 256 * i] = tile[layout_swizzle(tid + 256 * i)];
  } else {
#pragma unroll
    for (int i = 0; i < kLayoutPer; ++i) x[i] = src[s0 + tid + 256 * i];
#pragma unroll
    for (int i = 0; i < kLayoutPer; ++i) tile[layout_swizzle(tid + 256 * i)] = x[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kLayoutPer; ++i)
      dst[rc + ((uint64_t)(8 * i) << n)] = tile[layout_swizzle(sc | (spread16(r0 + 8 * i) << 1))];
  }
}

// Sum of |x|^2 over `count` complex elements in fp64, deterministic: a fixed
// grid of kSumBlocks CTAs each sums a fixed strided subset in a fixed order,
// then one CTA sums the partials in a fixed order.
constexpr int kSumBlocks = 1024;
constexpr int kSumThreads = 256;

// acc + |x|^2 as two fused multiply-adds: on GB300 the fp64 pipe, not
// memory, bounds this kernel, so it gets the fewest fp64 instructions
template <class T>
__device__ __forceinline__ double add_abs2(double acc, const T& x) {
  const double re = x.x, im = x.y;
  return __fma_rn(im, im, __fma_rn(re, re, acc));
}

__device__ __forceinline__ double block_sum(double v, double* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
  return t;
}

// Each thread keeps kSumUnroll loads in flight (independent partial sums,
// combined in a fixed order at the end).
constexpr int kSumUnroll = 8;

template <class T>
__global__ void __launch_bounds__(kSumThreads) k_sumsq_partial(const T* __restrict__ x, uint64_t count,
                                                               double* __restrict__ partial) {
  __shared__ double sh[kSumThreads / 32];
  double acc[kSumUnroll];
#pragma unroll
  for (int u = 0; u < kSumUnroll; ++u) acc[u] = 0.0;
  const uint64_t stride = (uint64_t)kSumBlocks * kSumThreads;
  uint64_t i = (uint64_t)blockIdx.x * kSumThreads + threadIdx.x;
  for (; i + (kSumUnroll - 1) * stride < count; i += kSumUnroll * stride) {
    T r[kSumUnroll];
#pragma unroll
    for (int u = 0; u < kSumUnroll; ++u) r[u] = __ldcs(x + i + u * stride);
#pragma unroll
    for (int u = 0; u < kSumUnroll; ++u) acc[u] = add_abs2(acc[u], r[u]);
  }
  for (; i < count; i += stride) acc[0] = add_abs2(acc[0], x[i]);   // tail: fewer than kSumUnroll
  double v = 0.0;
#pragma unroll
  for (int u = 0; u < kSumUnroll; ++u) v += acc[u];
  const double t = block_sum(v, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = t;
}

__global__ void __launch_bounds__(kSumThreads) k_sumsq_final(const double* __restrict__ partial,
                                                             double* __restrict__ out) {
  __shared__ double sh[kSumThreads / 32];
  double v = 0.0;
  for (int i = threadIdx.x; i < kSumBlocks; i += kSumThreads) v += partial[i];
  const double t = block_sum(v, sh);
  if (threadIdx.x == 0) *out = t;
}

template <class T>
cudaError_t launch_layout_t(const void* src, void* dst, int n, int to_string, cudaStream_t s) {
  const int k = n < 5 ? n : 5;
  const uint64_t blocks = 1ull << (2 * (n - k));
  const unsigned gx = blocks > 65536 ? 65536u : (unsigned)blocks;
  const dim3 grid(gx, (unsigned)(blocks / gx));
  const T* in = static_cast<const T*>(src);
  T* out = static_cast<T*>(dst);
  if (n >= 5) k_layout32<T><<<grid, 256, 0, s>>>(in, out, n, to_string);
  else k_layout<T><<<grid, 1u << (2 * k), 0, s>>>(in, out, n, k, to_string);
  return cudaGetLastError();
}

template <class T>
__global__ void __launch_bounds__(256) k_gather(const T* __restrict__ mat, const unsigned long long* __restrict__ pos,
                                                unsigned long long count, T* __restrict__ out) {
  const unsigned long long i = blockIdx.x * 256ull + threadIdx.x;
  if (i < count) out[i] = mat[pos[i]];
}

// ---------------------------------------------------------------- nonzero list
//
// The paper's output form (Alg. 1/2: the list L of strings with nonzero
// weight), in string order, the order independent of scheduling.  Blocks of
// 4^k consecutive string indices (k = 4: 16 x 16 positions of W), a warp a
// block, kNzChunk blocks a CTA: one pass counts each block's entries and each
// chunk's, one CTA turns the chunks' counts into offsets, and one pass writes
// the entries, of which only the blocks that have any are read again.  Bound
// by reading W once: n = 14 complex128, 53 entries, 4.3 GB counted in 0.58 ms
// (7.4 TB/s; a thread an element with a barrier a block: 1.18 ms), offsets
// 0.02 ms (one CTA over every block's count: 1.71 ms), written in 0.03 ms
// (W read again whole: 1.28 ms).
constexpr int kNzThreads = 256;
constexpr int kNzWarps = kNzThreads / 32;
constexpr int kNzChunk = 64;

template <class T>
__device__ __forceinline__ bool keep(const T& w, double tol) {
  const double re = w.x, im = w.y;
  return !(fabs(re) <= tol && fabs(im) <= tol);            // NaN is kept
}
// tol = 0 without the fp64 pipe: any bit but the sign's (NaN is kept)
__device__ __forceinline__ bool keep_bits(const double2& w) {
  return (((uint32_t)__double2hiint(w.x) | (uint32_t)__double2hiint(w.y)) << 1 | (uint32_t)__double2loint(w.x) |
          (uint32_t)__double2loint(w.y)) != 0u;
}
__device__ __forceinline__ bool keep_bits(const float2& w) {
  return (__float_as_uint(w.x) | __float_as_uint(w.y)) << 1 != 0u;
}

// RC position of block b's first element
__device__ __forceinline__ uint64_t block_base(int n, int k, uint64_t b) {
  const uint32_t ch = compact16((uint32_t)b) | (compact16((uint32_t)(b >> 32)) << 16);
  const uint32_t rh = compact16((uint32_t)(b >> 1)) | (compact16((uint32_t)(b >> 33)) << 16);
  return (((uint64_t)rh << k) << n) + ((uint64_t)ch << k);
}

constexpr int kNzPer = 8;                                  // elements of a block per lane

// Lane's elements of block b, e = lane + 32 i at row e >> k, column e & (2^k - 1);
// zeros past the block's 4^k elements.
template <class T>
__device__ __forceinline__ void load_block(const T* __restrict__ W, int n, int k, uint64_t b, uint32_t lane,
                                           T (&w)[kNzPer]) {
  const uint64_t base = block_base(n, k, b);
  const uint32_t K = 1u << k, cnt = 1u << (2 * k);
#pragma unroll
  for (int i = 0; i < kNzPer; ++i) {
    const uint32_t e = lane + 32u * i;
    w[i] = T{};
    if (e < cnt) w[i] = __ldg(W + base + ((uint64_t)(e >> k) << n) + (e & (K - 1u)));
  }
}

template <class T>
__global__ void __launch_bounds__(kNzThreads) k_nz_count(const T* __restrict__ W, int n, int k, double tol,
                                                         uint64_t nb, unsigned* __restrict__ counts,
                                                         unsigned long long* __restrict__ chunks) {
  __shared__ unsigned part[kNzWarps];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned sum = 0;
#pragma unroll 2
  for (int j = 0; j < kNzChunk / kNzWarps; ++j) {
    const uint64_t b = (uint64_t)blockIdx.x * kNzChunk + j * kNzWarps + warp;
    if (b >= nb) break;
    T w[kNzPer];
    load_block(W, n, k, b, lane, w);
    unsigned c = 0;
    if (tol == 0.0) {
#pragma unroll
      for (int i = 0; i < kNzPer; ++i) c += keep_bits(w[i]) ? 1u : 0u;
    } else {
#pragma unroll
      for (int i = 0; i < kNzPer; ++i) c += keep(w[i], tol) ? 1u : 0u;
    }
    c = __reduce_add_sync(0xffffffffu, c);
    if (lane == 0) counts[b] = c;
    sum += c;
  }
  if (lane == 0) part[warp] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long t = 0;
    for (int i = 0; i < kNzWarps; ++i) t += part[i];
    chunks[blockIdx.x] = t;
  }
}

// in-place exclusive scan of nc chunk counts (one CTA of 1024 threads), total into *total
__global__ void __launch_bounds__(1024) k_nz_scan(unsigned long long* __restrict__ chunks, uint64_t nc,
                                                  unsigned long long* __restrict__ total) {
  __shared__ unsigned long long part[32];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long run = 0;                               // entries before this round's chunks
  for (uint64_t i0 = 0; i0 < nc; i0 += 1024) {
    const uint64_t i = i0 + threadIdx.x;
    const unsigned long long c = i < nc ? chunks[i] : 0ull;
    unsigned long long inc = c;                             // inclusive over the warp, then the CTA
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned long long v = __shfl_up_sync(0xffffffffu, inc, d);
      if (lane >= (unsigned)d) inc += v;
    }
    if (lane == 31) part[warp] = inc;
    __syncthreads();
    unsigned long long w = part[lane];
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned long long v = __shfl_up_sync(0xffffffffu, w, d);
      if (lane >= (unsigned)d) w += v;
    }
    const unsigned long long all = __shfl_sync(0xffffffffu, w, 31);
    const unsigned long long before = __shfl_sync(0xffffffffu, w, warp ? warp - 1 : 0);
    if (i < nc) chunks[i] = run + (warp ? before : 0ull) + inc - c;
    run += all;
    __syncthreads();
  }
  if (threadIdx.x == 0) *total = run;
}

// Entries of a chunk's nonempty blocks, at the chunk's offset.
template <class T>
__global__ void __launch_bounds__(kNzThreads) k_nz_write(const T* __restrict__ W, int n, int k, double tol,
                                                         uint64_t nb, const unsigned* __restrict__ counts,
                                                         const unsigned long long* __restrict__ chunks,
                                                         unsigned long long capacity,
                                                         unsigned long long* __restrict__ strings,
                                                         T* __restrict__ weights) {
  __shared__ __align__(16) unsigned char raw[kNzWarps][256 * sizeof(T)];   // a block a warp, in string order
  __shared__ unsigned start[kNzChunk + 1];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint64_t b0 = (uint64_t)blockIdx.x * kNzChunk;
  if (warp == 0) {                                          // the blocks' offsets within the chunk
    const unsigned c0 = b0 + 2 * lane < nb ? counts[b0 + 2 * lane] : 0u;
    const unsigned c1 = b0 + 2 * lane + 1 < nb ? counts[b0 + 2 * lane + 1] : 0u;
    unsigned inc = c0 + c1;
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned v = __shfl_up_sync(0xffffffffu, inc, d);
      if (lane >= (unsigned)d) inc += v;
    }
    start[2 * lane] = inc - c0 - c1;
    start[2 * lane + 1] = inc - c1;
    if (lane == 31) start[kNzChunk] = inc;
  }
  __syncthreads();
  if (start[kNzChunk] == 0) return;
  T* const tile = reinterpret_cast<T*>(raw[warp]);
  const uint32_t K = 1u << k, cnt = 1u << (2 * k);
  const unsigned long long off = chunks[blockIdx.x];
  for (uint32_t j = warp; j < (uint32_t)kNzChunk; j += kNzWarps) {
    if (start[j + 1] == start[j]) continue;                 // (uniform over the warp)
    const uint64_t b = b0 + j;
    T w[kNzPer];
    load_block(W, n, k, b, lane, w);
    __syncwarp();                                           // the last block's reads are done
#pragma unroll
    for (int i = 0; i < kNzPer; ++i) {
      const uint32_t e = lane + 32u * i;
      if (e < cnt) tile[spread16(e & (K - 1u)) | (spread16(e >> k) << 1)] = w[i];
    }
    __syncwarp();
    unsigned long long pos = off + start[j];
    for (int i = 0; i < kNzPer; ++i) {
      const uint32_t e = lane + 32u * i;                    // string order
      const bool kp = e < cnt && keep(tile[e < cnt ? e : 0u], tol);
      const unsigned ball = __ballot_sync(0xffffffffu, kp);
      const unsigned long long p = pos + __popc(ball & ((1u << lane) - 1u));
      if (kp && p < capacity) {
        strings[p] = (b << (2 * k)) + e;
        weights[p] = tile[e];
      }
      pos += __popc(ball);
    }
  }
}

struct NzLayout {
  int k;
  uint64_t nb, nc;                                          // blocks, chunks
  unsigned* counts;
  unsigned long long* chunks;
};
NzLayout nz_layout(int n, void* ws) {
  NzLayout L;
  L.k = n < 4 ? n : 4;
  L.nb = 1ull << (2 * (n - L.k));
  L.nc = (L.nb + kNzChunk - 1) / kNzChunk;
  L.counts = static_cast<unsigned*>(ws);
  L.chunks = reinterpret_cast<unsigned long long*>(static_cast<char*>(ws) + ((L.nb * 4 + 255) & ~255ull));
  return L;
}

template <class T>
cudaError_t launch_nz_count_t(const void* W, int n, double tol, unsigned long long* total, void* ws, cudaStream_t s) {
  const NzLayout L = nz_layout(n, ws);
  k_nz_count<T><<<(unsigned)L.nc, kNzThreads, 0, s>>>(static_cast<const T*>(W), n, L.k, tol, L.nb, L.counts, L.chunks);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_nz_scan<<<1, 1024, 0, s>>>(L.chunks, L.nc, total);
  return cudaGetLastError();
}

template <class T>
cudaError_t launch_nz_write_t(const void* W, int n, double tol, unsigned long long* strings, void* weights,
                              unsigned long long capacity, void* ws, cudaStream_t s) {
  const NzLayout L = nz_layout(n, ws);
  k_nz_write<T><<<(unsigned)L.nc, kNzThreads, 0, s>>>(static_cast<const T*>(W), n, L.k, tol, L.nb, L.counts, L.chunks,
                                                      capacity, strings, static_cast<T*>(weights));
  return cudaGetLastError();
}

}  // namespace

size_t nonzero_workspace_bytes(int n) {
  const int k = n < 4 ? n : 4;
  const uint64_t blocks = 1ull << (2 * (n - k));
  return ((blocks * 4 + 255) & ~255ull) + blocks * 8;
}

cudaError_t launch_nonzero_count(const void* W, int n, int elem_bytes, double tol, unsigned long long* total, void* ws,
                                 cudaStream_t s) {
  return elem_bytes == 16 ? launch_nz_count_t<double2>(W, n, tol, total, ws, s)
                          : launch_nz_count_t<float2>(W, n, tol, total, ws, s);
}

cudaError_t launch_nonzero_write(const void* W, int n, int elem_bytes, double tol, unsigned long long* strings,
                                 void* weights, unsigned long long capacity, void* ws, cudaStream_t s) {
  return elem_bytes == 16 ? launch_nz_write_t<double2>(W, n, tol, strings, weights, capacity, ws, s)
                          : launch_nz_write_t<float2>(W, n, tol, strings, weights, capacity, ws, s);
}

cudaError_t launch_gather(const void* mat, const unsigned long long* pos, unsigned long long count, int elem_bytes,
                          void* out, cudaStream_t s) {
  if (count == 0) return cudaSuccess;
  const unsigned long long blocks = (count + 255) / 256;
  if (blocks > 0x7fffffffull) return cudaErrorInvalidValue;
  if (elem_bytes == 16)
    k_gather<double2><<<(unsigned)blocks, 256, 0, s>>>(static_cast<const double2*>(mat), pos, count,
                                                       static_cast<double2*>(out));
  else
    k_gather<float2><<<(unsigned)blocks, 256, 0, s>>>(static_cast<const float2*>(mat), pos, count,
                                                      static_cast<float2*>(out));
  return cudaGetLastError();
}

cudaError_t launch_layout(const void* src, void* dst, int n, int elem_bytes, int to_string, cudaStream_t s) {
  return elem_bytes == 16 ? launch_layout_t<double2>(src, dst, n, to_string, s)
                          : launch_layout_t<float2>(src, dst, n, to_string, s);
}

size_t sumsq_workspace_bytes() { return kSumBlocks * sizeof(double); }

cudaError_t launch_sumsq(const void* x, unsigned long long count, int elem_bytes, double* out, void* ws,
                         cudaStream_t s) {
  double* partial = static_cast<double*>(ws);
  if (elem_bytes == 16)
    k_sumsq_partial<double2><<<kSumBlocks, kSumThreads, 0, s>>>(static_cast<const double2*>(x), count, partial);
  else
    k_sumsq_partial<float2><<<kSumBlocks, kSumThreads, 0, s>>>(static_cast<const float2*>(x), count, partial);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_sumsq_final<<<1, kSumThreads, 0, s>>>(partial, out);
  return cudaGetLastError();
}

}  // namespace tpd
