// Sparse input: the decomposition of a matrix given by its nonzero entries
// (COO), level by level as in the paper's iterative algorithm (Alg. 2, the
// CMWs of Eq. 4), keeping only nonzero entries -- the zero-CMW pruning that
// gives the paper's O(m n p) cost for m nonzero entries and p contributing
// strings (Sec. IV).
//
// An entry is (key, value): key = the element's flat index r*N + c in the
// "RC" numbering, where after a qubit level beta the row / column bits
// (r_beta, c_beta) hold that level's Pauli label (I (0,0), X (0,1), Y (1,0),
// Z (1,1)) instead of the index bits.  One level maps an entry at (r_beta,
// c_beta) to two entries of its quad (Eq. 4 without the 1/2, applied once at
// the end as 2^-n):
//     a00 -> I +v, Z +v     a11 -> I +v, Z -v
//     a01 -> X +v, Y +iv    a10 -> X +v, Y -iv
// Entries with equal keys are summed in a hash table, zero sums dropped: one
// launch a level reads the table that the level before filled, drops its zero
// sums, empties it and adds the others' children to a second table.  The
// launches, not the entries, set the time of small problems, so the sort of
// the final list is one launch per doubling beyond 2048 entries, and a
// counter is touched once a CTA.  GB300, n = 14 Heisenberg chain (122,880
// entries, 53 strings): 0.70 -> 0.29 ms a call with its synchronisation, against
// an entry list between two launches a level (9 and 26 us), an atomic an entry on
// its counter and a launch per bitonic step, 80 launches against 27.  A level
// takes 5-11 us, round trips to L2 and little else: with the entries left in
// their slots' lanes it took 70-90 us, and with the values loaded one after
// another, at six CTAs an SM, 16-29 us.
//
// Exactness: values are int64 on one binary point per X-mask x = r xor c
// (x * 2^S_x, S_x = 1084 - n - the largest exponent among the entries of that
// X-mask, like a fixed-point pass with K = n).  A level never changes an
// entry's X-mask (Eq. 4: I, Z keep r_beta xor c_beta = 0, X, Y keep 1), so
// every sum adds values on one binary point: the sums are exact and
// independent of the order the atomics land in, and a weight's truncation
// error is bounded by its own X-mask's entries.  The weights are rounded to
// double once, at the end.  The output list is
// sorted by string index (bitonic sort), so it does not depend on scheduling.
#include <cuda_runtime.h>
#include <stdint.h>

#include "tpd_launch.h"

namespace tpd {

namespace {

constexpr uint32_t kEmpty = 0xFFFFFFFFu;      // keys are < 4^15

__device__ __forceinline__ uint32_t hash32(uint32_t k) {
  k ^= k >> 16; k *= 0x7feb352du; k ^= k >> 15; k *= 0x846ca68bu; k ^= k >> 16;
  return k;
}

// emax[x] = the largest exponent field among the entries of X-mask x = r xor c
// (emax: 2^n ints, zero on entry; the index is masked to n bits, so that rows
// or columns outside 0..2^n-1 cannot address outside the array)
__global__ void k_sp_emax(const int* __restrict__ rows, const int* __restrict__ cols,
                          const double2* __restrict__ vals, unsigned long long m, int n, int* __restrict__ emax) {
  const int xmask = (1 << n) - 1;
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < m;
       i += (unsigned long long)gridDim.x * blockDim.x) {
    const int ex = (int)((unsigned long long)__double_as_longlong(vals[i].x) >> 52) & 0x7FF;
    const int ey = (int)((unsigned long long)__double_as_longlong(vals[i].y) >> 52) & 0x7FF;
    const int e = max(ex, ey);
    // read first: an X-mask's entries mostly share a magnitude, and atomics on
    // one address (the diagonal's) serialise (26 -> 18 us for 122,880 entries)
    int* const p = emax + ((rows[i] ^ cols[i]) & xmask);
    if (e > *reinterpret_cast<const volatile int*>(p)) atomicMax(p, e);
  }
}

// x * 2^S truncated toward zero, S = 1084 - n - emax_eff (|result| < 2^(62-n)):
// x = m * 2^(max(e,1) - 1075), and (m << 11) >> rs = x * 2^S for
// rs = 2 + n + emax_eff - max(e, 1) >= 3
__device__ __forceinline__ long long sp_to_fixed(double x, int n, int emax_eff) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int e = (int)(bits >> 52) & 0x7FF;
  const unsigned long long mnt = (bits & 0x000FFFFFFFFFFFFFull) | ((unsigned long long)(e != 0) << 52);
  const unsigned rs = (unsigned)(2 + n + emax_eff - max(e, 1));
  unsigned long long mag;
  const unsigned long long ml = mnt << 11;                         // < 2^64
  asm("shr.b64 %0, %1, %2;" : "=l"(mag) : "l"(ml), "r"(rs));       // clamps above 64: 0
  const unsigned long long s = (unsigned long long)((long long)bits >> 63);
  return (long long)((mag ^ s) - s);
}

// v * 2^-T rounded to nearest even (integer instructions, normal range or Inf / subnormal)
__device__ __forceinline__ double sp_to_double(long long v, int T) {
  if (v == 0) return 0.0;
  const unsigned long long s = (unsigned long long)(v >> 63);
  unsigned long long a = ((unsigned long long)v ^ s) - s;
  const int lz = __clzll((long long)a);
  a <<= lz;
  const int be = 1086 - lz - T;
  unsigned long long bits;
  if (be >= 1) {
    unsigned long long mant = a >> 11;
    const unsigned rem = (unsigned)a & 0x7FFu;
    mant += (unsigned long long)((rem > 0x400u) | ((rem == 0x400u) & (unsigned)mant));
    bits = be > 2046 ? 0x7FF0000000000000ull : ((unsigned long long)(be - 1) << 52) + mant;
    if (bits > 0x7FF0000000000000ull) bits = 0x7FF0000000000000ull;
  } else {
    const int rsh = 12 - be;
    if (rsh > 64) bits = 0;
    else if (rsh == 64) bits = a > 0x8000000000000000ull ? 1ull : 0ull;
    else {
      const unsigned long long mant = a >> rsh, rem = a & ((1ull << rsh) - 1), half = 1ull << (rsh - 1);
      bits = mant + (unsigned long long)((rem > half) | ((rem == half) & (mant & 1ull)));
    }
  }
  return __longlong_as_double((long long)(bits | (s & 0x8000000000000000ull)));
}

__device__ __forceinline__ void sp_add(unsigned long long* __restrict__ tv, uint32_t slot, long long re, long long im) {
  atomicAdd(tv + 2ull * slot, (unsigned long long)re);         // two's complement: exact int64 sums
  atomicAdd(tv + 2ull * slot + 1, (unsigned long long)im);
}

// A key's first slot of the table that level beta fills, and the slot after
// another.  The level is part of the hash: one of an entry's children has the
// entry's own key, so with one hash for all levels the entries of one region of
// a table (those that a level past its capacity keeps, read in the table's
// order) crowd the same region of the next, and probes run as long as the
// table: n = 14, 2,000 random entries, 8 attempts of growing capacity 351 -> 4.0 ms;
// n = 11, 200,000 entries, 4 attempts 24 s -> 13 ms.
__device__ __forceinline__ uint32_t sp_slot(uint32_t key, int beta, uint32_t slots) {
  return __umulhi(hash32(key ^ ((uint32_t)beta * 0x9e3779b9u)), slots);
}
__device__ __forceinline__ uint32_t sp_next(uint32_t slot, uint32_t slots) { return slot + 1 == slots ? 0u : slot + 1; }

// one value into the table, probing from `slot` on
__device__ __noinline__ void sp_insert(uint32_t key, long long re, long long im, uint32_t* __restrict__ tkeys,
                                       unsigned long long* __restrict__ tv, uint32_t slot, uint32_t slots,
                                       unsigned long long* __restrict__ overflow) {
  for (uint32_t probe = 0; probe < slots; ++probe) {
    const uint32_t prev = atomicCAS(tkeys + slot, kEmpty, key);
    if (prev == kEmpty || prev == key) {
      sp_add(tv, slot, re, im);
      return;
    }
    slot = sp_next(slot, slots);
  }
  atomicExch(overflow, 1ull);                                  // table full (cannot happen when sized 2x)
}

// Level beta of one entry: its two children into the table.  Both first probes
// are in flight at once, and no lane waits for another label's: a probe is a
// round trip to L2, and a level is little else.
__device__ __forceinline__ void sp_children(uint32_t k, long long re, long long im, int n, int beta,
                                            uint32_t* __restrict__ tkeys, unsigned long long* __restrict__ tv,
                                            uint32_t slots, unsigned long long* __restrict__ overflow) {
  const uint32_t cb = (k >> beta) & 1u, rb = (k >> (n + beta)) & 1u;
  const uint32_t kI = k & ~((1u << beta) | (1u << (n + beta)));
  const uint32_t kX = kI | (1u << beta), kY = kI | (1u << (n + beta)), kZ = kX | kY;
  // I += v and Z +- v (a00 / a11), or X += v and Y +- i v (a01 / a10)
  const bool diag = rb == cb;
  const uint32_t k1 = diag ? kI : kX, k2 = diag ? kZ : kY;
  const long long re2 = diag ? (rb ? -re : re) : (cb ? -im : im);
  const long long im2 = diag ? (rb ? -im : im) : (cb ? re : -re);
  const uint32_t s1 = sp_slot(k1, beta, slots), s2 = sp_slot(k2, beta, slots);
  const uint32_t p1 = atomicCAS(tkeys + s1, kEmpty, k1);
  const uint32_t p2 = atomicCAS(tkeys + s2, kEmpty, k2);
  if (p1 == kEmpty || p1 == k1) sp_add(tv, s1, re, im);
  else sp_insert(k1, re, im, tkeys, tv, sp_next(s1, slots), slots, overflow);
  if (p2 == kEmpty || p2 == k2) sp_add(tv, s2, re2, im2);
  else sp_insert(k2, re2, im2, tkeys, tv, sp_next(s2, slots), slots, overflow);
}

// Counters (unsigned long long): [0] overflow flag, [1 + beta] entries
// entering level beta (beta = 0..n-1), [1 + n] the final entries.
constexpr int kSpCounters = 18;                                // n <= 15

// Slots of the table that level beta fills: twice its children at most.  They
// are two per entry, and the entries of level beta (counted only while they are
// read) at most two per entry of the level before, so later levels of a list
// that shrinks scan, and spread over, a table that shrinks with it (the chain's
// thirteen: 1.0 million slots each otherwise).
__device__ __forceinline__ uint32_t sp_slots(const unsigned long long* __restrict__ ctr, int beta, uint32_t slots) {
  const unsigned long long need = beta == 0 ? 4 * ctr[1] : 8 * ctr[beta];
  unsigned long long p = 1024;
  while (p < need && p < slots) p <<= 1;
  return p < slots ? (uint32_t)p : slots;
}

// the input's entries (key = r*N + c, value on its X-mask's binary point) through level 0
__global__ void k_sp_first(const int* __restrict__ rows, const int* __restrict__ cols, const double2* __restrict__ vals,
                           unsigned long long m, unsigned long long cap, int n, const int* __restrict__ emax,
                           uint32_t* __restrict__ tkeys, unsigned long long* __restrict__ tv, uint32_t slots,
                           unsigned long long* __restrict__ ctr) {
  const unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
  if (i == 0 && m > cap) ctr[0] = 1ull;
  if (i >= m || i >= cap) return;
  const uint32_t size = sp_slots(ctr, 0, slots);
  const int r = rows[i], c = cols[i];
  const int emax_eff = max(emax[(r ^ c) & ((1 << n) - 1)], 1);
  sp_children(((uint32_t)r << n) | (uint32_t)c, sp_to_fixed(vals[i].x, n, emax_eff), sp_to_fixed(vals[i].y, n, emax_eff),
              n, 0, tkeys, tv, size, ctr);
}

// the entries of the first level (the input's nonzeros, at most the capacity)
__global__ void k_sp_start(unsigned long long* ctr, unsigned long long m, unsigned long long cap) {
  ctr[1] = m < cap ? m : cap;
}

constexpr int kSpThreads = 256;
constexpr int kSpSlots = 4;                                    // table slots per thread

// The thread's occupied slots of a table, emptied, their zero sums dropped
// (zero CMWs: pruned); returns how many it keeps in key / re / im.
__device__ __forceinline__ int sp_take(uint32_t* __restrict__ tkeys, unsigned long long* __restrict__ tv, uint32_t slots,
                                       uint32_t (&key)[kSpSlots], long long (&re)[kSpSlots], long long (&im)[kSpSlots]) {
  const unsigned long long s0 = (unsigned long long)blockIdx.x * (kSpThreads * kSpSlots) + threadIdx.x;
#pragma unroll
  for (int k = 0; k < kSpSlots; ++k) {
    const unsigned long long s = s0 + k * kSpThreads;
    key[k] = s < slots ? tkeys[s] : kEmpty;
  }
  // every value in flight before the first slot is emptied
#pragma unroll
  for (int k = 0; k < kSpSlots; ++k) {
    re[k] = im[k] = 0;
    if (key[k] != kEmpty) {
      const longlong2 v = *reinterpret_cast<const longlong2*>(tv + 2 * (s0 + k * kSpThreads));
      re[k] = v.x;
      im[k] = v.y;
    }
  }
  int kept = 0;
#pragma unroll
  for (int k = 0; k < kSpSlots; ++k) {
    if (key[k] == kEmpty) continue;
    const unsigned long long s = s0 + k * kSpThreads;
    tkeys[s] = kEmpty;
    *reinterpret_cast<ulonglong2*>(tv + 2 * s) = make_ulonglong2(0ull, 0ull);
    if ((re[k] | im[k]) == 0) key[k] = kEmpty;
    else ++kept;
  }
  return kept;
}

// The CTA's entries counted into the level's count: their first position,
// *at the thread's first among them, *fit how many the capacity has room for.
// The CTAs' positions follow one another, so the entries below the capacity
// have no gaps.
__device__ __forceinline__ unsigned long long sp_count(int kept, unsigned long long* __restrict__ count,
                                                       unsigned long long cap, unsigned long long* __restrict__ overflow,
                                                       unsigned* at, unsigned* fit) {
  __shared__ unsigned part[kSpThreads / 32];
  __shared__ unsigned long long first;
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned inc = (unsigned)kept;
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned v = __shfl_up_sync(0xffffffffu, inc, d);
    if (lane >= (unsigned)d) inc += v;
  }
  if (lane == 31) part[warp] = inc;
  __syncthreads();
  unsigned before = 0, total = 0;
  for (unsigned w = 0; w < kSpThreads / 32; ++w) {
    if (w < warp) before += part[w];
    total += part[w];
  }
  if (threadIdx.x == 0) {
    first = total ? atomicAdd(count, (unsigned long long)total) : 0ull;
    if (first + total > cap) atomicExch(overflow, 1ull);
  }
  __syncthreads();
  *at = before + inc - (unsigned)kept;
  *fit = first >= cap ? 0u : (unsigned)min((unsigned long long)total, cap - first);
  return first;
}

// level beta (1..n-1): the entries that level beta - 1 left in one table into
// the other (count: ctr + 1 + beta)
__global__ void __launch_bounds__(kSpThreads, 8) k_sp_step(uint32_t* __restrict__ tkeys, unsigned long long* __restrict__ tv,
                                                        uint32_t slots, unsigned long long* __restrict__ ctr,
                                                        unsigned long long cap, int n, int beta,
                                                        uint32_t* __restrict__ ukeys, unsigned long long* __restrict__ uv) {
  const uint32_t from = sp_slots(ctr, beta - 1, slots);
  if ((unsigned long long)blockIdx.x * (kSpThreads * kSpSlots) >= from) return;
  uint32_t key[kSpSlots];
  long long re[kSpSlots], im[kSpSlots];
  const int kept = sp_take(tkeys, tv, from, key, re, im);
  if (!__syncthreads_or(kept)) return;
  unsigned at, fit;
  sp_count(kept, ctr + 1 + beta, cap, ctr, &at, &fit);        // entries past the capacity are lost (the status says so)
  // The kept entries side by side, then one a thread: in the table they are
  // few and far between, and a warp would wait for each of its lanes' slots.
  __shared__ uint32_t lkey[kSpThreads * kSpSlots];
  __shared__ longlong2 lval[kSpThreads * kSpSlots];
#pragma unroll
  for (int k = 0; k < kSpSlots; ++k)
    if (key[k] != kEmpty) {
      lkey[at] = key[k];
      lval[at] = make_longlong2(re[k], im[k]);
      ++at;
    }
  __syncthreads();
  const uint32_t size = sp_slots(ctr, beta, slots);
  for (unsigned i = threadIdx.x; i < fit; i += kSpThreads)
    sp_children(lkey[i], lval[i].x, lval[i].y, n, beta, ukeys, uv, size, ctr);
}

// RC key -> base-4 string index (bit 2b = c_b, bit 2b+1 = r_b)
__device__ __forceinline__ unsigned long long sp_string(uint32_t key, int n) {
  unsigned long long s = 0;
  for (int b = 0; b < n; ++b) {
    s |= (unsigned long long)((key >> b) & 1u) << (2 * b);
    s |= (unsigned long long)((key >> (n + b)) & 1u) << (2 * b + 1);
  }
  return s;
}

// the last level's table -> the final entries (any order) and their sort keys
__global__ void __launch_bounds__(kSpThreads, 8) k_sp_final(uint32_t* __restrict__ tkeys,
                                                         unsigned long long* __restrict__ tv, uint32_t slots,
                                                         unsigned long long* __restrict__ ctr, unsigned long long cap,
                                                         int n, uint32_t* __restrict__ keys, longlong2* __restrict__ v,
                                                         unsigned long long* __restrict__ skey,
                                                         uint32_t* __restrict__ sidx) {
  const uint32_t from = sp_slots(ctr, n - 1, slots);
  if ((unsigned long long)blockIdx.x * (kSpThreads * kSpSlots) >= from) return;
  uint32_t key[kSpSlots];
  long long re[kSpSlots], im[kSpSlots];
  const int kept = sp_take(tkeys, tv, from, key, re, im);
  if (!__syncthreads_or(kept)) return;
  unsigned at, fit;
  unsigned long long pos = sp_count(kept, ctr + 1 + n, cap, ctr, &at, &fit) + at;
#pragma unroll
  for (int k = 0; k < kSpSlots; ++k)
    if (key[k] != kEmpty && pos < cap) {
      keys[pos] = key[k];
      v[pos] = make_longlong2(re[k], im[k]);
      skey[pos] = sp_string(key[k], n);
      sidx[pos] = (uint32_t)pos;
      ++pos;
    }
}


// The final entries, sorted by string index: a bitonic sort of chunks of
// kSpChunk keys in shared memory, then merges of pairs of sorted runs, each
// key to its rank in both, between two buffers.  The number of entries, E, is
// read on the device: launches for longer runs than there are return at once,
// so the host plans the launches for the largest possible E.
constexpr int kSpChunk = 2048;                 // keys per CTA in shared memory
constexpr int kSpLocalThreads = kSpChunk / 2;  // one compare-exchange pair per thread

// entries of the final list: those that fit
__device__ __forceinline__ unsigned long long sp_entries(const unsigned long long* __restrict__ ctr, int n,
                                                         unsigned long long cap) {
  return min(ctr[1 + n], cap);
}

// one merge: runs of h keys (the last one shorter) in (skey, sidx) to runs of 2 h in (okey, oidx)
__global__ void k_sp_merge(const unsigned long long* __restrict__ skey, const uint32_t* __restrict__ sidx,
                           unsigned long long* __restrict__ okey, uint32_t* __restrict__ oidx,
                           const unsigned long long* __restrict__ ctr, int n, unsigned long long cap,
                           unsigned long long h) {
  const unsigned long long E = sp_entries(ctr, n, cap);
  if (h >= E) return;
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < E;
       i += (unsigned long long)gridDim.x * blockDim.x) {
    const unsigned long long key = skey[i];
    const unsigned long long base = i & ~(2 * h - 1), mid = base + h;
    // keys before this one in the other run (equal keys, from rows or columns
    // out of range alone: the left run's first), so that every place is taken once
    const bool left = i < mid;
    unsigned long long lo = left ? min(mid, E) : base, hi = left ? min(mid + h, E) : mid;
    const unsigned long long lo0 = lo;
    while (lo < hi) {
      const unsigned long long m = (lo + hi) >> 1;
      if (left ? skey[m] < key : skey[m] <= key) lo = m + 1;
      else hi = m;
    }
    const unsigned long long pos = base + (i - (left ? base : mid)) + (lo - lo0);
    okey[pos] = key;
    oidx[pos] = sidx[i];
  }
}

// each CTA's chunk sorted in shared memory (padded with the largest key to a power of two)
__global__ void __launch_bounds__(kSpLocalThreads) k_sp_local(unsigned long long* __restrict__ skey,
                                                              uint32_t* __restrict__ sidx,
                                                              const unsigned long long* __restrict__ ctr, int n,
                                                              unsigned long long cap) {
  __shared__ unsigned long long sk[kSpChunk];
  __shared__ uint32_t si[kSpChunk];
  const unsigned long long E = sp_entries(ctr, n, cap);
  const unsigned long long base = (unsigned long long)blockIdx.x * kSpChunk;
  if (base >= E) return;
  const unsigned cnt = (unsigned)min((unsigned long long)kSpChunk, E - base);
  unsigned P = 1;
  while (P < cnt) P <<= 1;
  for (unsigned t = threadIdx.x; t < P; t += blockDim.x) {
    sk[t] = t < cnt ? skey[base + t] : ~0ull;
    si[t] = t < cnt ? sidx[base + t] : 0u;
  }
  __syncthreads();
  for (unsigned k = 2; k <= P; k <<= 1) {
    for (unsigned j = k >> 1; j > 0; j >>= 1) {
      const unsigned t = threadIdx.x;
      const unsigned i = (t / j) * 2 * j + (t % j);
      const unsigned l = i + j;
      if (l < P) {
        const bool up = (i & k) == 0;
        const unsigned long long a = sk[i], b = sk[l];
        if ((a > b) == up) {
          sk[i] = b; sk[l] = a;
          const uint32_t x = si[i]; si[i] = si[l]; si[l] = x;
        }
      }
      __syncthreads();
    }
  }
  for (unsigned t = threadIdx.x; t < cnt; t += blockDim.x) { skey[base + t] = sk[t]; sidx[base + t] = si[t]; }
}

// the sorted list (after an odd number of merges it is in the second buffer), its length and the status
__global__ void k_sp_emit(const uint32_t* __restrict__ keys, const longlong2* __restrict__ v,
                          const unsigned long long* __restrict__ ctr, unsigned long long cap,
                          const unsigned long long* __restrict__ skey, const uint32_t* __restrict__ sidx,
                          const unsigned long long* __restrict__ skey2, const uint32_t* __restrict__ sidx2, int n,
                          const int* __restrict__ emax, unsigned long long capacity,
                          unsigned long long* __restrict__ strings, double2* __restrict__ weights,
                          unsigned long long* __restrict__ out_count, unsigned* __restrict__ status) {
  const unsigned long long E = sp_entries(ctr, n, cap);
  int merges = 0;
  for (unsigned long long h = kSpChunk; h < E; h <<= 1) ++merges;
  if (merges & 1) { skey = skey2; sidx = sidx2; }
  const uint32_t xmask = (1u << n) - 1;
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < E && i < capacity;
       i += (unsigned long long)gridDim.x * blockDim.x) {
    const uint32_t at = sidx[i];
    if (at >= E) continue;                                     // (never: the sort is a permutation)
    const uint32_t key = keys[at];
    const longlong2 x = v[at];
    // S_x of the input, and the 1/2 of Eq. 4 per level (the labels keep x = r xor c)
    const int T = 1084 - max(emax[((key >> n) ^ key) & xmask], 1);
    strings[i] = skey[i];
    weights[i] = make_double2(sp_to_double(x.x, T), sp_to_double(x.y, T));
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *out_count = E;
    // TPD_ERR_WORKSPACE if some level had more entries than the capacity
    if (status) *status = ctr[0] ? 4u : 0u;
  }
}

unsigned grid_for(unsigned long long items) {
  unsigned long long b = (items + 255) / 256;
  if (b < 1) b = 1;
  return (unsigned)(b > 4096 ? 4096 : b);
}

}  // namespace

// Workspace: counters, X-mask maxima | two hash tables' keys | their values.  A
// level's table takes at most twice its entries; 2.5 slots an entry keep the
// linear probes short (load 0.8; with two slots a level that just passes the
// capacity fills its table: 10 times the time over attempts of growing
// capacity).  The last level leaves one table to be read and one free: the
// final entries and their sort keys go into the free one's values (32 of its 40
// bytes an entry), the second sort buffer into the other's, empty by then.
struct SparseLayout {
  size_t ctr, emax, tkeys, tvals, total;
  unsigned long long entries, slots, list;   // list: final entries there is room for (all, but for entries > 2^31)
};

static SparseLayout sparse_layout(unsigned long long max_entries) {
  auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
  SparseLayout L;
  L.entries = max_entries < 1 ? 1 : max_entries;
  L.slots = 2 * L.entries + L.entries / 2;
  if (L.slots > 0xFFFFFFFFull) L.slots = 0xFFFFFFFFull;      // (a matrix has at most 2^30 entries)
  L.list = L.entries < L.slots / 2 ? L.entries : L.slots / 2;
  size_t off = 0;
  L.ctr = off; off += al(kSpCounters * sizeof(unsigned long long));
  L.emax = off; off += al(sizeof(int) << 15);     // one per X-mask, n <= 15
  L.tkeys = off; off += al(2 * L.slots * 4);
  L.tvals = off; off += al(2 * L.slots * 16);
  L.total = off;
  return L;
}

size_t sparse_workspace_bytes(unsigned long long max_entries) { return sparse_layout(max_entries).total; }

cudaError_t launch_sparse(const int* rows, const int* cols, const void* vals, unsigned long long m, int n,
                          unsigned long long max_entries, unsigned long long* strings, void* weights,
                          unsigned long long capacity, unsigned long long* count, void* ws, unsigned* status,
                          cudaStream_t s) {
  const SparseLayout L = sparse_layout(max_entries);
  char* w = static_cast<char*>(ws);
  unsigned long long* ctr = reinterpret_cast<unsigned long long*>(w + L.ctr);   // see kSpCounters
  int* emax = reinterpret_cast<int*>(w + L.emax);
  const uint32_t slots = (uint32_t)L.slots;
  uint32_t* tkeys[2] = {reinterpret_cast<uint32_t*>(w + L.tkeys), nullptr};
  unsigned long long* tv[2] = {reinterpret_cast<unsigned long long*>(w + L.tvals), nullptr};
  tkeys[1] = tkeys[0] + L.slots;
  tv[1] = tv[0] + 2 * L.slots;
  const unsigned long long cap = L.entries;
  cudaError_t e;
  // counters and X-mask maxima; both tables start empty, and every read leaves its table so
  if ((e = cudaMemsetAsync(w, 0, L.tkeys, s)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(tkeys[0], 0xFF, 2 * L.slots * 4, s)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(tv[0], 0, 2 * L.slots * 16, s)) != cudaSuccess) return e;
  const unsigned long long m0 = m < cap ? m : cap;
  if (m0 > 0) {
    const double2* val = static_cast<const double2*>(vals);
    k_sp_start<<<1, 1, 0, s>>>(ctr, m, cap);
    k_sp_emax<<<grid_for(m0), 256, 0, s>>>(rows, cols, val, m0, n, emax);
    k_sp_first<<<(unsigned)((m0 + 255) / 256), 256, 0, s>>>(rows, cols, val, m, cap, n, emax, tkeys[0], tv[0],
                                                          slots, ctr);
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const unsigned tgrid = (unsigned)((L.slots + kSpThreads * kSpSlots - 1) / (kSpThreads * kSpSlots));
  for (int beta = 1; beta < n; ++beta) {
    const int from = (beta - 1) & 1;
    k_sp_step<<<tgrid, kSpThreads, 0, s>>>(tkeys[from], tv[from], slots, ctr, cap, n, beta, tkeys[from ^ 1],
                                           tv[from ^ 1]);
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const int lastt = (n - 1) & 1;                   // the last level's table; the other one is free
  longlong2* v = reinterpret_cast<longlong2*>(tv[lastt ^ 1]);
  unsigned long long* skey = reinterpret_cast<unsigned long long*>(v + L.list);
  uint32_t* keys = reinterpret_cast<uint32_t*>(skey + L.list);
  uint32_t* sidx = keys + L.list;
  unsigned long long* skey2 = tv[lastt];           // once k_sp_final has read it
  uint32_t* sidx2 = reinterpret_cast<uint32_t*>(skey2 + L.list);
  k_sp_final<<<tgrid, kSpThreads, 0, s>>>(tkeys[lastt], tv[lastt], slots, ctr, L.list, n, keys, v, skey, sidx);
  const unsigned chunks = (unsigned)((L.list + kSpChunk - 1) / kSpChunk);
  k_sp_local<<<chunks, kSpLocalThreads, 0, s>>>(skey, sidx, ctr, n, L.list);
  int at = 0;
  for (unsigned long long h = kSpChunk; h < L.list; h <<= 1, at ^= 1)
    k_sp_merge<<<grid_for(L.list), 256, 0, s>>>(at ? skey2 : skey, at ? sidx2 : sidx, at ? skey : skey2,
                                                at ? sidx : sidx2, ctr, n, L.list, h);
  k_sp_emit<<<grid_for(L.list), 256, 0, s>>>(keys, v, ctr, L.list, skey, sidx, skey2, sidx2, n, emax, capacity, strings,
                                          static_cast<double2*>(weights), count, status);
  return cudaGetLastError();
}

}  // namespace tpd
