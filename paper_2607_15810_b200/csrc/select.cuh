// Selection of the n_sel largest of C order-preserving 64-bit keys by one thread block: a search for
// the threshold instead of a rank per key, so that any kernel that needs the selection can make it
// for itself and no launch is spent on it.
#pragma once
#include "common.cuh"

namespace quads {

struct SelectScratch {
  unsigned long long mn[32], mx[32];
  uint32_t cnt[3];
};

// Key j is selected iff key > thr, or key == thr and j < tie_end (ties go to the lower index).
struct Selection {
  unsigned long long thr;
  int tie_end;
  __device__ __forceinline__ bool has(unsigned long long key, int j) const {
    return key > thr || (key == thr && j < tie_end);
  }
};

// Block-wide sum of a packed pair of counts, one barrier per call.  Three counters take turns: while
// counter i is added to, the one of the next call is cleared; the last reads of that one lie a barrier
// back.
template <int kThreads>
__device__ __forceinline__ uint32_t block_count(uint32_t c, int it, SelectScratch* s) {
  c = __reduce_add_sync(0xFFFFFFFFu, c);
  if (threadIdx.x == 0) s->cnt[(it + 1) % 3] = 0;
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(&s->cnt[it % 3], c);
  __syncthreads();
  return s->cnt[it % 3];
}

// All kThreads threads call it with the same arguments, after a barrier behind the stores to `sc`
// (shared memory, C <= 16384).  Every round tests two thresholds between the bounds (at equal distances
// in exponent while the bounds are far apart, else in value) and stops at the first that exactly n_sel keys
// reach: about a dozen rounds of one barrier (~0.06 us each) for the score distributions met here, 41
// at most; equal keys across the boundary cost fourteen more, for the index.
template <int kThreads>
__device__ Selection select_largest(const unsigned long long* sc, int C, int n_sel, SelectScratch* s) {
  Selection r;
  if (n_sel >= C) { r.thr = 0; r.tie_end = 0x7FFFFFFF; return r; }
  if (n_sel <= 0) { r.thr = ~0ull; r.tie_end = 0; return r; }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long mn = ~0ull, mx = 0;
  for (int i = threadIdx.x; i < C; i += kThreads) { mn = min(mn, sc[i]); mx = max(mx, sc[i]); }
  constexpr int kHeld = 4;                    // keys a thread keeps in registers (0 is below every threshold tested)
  unsigned long long held[kHeld];
#pragma unroll
  for (int u = 0; u < kHeld; ++u) held[u] = (int)threadIdx.x + u * kThreads < C ? sc[threadIdx.x + u * kThreads] : 0ull;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    mn = min(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, o));
    mx = max(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
  }
  if (lane == 0) { s->mn[warp] = mn; s->mx[warp] = mx; }
  if (threadIdx.x < 3) s->cnt[threadIdx.x] = 0;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kThreads / 32; ++w) { mn = min(mn, s->mn[w]); mx = max(mx, s->mx[w]); }
  // invariant: at least n_sel keys are >= lo, fewer than n_sel (c_hi of them) are >= hi
  unsigned long long lo = mn, hi = mx + 1;
  int c_hi = 0, it = 0;
  while (hi - lo > 1) {
    unsigned long long m1, m2;
    if ((hi >> 2) > lo) {
      const int a = 63 - __clzll((long long)(lo | 1)), w = (63 - __clzll((long long)hi)) - a;   // w >= 1
      m1 = min(max(1ull << (a + (w + 2) / 3), lo + 1), hi - 1);
      m2 = min(max(1ull << (a + (2 * w + 2) / 3), m1), hi - 1);
    } else {
      const unsigned long long d = hi - lo, step = max((d >> 2) + (d >> 4), 1ull);
      m1 = lo + step;
      m2 = hi - step;
    }
    uint32_t c = 0;
#pragma unroll
    for (int u = 0; u < kHeld; ++u) c += (held[u] >= m1 ? 1u : 0u) + (held[u] >= m2 ? 0x10000u : 0u);
    for (int i = threadIdx.x + kHeld * kThreads; i < C; i += kThreads) {
      const unsigned long long k = sc[i];
      c += (k >= m1 ? 1u : 0u) + (k >= m2 ? 0x10000u : 0u);
    }
    c = block_count<kThreads>(c, it++, s);
    const int c1 = (int)(c & 0xFFFFu), c2 = (int)(c >> 16);
    if (c1 == n_sel || c2 == n_sel) { r.thr = c2 == n_sel ? m2 : m1; r.tie_end = 0x7FFFFFFF; return r; }
    if (c2 > n_sel) { lo = m2; }
    else if (c1 > n_sel) { lo = m1; hi = m2; c_hi = c2; }
    else { hi = m1; c_hi = c1; }
  }
  // keys equal to lo straddle the boundary (or exactly fill it): the n_sel - c_hi of lowest index
  r.thr = lo;
  const int need = n_sel - c_hi;
  int i_lo = 0, i_hi = C;                     // fewer than `need` of them lie below i_lo, at least `need` below i_hi
  while (i_hi - i_lo > 1) {
    const int m = (i_lo + i_hi) >> 1;
    uint32_t c = 0;
    for (int i = threadIdx.x; i < m; i += kThreads) c += sc[i] == lo ? 1u : 0u;
    c = block_count<kThreads>(c, it++, s);
    if ((int)c >= need) i_hi = m; else i_lo = m;
  }
  r.tie_end = i_hi;
  return r;
}

}  // namespace quads
