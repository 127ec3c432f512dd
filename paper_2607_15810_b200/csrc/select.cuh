// Selection of the n_sel largest of C order-preserving 64-bit keys by one thread block, so that any
// kernel that needs the selection can make it for itself and no launch is spent on it.
#pragma once
#include "common.cuh"

namespace quads {

constexpr int kSelList = 512;                 // keys around the boundary that are listed and sorted out by one warp

// Key j is selected iff key > thr, or key == thr and j < tie_end (ties go to the lower index).
struct Selection {
  unsigned long long thr;
  int tie_end;
  __device__ __forceinline__ bool has(unsigned long long key, int j) const {
    return key > thr || (key == thr && j < tie_end);
  }
};

struct SelectScratch {
  uint32_t key[2][kSelList];
  int idx[2][kSelList];
  uint32_t cnt[3][32];
  int n_list;
  Selection result;
};

// Bounds of the boundary in a monotone 32-bit image of the keys: c_lo >= n keys are >= lo, c_hi < n are >= hi.
struct SelectBounds {
  uint32_t lo, hi;
  int c_lo, c_hi;
};

// One round of tightening by a warp: lane l has counted c keys >= its own threshold t (0: none).
__device__ __forceinline__ void select_tighten(SelectBounds& b, uint32_t t, int c, int n) {
  const bool above = c >= n;                                 // the boundary is at or above t
  b.lo = max(b.lo, __reduce_max_sync(0xFFFFFFFFu, above ? t : 0u));
  b.c_lo = min(b.c_lo, (int)__reduce_min_sync(0xFFFFFFFFu, (unsigned)(above ? c : 0x7FFFFFFF)));
  b.hi = min(b.hi, __reduce_min_sync(0xFFFFFFFFu, above ? 0xFFFFFFFFu : t));
  b.c_hi = max(b.c_hi, (int)__reduce_max_sync(0xFFFFFFFFu, (unsigned)(above ? 0 : c)));
}

__device__ __forceinline__ int select_count4(const uint4& k, uint32_t t) {
  return (k.x >= t ? 1 : 0) + (k.y >= t ? 1 : 0) + (k.z >= t ? 1 : 0) + (k.w >= t ? 1 : 0);
}

// Exact search among more than kSelList keys whose images are equal (all of them at `image`): by value, then by
// index, one count over the block per bit.  Degenerate inputs only (hundreds of equal channels).
template <typename Count>
__device__ Selection select_ties(const unsigned long long* sc, const uint32_t* k32, uint32_t image, int C, int need, Count count) {
  unsigned long long lo = 0, hi = 1ull << 63;                // at least `need` are >= lo, fewer are >= hi
  int c_hi = 0;
  while (hi - lo > 1) {
    const unsigned long long m = lo + ((hi - lo) >> 1);
    const int c = count([&](int i) { return k32[i] == image && sc[i] >= m; });
    if (c >= need) lo = m; else { hi = m; c_hi = c; }
  }
  int a = 0, b = C;
  while (b - a > 1) {
    const int m = (a + b) >> 1;
    if (count([&](int i) { return i < m && sc[i] == lo; }) >= need - c_hi) b = m; else a = m;
  }
  Selection r;
  r.thr = lo;
  r.tie_end = b;
  return r;
}

// All threads of the block call it with the same arguments, after a barrier behind the stores to `sc`
// (shared memory); it returns behind another one.  C is a multiple of 128, at most 16384; the block has at
// least 128 threads, a multiple of 32; `k32` is scratch of C words, 16-byte aligned.  kDoubleKeys: the keys are the
// bit patterns of non-negative doubles, else integers.
//   1. Every lane of a warp takes one of 32 sampled keys as its threshold and counts the keys above it in the
//      warp's share, on 32-bit images of the keys (float, rounded down): the boundary lies between two
//      neighbouring samples, which leaves C / 16 keys or so.
//   2. Those are listed, and one warp repeats the step on the list until at most 32 are left, which it ranks
//      by exact key and index.
// Three block barriers and no long serial chain, where a bisection pays one barrier and some hundred
// dependent instructions per halving (measured in front_small_kernel at C = 2048: 8 000 to 21 000 cycles).
template <bool kDoubleKeys>
__device__ Selection select_largest(const unsigned long long* sc, uint32_t* k32, int C, int n_sel, SelectScratch* s) {
  Selection r;
  if (n_sel >= C) { r.thr = 0; r.tie_end = 0x7FFFFFFF; return r; }
  if (n_sel <= 0) { r.thr = ~0ull; r.tie_end = 0; return r; }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nt = blockDim.x, nw = nt >> 5;
  for (int i = threadIdx.x; i < C; i += nt) {
    const unsigned long long k = sc[i];
    k32[i] = __float_as_uint(kDoubleKeys ? __double2float_rz(__longlong_as_double((long long)k)) : __ull2float_rz(k));
  }
  if (threadIdx.x < 96) (&s->cnt[0][0])[threadIdx.x] = 0;
  if (threadIdx.x == 0) s->n_list = 0;
  __syncthreads();
  SelectBounds b{0u, 0xFFFFFFFFu, C, 0};
  const uint4* k4 = reinterpret_cast<const uint4*>(k32);
  int round = 0;
  uint32_t t = k32[(int)(((unsigned)lane * (unsigned)C) >> 5) + (C >> 6)];     // sampled thresholds
  for (;;) {
    int c = 0;
    for (int i = warp; i < (C >> 2); i += nw) c += select_count4(k4[i], t);    // (broadcast reads)
    uint32_t* cnt = s->cnt[round % 3];
    if (c) atomicAdd(cnt + lane, (uint32_t)c);
    __syncthreads();
    select_tighten(b, t, (int)cnt[lane], n_sel);
    if (b.c_lo - b.c_hi <= kSelList || b.hi - b.lo <= 1) break;
    // still many (rare): thresholds at equal distances between the bounds
    ++round;
    if (warp == 0) s->cnt[(round + 1) % 3][lane] = 0;
    t = b.lo + (uint32_t)(((unsigned long long)(b.hi - b.lo) * (unsigned)(lane + 1)) / 33u);
  }
  int m = b.c_lo - b.c_hi;
  if (m > kSelList) {
    const int need = n_sel - b.c_hi;
    const Selection e = select_ties(sc, k32, b.lo, C, need, [&](auto pred) {
      __syncthreads();                                       // the previous count has been read
      if (threadIdx.x == 0) s->n_list = 0;
      __syncthreads();
      int c = 0;
      for (int i = threadIdx.x; i < C; i += nt) c += pred(i) ? 1 : 0;
      c = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)c);
      if (lane == 0 && c) atomicAdd(&s->n_list, c);
      __syncthreads();
      return s->n_list;
    });
    __syncthreads();
    return e;
  }
  for (int i0 = warp * 32; i0 < C; i0 += nt) {
    const uint32_t k = k32[i0 + lane];
    const bool in = k >= b.lo && k < b.hi;
    const uint32_t who = __ballot_sync(0xFFFFFFFFu, in);
    if (who == 0) continue;
    int base = 0;
    if (lane == 0) base = atomicAdd(&s->n_list, __popc(who));
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    if (in) {
      const int p = base + __popc(who & ((1u << lane) - 1u));
      s->key[0][p] = k;
      s->idx[0][p] = i0 + lane;
    }
  }
  __syncthreads();
  if (warp == 0) {
    int cur = 0;
    while (m > 32) {
      const uint32_t* lk = s->key[cur];
      const int* li = s->idx[cur];
      const uint32_t tt = lk[(lane * m) >> 5];
      int c = 0;
      for (int i = 0; i < m; ++i) c += lk[i] >= tt ? 1 : 0;
      SelectBounds d{b.lo, b.hi, b.c_lo, b.c_hi};
      select_tighten(d, tt, c + b.c_hi, n_sel);
      const int left = d.c_lo - d.c_hi;
      if (left == m) break;                                  // equal images: ranked in the loop below
      int n = 0;
      for (int i0 = 0; i0 < m; i0 += 32) {
        const bool here = i0 + lane < m;
        const uint32_t k = here ? lk[i0 + lane] : 0u;
        const bool in = here && k >= d.lo && k < d.hi;
        const uint32_t who = __ballot_sync(0xFFFFFFFFu, in);
        if (in) {
          const int p = n + __popc(who & ((1u << lane) - 1u));
          s->key[cur ^ 1][p] = k;
          s->idx[cur ^ 1][p] = li[i0 + lane];
        }
        n += __popc(who);
      }
      __syncwarp();
      b = d;
      m = left;
      cur ^= 1;
    }
    const int* li = s->idx[cur];
    const int need = n_sel - b.c_hi;                         // the boundary is the candidate with need - 1 before it
    for (int i0 = 0; i0 < m; i0 += 32) {
      const bool on = i0 + lane < m;
      const int idx = on ? li[i0 + lane] : 0;
      const unsigned long long k = sc[idx];
      int rank = 0;
      for (int j = 0; j < m; ++j) {
        const int ij = li[j];
        const unsigned long long kj = sc[ij];
        rank += (kj > k || (kj == k && ij < idx)) ? 1 : 0;
      }
      if (on && rank == need - 1) { s->result.thr = k; s->result.tie_end = idx + 1; }
    }
  }
  __syncthreads();
  return s->result;
}

}  // namespace quads
