// Selection of the n_sel largest of C order-preserving 64-bit keys by one thread block, so that any
// kernel that needs the selection can make it for itself and no launch is spent on it.
#pragma once
#include "common.cuh"

namespace quads {

constexpr int kSelBins = 1024;
constexpr int kSelFew = 128;                  // so few keys in the boundary's bin are ranked among each other
constexpr int kSelList = 512;                 // (more of them only when their images are equal)

// Key j is selected iff key > thr, or key == thr and j < tie_end (ties go to the lower index).
struct Selection {
  unsigned long long thr;
  int tie_end;
  __device__ __forceinline__ bool has(unsigned long long key, int j) const {
    return key > thr || (key == thr && j < tie_end);
  }
};

struct SelectScratch {
  uint32_t hist[kSelBins];
  uint32_t mn[32], mx[32], sum[32];
  int n_list;
  struct __align__(16) Entry { unsigned long long key; int idx; int pad; } list[kSelList];
  Selection result;
};

// Monotone 32-bit image of a key: the high word of a double (its exponent and 20 bits), or, for an integer, the
// position of its leading one and the 26 bits behind it.
template <bool kDoubleKeys>
__device__ __forceinline__ uint32_t select_image(unsigned long long k) {
  if (kDoubleKeys) return (uint32_t)(k >> 32);
  const int lz = __clzll((long long)(k | 1ull));
  return ((uint32_t)(64 - lz) << 26) - (1u << 26) + ((uint32_t)((k << lz) >> 37) & 0x3FFFFFFu);
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

// `nt` threads of a block (128 or more, a multiple of 32; `tid` = 0 .. nt - 1, `sync` is a barrier over them) call it
// with the same arguments, after a barrier behind the stores to `sc` (shared memory); it returns behind another
// one.  C is a multiple of 128, at most 16384; `k32` is scratch of C words.  kDoubleKeys: the keys are the bit patterns
// of non-negative doubles, else integers.
//   1. A histogram of 1024 bins over the range of the keys' 32-bit images tells which bin the boundary lies in; while
//      that bin holds many keys it is divided again (outliers stretch the range of the first one).
//   2. Its keys are listed and ranked among each other by exact key and index.
// Latency bounds it: a handful of barriers and little code, because code that runs once per launch is fetched
// cold.  In front_small_kernel (1024 threads, C = 2048) it takes 6 300 cycles; a bisection with one barrier and some
// hundred dependent instructions per halving took 8 000 to 21 000, 32 sampled thresholds instead of the bins 7 500.
template <bool kDoubleKeys, typename Sync>
__device__ Selection select_largest(const unsigned long long* sc, uint32_t* k32, int C, int n_sel, SelectScratch* s, int tid, int nt,
                                    Sync sync) {
  Selection r;
  if (n_sel >= C) { r.thr = 0; r.tie_end = 0x7FFFFFFF; return r; }
  if (n_sel <= 0) { r.thr = ~0ull; r.tie_end = 0; return r; }
  const int lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  uint32_t mn = 0xFFFFFFFFu, mx = 0u;
  for (int i = tid; i < C; i += nt) {
    const uint32_t k = select_image<kDoubleKeys>(sc[i]);
    k32[i] = k;
    mn = min(mn, k);
    mx = max(mx, k);
  }
  for (int i = tid; i < kSelBins; i += nt) s->hist[i] = 0;
  mn = __reduce_min_sync(0xFFFFFFFFu, mn);
  mx = __reduce_max_sync(0xFFFFFFFFu, mx);
  if (lane == 0) { s->mn[warp] = mn; s->mx[warp] = mx; }
  if (tid == 0) s->n_list = 0;
  sync();
  uint32_t lo = __reduce_min_sync(0xFFFFFFFFu, lane < nw ? s->mn[lane] : 0xFFFFFFFFu);
  uint32_t range = __reduce_max_sync(0xFFFFFFFFu, lane < nw ? s->mx[lane] : 0u) - lo;
  int need = n_sel, m, shift;                  // `need` of the m keys with lo <= image <= lo + range are selected
  for (;;) {
    shift = max(0, 22 - __clz((int)range));
    for (int i = tid; i < C; i += nt) {
      const uint32_t d = k32[i] - lo;
      if (d <= range) atomicAdd(&s->hist[d >> shift], 1u);
    }
    sync();
    for (int w = warp; w < kSelBins / 32; w += nw) {
      const uint32_t v = __reduce_add_sync(0xFFFFFFFFu, s->hist[w * 32 + lane]);
      if (lane == 0) s->sum[w] = v;
    }
    sync();
    // the last group of 32 bins, then the last bin, with at least `need` keys at or above it
    int pos = 0, above = 0;
    const uint32_t* v = s->sum;
#pragma unroll 1
    for (int level = 0; level < 2; ++level) {
      const int own = (int)v[pos + lane];
      int a = own;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_down_sync(0xFFFFFFFFu, a, o);
        if (lane + o < 32) a += t;
      }
      const int l = __popc(__ballot_sync(0xFFFFFFFFu, a + above >= need)) - 1;
      m = __shfl_sync(0xFFFFFFFFu, own, l);
      above += __shfl_sync(0xFFFFFFFFu, a, l) - m;
      pos = (pos + l) * 32;
      v = s->hist;
    }
    pos >>= 5;
    need -= above;
    lo += (uint32_t)pos << shift;
    range = (1u << shift) - 1u;
    if (m <= kSelFew || shift == 0) break;
    sync();
    for (int i = tid; i < kSelBins; i += nt) s->hist[i] = 0;
    sync();
  }
  if (m > kSelList) {
    r = select_ties(sc, k32, lo, C, need, [&](auto pred) {
      sync();                                       // the previous count has been read
      if (tid == 0) s->n_list = 0;
      sync();
      int c = 0;
      for (int i = tid; i < C; i += nt) c += pred(i) ? 1 : 0;
      c = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)c);
      if (lane == 0 && c) atomicAdd(&s->n_list, c);
      sync();
      return s->n_list;
    });
    sync();
    return r;
  }
  for (int i = tid; i < C; i += nt)
    if (k32[i] - lo <= range) {
      const int p = atomicAdd(&s->n_list, 1);
      s->list[p].key = sc[i];
      s->list[p].idx = i;
    }
  sync();
  // eight threads per candidate count the candidates selected before it; the boundary has need - 1 of them
  for (int i0 = 0; i0 < m; i0 += nt >> 3) {
    const int me = i0 + (tid >> 3);
    const SelectScratch::Entry e = s->list[min(me, m - 1)];
    int rank = 0;
#pragma unroll 4
    for (int j = tid & 7; j < m; j += 8) {
      const SelectScratch::Entry o = s->list[j];
      rank += (o.key > e.key ? 1 : 0) + ((o.key == e.key ? 1 : 0) & (o.idx < e.idx ? 1 : 0));
    }
    rank += __shfl_xor_sync(0xFFFFFFFFu, rank, 1);
    rank += __shfl_xor_sync(0xFFFFFFFFu, rank, 2);
    rank += __shfl_xor_sync(0xFFFFFFFFu, rank, 4);
    if (me < m && rank == need - 1 && (tid & 7) == 0) { s->result.thr = e.key; s->result.tie_end = e.idx + 1; }
  }
  sync();
  return s->result;
}

// By a whole block.
template <bool kDoubleKeys>
__device__ __forceinline__ Selection select_largest(const unsigned long long* sc, uint32_t* k32, int C, int n_sel, SelectScratch* s) {
  return select_largest<kDoubleKeys>(sc, k32, C, n_sel, s, (int)threadIdx.x, (int)blockDim.x, [] { __syncthreads(); });
}

// The site-2 selection made by the kernel that uses it: loads the C integer totals, selects, and leaves the nibble
// masks of the selected channels in `nib` (C / 8 words); `scratch` holds 12 C bytes and a SelectScratch behind
// them.  mask_out (or NULL) gets the mask as bytes.  Ends behind a barrier.
template <typename Sync>
__device__ __forceinline__ void select_nibble_masks(const unsigned long long* totals, int C, int n_sel, uint8_t* scratch, uint32_t* nib,
                                                    uint8_t* mask_out, int tid, int nt, Sync sync) {
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(scratch);
  uint32_t* images = reinterpret_cast<uint32_t*>(scratch + (size_t)C * 8);
  SelectScratch* ss = reinterpret_cast<SelectScratch*>(scratch + (size_t)C * 12);
  for (int i = tid; i < C; i += nt) keys[i] = __ldcg(totals + i);
  sync();
  const Selection sel = select_largest<false>(keys, images, C, n_sel, ss, tid, nt, sync);
  for (int w = tid; w < (C >> 3); w += nt) {
    uint32_t m = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) m |= sel.has(keys[8 * w + i], 8 * w + i) ? 0xFu << (4 * i) : 0u;
    nib[w] = m;
  }
  if (mask_out)
    for (int i = tid; i < C; i += nt) mask_out[i] = sel.has(keys[i], i) ? 1 : 0;
  sync();
}

// One warp clears the codes of unselected channels in `rows` rows of a 128-byte-swizzled residual tile (128 bytes = 256
// channels per row, 1024-byte aligned) in shared memory; `nib` points at the tile's first channel's mask word and
// `chunks` (8 or fewer) of its 16-byte chunks exist.  The caller fences and signals.
__device__ __forceinline__ void mask_tile(uint32_t tile, int rows, int chunks, const uint32_t* nib, int lane) {
  const int c = lane & 7;
  if (c >= chunks) return;
  const uint4 m = reinterpret_cast<const uint4*>(nib)[c];
  if ((m.x & m.y & m.z & m.w) == 0xFFFFFFFFu) return;        // every channel of this chunk is selected
  for (int r0 = lane >> 3; r0 < rows; r0 += 32) {
    uint4 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int r = r0 + 4 * u;
      if (r < rows)
        asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v[u].x), "=r"(v[u].y), "=r"(v[u].z), "=r"(v[u].w)
                     : "r"(tile + r * 128 + ((c ^ (r & 7)) << 4)));
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int r = r0 + 4 * u;
      if (r < rows)
        asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(tile + r * 128 + ((c ^ (r & 7)) << 4)), "r"(v[u].x & m.x),
                     "r"(v[u].y & m.y), "r"(v[u].z & m.z), "r"(v[u].w & m.w) : "memory");
    }
  }
}

}  // namespace quads
