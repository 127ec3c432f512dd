// Top-k routing, per-expert histogram, exclusive scan and the stable dispatch permutation by a group of
// thread blocks that are resident together, as one role of a larger kernel (it shares the launch with the
// quantization of x, which does not depend on it).  Integer outputs are deterministic: assignments
// (token, slot) end up sorted by (expert, token, slot).
#pragma once
#include "kernels.cuh"

namespace quads {

// Bounded wait until `n` thread blocks have counted themselves in (the caller's other threads wait at a barrier).
__device__ __forceinline__ void grid_wait(const unsigned int* arrivals, uint32_t n, int32_t* status) {
  const long long t0 = clock64();
  while (ld_acquire_u32(arrivals) < n) {
    __nanosleep(100);
    if (clock64() - t0 > 4000000000ll) { atomicExch(status, (int32_t)QUADS_ERR_TIMEOUT); break; }
  }
}

constexpr int kRouteThreads = 256;
constexpr int kRouteWarps = kRouteThreads / 32;

struct RouteShared {
  uint32_t words[kMaxExperts];            // assignment bits of the 32 tokens of a chunk, per expert
  int part[2][kRouteThreads];
  int base[kMaxExperts], off[kMaxExperts], tile0[kMaxExperts], total[kMaxExperts];
  int wsum[2][kRouteWarps];
};

// Routes tokens t0 .. t0 + 8 * (TW - 1), one warp: top-k by logit on order-preserving integer keys, ties to
// the lower expert id, two warp reductions per slot; TW independent chains hide their latency.  Softmax over all
// experts at the chosen ones, optionally renormalised.  Lane s ends up with slot s.  Assignments are counted in
// `counts` [E].
template <int NJ, int TW>
__device__ __forceinline__ void route_tokens(const RouteArgs& p, int t0, int t_end, int32_t* counts) {
  const int lane = threadIdx.x & 31;
  float v[TW][NJ];
  uint32_t my_key[TW];
  int my_id[TW];
#pragma unroll
  for (int a = 0; a < TW; ++a) {
    const int t = t0 + a * kRouteWarps;
    my_key[a] = 0; my_id[a] = 0;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const int e = j * 32 + lane;
      v[a][j] = (t < t_end && e < p.E) ? p.logits[(size_t)t * p.E + e] + 0.f : -INFINITY;   // -0 counts as +0
    }
  }
  uint32_t key[TW][NJ];
#pragma unroll
  for (int a = 0; a < TW; ++a)
#pragma unroll
    for (int j = 0; j < NJ; ++j) key[a][j] = j * 32 + lane < p.E ? float_key(v[a][j]) : 0u;
  for (int k = 0; k < p.topk; ++k) {
    uint32_t g[TW];
#pragma unroll
    for (int a = 0; a < TW; ++a) {
      uint32_t m = key[a][0];
#pragma unroll
      for (int j = 1; j < NJ; ++j) m = max(m, key[a][j]);
      g[a] = __reduce_max_sync(0xFFFFFFFFu, m);
    }
#pragma unroll
    for (int a = 0; a < TW; ++a) {
      uint32_t e1 = 0x7FFFFFFFu;
#pragma unroll
      for (int j = NJ - 1; j >= 0; --j)
        if (key[a][j] == g[a]) e1 = (uint32_t)(j * 32 + lane);
      const int be = (int)__reduce_min_sync(0xFFFFFFFFu, e1);
      if (lane == k) { my_key[a] = g[a]; my_id[a] = be; }
#pragma unroll
      for (int j = 0; j < NJ; ++j)
        if (j * 32 + lane == be) key[a][j] = 0u;                         // remove the winner
    }
  }
#pragma unroll
  for (int a = 0; a < TW; ++a) {
    const int t = t0 + a * kRouteWarps;
    if (t >= t_end) continue;                                            // (the whole warp)
    const float gv = __uint_as_float((my_key[a] & 0x80000000u) ? (my_key[a] & 0x7FFFFFFFu) : ~my_key[a]);
    const float mx = __shfl_sync(0xFFFFFFFFu, gv, 0);
    const float ex = lane < p.topk ? expf(gv - mx) : 0.f;
    float sum = ex;                                                      // renormalised: over the chosen ones only
    if (!p.renormalize) {
      sum = 0.f;
#pragma unroll
      for (int j = 0; j < NJ; ++j) sum += j * 32 + lane < p.E ? expf(v[a][j] - mx) : 0.f;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
    const float w = ex / sum;
    if (lane < p.topk) {
      const size_t flat = (size_t)t * p.topk + lane;
      p.ids[flat] = my_id[a];
      p.wts[flat] = w;
      if (p.ids_out) p.ids_out[flat] = my_id[a];
      if (p.wts_out) p.wts_out[flat] = w;
      if (my_id[a] >= p.e_lo && my_id[a] < p.e_hi) atomicAdd(counts + my_id[a], 1);   // only this call's experts get rows
    }
  }
}

// Both parts deal the tokens to `n_groups` consecutive ranges.
//
// Part 1, by CTA `cta` of the `n_cta` CTAs of the kernel: top-k of a piece of a range's tokens, counted per (range,
// expert).  Every CTA takes a piece, before its own work: left to a few CTAs beside ones that are bound by
// instruction issue, 56 tokens per CTA took 30 us.
template <int NJ>
__device__ __forceinline__ void route_part1(const RouteArgs& p, int cta, int n_cta, int n_groups) {
  const int group = cta % n_groups, sub = cta / n_groups, n_sub = n_cta / n_groups;
  if (sub < n_sub) {
    const int warp = threadIdx.x >> 5;
    const int per = (p.T + n_groups - 1) / n_groups, per_sub = (per + n_sub - 1) / n_sub;
    const int g_end = min(p.T, (group + 1) * per);
    const int t0 = group * per + sub * per_sub, t_end = min(g_end, t0 + per_sub);
    int32_t* counts = p.counts + (size_t)group * p.E;
    if (per_sub <= kRouteWarps) {
      if (t0 + warp < t_end) route_tokens<NJ, 1>(p, t0 + warp, t_end, counts);
    } else {
      for (int t = t0 + warp; t < t_end; t += 2 * kRouteWarps) route_tokens<NJ, 2>(p, t, t_end, counts);
    }
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) atomicAdd(p.arrivals, 1u);
}

// Part 2, by CTA `cta` of `n_groups` (kRouteThreads threads each), one per range: after a bounded wait for part 1
// adds the ranges' counts up -- totals, and those of the ranges before its own -- scans over the experts, and hands
// out rows to its assignments: a token's row inside an expert is the expert's start plus the population count
// of the assignment bits before it.  Latency-bound: at 8192 tokens and 128 experts a CTA reads 148 x 128 counts.
template <int NJ>
__device__ void route_part2(const RouteArgs& p, int cta, int n_groups, uint32_t n_arrivals, RouteShared* s) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int E = p.E, topk = p.topk, n_cta = n_groups;
  const int per = (p.T + n_cta - 1) / n_cta;
  const int t_begin = min(p.T, cta * per), t_end = min(p.T, t_begin + per);
  if (threadIdx.x == 0) grid_wait(p.arrivals, n_arrivals, p.status);
  __syncthreads();
  // ---- totals and this CTA's first row per expert: the CTAs' counts dealt to 256 / 32 NJ groups of threads
  constexpr int kGroups = kRouteThreads / (32 * NJ);
  {
    const int e = threadIdx.x % (32 * NJ), g = threadIdx.x / (32 * NJ);
    int tot = 0, pre = 0;
    if (e < E) {
      int c = g;
      for (; c + 15 * kGroups < n_cta; c += 16 * kGroups) {
        int v[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u] = __ldcg(p.counts + (size_t)(c + u * kGroups) * E + e);
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          tot += v[u];
          pre += c + u * kGroups < cta ? v[u] : 0;
        }
      }
      for (; c < n_cta; c += kGroups) {
        const int v = __ldcg(p.counts + (size_t)c * E + e);
        tot += v;
        pre += c < cta ? v : 0;
      }
    }
    s->part[0][threadIdx.x] = tot;
    s->part[1][threadIdx.x] = pre;
  }
  __syncthreads();
  const int slot_rows = p.slot_rows, group_rows = slot_rows * p.tile_group;
  int cnt = 0, tiles = 0, inc_c = 0, inc_t = 0;
  {
    const int e = threadIdx.x;
    int pre = 0;
    if (e < E) {
#pragma unroll
      for (int g = 0; g < kGroups; ++g) { cnt += s->part[0][g * 32 * NJ + e]; pre += s->part[1][g * 32 * NJ + e]; }
      s->base[e] = pre;
      s->total[e] = cnt;
    }
    tiles = (cnt + group_rows - 1) / group_rows * p.tile_group;
    inc_c = cnt; inc_t = tiles;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int a = __shfl_up_sync(0xFFFFFFFFu, inc_c, o), b = __shfl_up_sync(0xFFFFFFFFu, inc_t, o);
      if (lane >= o) { inc_c += a; inc_t += b; }
    }
    if (lane == 31) { s->wsum[0][warp] = inc_c; s->wsum[1][warp] = inc_t; }
  }
  __syncthreads();
  {
    const int e = threadIdx.x;
    int off = inc_c - cnt, tp = inc_t - tiles;
    for (int w = 0; w < warp; ++w) { off += s->wsum[0][w]; tp += s->wsum[1][w]; }
    if (e < E) {
      s->off[e] = off;
      s->tile0[e] = tp;
      if (cta == 0) {
        p.offsets[e] = off;
        p.tile_prefix[e] = tp;
        if (p.offsets_out) p.offsets_out[e] = off;
        if (e == E - 1) {
          p.offsets[E] = off + cnt;
          p.tile_prefix[E] = tp + tiles;
          if (p.offsets_out) p.offsets_out[E] = off + cnt;
          p.header[kHdrMTiles] = tp + tiles;
          p.header[kHdrAssignments] = off + cnt;
        }
      }
    }
  }
  __syncthreads();
  // ---- tile tables: expert e by CTA e mod n_cta
  for (int e = cta; e < E; e += n_cta) {
    const int n = s->total[e], tp = s->tile0[e], nt = (n + group_rows - 1) / group_rows * p.tile_group;
    for (int m = threadIdx.x; m < nt; m += kRouteThreads) {
      p.tile_expert[tp + m] = e;
      p.tile_rows[tp + m] = max(0, min(slot_rows, n - m * slot_rows));
    }
  }
  // ---- rows, 32 tokens at a time
  for (int c0 = t_begin; c0 < t_end; c0 += 32) {
    const int n = min(32, t_end - c0) * topk;
    for (int e = threadIdx.x; e < E; e += kRouteThreads) s->words[e] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += kRouteThreads) {
      const int e = __ldcg(p.ids + (size_t)c0 * topk + i);
      if (e >= p.e_lo && e < p.e_hi) atomicOr(&s->words[e], 1u << (i / topk));
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += kRouteThreads) {
      const int flat = c0 * topk + i, t = i / topk;
      const int e = __ldcg(p.ids + flat);
      if (e < p.e_lo || e >= p.e_hi) { p.pos_pad[flat] = -1; continue; }   // another call's expert (expert-sharded execution)
      const int r = s->base[e] + __popc(s->words[e] & ((1u << t) - 1u));
      const int row = s->off[e] + r;
      p.perm[row] = flat;
      if (p.perm_out) p.perm_out[row] = flat;
      const int slot = r / slot_rows, pos = (s->tile0[e] + slot) * 128 + (r - slot * slot_rows);
      p.pos_pad[flat] = pos;
      p.row_token[pos] = c0 + t;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < E; e += kRouteThreads) s->base[e] += __popc(s->words[e]);
    __syncthreads();
  }
}

}  // namespace quads
