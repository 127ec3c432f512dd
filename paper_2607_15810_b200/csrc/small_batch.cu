// The front of a call with few tokens, each half of it in ONE thread-block cluster, so that the steps meet
// at cluster barriers (a few hundred nanoseconds, distributed shared memory) instead of at kernel
// boundaries (two to three microseconds each):
//   route_small_kernel  top-k routing, per-expert counts, scan, dispatch order;
//   front_small_kernel  tensor amax, quantization of x and of its residual, channel scores, selection,
//                       masked copies in dispatch order.
// What bounds them is latency: at decode sizes they move a few megabytes at most, which stay in L2 and
// shared memory.  Larger batches use the grid-wide kernels of front.cu (api.cu holds the rule): a cluster is 16 of the 148 SMs.
#include <algorithm>
#include <atomic>

#include "kernels.cuh"
#include "select.cuh"
#include "tcgen05.cuh"

namespace quads {
namespace {

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void st_cluster_u32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void st_cluster_u64(uint32_t addr, unsigned long long v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
// 32 bytes, kept in L1: the amax pass and the quantization read the same block.
__device__ __forceinline__ void ldg256_l1(const void* p, uint4& a, uint4& b) {
  asm volatile("ld.global.nc.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w) : "l"(p));
}
constexpr int kSmallRouteThreads = 512;                         // 16 warps: a warp per token, four per scheduler
constexpr int kRouteTokens = kSmallRouteThreads / 32;           // tokens of a word of the assignment bit matrix
constexpr int kRouteWords = kSmallRouteMaxTokens / kRouteTokens;

// One warp per token (TW tokens).  The assignments are a bit matrix, words[t / 16][expert] bit t % 16: an expert's
// count is a population count over its words, and the row of token t inside an expert is the population count
// below bit t, which is the (expert, token, slot) order without a sort.
// Every CTA sends its words to the others, then scans all experts for itself.
template <int NJ, int TW>
__global__ void __launch_bounds__(kSmallRouteThreads)
route_small_kernel(const SmallRouteArgs p) {
  pdl_sync();
  __shared__ uint32_t words[kRouteWords][kMaxExperts];
  __shared__ int s_off[kMaxExperts], s_tile[kMaxExperts], s_base[kMaxExperts];
  __shared__ int wsum[2][8];
  const int rank = (int)cluster_ctarank(), n_cta = (int)gridDim.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int E = p.E, topk = p.topk;
  cluster_arrive();                                        // (waited for before the first remote store)
  for (int i = threadIdx.x; i < TW * kMaxExperts; i += kSmallRouteThreads) words[rank * TW + i / kMaxExperts][i % kMaxExperts] = 0;
  // Top-k on order-preserving integer keys, two warp reductions per slot; softmax only for the chosen ones.
  float v[TW][NJ], my_w[TW];
  int my_id[TW];
#pragma unroll
  for (int a = 0; a < TW; ++a) {
    const int t = (rank * TW + a) * kRouteTokens + warp;
    my_w[a] = 0.f; my_id[a] = 0;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const int e = j * 32 + lane;
      v[a][j] = (t < p.T && e < E) ? p.logits[(size_t)t * E + e] + 0.f : -INFINITY;   // -0 counts as +0
    }
  }
  __syncthreads();                                         // the words are zero
#pragma unroll
  for (int a = 0; a < TW; ++a) {
    const int t = (rank * TW + a) * kRouteTokens + warp;
    if (t >= p.T) continue;                                // (the whole warp)
    uint32_t key[NJ];
#pragma unroll
    for (int j = 0; j < NJ; ++j) key[j] = j * 32 + lane < E ? float_key(v[a][j]) : 0u;
    uint32_t my_key = 0;
    for (int s = 0; s < topk; ++s) {
      uint32_t m = key[0];
#pragma unroll
      for (int j = 1; j < NJ; ++j) m = max(m, key[j]);
      const uint32_t g = __reduce_max_sync(0xFFFFFFFFu, m);
      uint32_t e1 = 0x7FFFFFFFu;
#pragma unroll
      for (int j = NJ - 1; j >= 0; --j)
        if (key[j] == g) e1 = (uint32_t)(j * 32 + lane);
      const int be = (int)__reduce_min_sync(0xFFFFFFFFu, e1);            // ties to the lower expert id
      if (lane == s) { my_key = g; my_id[a] = be; }
#pragma unroll
      for (int j = 0; j < NJ; ++j)
        if (j * 32 + lane == be) key[j] = 0u;                            // remove the winner
    }
    const float gv = __uint_as_float((my_key & 0x80000000u) ? (my_key & 0x7FFFFFFFu) : ~my_key);
    const float mx = __shfl_sync(0xFFFFFFFFu, gv, 0);
    float sum = 0.f;
#pragma unroll
    for (int j = 0; j < NJ; ++j) sum += j * 32 + lane < E ? expf(v[a][j] - mx) : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
    float w = lane < topk ? expf(gv - mx) / sum : 0.f;
    if (p.renormalize) {
      float ws = 0.f;
      for (int s = 0; s < topk; ++s) ws += __shfl_sync(0xFFFFFFFFu, w, s);
      w = w / ws;
    }
    my_w[a] = w;
    if (lane < topk && my_id[a] >= p.e_lo && my_id[a] < p.e_hi) atomicOr(&words[rank * TW + a][my_id[a]], 1u << warp);
  }
  __syncthreads();
  cluster_wait();                                          // every CTA of the cluster has started
  if (n_cta > 1)
    for (int i = threadIdx.x; i < TW * E * n_cta; i += kSmallRouteThreads) {
      const int c = i / (TW * E), k = i - c * (TW * E), a = k / E, e = k - a * E;
      if (c != rank) st_cluster_u32(map_to_cta(smem_u32(&words[rank * TW + a][e]), (uint32_t)c), words[rank * TW + a][e]);
    }
  cluster_arrive();
  cluster_wait();
  // ---- counts, exclusive scans over the experts (threads 0..255), this CTA's first row in every expert
  const int n_words = n_cta * TW;
  int cnt = 0, base = 0, tiles = 0, inc_c = 0, inc_t = 0;
  if (threadIdx.x < 256) {
    const int e = threadIdx.x;
    if (e < E)
      for (int w = 0; w < n_words; ++w) {
        const int c = __popc(words[w][e]);
        cnt += c;
        if (w < rank * TW) base += c;
      }
    tiles = (cnt + p.slot_rows - 1) / p.slot_rows;
    inc_c = cnt; inc_t = tiles;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int a = __shfl_up_sync(0xFFFFFFFFu, inc_c, o), b = __shfl_up_sync(0xFFFFFFFFu, inc_t, o);
      if (lane >= o) { inc_c += a; inc_t += b; }
    }
    if (lane == 31) { wsum[0][warp] = inc_c; wsum[1][warp] = inc_t; }
  }
  __syncthreads();
  if (threadIdx.x < 256) {
    const int e = threadIdx.x;
    int off = inc_c - cnt, tp = inc_t - tiles;
    for (int w = 0; w < warp; ++w) { off += wsum[0][w]; tp += wsum[1][w]; }
    if (e < E) {
      s_off[e] = off; s_tile[e] = tp; s_base[e] = base;
      if (rank == 0) {
        p.offsets[e] = off;
        p.tile_prefix[e] = tp;
        if (p.offsets_out) p.offsets_out[e] = off;
        for (int m = 0; m < tiles; ++m) {
          p.tile_expert[tp + m] = e;
          p.tile_rows[tp + m] = min(p.slot_rows, cnt - m * p.slot_rows);
        }
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
  // words of the call that start at zero: the status word and the column totals of site 2
  if (rank == n_cta - 1) {
    if (threadIdx.x < kHdrWords - kHdrStatus) p.header[kHdrStatus + threadIdx.x] = 0;
    for (int i = threadIdx.x; i < p.n_zero; i += kSmallRouteThreads) p.zero_u64[i] = 0ull;
  }
  // ---- rows (and the stores that the barriers above would have waited for)
#pragma unroll
  for (int a = 0; a < TW; ++a) {
    const int t = (rank * TW + a) * kRouteTokens + warp;
    if (t >= p.T || lane >= topk) continue;
    const int flat = t * topk + lane;
    const int e = my_id[a];
    p.wts[flat] = my_w[a];
    if (p.ids_out) p.ids_out[flat] = e;
    if (p.wts_out) p.wts_out[flat] = my_w[a];
    if (e < p.e_lo || e >= p.e_hi) { p.pos_pad[flat] = -1; continue; }      // another call's expert (expert-sharded execution)
    int r = s_base[e] + __popc(words[rank * TW + a][e] & ((1u << warp) - 1u));
#pragma unroll
    for (int b = 0; b < TW; ++b)
      if (b < a) r += __popc(words[rank * TW + b][e]);
    const int slot = r / p.slot_rows, row = s_off[e] + r, pos = (s_tile[e] + slot) * 128 + (r - slot * p.slot_rows);
    p.perm[row] = flat;
    if (p.perm_out) p.perm_out[row] = flat;
    p.pos_pad[flat] = pos;
    p.row_token[pos] = t;
  }
}

// Site 13 of a small batch.  A CTA owns whole columns: units of 128 channels (8 scale blocks) for all rows, so
// that channel scores need no reduction across CTAs, only an exchange of finished scores; thread = (block of
// the unit, row group).  The CTA keeps the residual's codes in shared memory until the selection is known.
// Two forms of output: token order with linear scales (for the GEMM that gathers its rows), or dispatched
// copies with tiled scales, for which the codes of x and all scales are kept until then as well.
// dynamic shared memory: H keys | 32 x 128 partial sums, later the H images of the selection | per (unit, row):
// 64 B codes of the residual and, for dispatched copies, 64 B of x, 8 + 8 scale bytes.
__global__ void __launch_bounds__(kSmallThreads)
front_small_kernel(const SmallFrontArgs p) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ uint32_t amax_all[16];
  __shared__ uint32_t wmax[32];
  __shared__ SelectScratch scratch;
  __shared__ double red2[8][128];
  __shared__ __align__(16) uint32_t nib[kSmallMaxUnits * 16];
  const int rank = (int)cluster_ctarank(), n_cta = (int)gridDim.x;
  const int T = p.T, H = p.H, units = H >> 7;
  const int upc = (units + n_cta - 1) / n_cta;             // units per CTA
  const int n_my = rank < units ? (units - rank + n_cta - 1) / n_cta : 0;      // units rank, rank + n_cta, ...
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(smem);
  float* red = reinterpret_cast<float*>(smem + (size_t)H * 8);
  uint8_t* st_r = smem + (size_t)H * 8 + max(32 * 128, H) * 4;
  uint8_t* st_x = st_r + (size_t)upc * T * 64;
  uint8_t* sf_x = st_x + (size_t)upc * T * 64;
  uint8_t* sf_r = sf_x + (size_t)upc * T * 8;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int blk = threadIdx.x & 7, rg = threadIdx.x >> 3;
  // In front of a MoE layer the preceding kernel is route_small_kernel, which has itself waited for whatever
  // produced x: only the dispatch order has to be waited for, later on.
  if (!p.after_routing) pdl_sync();
  cluster_arrive();
  bool started = false;                                    // the wait that belongs to this arrive has been made
  float gs;
  if (p.gs_in) {
    gs = p.gs_in[0];
  } else {
    uint32_t m = 0;
    for (int ui = 0; ui < n_my; ++ui)
      for (int r = rg; r < T; r += kSmallThreads / 8) {
        uint4 v0, v1;
        ldg256_l1(p.x + (size_t)r * H + (rank + ui * n_cta) * 128 + blk * 16, v0, v1);
        m = __vmaxu2(m, __vmaxu2(absmax8(v0), absmax8(v1)));
      }
    m = __reduce_max_sync(0xFFFFFFFFu, max(m & 0xFFFFu, m >> 16));
    if (lane == 0) wmax[warp] = m;
    __syncthreads();
    cluster_wait();
    started = true;
    if (warp == 0) {
      const uint32_t t = __reduce_max_sync(0xFFFFFFFFu, wmax[lane]);
      if (lane < n_cta) st_cluster_u32(map_to_cta(smem_u32(&amax_all[rank]), (uint32_t)lane), t);
    }
    cluster_arrive();
    cluster_wait();
    uint32_t bits = 0;
    for (int c = 0; c < n_cta; ++c) bits = max(bits, amax_all[c]);
    bits <<= 16;
    if (rank == 0 && threadIdx.x == 0) p.amax_bits[0] = bits;
    const float amax = __uint_as_float(bits);
    gs = amax > 0.f ? __fdiv_rn(amax, kGlobalDiv) : 1.0f;
  }
  if (rank == 0 && threadIdx.x == 0) {
    if (p.gs_store) p.gs_store[0] = gs;
    if (!p.after_routing) p.header[kHdrStatus] = 0;
  }
  QuantCtx qc;                                             // (a reciprocal table costs more than a few blocks' divisions)
  quant_ctx_scalars(qc, gs);
  qc.inv_lut = nullptr;
  if (!started) cluster_wait();
  const int n_warps = min(32, (T * 8 + 31) / 32);          // warps that hold rows
  for (int ui = 0; ui < n_my; ++ui) {
    const int u = rank + ui * n_cta;
    float acc[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i] = 0.f;
    for (int r = rg; r < T; r += kSmallThreads / 8) {
      uint4 v0, v1;
      ldg256_l1(p.x + (size_t)r * H + u * 128 + blk * 16, v0, v1);
      float f[16];
      unpack8(v0, f);
      unpack8(v1, f + 8);
      const BlockQ bq = quantize_block<false>(f, qc);
      const int idx = ui * T + r;
      const size_t qo = (size_t)r * (H >> 1) + u * 64 + blk * 8, so = (size_t)r * (H >> 4) + u * 8 + blk;
      if (p.token_order) {
        *reinterpret_cast<uint2*>(p.xq_pad + qo) = make_uint2(bq.lo, bq.hi);
        p.xsf[so] = (uint8_t)bq.sf8;
      } else {
        reinterpret_cast<uint2*>(st_x)[idx * 8 + blk] = make_uint2(bq.lo, bq.hi);
        sf_x[idx * 8 + blk] = (uint8_t)bq.sf8;
      }
      if (p.xq_exp) *reinterpret_cast<uint2*>(p.xq_exp + qo) = make_uint2(bq.lo, bq.hi);
      if (p.xsf_exp) p.xsf_exp[so] = (uint8_t)bq.sf8;
      if (p.n_sel > 0) {
        float o[16];
        residual_block(bq, f, o);
        add_squares(o, acc);
        const BlockQ br = quantize_block<false>(o, qc);
        reinterpret_cast<uint2*>(st_r)[idx * 8 + blk] = make_uint2(br.lo, br.hi);
        if (p.token_order) p.rsf[so] = (uint8_t)br.sf8;
        else sf_r[idx * 8 + blk] = (uint8_t)br.sf8;
        if (p.rsf_exp) p.rsf_exp[so] = (uint8_t)br.sf8;
      }
    }
    if (p.n_sel > 0) {
      // column scores: the four row groups of a warp, then (float64) four warps each, then the eight groups of warps
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        acc[i] += __shfl_xor_sync(0xFFFFFFFFu, acc[i], 8);
        acc[i] += __shfl_xor_sync(0xFFFFFFFFu, acc[i], 16);
      }
      if (lane < 8 && warp < n_warps) {
        float4* d = reinterpret_cast<float4*>(red + warp * 128 + blk * 16);
        d[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
        d[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
        d[2] = make_float4(acc[8], acc[9], acc[10], acc[11]);
        d[3] = make_float4(acc[12], acc[13], acc[14], acc[15]);
      }
      __syncthreads();
      {
        const int c = threadIdx.x & 127, w0 = (threadIdx.x >> 7) * 4;
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < 4; ++w)
          if (w0 + w < n_warps) s += (double)red[(w0 + w) * 128 + c];
        red2[w0 / 4][c] = s;
      }
      __syncthreads();
      if (threadIdx.x < 128) {
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < 8; ++w) s += red2[w][threadIdx.x];
        keys[u * 128 + threadIdx.x] = (unsigned long long)__double_as_longlong(s);   // order-preserving: s >= 0
      }
      __syncthreads();
      for (int i = threadIdx.x; i < 128 * n_cta; i += kSmallThreads) {
        const int c = i >> 7, k = u * 128 + (i & 127);
        if (c != rank) st_cluster_u64(map_to_cta(smem_u32(&keys[k]), (uint32_t)c), keys[k]);
      }
    }
  }
  cluster_arrive();
  if (p.after_routing) pdl_sync();                         // the dispatch order is there; what follows may start
  cluster_wait();
  if (p.n_sel > 0) {
    const Selection sel = select_largest<true>(keys, reinterpret_cast<uint32_t*>(red), H, p.n_sel, &scratch);
    for (int i = threadIdx.x; i < n_my * 16; i += kSmallThreads) {
      const int ch = (rank + (i >> 4) * n_cta) * 128 + (i & 15) * 8;
      uint32_t m = 0;
#pragma unroll
      for (int k = 0; k < 8; ++k) m |= sel.has(keys[ch + k], ch + k) ? 0xFu << (4 * k) : 0u;
      nib[i] = m;
    }
    if (p.mask_out)
      for (int i = threadIdx.x; i < n_my * 128; i += kSmallThreads) {
        const int ch = (rank + (i >> 7) * n_cta) * 128 + (i & 127);
        p.mask_out[ch] = sel.has(keys[ch], ch) ? 1 : 0;
      }
  }
  __syncthreads();
  const int kt_count = H >> 6;
  for (int ui = 0; ui < n_my; ++ui) {
    const int u = rank + ui * n_cta;
    // ---- the masked residual in token order: the operand itself (stored negated), and the verification export
    if (p.n_sel > 0 && (p.token_order || p.rq_exp))
      for (int i = threadIdx.x; i < T * 4; i += kSmallThreads) {
        const int r = i >> 2, q = i & 3;
        uint4 v = reinterpret_cast<const uint4*>(st_r)[(ui * T + r) * 4 + q];
        const uint4 m = reinterpret_cast<const uint4*>(nib)[ui * 4 + q];
        v.x &= m.x; v.y &= m.y; v.z &= m.z; v.w &= m.w;
        const size_t o = (size_t)r * (H >> 1) + u * 64 + q * 16;
        if (p.rq_exp) *reinterpret_cast<uint4*>(p.rq_exp + o) = v;
        v.x ^= 0x88888888u; v.y ^= 0x88888888u; v.z ^= 0x88888888u; v.w ^= 0x88888888u;
        if (p.token_order) *reinterpret_cast<uint4*>(p.rq_pad + o) = v;
      }
    if (p.token_order) continue;
    // ---- dispatched copies: four threads per assignment, 16 bytes of codes each, the residual masked and
    // stored negated; the four also carry the two scale words of either operand
    const int A = T * p.topk;
    for (int i = threadIdx.x; i < A * 4; i += kSmallThreads) {
      const int flat = i >> 2, q = i & 3;
      const int pos = p.pos_pad ? __ldg(p.pos_pad + flat) : flat;
      if (pos < 0) continue;
      const int idx = ui * T + (p.topk == 1 ? flat : flat / p.topk);
      const size_t po = (size_t)pos * (H >> 1) + u * 64 + q * 16;
      *reinterpret_cast<uint4*>(p.xq_pad + po) = reinterpret_cast<const uint4*>(st_x)[idx * 4 + q];
      if (p.n_sel > 0) {
        uint4 v = reinterpret_cast<const uint4*>(st_r)[idx * 4 + q];
        const uint4 m = reinterpret_cast<const uint4*>(nib)[ui * 4 + q];
        v.x = (v.x & m.x) ^ 0x88888888u; v.y = (v.y & m.y) ^ 0x88888888u;
        v.z = (v.z & m.z) ^ 0x88888888u; v.w = (v.w & m.w) ^ 0x88888888u;
        *reinterpret_cast<uint4*>(p.rq_pad + po) = v;
      }
      const size_t so = sf_tiled_offset(pos, u * 8 + (q & 1) * 4, kt_count);
      if (q < 2) *reinterpret_cast<uint32_t*>(p.xsf + so) = reinterpret_cast<const uint32_t*>(sf_x)[idx * 2 + q];
      else if (p.n_sel > 0) *reinterpret_cast<uint32_t*>(p.rsf + so) = reinterpret_cast<const uint32_t*>(sf_r)[idx * 2 + (q & 1)];
    }
  }
}

size_t front_small_smem(int T, int H, int n_cta, bool token_order) {
  const int units = H / 128, upc = (units + n_cta - 1) / n_cta;
  return (size_t)H * 8 + std::max(32 * 128, H) * 4 + (size_t)upc * T * (token_order ? 64 : 64 + 64 + 8 + 8);
}

constexpr int kFrontMaxSmem = 200 * 1024;

// Largest cluster front_small_kernel can be launched with on the current device: 16 CTAs where the device
// schedules clusters beyond the portable size, else 8.
int front_cluster_limit() {
  static std::atomic<int> per_device[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 8;
  int v = per_device[dev].load();
  if (v == 0) {
    v = 8;
    if (cudaFuncSetAttribute(front_small_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        set_max_dynamic_smem<front_small_kernel>(kFrontMaxSmem) == cudaSuccess) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(16);
      cfg.blockDim = dim3(kSmallThreads);
      cfg.dynamicSmemBytes = kFrontMaxSmem;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = 16; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, front_small_kernel, &cfg) == cudaSuccess && n > 0) v = 16;
    }
    (void)cudaGetLastError();                              // a refused query is an answer, not an error of the call
    per_device[dev].store(v);
  }
  return v;
}

int front_ctas(int H) {
  const int limit = front_cluster_limit();
  int n = 1;
  while (n < limit && n < H / 128) n *= 2;
  return n;
}

template <int NJ, int TW>
quads_status launch_route_tw(const SmallRouteArgs& a, cudaStream_t st) {
  static std::atomic<bool> wide[64];                       // clusters beyond the portable size allowed for this kernel
  int n = 1, dev = 0;
  while (n * TW * kRouteTokens < a.T) n *= 2;
  if (n > 8) {
    QUADS_CUDA_OK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return QUADS_ERR_CUDA;
    if (!wide[dev].load()) {
      QUADS_CUDA_OK(cudaFuncSetAttribute(route_small_kernel<NJ, TW>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
      wide[dev].store(true);
    }
  }
  QUADS_CUDA_OK(launch_cluster(route_small_kernel<NJ, TW>, n, kSmallRouteThreads, 0, st, a));
  return QUADS_OK;
}

template <int NJ>
quads_status launch_route_nj(const SmallRouteArgs& a, cudaStream_t st) {
  return a.T <= kRouteTokens * front_cluster_limit() ? launch_route_tw<NJ, 1>(a, st) : launch_route_tw<NJ, 2>(a, st);
}

}  // namespace

bool route_small_fits(int T) { return T <= 2 * kRouteTokens * front_cluster_limit(); }

bool front_small_fits(int T, int H, bool token_order) {
  const int n = front_ctas(H), upc = (H / 128 + n - 1) / n;
  return route_small_fits(T) && upc <= kSmallMaxUnits && front_small_smem(T, H, n, token_order) <= (size_t)kFrontMaxSmem;
}

quads_status launch_route_small(const SmallRouteArgs& a, cudaStream_t st) {
  return a.E <= 32 ? launch_route_nj<1>(a, st)
                   : (a.E <= 64 ? launch_route_nj<2>(a, st) : (a.E <= 128 ? launch_route_nj<4>(a, st) : launch_route_nj<8>(a, st)));
}

quads_status launch_front_small(const SmallFrontArgs& a, cudaStream_t st) {
  QUADS_CUDA_OK(set_max_dynamic_smem<front_small_kernel>(kFrontMaxSmem));
  const int n = front_ctas(a.H);
  QUADS_CUDA_OK(launch_cluster(front_small_kernel, n, kSmallThreads, front_small_smem(a.T, a.H, n, a.token_order != 0), st, a));
  return QUADS_OK;
}

}  // namespace quads
