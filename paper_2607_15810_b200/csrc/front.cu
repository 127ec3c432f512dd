// The front of a MoE call or a dense projection of more than a few tokens (small_batch.cu has the others):
//   front_kernel        routing and quantization, two independent roles of one cooperative launch;
//   quant_rows_kernel   the quantization role alone (dense projections have no routing);
//   dispatch_kernel     the copies of codes and scales in dispatch order, and the channel selection.
#include <algorithm>
#include <atomic>

#include "routing.cuh"

namespace quads {

// ---------------------------------------------------------------------------
// Site-13 quantization pass, token order.  For every row and 16-channel block:
// Q_A(x) codes + scale; the residual Q_A(x) - x in float32 (Eq. residual-def);
// its squared sum per channel (Eq. channel-score); and the residual's own
// quantization with the same per-tensor scale (the mask of Eq. residual-recon is
// applied later: quantizing the residual does not depend on the selection).
//
// A CTA owns bw blocks of 16 channels (8, 16 or 32, see plan_quant) for a range of rows;
// thread = (block, row lane).  The grid is what is resident at once, so that the amax of x can be the
// first phase of the same launch: the CTAs meet at a counter (bounded wait) and read their rows again, out of L2.
// A CTA adds its row lanes' column sums up in shared memory and leaves one float32 per channel; the last CTA of a
// column group to finish adds the row ranges up in float64, in their order, so that the scores keep their
// relative precision whatever the range of x and its scale, and do not depend on who finishes when.  Fixed-point
// totals, one reduction per CTA and channel, cost 1 to 2 us less (dense 8192 x 4096 -> 4096 157.4 us, 158.6 so; 1200 x
// 512 -> 128 18.5, 20.5; a MoE layer of 1500 tokens the same), but need a bound on the residual, which a given
// scale that x exceeds does not have, and lose channels that are small beside an outlier.
// Bound by the arithmetic, about 240 cycles per warp and block with its loads, 64 of them in the two conversions to E2M1, and by
// reading x a second time out of L2 (some 6.6 TB/s).
// Dense projection 8192 x 4096 -> 4096: amax, quantization, score reduction, ranking and copy took 16 + 27 + 12 +
// 12 + 28 us as kernels of their own; this one takes about 40 and the in-place mask behind it 10 (whole call
// 205 -> 159 us).
// Scales are stored linear [T, H/16], or tiled when the rows are a dense projection's operand as they are.
// ---------------------------------------------------------------------------
struct QuantShared {
  float gs;
  int last;
  uint32_t wmax[8];
  float inv_lut[128];
  __align__(16) float red[256 * 16];
};

// Adds up the partial scores of a column group (n_ch = 128, 256 or 512 channels, `part` its first one's, rows of H), one
// row per row range.  Thread = (four channels, every n-th row); latency-bound, eight loads in flight.
__device__ __forceinline__ void sum_partial_scores(const float* part, int n_rg, int H, int n_ch, unsigned long long* keys, double* red) {
  const int quads = n_ch >> 2, q = threadIdx.x % quads, sl = threadIdx.x / quads, n_sl = 256 / quads;
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
  for (int r = sl; r < n_rg; r += 8 * n_sl) {
    float4 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      v[u] = r + u * n_sl < n_rg ? __ldcg(reinterpret_cast<const float4*>(part + (size_t)(r + u * n_sl) * H) + q)
                                 : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < 8; ++u) { a0 += (double)v[u].x; a1 += (double)v[u].y; a2 += (double)v[u].z; a3 += (double)v[u].w; }
  }
  double* d = red + sl * n_ch + 4 * q;
  d[0] = a0; d[1] = a1; d[2] = a2; d[3] = a3;
  __syncthreads();
  for (int c = threadIdx.x; c < n_ch; c += 256) {
    double t = 0.0;
    for (int l = 0; l < n_sl; ++l) t += red[l * n_ch + c];
    keys[c] = (unsigned long long)__double_as_longlong(t);   // order-preserving: t >= 0
  }
}

// CTA `cta` of `n_cta`.
__device__ __forceinline__ void quant_role(const QuantRowsArgs& p, int cta, int n_cta, QuantShared* s) {
  const int H = p.H, k16 = H >> 4;
  const int col = cta % p.n_col, rg = cta / p.n_col;
  const int blk = threadIdx.x % p.bw, lane_r = threadIdx.x / p.bw, lanes = 256 / p.bw;
  const int kb = col * p.bw + blk;
  const int r0 = rg * p.rows_per_cta + lane_r, r1 = min(p.T, (rg + 1) * p.rows_per_cta);
  const uint16_t* xk = p.x + kb * 16;
  if (!p.gs_in && p.amax_parts) {
    uint32_t m = 0;
    for (int i = threadIdx.x; i < p.n_amax_parts; i += 256) m = max(m, __ldcg(p.amax_parts + i));
    m = __reduce_max_sync(0xFFFFFFFFu, m);
    if ((threadIdx.x & 31) == 0) s->wmax[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t tm = 0;
      for (int i = 0; i < 8; ++i) tm = max(tm, s->wmax[i]);
      if (cta == 0) p.amax_bits[0] = tm;
      s->gs = gs_from_amax_bits(tm);
    }
    __syncthreads();
  } else if (!p.gs_in) {
    uint32_t m = 0;
    int r = r0;
    for (; r + 3 * lanes < r1; r += 4 * lanes) {
      uint4 v[8];
#pragma unroll
      for (int u = 0; u < 4; ++u) ldg256_keep(xk + (size_t)(r + u * lanes) * H, v[2 * u], v[2 * u + 1]);
#pragma unroll
      for (int u = 0; u < 8; ++u) m = __vmaxu2(m, absmax8(v[u]));
    }
    for (; r < r1; r += lanes) {
      uint4 v0, v1;
      ldg256_keep(xk + (size_t)r * H, v0, v1);
      m = __vmaxu2(m, __vmaxu2(absmax8(v0), absmax8(v1)));
    }
    m = __reduce_max_sync(0xFFFFFFFFu, max(m & 0xFFFFu, m >> 16));
    if ((threadIdx.x & 31) == 0) s->wmax[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t tm = 0;
      for (int i = 0; i < 8; ++i) tm = max(tm, s->wmax[i]);
      if (tm) atomicMax(p.amax_bits, tm << 16);
      __threadfence();
      atomicAdd(p.arrivals, 1u);
      grid_wait(p.arrivals, (uint32_t)n_cta, p.status);
      s->gs = gs_from_amax_bits(ld_relaxed_u32(p.amax_bits));
    }
    __syncthreads();
  } else {
    if (threadIdx.x == 0) s->gs = p.gs_in[0];
    __syncthreads();
  }
  const float gs = s->gs;
  if (p.gs_store && cta == 0 && threadIdx.x == 0) p.gs_store[0] = gs;
  if (threadIdx.x < 128) s->inv_lut[threadIdx.x] = quant_inv_entry(threadIdx.x, gs);
  __syncthreads();
  QuantCtx qc;
  quant_ctx_scalars(qc, gs);
  qc.inv_lut = s->inv_lut;
  float acc[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) acc[i] = 0.f;
  uint4 n0 = make_uint4(0, 0, 0, 0), n1 = n0;
  if (r0 < r1) ldg256(xk + (size_t)r0 * H, n0, n1);
  for (int r = r0; r < r1; r += lanes) {
    const uint4 v0 = n0, v1 = n1;
    if (r + lanes < r1) ldg256(xk + (size_t)(r + lanes) * H, n0, n1);   // next block, ahead of this one's arithmetic
    float f[16], o[16];
    unpack8(v0, f);
    unpack8(v1, f + 8);
    const BlockQ bq = quantize_block(f, qc);
    const size_t qo = (size_t)r * (H >> 1) + kb * 8, so = (size_t)r * k16 + kb;
    const size_t so_op = p.sf_tiled ? sf_tiled_offset(r, kb, H >> 6) : so;
    *reinterpret_cast<uint2*>(p.xq + qo) = make_uint2(bq.lo, bq.hi);
    p.xsf[so_op] = (uint8_t)bq.sf8;
    if (p.xq_exp) *reinterpret_cast<uint2*>(p.xq_exp + qo) = make_uint2(bq.lo, bq.hi);
    if (p.xsf_exp) p.xsf_exp[so] = (uint8_t)bq.sf8;
    if (p.with_residual) {
      residual_block(bq, f, o);
      add_squares(o, acc);
      const BlockQ br = quantize_block(o, qc);
      *reinterpret_cast<uint2*>(p.rq + qo) = make_uint2(br.lo, br.hi);
      p.rsf[so_op] = (uint8_t)br.sf8;
      if (p.rsf_exp) p.rsf_exp[so] = (uint8_t)br.sf8;
    }
  }
  if (!p.with_residual) return;
  // column sums: the CTA's row lanes, then (by the last CTA) the row ranges
  const int n_ch = p.bw * 16, n_rg = n_cta / p.n_col;        // channels of this CTA, row ranges
  float4* d = reinterpret_cast<float4*>(s->red + threadIdx.x * 16);
#pragma unroll
  for (int i = 0; i < 4; ++i) d[i] = make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
  __syncthreads();
  for (int c = threadIdx.x; c < n_ch; c += 256) {
    double t = 0.0;
#pragma unroll 8
    for (int l = 0; l < lanes; ++l) t += (double)s->red[l * n_ch + c];
    p.partials[(size_t)rg * H + col * n_ch + c] = (float)t;
  }
  __syncthreads();
  if (threadIdx.x == 0) {                                    // (releases what the barrier ordered before it)
    uint32_t before;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(before) : "l"(p.col_arrivals + col) : "memory");
    s->last = before == (uint32_t)n_rg - 1u;
  }
  __syncthreads();
  if (s->last) sum_partial_scores(p.partials + col * n_ch, n_rg, H, n_ch, p.keys + col * n_ch, reinterpret_cast<double*>(s->red));
}

__global__ void __launch_bounds__(256, kQuantRowsPerSm) quant_rows_kernel(const QuantRowsArgs p) {
  pdl_sync();
  __shared__ QuantShared s;
  quant_role(p, (int)blockIdx.x, (int)gridDim.x, &s);
}

// All CTAs route a few tokens first; then the first n_groups (one per SM) hand out the rows while the others, three
// per SM beside them, quantize: the roles need nothing of one another, each has its own counters to meet at.
// As five kernels on two streams (route, scan, permute beside quantize, rank) the last of them ended 44 us after
// the call's start at 8192 tokens, because the quantization held the SMs; here codes, scores and tables are
// there after 30 us (1500 tokens: 14 instead of 30).  Asking L2 for x before the tokens are routed gains nothing up to 4096 x
// 4096 and loses beyond, where the lines it is asked to keep are evicted unread or evict others (this kernel with a cold
// cache, 8192 x 4096 53 us, 57 so; 16384 x 4096 92 and 108; with a given scale 39 and 47).
template <int NJ>
__global__ void __launch_bounds__(256, kQuantRowsPerSm)
front_kernel(const QuantRowsArgs q, const RouteArgs r, int n_groups) {
  pdl_sync();
  __shared__ union { QuantShared q; RouteShared r; } s;
  route_part1<NJ>(r, (int)blockIdx.x, (int)gridDim.x, n_groups);
  if ((int)blockIdx.x < n_groups) route_part2<NJ>(r, (int)blockIdx.x, n_groups, gridDim.x, &s.r);
  else quant_role(q, (int)blockIdx.x - n_groups, (int)gridDim.x - n_groups, &s.q);
}

// ---------------------------------------------------------------------------
// Site-13 dispatch, driven by the DESTINATION: the tiles of the padded dispatch order are cut into slabs of 512
// channels; a CTA gathers a slab's rows from the token-order arrays (which stay in L2: every token row is
// read top-k times) and writes its codes and its eight scale atoms as whole regions.  Written from the
// source side instead (one thread per token chunk), every 512-byte scale atom is touched by 128 different
// tokens at 128 different times, 4 bytes each: partially written sectors get evicted and the memory system
// pays for them.
// kResid = false copies Q(x), and ranks the channels on the side (every CTA a few of them), so that the mask is there
// for kResid = true, which copies the residual: masked on the way (Eq. residual-recon: codes of unselected
// channels are cleared) and stored NEGATED (sign bits flipped), so that the GEMM can accumulate
// W Q(x) + W (-M Q(dx)) with two plain MMAs.
// Bound by the writes (75 MB each at 8192 tokens x 8 x 2048 channels).  A ranking kernel and copies with one CTA
// per tile (half of the last wave idle) took 6 + 21 + 21 us; these are 18 (ranking included) + 16.
// dynamic shared memory: two sets of eight scale atoms, H / 8 mask words.
// ---------------------------------------------------------------------------
constexpr int kSlabChunks = 16;                      // 16-byte chunks of codes (32 channels each) per row and slab
constexpr int kSlabAtoms = 8;
constexpr int kRankBatch = 4;                        // channels a CTA ranks in one pass over the scores

// rank_j = #{i : s_i > s_j, or s_i == s_j and i < j}; channel j is selected iff rank_j < n_sel (the n_sel largest, ties
// to the lower index; Eq. channel-select).
__device__ __forceinline__ void rank_channels(const DispatchArgs& p, int* rank_sh) {
  const int H = p.H;
  if (threadIdx.x < kRankBatch) rank_sh[threadIdx.x] = 0;
  __syncthreads();
  for (int j0 = blockIdx.x * kRankBatch; j0 < H; j0 += gridDim.x * kRankBatch) {
    unsigned long long mine[kRankBatch];
    int cnt[kRankBatch];
#pragma unroll
    for (int k = 0; k < kRankBatch; ++k) {
      mine[k] = __ldcg(p.keys + j0 + k);             // (H is a multiple of 128)
      cnt[k] = 0;
    }
#pragma unroll 4
    for (int i = threadIdx.x; i < H; i += kDispatchThreads) {
      const unsigned long long si = __ldcg(p.keys + i);
#pragma unroll
      for (int k = 0; k < kRankBatch; ++k) cnt[k] += (si > mine[k] || (si == mine[k] && i < j0 + k)) ? 1 : 0;
    }
#pragma unroll
    for (int k = 0; k < kRankBatch; ++k) {
      const int t = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)cnt[k]);
      if ((threadIdx.x & 31) == 0 && t) atomicAdd(rank_sh + k, t);
    }
    __syncthreads();
    if (threadIdx.x < kRankBatch) {
      p.mask[j0 + threadIdx.x] = rank_sh[threadIdx.x] < p.n_sel ? 1 : 0;
      rank_sh[threadIdx.x] = 0;
    }
    __syncthreads();
  }
}

template <bool kResid>
__global__ void __launch_bounds__(kDispatchThreads, kDispatchPerSm)
dispatch_kernel(const DispatchArgs p) {
  static_assert(kDispatchThreads == 512, "four 16-byte chunks and one 8-byte piece of scales per thread");
  pdl_sync();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int tok[2][128];
  __shared__ int rank_sh[kRankBatch];
  const int H = p.H, per_row = H >> 5, kt_count = H >> 6;
  uint32_t* nib = reinterpret_cast<uint32_t*>(smem_raw + 2 * kSlabAtoms * 512);
  if (kResid) {
    for (int w = threadIdx.x; w < (H >> 3); w += kDispatchThreads)
      nib[w] = nibble_mask8(__ldg(reinterpret_cast<const uint2*>(p.mask) + w));
  } else if (p.n_sel > 0) {
    rank_channels(p, rank_sh);
  }
  const uint8_t *src = kResid ? p.rq : p.xq, *src_sf = kResid ? p.rsf : p.xsf;
  uint8_t *dst = kResid ? p.rq_pad : p.xq_pad, *dst_sf = kResid ? p.rsf_tiled : p.xsf_tiled;
  const int n_slabs = (per_row + kSlabChunks - 1) / kSlabChunks;
  const int n_items = p.header[kHdrMTiles] * n_slabs;
  int buf = 0;
  for (int item = blockIdx.x; item < n_items; item += gridDim.x, buf ^= 1) {
    const int mt = item / n_slabs, sl = item - mt * n_slabs;
    const int n_rows = p.tile_rows[mt];
    if (threadIdx.x < 128) tok[buf][threadIdx.x] = threadIdx.x < n_rows ? p.row_token[mt * 128 + threadIdx.x] : -1;
    __syncthreads();                                 // (and the atoms of two items ago have been written out)
    const int c0 = sl * kSlabChunks, nc = min(kSlabChunks, per_row - c0), k0 = sl * kSlabAtoms, nk = nc >> 1;
    // ---- loads: codes (thread = chunk threadIdx % 16 of rows threadIdx / 16 + 32 u), scales (two atoms of a row)
    const int c = threadIdx.x & 15, r_of = threadIdx.x >> 4;
    uint4 v[4];
    bool on[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int t = tok[buf][r_of + 32 * u];
      on[u] = t >= 0 && c < nc;
      if (on[u]) v[u] = __ldg(reinterpret_cast<const uint4*>(src + (size_t)t * (H >> 1) + (size_t)(c0 + c) * 16));
    }
    const int sr = threadIdx.x >> 2, pc = threadIdx.x & 3, st = tok[buf][sr];
    uint2 sv = make_uint2(0, 0);                     // (padding rows get zero scales)
    if (st >= 0 && 2 * pc < nk) sv = __ldg(reinterpret_cast<const uint2*>(src_sf + (size_t)st * (H >> 4) + (size_t)(k0 + 2 * pc) * 4));
    uint8_t* atoms = smem_raw + buf * (kSlabAtoms * 512);
    {
      uint32_t* a = reinterpret_cast<uint32_t*>(atoms + 2 * pc * 512 + (sr & 31) * 16 + (sr >> 5) * 4);
      a[0] = sv.x; a[128] = sv.y;
    }
    __syncthreads();
    // ---- stores
    if (threadIdx.x < nk * 32)
      __stcs(reinterpret_cast<uint4*>(dst_sf + ((size_t)mt * kt_count + k0) * 512u) + threadIdx.x, reinterpret_cast<const uint4*>(atoms)[threadIdx.x]);
    uint4 m = make_uint4(0, 0, 0, 0);
    if (kResid && c < nc) m = reinterpret_cast<const uint4*>(nib)[c0 + c];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (on[u]) {
        if (kResid) {
          v[u].x = (v[u].x & m.x) ^ 0x88888888u; v[u].y = (v[u].y & m.y) ^ 0x88888888u;
          v[u].z = (v[u].z & m.z) ^ 0x88888888u; v[u].w = (v[u].w & m.w) ^ 0x88888888u;
        }
        __stcs(reinterpret_cast<uint4*>(dst + (size_t)(mt * 128 + r_of + 32 * u) * (H >> 1) + (size_t)(c0 + c) * 16), v[u]);
      }
  }
}

namespace {

// Resident CTAs per SM of a kernel (same on every sm_100 device).
template <typename K>
cudaError_t resident_per_sm(K kernel, int threads, std::atomic<int>* cache, int* out) {
  int v = cache->load();
  if (v == 0) {
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, kernel, threads, 0);
    if (e != cudaSuccess) return e;
    if (v < 1) return cudaErrorLaunchOutOfResources;
    cache->store(v);
  }
  *out = v;
  return cudaSuccess;
}

// Column groups and row ranges of the quantization role on at most `ctas` CTAs; returns the CTAs used.  Of the widths
// that divide a row the one with the least time: rounds of 256 blocks per CTA (some 2 us each with four CTAs per
// SM), and batches of partial scores that a group's last CTA adds up (some 0.4 us each).
int plan_quant(QuantRowsArgs* q, int ctas) {
  const int blocks = q->H / 16;
  ctas = std::min(ctas, kQuantCtasMax);
  int best = 0, n_used = 1;
  for (int bw = 8; bw <= 32 && blocks % bw == 0; bw *= 2) {
    const int n_col = blocks / bw, lanes = 256 / bw;  // each range at least a row per row lane
    const int n_rg = std::max(1, std::min(ctas / n_col, (q->T + lanes - 1) / lanes));
    const int rounds = ((q->T + n_rg - 1) / n_rg + lanes - 1) / lanes, rows = rounds * lanes, used = (q->T + rows - 1) / rows;
    const int cost = 5 * rounds + (used * bw + 511) / 512;
    if (bw > 8 && cost >= best) continue;
    best = cost;
    q->bw = bw; q->n_col = n_col; q->rows_per_cta = rows;
    n_used = used;
  }
  return n_used * q->n_col;
}

template <int NJ>
quads_status launch_front_nj(QuantRowsArgs q, RouteArgs r, int sm_count, cudaStream_t st) {
  static std::atomic<int> cache{0};
  int per_sm = 0;
  QUADS_CUDA_OK(resident_per_sm(front_kernel<NJ>, 256, &cache, &per_sm));
  if (per_sm < 2) return QUADS_ERR_CUDA;
  int n_groups = std::min(std::min(sm_count, kRouteCtasMax), (r.T + kRouteWarps - 1) / kRouteWarps);
  const int n_quant = plan_quant(&q, (per_sm - 1) * sm_count);
  void* args[] = {&q, &r, &n_groups};
  QUADS_CUDA_OK(cudaLaunchCooperativeKernel(reinterpret_cast<void*>(front_kernel<NJ>), dim3(n_groups + n_quant), dim3(256), args, 0, st));
  note_launch();
  return QUADS_OK;
}

}  // namespace

quads_status launch_front(const QuantRowsArgs& q, const RouteArgs& r, int sm_count, cudaStream_t st) {
  return r.E <= 32 ? launch_front_nj<1>(q, r, sm_count, st)
                   : (r.E <= 64 ? launch_front_nj<2>(q, r, sm_count, st)
                                : (r.E <= 128 ? launch_front_nj<4>(q, r, sm_count, st) : launch_front_nj<8>(q, r, sm_count, st)));
}

quads_status launch_quant_rows(const QuantRowsArgs& args, int sm_count, cudaStream_t st) {
  static std::atomic<int> cache{0};
  QuantRowsArgs q = args;
  int per_sm = 0;
  QUADS_CUDA_OK(resident_per_sm(quant_rows_kernel, 256, &cache, &per_sm));
  const int n = plan_quant(&q, per_sm * sm_count);
  if (!q.gs_in && !q.amax_parts) {                   // its CTAs wait for one another
    void* kargs[] = {&q};
    QUADS_CUDA_OK(cudaLaunchCooperativeKernel(reinterpret_cast<void*>(quant_rows_kernel), dim3(n), dim3(256), kargs, 0, st));
    note_launch();
  } else {
    QUADS_CUDA_OK(launch_kernel(quant_rows_kernel, dim3(n), dim3(256), (size_t)0, st, q));
  }
  return QUADS_OK;
}

quads_status launch_dispatch(const DispatchArgs& p, int m_tiles_max, int sm_count, cudaStream_t st) {
  const int64_t items = (int64_t)m_tiles_max * ((p.H / 32 + kSlabChunks - 1) / kSlabChunks);
  const int grid = (int)std::min<int64_t>(items, kDispatchPerSm * sm_count);
  const int atoms = 2 * kSlabAtoms * 512;
  QUADS_CUDA_OK(launch_kernel(dispatch_kernel<false>, dim3(grid), dim3(kDispatchThreads), (size_t)atoms, st, p));
  if (p.n_sel > 0) QUADS_CUDA_OK(launch_kernel(dispatch_kernel<true>, dim3(grid), dim3(kDispatchThreads), (size_t)(atoms + p.H / 2), st, p));
  return QUADS_OK;
}

}  // namespace quads
