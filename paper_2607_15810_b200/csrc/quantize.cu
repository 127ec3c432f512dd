// Streaming kernels: tensor amax, NVFP4 quantize / fake-quant / decode, channel statistics, selection and masking of a
// residual in place, the weighted sum over a token's experts, verification exports, mismatch norms.
// All HBM- or latency-bound; no tensor cores here.
#include "kernels.cuh"
#include "select.cuh"
#include "tcgen05.cuh"

namespace quads {

// ---------------------------------------------------------------------------
// amax over bf16 tensors.  gridDim.y = tensor; magnitudes compared as 15-bit
// integers (two per 32-bit word); result = bf16 bit pattern << 16 = float bits.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) amax_kernel(const uint16_t* __restrict__ x, int64_t rows, int64_t K,
                                                   int64_t ld, int64_t tensor_stride,
                                                   uint32_t* __restrict__ amax_bits) {
  pdl_sync();
  const uint16_t* base = x + (size_t)blockIdx.y * tensor_stride;
  const int64_t k8 = K >> 3;
  const int64_t chunks = rows * k8;
  uint32_t m = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  if (ld == K) {
    const uint4* p = reinterpret_cast<const uint4*>(base);
    int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (; c + 3 * stride < chunks; c += 4 * stride) {
      uint4 v0 = __ldg(p + c), v1 = __ldg(p + c + stride), v2 = __ldg(p + c + 2 * stride),
            v3 = __ldg(p + c + 3 * stride);
      uint32_t a = __vmaxu2(__vmaxu2(v0.x & 0x7FFF7FFFu, v0.y & 0x7FFF7FFFu),
                            __vmaxu2(v0.z & 0x7FFF7FFFu, v0.w & 0x7FFF7FFFu));
      uint32_t b = __vmaxu2(__vmaxu2(v1.x & 0x7FFF7FFFu, v1.y & 0x7FFF7FFFu),
                            __vmaxu2(v1.z & 0x7FFF7FFFu, v1.w & 0x7FFF7FFFu));
      uint32_t c2 = __vmaxu2(__vmaxu2(v2.x & 0x7FFF7FFFu, v2.y & 0x7FFF7FFFu),
                             __vmaxu2(v2.z & 0x7FFF7FFFu, v2.w & 0x7FFF7FFFu));
      uint32_t d = __vmaxu2(__vmaxu2(v3.x & 0x7FFF7FFFu, v3.y & 0x7FFF7FFFu),
                            __vmaxu2(v3.z & 0x7FFF7FFFu, v3.w & 0x7FFF7FFFu));
      m = __vmaxu2(m, __vmaxu2(__vmaxu2(a, b), __vmaxu2(c2, d)));
    }
    for (; c < chunks; c += stride) {
      uint4 v = __ldg(p + c);
      m = __vmaxu2(m, __vmaxu2(__vmaxu2(v.x & 0x7FFF7FFFu, v.y & 0x7FFF7FFFu),
                               __vmaxu2(v.z & 0x7FFF7FFFu, v.w & 0x7FFF7FFFu)));
    }
  } else {
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < chunks; c += stride) {
      const int64_t r = c / k8, cc = c - r * k8;
      uint4 v = __ldg(reinterpret_cast<const uint4*>(base + r * ld + cc * 8));
      m = __vmaxu2(m, __vmaxu2(__vmaxu2(v.x & 0x7FFF7FFFu, v.y & 0x7FFF7FFFu),
                               __vmaxu2(v.z & 0x7FFF7FFFu, v.w & 0x7FFF7FFFu)));
    }
  }
  uint32_t s = max(m & 0xFFFFu, m >> 16);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s = max(s, __shfl_xor_sync(0xFFFFFFFFu, s, o));
  __shared__ uint32_t wmax[8];
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t t = 0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t = max(t, wmax[i]);
    if (t) atomicMax(amax_bits + blockIdx.y, t << 16);
  }
}

// ---------------------------------------------------------------------------
// Fused amax + NVFP4 quantize / fake-quant in ONE cooperative launch.
// The CTAs form `n_groups` groups (CTA c belongs to group c % n_groups, so every
// group spans all SMs).  A group takes tensors group, group + n_groups, ...:
//   phase 1  its CTAs stream the tensor once (kept in L2: evict_last), reduce
//            |x| max, publish it with atomicMax and meet at a per-tensor counter;
//   phase 2  they read the tensor again (from L2), quantize, and stream the
//            outputs out (evict_first).
// Other groups overlap their phases with this group's barrier wait.  DRAM sees
// each input byte once: 2 B read + the outputs per element.
// `amax_bits` and `counters` (one word each per tensor) must be zero on entry.
// ---------------------------------------------------------------------------
// First pass of the single-tensor quantizer: CTA b leaves the |x| maximum of its share in
// partials[b] (every CTA stores, so the array needs no initialisation and there is no atomic);
// the 32-byte loads ask L2 to keep the lines for the pass that follows.  `zero0` (or NULL) is a word
// that it clears; kClear: in front of a dense projection it clears all the words that the call starts at zero (n0 and n1 of them, by CTA 0).
template <bool kClear>
__global__ void __launch_bounds__(256) amax_partial_kernel(const uint16_t* __restrict__ x, int64_t rows, int64_t K,
                                                           int64_t ld, uint32_t* __restrict__ partials, uint32_t* __restrict__ zero0,
                                                           int n0, uint32_t* __restrict__ zero1, int n1) {
  pdl_sync();
  if (kClear && blockIdx.x == 0) {
    for (int i = threadIdx.x; i < n0; i += 256) zero0[i] = 0u;
    for (int i = threadIdx.x; i < n1; i += 256) zero1[i] = 0u;
  }
  const int64_t k16 = K >> 4, nblk = rows * k16;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  uint32_t m = 0;
  int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (ld == K) {
    for (; b + 3 * stride < nblk; b += 4 * stride) {
      uint4 a0, a1, b0, b1, c0, c1, d0, d1;
      ldg256_keep(x + b * 16, a0, a1);
      ldg256_keep(x + (b + stride) * 16, b0, b1);
      ldg256_keep(x + (b + 2 * stride) * 16, c0, c1);
      ldg256_keep(x + (b + 3 * stride) * 16, d0, d1);
      m = __vmaxu2(m, __vmaxu2(__vmaxu2(__vmaxu2(absmax8(a0), absmax8(a1)), __vmaxu2(absmax8(b0), absmax8(b1))),
                               __vmaxu2(__vmaxu2(absmax8(c0), absmax8(c1)), __vmaxu2(absmax8(d0), absmax8(d1)))));
    }
  }
  for (; b < nblk; b += stride) {
    const int64_t r = b / k16, kb = b - r * k16;
    uint4 a0, a1;
    ldg256_keep(x + r * ld + kb * 16, a0, a1);
    m = __vmaxu2(m, __vmaxu2(absmax8(a0), absmax8(a1)));
  }
  uint32_t sm = max(m & 0xFFFFu, m >> 16);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sm = max(sm, __shfl_xor_sync(0xFFFFFFFFu, sm, o));
  __shared__ uint32_t wmax[8];
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = sm;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t t = 0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t = max(t, wmax[i]);
    partials[blockIdx.x] = t << 16;
    if (!kClear && zero0 && blockIdx.x == 0) *zero0 = 0u;
  }
}

template __global__ void amax_partial_kernel<false>(const uint16_t*, int64_t, int64_t, int64_t, uint32_t*, uint32_t*, int, uint32_t*, int);
template __global__ void amax_partial_kernel<true>(const uint16_t*, int64_t, int64_t, int64_t, uint32_t*, uint32_t*, int, uint32_t*, int);

// Where the quantizer's outputs of one tensor go (any pointer may be null).
struct QuantSink {
  uint8_t* q;        // packed codes: block b owns bytes [8b, 8b+8)
  uint8_t* sf;       // scale bytes, linear ([b]) or tiled
  uint16_t* fq;      // dequantized bf16: block b owns bytes [32b, 32b+32)
  int sf_tiled;
  uint32_t k16;      // blocks per row
  int kt_count;      // scale atoms per row tile
  uint32_t div_m;    // floor(b / k16) = (b * div_m) >> div_s for every block index b < 2^31
  int div_s;
};

// The multiplier / shift pair of the division by k16 above (round-up method on 31-bit dividends).
__device__ __forceinline__ void quant_sink_divisor(QuantSink& o) {
  const int l = o.k16 > 1 ? 32 - __clz((int)(o.k16 - 1)) : 0;   // ceil(log2(k16))
  o.div_s = 31 + l;
  o.div_m = (uint32_t)((((unsigned long long)1 << o.div_s) + o.k16 - 1) / o.k16);
}

// Quantize block b (16 bf16 values in v0 | v1) and stream the outputs out.
template <bool kLut>
__device__ __forceinline__ void emit_block(const QuantSink& o, const QuantCtx& qc, int64_t b, const uint4& v0,
                                           const uint4& v1) {
  float f[16];
  unpack8(v0, f);
  unpack8(v1, f + 8);
  const BlockQ bq = quantize_block<kLut>(f, qc);
  if (o.q) __stcs(reinterpret_cast<uint2*>(o.q + b * 8), make_uint2(bq.lo, bq.hi));
  if (o.sf) {
    if (o.sf_tiled) {
      const uint32_t bu = (uint32_t)b;
      const uint32_t r = (uint32_t)(((unsigned long long)bu * o.div_m) >> o.div_s), kb = bu - r * o.k16;
      const uint32_t tile = (r >> 7) * (uint32_t)o.kt_count + (kb >> 2);
      o.sf[(size_t)tile * 512u + ((r & 31u) * 16u + ((r >> 5) & 3u) * 4u + (kb & 3u))] = (uint8_t)bq.sf8;
    } else {
      o.sf[b] = (uint8_t)bq.sf8;
    }
  }
  if (o.fq) {
    float d[16];
    dequant_block(bq, d);
    uint32_t w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = f32x2_to_bf16x2(d[2 * i], d[2 * i + 1]);
    stg256_stream(o.fq + b * 16, w);
  }
}

// With given scales there are no arrivals to count: `counters` (or NULL) is then a word that the kernel clears.  (As one more parameter it
// cost every call 0.37 us of host time.)
__global__ void __launch_bounds__(256, 4)
fused_quantize_kernel(const uint16_t* __restrict__ x, int64_t rows, int64_t K, int64_t ld, int64_t tensor_stride,
                      int n_tensors, const float* __restrict__ gs_in, uint32_t* __restrict__ amax_bits,
                      uint32_t* __restrict__ counters, uint8_t* __restrict__ q, uint8_t* __restrict__ sf,
                      uint16_t* __restrict__ fq, float* __restrict__ gs_out, int sf_tiled, int64_t sf_tensor_stride,
                      int n_groups, long long wait_cycles, int extra_arrivals, const uint32_t* __restrict__ amax_parts,
                      int n_amax_parts) {
  pdl_sync();
  if (gs_in && counters && blockIdx.x == 0 && threadIdx.x == 0) *counters = 0u;
  const int group = blockIdx.x % n_groups;
  const int rank = blockIdx.x / n_groups;
  const int gsize = ((int)gridDim.x - group + n_groups - 1) / n_groups;
  const int64_t k16 = K >> 4;
  const int64_t nblk = rows * k16;
  const int64_t gthreads = (int64_t)gsize * blockDim.x;
  const int64_t gtid = (int64_t)rank * blockDim.x + threadIdx.x;
  __shared__ uint32_t wmax[8];
  __shared__ float gs_sh;
  __shared__ float inv_lut[128];
  for (int t = group; t < n_tensors; t += n_groups) {
    const uint16_t* base = x + (size_t)t * tensor_stride;
    float gs;
    if (gs_in) {
      gs = gs_in[t];
    } else if (amax_parts) {
      // the tensor's amax was reduced to `n_amax_parts` partial maxima by the preceding kernel
      uint32_t m = 0;
      for (int i = threadIdx.x; i < n_amax_parts; i += blockDim.x) m = max(m, amax_parts[i]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
      if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = m;
      __syncthreads();
      if (threadIdx.x == 0) {
        uint32_t tm = 0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) tm = max(tm, wmax[i]);
        gs_sh = gs_from_amax_bits(tm);
      }
      __syncthreads();
      gs = gs_sh;
      __syncthreads();
    } else {
      // ---- phase 1: tensor amax, one 32-byte block per load
      uint32_t m = 0;
      if (ld == K) {
        int64_t b = gtid;
        for (; b + 3 * gthreads < nblk; b += 4 * gthreads) {
          uint4 a0, a1, b0, b1, c0, c1, d0, d1;
          ldg256_keep(base + b * 16, a0, a1);
          ldg256_keep(base + (b + gthreads) * 16, b0, b1);
          ldg256_keep(base + (b + 2 * gthreads) * 16, c0, c1);
          ldg256_keep(base + (b + 3 * gthreads) * 16, d0, d1);
          m = __vmaxu2(m, __vmaxu2(__vmaxu2(__vmaxu2(absmax8(a0), absmax8(a1)), __vmaxu2(absmax8(b0), absmax8(b1))),
                                   __vmaxu2(__vmaxu2(absmax8(c0), absmax8(c1)), __vmaxu2(absmax8(d0), absmax8(d1)))));
        }
        for (; b < nblk; b += gthreads) {
          uint4 a0, a1;
          ldg256_keep(base + b * 16, a0, a1);
          m = __vmaxu2(m, __vmaxu2(absmax8(a0), absmax8(a1)));
        }
      } else {
        for (int64_t b = gtid; b < nblk; b += gthreads) {
          const int64_t r = b / k16, kb = b - r * k16;
          uint4 a0, a1;
          ldg256_keep(base + r * ld + kb * 16, a0, a1);
          m = __vmaxu2(m, __vmaxu2(absmax8(a0), absmax8(a1)));
        }
      }
      uint32_t sm = max(m & 0xFFFFu, m >> 16);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sm = max(sm, __shfl_xor_sync(0xFFFFFFFFu, sm, o));
      if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = sm;
      __syncthreads();
      if (threadIdx.x == 0) {
        uint32_t tm = 0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) tm = max(tm, wmax[i]);
        if (tm) atomicMax(amax_bits + t, tm << 16);
        __threadfence();
        atomicAdd(counters + t, 1u);
        // bounded wait for the rest of the group (cooperative launch: all CTAs are resident)
        const long long t0 = clock64();
        bool gave_up = false;
        // (extra_arrivals is zero except under the test hook that makes this wait run out)
        while (atomicAdd(counters + t, 0u) < (uint32_t)(gsize + extra_arrivals)) {
          __nanosleep(64);
          if (clock64() - t0 > wait_cycles) { gave_up = true; break; }
        }
        __threadfence();
        // (the count only grows, so if one CTA of the group gives up on it, all do: NaN marks the tensor)
        gs_sh = gave_up ? __int_as_float(0x7FC00000) : gs_from_amax_bits(atomicAdd(amax_bits + t, 0u));
      }
      __syncthreads();
      gs = gs_sh;
      __syncthreads();
    }
    if (gs_out && rank == 0 && threadIdx.x == 0) gs_out[t] = gs;
    __syncthreads();                              // the previous tensor's table is no longer read
    if (threadIdx.x < 128) inv_lut[threadIdx.x] = quant_inv_entry(threadIdx.x, gs);
    __syncthreads();
    QuantCtx qc;
    quant_ctx_scalars(qc, gs);
    qc.inv_lut = inv_lut;
    // ---- phase 2: quantize (16-element blocks), stream the outputs
    uint8_t* qt = q ? q + (size_t)t * rows * (K >> 1) : nullptr;
    uint8_t* sft = sf ? sf + (size_t)t * sf_tensor_stride : nullptr;
    uint16_t* fqt = fq ? fq + (size_t)t * rows * K : nullptr;
    const int kt_count = (int)((K + 63) >> 6);
    const bool contiguous = (ld == K);
    const uint32_t k16u = (uint32_t)k16;
    QuantSink sink{qt, sft, fqt, sf_tiled, k16u, kt_count, 0, 0};
    quant_sink_divisor(sink);
    auto emit = [&](int64_t b, const uint4& v0, const uint4& v1) { emit_block<true>(sink, qc, b, v0, v1); };
    auto src_of = [&](int64_t b) -> const uint16_t* {
      if (contiguous) return base + b * 16;
      const int64_t r = b / k16, kb = b - r * k16;
      return base + r * ld + kb * 16;
    };
    int64_t b = gtid;
    for (; b + 3 * gthreads < nblk; b += 4 * gthreads) {     // four loads in flight per thread
      uint4 a0, a1, c0, c1, d0, d1, e0, e1;
      ldg256_stream(src_of(b), a0, a1);
      ldg256_stream(src_of(b + gthreads), c0, c1);
      ldg256_stream(src_of(b + 2 * gthreads), d0, d1);
      ldg256_stream(src_of(b + 3 * gthreads), e0, e1);
      emit(b, a0, a1);
      emit(b + gthreads, c0, c1);
      emit(b + 2 * gthreads, d0, d1);
      emit(b + 3 * gthreads, e0, e1);
    }
    for (; b < nblk; b += gthreads) {
      uint4 a0, a1;
      ldg256_stream(src_of(b), a0, a1);
      emit(b, a0, a1);
    }
  }
}

// ---------------------------------------------------------------------------
// Fused amax + fake-quant for a batch of tensors (expert weights), one persistent CTA per SM made
// of kRingGroups independent pipelines: 7 consumer warps and one producer warp each.  A tensor is
// cut into one contiguous share per CTA and a share into chunks of 448 blocks (14 KB, two blocks
// per consumer lane; a bulk copy costs the SM about 50 ns whatever its size and every chunk costs
// every warp some bookkeeping, so small chunks cannot keep up), dealt to the groups round-robin.
// A group works through two streams of its chunks, both in tensor order:
//   A  reduce |x| max over the chunk; when the last consumer warp of the CTA gets to the end of a
//      tensor, the CTA's maximum is published and the CTA counted in at the tensor's arrival word;
//   Q  quantize the chunk with the tensor's scale, known once all CTAs have arrived.
// The streams are interleaved chunk by chunk with A `lead` chunks ahead (more than a tensor, so
// that a scale is normally known long before Q needs it), which keeps DRAM reads (A) and writes
// (Q) flowing at the same time instead of in chip-wide bursts.  The producer walks the same list
// kRingDepth chunks ahead and fills the group's ring of shared-memory stages with bulk
// asynchronous copies (A's copy fetches from DRAM and asks L2 to keep the lines, Q's copy finds
// them in L2), so no consumer waits for DRAM.  Between copies the producers also do the talking
// between CTAs (tensor t belongs to producer t mod kRingGroups): they publish the CTA's
// maxima, watch the arrival words and post each scale on a shared-memory board, where the
// consumers find it -- one reader per tensor and CTA, because thousands of readers of one
// address queue up at its L2 slice.
// For small tensors the grid is cut into `split` sets of CTAs and tensor t goes to set t mod split,
// so that a CTA's share stays a few chunks long.
// `pair` holds {amax bits, arrivals} per tensor, zero on entry.  Waits are bounded; a warp that
// gives up raises a flag that stops the CTA, and NaN is written to the scales not yet posted.
// ---------------------------------------------------------------------------
constexpr int kRingBoard = 32;                                  // tensors in flight per CTA, at most half of this
constexpr int kRingGroups = 4;
constexpr int kRingGroupWarps = kRingThreads / 32 / kRingGroups;   // 8: 7 consumers + the producer
constexpr int kRingConsumers = kRingGroupWarps - 1;
constexpr int kRingLaneBlocks = 2;                              // blocks per consumer lane and chunk
constexpr int kRingPassBlocks = kRingConsumers * 32;            // blocks a group takes in one pass over its lanes
constexpr int kRingChunkBlocks = kRingPassBlocks * kRingLaneBlocks;
static_assert(kRingChunkBlocks * 32 == kRingChunkBytes, "chunk size");
struct RingShared {
  unsigned long long board[kRingBoard];   // {tensor index + 1, amax bits} once known to this CTA
  unsigned long long pub[kRingBoard];     // {tensor index + 1, this CTA's |x| max} waiting to be published
  uint32_t cta_max[kRingBoard];
  uint32_t amax_cnt[kRingBoard];
  uint64_t full[kRingGroups][kRingDepth];   // mbarriers: chunk landed
  uint64_t empty[kRingGroups][kRingDepth];  // mbarriers: all consumer warps have left the stage
  int abort_flag;
};
static_assert(sizeof(RingShared) <= kRingHeaderBytes, "header region too small");

// Non-blocking test of an mbarrier phase (try_wait may park the thread for a while, which a
// thread with other duties in its wait loop cannot afford).
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{ .reg .pred p; mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ void bulk_load_hint(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar,
                                               uint64_t policy) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar), "l"(policy) : "memory");
}

// A group's work list, in the order it is both fetched and consumed.
enum { kItemA = 0, kItemQ = 1, kItemEndA = 2 };                 // kItemEndA: no chunk, tensor t's A stream is complete
struct RingItems {
  int n, lead, cnt, group;  // tensors, A's lead over Q in chunks, blocks in the CTA's share, group index
  int ta, ka, tq, kq, ahead;
  int kind, t, blk0, nb;    // current item
  __device__ __forceinline__ void reset(int n_, int lead_, int cnt_, int group_) {
    n = n_; lead = lead_; cnt = cnt_; group = group_; ta = ka = tq = kq = ahead = 0;
  }
  // first block (within the CTA's share) of the group's chunk k of tensor t, or >= cnt
  __device__ __forceinline__ int chunk_first(int tt, int kk) const {
    return (kk * kRingGroups + ((group + tt) & (kRingGroups - 1))) * kRingChunkBlocks;   // the ragged last round rotates
  }
  __device__ __forceinline__ bool next() {
    if (ta < n && chunk_first(ta, ka) >= cnt) {                  // A has run off the end of a tensor
      kind = kItemEndA; t = ta; ++ta; ka = 0;
      return true;
    }
    while (tq < n && chunk_first(tq, kq) >= cnt) { ++tq; kq = 0; }
    const bool q_ok = tq < n && tq < ta;                         // the group has finished A of that tensor
    if (ta < n && (!q_ok || ahead < lead) && ta - tq < kRingBoard / 2) {
      kind = kItemA; t = ta; blk0 = chunk_first(ta, ka); ++ka; ++ahead;
    } else if (q_ok) {
      kind = kItemQ; t = tq; blk0 = chunk_first(tq, kq); ++kq; --ahead;
    } else {
      return false;
    }
    nb = min(kRingChunkBlocks, cnt - blk0);
    return true;
  }
};

__global__ void __launch_bounds__(kRingThreads, 1)
fake_quant_ring_kernel(const uint16_t* __restrict__ x, int64_t nblk, int64_t tensor_stride, int n_tensors_all,
                       uint32_t* __restrict__ pair, int per, int lead, int split, uint8_t* __restrict__ q,
                       uint8_t* __restrict__ sf, uint16_t* __restrict__ fq, float* __restrict__ gs_out, int sf_tiled,
                       int64_t sf_tensor_stride, uint32_t k16, int kt_count) {
  extern __shared__ __align__(128) uint8_t smem[];
  RingShared* sh = reinterpret_cast<RingShared*>(smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Warp 8g + 7 is the producer of group g, so all four producers sit on one warp scheduler
  // (measured 4 % faster than one producer per scheduler).
  const int group = warp / kRingGroupWarps, warp_g = warp % kRingGroupWarps;
  const bool is_producer = warp_g == kRingConsumers;
  uint8_t* stage0 = smem + kRingHeaderBytes + (size_t)group * kRingDepth * kRingChunkBytes;
  const uint32_t stage0_u32 = smem_u32(stage0);
  const uint32_t full0 = smem_u32(&sh->full[group][0]), empty0 = smem_u32(&sh->empty[group][0]);
  // The CTAs form `split` sets; set s takes tensors s, s + split, ... (small tensors: a share of a
  // few chunks per CTA keeps the lanes busy and halves the number of CTAs a scale has to wait for).
  // Below, tensors are numbered within the set; glob() gives the caller's index.
  const int ctas_per_tensor = (int)gridDim.x / split;
  const int set = (int)blockIdx.x / ctas_per_tensor, cta_in_set = (int)blockIdx.x % ctas_per_tensor;
  const int n_tensors = set < n_tensors_all ? (n_tensors_all - set + split - 1) / split : 0;
  auto glob = [&](int t) -> size_t { return (size_t)set + (size_t)split * (size_t)t; };
  const int64_t start = (int64_t)cta_in_set * per;               // first block of this CTA's share
  const int64_t left = nblk - start;
  const int cnt = left <= 0 ? 0 : (left < per ? (int)left : per);  // blocks in the share (same for every tensor)
  volatile int* abort_flag = &sh->abort_flag;

  if (threadIdx.x < kRingBoard) {
    sh->board[threadIdx.x] = 0; sh->pub[threadIdx.x] = 0; sh->cta_max[threadIdx.x] = 0; sh->amax_cnt[threadIdx.x] = 0;
  }
  if (threadIdx.x == 0) {
    for (int g = 0; g < kRingGroups; ++g)
      for (int s = 0; s < kRingDepth; ++s) {
        mbar_init(smem_u32(&sh->full[g][s]), 1);
        mbar_init(smem_u32(&sh->empty[g][s]), kRingConsumers);
      }
    sh->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  auto wait_bar = [&](uint32_t bar, uint32_t parity) -> bool {   // bounded; false after giving up
    if (mbar_try(bar, parity)) return true;
    const uint64_t t0 = globaltimer();
    uint32_t spins = 0;
    while (!mbar_try(bar, parity)) {
      if ((++spins & 255u) == 0) {
        if (*abort_flag) return false;
        if (globaltimer() - t0 > kWaitNs) { *abort_flag = 1; return false; }
      }
    }
    return true;
  };

  if (cnt == 0) {
    // A CTA beyond the end of the tensors (fewer blocks than CTAs): nothing to reduce or quantize,
    // but every tensor still waits for this CTA's arrival.
    if (is_producer && lane == 0)
      for (int t = group; t < n_tensors; t += kRingGroups) atomicAdd(pair + 2 * glob(t) + 1, 1u);
    return;
  }
  if (is_producer) {
    // =========================== producer (one lane)
    if (lane != 0) return;
    uint64_t keep, stream;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(keep));
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(stream));
    int watch = group;                                           // the tensor whose arrival word this producer reads next
    uint32_t seen = 0;
    bool asked = false;
    long long asked_at = 0;
    // One look at the arrival word of tensor `watch`; posts the scale once every CTA has arrived.
    // The load is issued in one call and its value used in a later one, when it has had the time
    // to return, so a call never waits.
    int owed = group;                                            // the tensor this producer publishes next
    auto watch_step = [&]() {
      if (owed < n_tensors) {
        const unsigned long long pv = *reinterpret_cast<volatile unsigned long long*>(&sh->pub[owed & (kRingBoard - 1)]);
        if ((uint32_t)(pv >> 32) == (uint32_t)owed + 1u) {       // the CTA is through with A of that tensor
          *reinterpret_cast<volatile unsigned long long*>(&sh->pub[owed & (kRingBoard - 1)]) = 0;   // slot free again
          uint32_t* pr = pair + 2 * glob(owed);
          if ((uint32_t)pv) atomicMax(pr, (uint32_t)pv << 16);
          __threadfence();
          atomicAdd(pr + 1, 1u);
          owed += kRingGroups;
        }
      }
      if (watch >= n_tensors) return;
      if (asked && clock64() - asked_at < 2000) return;
      if (asked && seen == (uint32_t)ctas_per_tensor) {
        const uint32_t amax_b = ld_relaxed_u32(pair + 2 * glob(watch));   // ordered after the acquire load above
        if (gs_out && cta_in_set == 0) gs_out[glob(watch)] = gs_from_amax_bits(amax_b);
        sh->board[watch & (kRingBoard - 1)] = ((unsigned long long)((uint32_t)watch + 1u) << 32) | amax_b;
        watch += kRingGroups;
        asked = false;
        if (watch >= n_tensors) return;
      }
      // (a CTA publishes its maximum, fences, then counts itself in: once this acquire load shows every arrival, a
      // later load of the amax word returns the final maximum)
      seen = ld_acquire_u32(pair + 2 * glob(watch) + 1);
      asked = true;
      asked_at = clock64();
    };
    RingItems pi;
    pi.reset(n_tensors, lead, cnt, group);
    int issued = 0;
    bool ok = true;
    while (ok && pi.next()) {
      if (pi.kind == kItemEndA) continue;
      const int s = issued % kRingDepth;
      if (issued >= kRingDepth) {                                // the stage's previous chunk must have been left by all
        const uint32_t bar = empty0 + 8 * s, parity = (uint32_t)(issued / kRingDepth - 1) & 1u;
        const uint64_t t0 = globaltimer();
        uint32_t spins = 0;
        while (!mbar_test(bar, parity)) {
          watch_step();                                          // consumers may be waiting for a scale meanwhile
          __nanosleep(40);                                       // (neutral for speed; leaves the issue slots alone)
          if ((++spins & 1023u) == 0 && (*abort_flag || globaltimer() - t0 > kWaitNs)) { *abort_flag = 1; ok = false; break; }
        }
        if (!ok) break;
      }
      const uint32_t bytes = (uint32_t)pi.nb * 32u;
      mbar_expect_tx(full0 + 8 * s, bytes);
      bulk_load_hint(stage0_u32 + s * kRingChunkBytes, x + glob(pi.t) * tensor_stride + (size_t)(start + pi.blk0) * 16,
                     bytes, full0 + 8 * s, pi.kind == kItemA ? keep : stream);
      ++issued;
      watch_step();
    }
    // the remaining scales of this producer's tensors
    const uint64_t t0 = globaltimer();
    while (ok && (watch < n_tensors || owed < n_tensors)) {
      watch_step();
      __nanosleep(64);
      if (*abort_flag || globaltimer() - t0 > kWaitNs) { *abort_flag = 1; ok = false; }
    }
    if (!ok) {
      // gave up: mark the scales not posted, and let the copies in flight land (bounded) before leaving
      if (gs_out)
        for (int t = watch; t < n_tensors; t += kRingGroups) gs_out[glob(t)] = __int_as_float(0x7FC00000);
      for (int d = issued < kRingDepth ? 0 : issued - kRingDepth; d < issued; ++d) {
        const uint32_t bar = full0 + 8 * (d % kRingDepth), parity = (uint32_t)(d / kRingDepth) & 1u;
        const uint64_t t1 = globaltimer();
        while (!mbar_try(bar, parity) && globaltimer() - t1 < 100000000ull) {}
      }
    }
    return;
  }

  // =========================== consumers
  const int lane_c = warp_g * 32 + lane;                         // lane within the group's consumers
  RingItems ci;
  ci.reset(n_tensors, lead, cnt, group);
  QuantSink sink0{q, sf, fq, sf_tiled, k16, kt_count, 0, 0};
  quant_sink_divisor(sink0);
  QuantSink sink = sink0;
  QuantCtx qc;
  qc.inv_lut = nullptr;
  int consumed = 0;
  int cur_q = -1;                                                // tensor whose scale is in qc
  uint32_t m = 0;                                                // running |x| max (two 15-bit magnitudes) of the A tensor
  while (ci.next()) {
    if (ci.kind == kItemEndA) {
      // ---- this warp is through with A of tensor t; the last consumer warp of the CTA publishes
      uint32_t wm = max(m & 0xFFFFu, m >> 16);
      m = 0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) wm = max(wm, __shfl_xor_sync(0xFFFFFFFFu, wm, o));
      if (lane == 0) {
        const int s = ci.t & (kRingBoard - 1);
        if (wm) atomicMax(&sh->cta_max[s], wm);
        __threadfence_block();
        if (atomicAdd(&sh->amax_cnt[s], 1u) == (uint32_t)(kRingGroups * kRingConsumers - 1)) {
          __threadfence_block();
          // hand the CTA's maximum to the producer that owns the tensor: a fence between the two
          // global atomics would make THIS warp wait for all its output stores in flight
          const uint32_t tm = atomicExch(&sh->cta_max[s], 0u);
          atomicExch(&sh->amax_cnt[s], 0u);
          volatile unsigned long long* slot = reinterpret_cast<volatile unsigned long long*>(&sh->pub[s]);
          if (*slot != 0) {                                      // the producer has not taken tensor t - 32 yet
            const uint64_t t0 = globaltimer();
            uint32_t spins = 0;
            while (*slot != 0)
              if ((++spins & 63u) == 0 && (*abort_flag || globaltimer() - t0 > kWaitNs)) { *abort_flag = 1; break; }
          }
          *slot = ((unsigned long long)((uint32_t)ci.t + 1u) << 32) | tm;
        }
      }
      continue;
    }
    if (ci.kind == kItemQ && ci.t != cur_q) {
      // ---- a new tensor's scale, from the board
      const int t = ci.t;
      uint32_t amax_b = 0xFFFFFFFFu;                             // (never an amax pattern)
      if (lane == 0) {
        const uint32_t tag = (uint32_t)t + 1u;
        volatile unsigned long long* board = &sh->board[t & (kRingBoard - 1)];
        unsigned long long b = *board;
        if ((uint32_t)(b >> 32) != tag) {
          const uint64_t t0 = globaltimer();
          uint32_t spins = 0;
          while ((uint32_t)((b = *board) >> 32) != tag) {
            if ((++spins & 63u) == 0 && (*abort_flag || globaltimer() - t0 > kWaitNs)) { *abort_flag = 1; break; }
          }
        }
        if ((uint32_t)(b >> 32) == tag) amax_b = (uint32_t)b;
      }
      amax_b = __shfl_sync(0xFFFFFFFFu, amax_b, 0);
      if (amax_b == 0xFFFFFFFFu) break;
      cur_q = t;
      quant_ctx_scalars(qc, gs_from_amax_bits(amax_b));
      sink = sink0;
      if (sink.q) sink.q += glob(t) * nblk * 8;
      if (sink.sf) sink.sf += glob(t) * sf_tensor_stride;
      if (sink.fq) sink.fq += glob(t) * nblk * 16;
    }
    const int s = consumed % kRingDepth;
    if (!wait_bar(full0 + 8 * s, (uint32_t)(consumed / kRingDepth) & 1u)) break;
    const uint8_t* st = stage0 + s * kRingChunkBytes;
    if (ci.kind == kItemA) {
#pragma unroll
      for (int h = 0; h < kRingLaneBlocks; ++h) {
        const int bl = lane_c + h * kRingPassBlocks;
        if (bl < ci.nb) {
          const uint4* v = reinterpret_cast<const uint4*>(st + bl * 32);
          m = __vmaxu2(m, __vmaxu2(absmax8(v[0]), absmax8(v[1])));
        }
      }
    } else {
#pragma unroll
      for (int h = 0; h < kRingLaneBlocks; ++h) {
        const int bl = lane_c + h * kRingPassBlocks;
        if (bl < ci.nb) {
          const uint4* v = reinterpret_cast<const uint4*>(st + bl * 32);
          const uint4 v0 = v[0], v1 = v[1];
          emit_block<false>(sink, qc, start + ci.blk0 + bl, v0, v1);
        }
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(empty0 + 8 * s);                  // this warp has left the stage
    ++consumed;
  }
}

// ---------------------------------------------------------------------------
// NVFP4 -> bf16 decode of packed tensors (what a rollout engine's weight loader, or a W4A16
// path, reads): value(code) * (E4M3 block scale * per-tensor scale), one float32 multiply,
// rounded to bf16 -- the decode that the weight fake-quant's bf16 output is defined by.
// blockIdx.y = tensor; a thread decodes 16-element blocks, 8 B of codes + 1 B of scale in, one 32-byte store out,
// four blocks in flight.  In the one-sided dense projection the result is read back out of L2 by the product
// behind it (no streaming hint on the stores).  4096 x 4096 in front of that product: 11.5 us with one block at
// a time and a 64-bit division for its tensor, 7.5 now (43 MB: 6.6 us).  `zero` (or NULL) is a word the kernel clears.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
dequantize_kernel(const uint8_t* __restrict__ q, const uint8_t* __restrict__ sf, const float* __restrict__ gs,
                  int64_t nblk, uint32_t k16, int kt_count, int sf_tiled, int64_t sf_tensor_stride,
                  uint16_t* __restrict__ out, int32_t* __restrict__ zero) {
  pdl_sync();
  if (zero && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *zero = 0;
  QuantSink geo{nullptr, nullptr, nullptr, sf_tiled, k16, kt_count, 0, 0};
  quant_sink_divisor(geo);
  const size_t t = blockIdx.y;
  const uint2* qt = reinterpret_cast<const uint2*>(q) + t * (size_t)nblk;
  const uint8_t* sft = sf + t * (size_t)sf_tensor_stride;
  uint16_t* ot = out + t * (size_t)nblk * 16;
  const float g = gs[t];
  const uint32_t n = (uint32_t)nblk, step = gridDim.x * 256u;         // n < 2^31
  for (uint32_t b0 = blockIdx.x * 256u + threadIdx.x; b0 < n; b0 += 4 * step) {
    uint2 codes[4];
    uint32_t scale[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t b = b0 + u * step;
      if (b < n) {
        size_t so = b;
        if (sf_tiled) {
          const uint32_t r = (uint32_t)(((unsigned long long)b * geo.div_m) >> geo.div_s), kb = b - r * k16;
          so = (size_t)((r >> 7) * (uint32_t)kt_count + (kb >> 2)) * 512u + ((r & 31u) * 16u + ((r >> 5) & 3u) * 4u + (kb & 3u));
        }
        codes[u] = __ldcs(qt + b);
        scale[u] = __ldg(sft + so);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t b = b0 + u * step;
      if (b >= n) break;
      BlockQ bq;
      bq.lo = codes[u].x;
      bq.hi = codes[u].y;
      bq.sf8 = scale[u];
      bq.d = __fmul_rn(e4m3_to_f32(bq.sf8), g);
      float d[16];
      dequant_block(bq, d);
      uint32_t w[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) w[i] = f32x2_to_bf16x2(d[2 * i], d[2 * i + 1]);
      stg256(ot + (size_t)b * 16, w);
    }
  }
}

// Statistics only (quads_rac_channel_scores): the squared residual sums of a CTA's rows, one partial row per CTA.
__global__ void __launch_bounds__(256)
channel_stats_kernel(const uint16_t* __restrict__ x, int T, int H, const float* __restrict__ gs_in,
                     const uint32_t* __restrict__ amax_bits, int rows_per_cta, float* __restrict__ partials) {
  pdl_sync();
  const int k16 = H >> 4;
  const int r0 = blockIdx.x * rows_per_cta;
  const int r1 = min(T, r0 + rows_per_cta);
  const float gs = gs_in ? gs_in[0] : gs_from_amax_bits(amax_bits[0]);
  __shared__ float inv_lut[128];
  for (int i = threadIdx.x; i < 128; i += blockDim.x) inv_lut[i] = quant_inv_entry(i, gs);
  __syncthreads();
  QuantCtx qc;
  quant_ctx_scalars(qc, gs);
  qc.inv_lut = inv_lut;
  for (int kb = threadIdx.x; kb < k16; kb += blockDim.x) {
    float acc[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i] = 0.f;
    uint4 n0 = make_uint4(0, 0, 0, 0), n1 = n0;
    if (r0 < r1) ldg256(x + (size_t)r0 * H + kb * 16, n0, n1);
    for (int r = r0; r < r1; ++r) {
      const uint4 v0 = n0, v1 = n1;
      if (r + 1 < r1) ldg256(x + (size_t)(r + 1) * H + kb * 16, n0, n1);
      float f[16], o[16];
      unpack8(v0, f);
      unpack8(v1, f + 8);
      residual_block(quantize_block(f, qc), f, o);
      add_squares(o, acc);
    }
    float4* dst = reinterpret_cast<float4*>(partials + (size_t)blockIdx.x * H + kb * 16);
    dst[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
    dst[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
    dst[2] = make_float4(acc[8], acc[9], acc[10], acc[11]);
    dst[3] = make_float4(acc[12], acc[13], acc[14], acc[15]);
  }
}

// Channel scores (Eq. channel-score).  The partial rows are split into
// kScoreSlices contiguous slices; CTA (column group, slice) adds its slice's
// rows in float64.  The CTA of a column group that finishes last adds the
// slice sums in slice order (a fixed order, whichever CTA does it) and stores
// the group's 32 scores as order-preserving 64-bit keys (scores are >= 0).
// grid = (ceil(C/32), kScoreSlices), 256 threads = 32 columns x 8 row lanes.
// `counters` (one per column group) must be zero on entry.
__global__ void __launch_bounds__(256)
score_reduce_kernel(const float* __restrict__ partials, int n_part, int C, double* __restrict__ slice_sums,
                    unsigned int* __restrict__ counters, unsigned long long* __restrict__ score_keys) {
  pdl_sync();
  const int per = (n_part + kScoreSlices - 1) / kScoreSlices;
  const int p0 = blockIdx.y * per, p1 = min(n_part, p0 + per);
  const int col = blockIdx.x * 32 + (threadIdx.x & 31);
  const int rl = threadIdx.x >> 5;
  double s = 0.0;
  if (col < C)
    for (int p = p0 + rl; p < p1; p += 8) s += (double)partials[(size_t)p * C + col];
  __shared__ double sm[8][32];
  __shared__ unsigned int last;
  sm[rl][threadIdx.x & 31] = s;
  __syncthreads();
  if (rl == 0 && col < C) {
    double t = 0.0;
#pragma unroll
    for (int i = 0; i < 8; ++i) t += sm[i][threadIdx.x & 31];
    slice_sums[(size_t)blockIdx.y * C + col] = t;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(counters + blockIdx.x, 1u);
  __syncthreads();
  if (last == kScoreSlices - 1 && rl == 0 && col < C) {
    __threadfence();
    double t = 0.0;
#pragma unroll
    for (int i = 0; i < kScoreSlices; ++i) t += __ldcg(slice_sums + (size_t)i * C + col);
    score_keys[col] = (unsigned long long)__double_as_longlong(t);
  }
}

// Ascending list of the selected channels (verification export only).  One CTA.
__global__ void __launch_bounds__(1024)
sel_list_kernel(const uint8_t* __restrict__ mask, int C, int32_t* __restrict__ sel_export) {
  pdl_sync();
  __shared__ int chunk_tot[1024];
  const int tid = threadIdx.x, nt = blockDim.x;
  const int per = (C + nt - 1) / nt;
  const int c0 = tid * per, c1 = min(C, c0 + per);
  int cnt = 0;
  for (int i = c0; i < c1; ++i) cnt += mask[i];
  chunk_tot[tid] = cnt;
  __syncthreads();
  if (tid == 0) {
    int run = 0;
    for (int i = 0; i < nt; ++i) { const int c = chunk_tot[i]; chunk_tot[i] = run; run += c; }
  }
  __syncthreads();
  int pos = chunk_tot[tid];
  for (int i = c0; i < c1; ++i)
    if (mask[i]) sel_export[pos++] = i;
}

// Clears n 16-byte words.  A memset operation in its place starts 1 us later behind the preceding kernel and holds the
// following one back for another 2.4 us (1500 tokens: 135.2 us per call, 133.2 with this kernel; dense 8192 x 4096 x 4096:
// 166.5, 164.3).
__global__ void __launch_bounds__(256)
clear_kernel(uint4* __restrict__ p, int n) {
  pdl_sync();
  for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) p[i] = make_uint4(0, 0, 0, 0);
}

// Verification export of the masked residual's codes in token order (Eq. residual-recon: codes of unselected
// channels cleared), from codes stored with `flip` XORed into every word.  One thread per (token, 32 channels).
__global__ void __launch_bounds__(256)
export_residual_kernel(int T, int H, const uint8_t* __restrict__ mask, uint32_t flip, const uint8_t* __restrict__ rq,
                       uint8_t* __restrict__ rq_exp) {
  pdl_sync();
  const int per_row = H >> 5;
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= (int64_t)T * per_row) return;
  const int t = (int)(g / per_row), c = (int)(g - (int64_t)t * per_row);
  const size_t co = (size_t)t * (H >> 1) + c * 16;
  uint4 v = *reinterpret_cast<const uint4*>(rq + co);
  const uint8_t* m = mask + c * 32;
  v.x = (v.x ^ flip) & nibble_mask8(m); v.y = (v.y ^ flip) & nibble_mask8(m + 8);
  v.z = (v.z ^ flip) & nibble_mask8(m + 16); v.w = (v.w ^ flip) & nibble_mask8(m + 24);
  *reinterpret_cast<uint4*>(rq_exp + co) = v;
}

// Site-2 selection and masking in one launch: every CTA finds the selection's threshold for itself (C
// scores, 8 C bytes out of L2), turns it into nibble masks in shared memory and clears, in place,
// the codes of unselected channels in its share of the valid rows of the padded [rows, C/2] code matrix.
// A thread keeps its 16-byte column chunk and walks down the rows, eight of them in flight; the first
// eight are fetched before the search, which hides their latency.  CTA 0 also exports the mask when asked
// to.  Rows beyond a tile's valid ones are left alone: with few rows per expert they are most of the matrix.
// Latency-bound: one CTA of 1024 threads per SM (8192 tokens, 25 MB of codes: 18 us in a loop; with 512 threads 26, a
// ranking kernel and a mask kernel behind it took 19; eight CTAs of 256 threads per SM, each repeating the
// search, cost a decode layer 7 us more than those two did).
// The scores are integer totals (site 2) or float64 bit patterns (site 13).  With n_rows_fixed > 0 the matrix has that many
// rows, all valid (site 13 in token order, dense projections); `flip` is XORed
// into every word of the result (the residual operand is stored negated).
// dynamic shared memory: C keys of 8 bytes, C words of scratch, C / 8 mask words.
template <bool kDoubleKeys>
__global__ void __launch_bounds__(kSelectThreads)
select_mask_kernel(uint8_t* __restrict__ codes, int n_rows_fixed, uint32_t flip, const int32_t* __restrict__ header,
                   const int32_t* __restrict__ tile_rows,
                   const unsigned long long* __restrict__ score_keys, int C, int n_sel, uint8_t* __restrict__ mask_out) {
  pdl_sync();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned long long* sc = reinterpret_cast<unsigned long long*>(smem_raw);
  uint32_t* images = reinterpret_cast<uint32_t*>(smem_raw + (size_t)C * 8);
  uint32_t* nib = images + C;
  __shared__ SelectScratch scratch;
  for (int i = threadIdx.x; i < C; i += kSelectThreads) sc[i] = __ldcg(score_keys + i);
  const int per_row = C >> 5;
  const int n_rows = n_rows_fixed > 0 ? n_rows_fixed : header[kHdrMTiles] * 128;
  const int cols = min(per_row, kSelectThreads), rows_per_pass = kSelectThreads / cols;
  const int rl = threadIdx.x / cols;
  const int first = rl < rows_per_pass ? blockIdx.x * rows_per_pass + rl : n_rows;
  const int step = gridDim.x * rows_per_pass;
  uint4 v[8];
  uint32_t on = 0;                                             // bit u: row u of the batch is a valid one
  auto fetch = [&](int c, int r0) {
    on = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int r = r0 + u * step;
      if (r < n_rows && (n_rows_fixed > 0 || (r & 127) < __ldg(tile_rows + (r >> 7)))) on |= 1u << u;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (on >> u & 1) v[u] = __ldcg(reinterpret_cast<const uint4*>(codes + (size_t)(r0 + u * step) * (C >> 1)) + c);
  };
  const int c_first = threadIdx.x % cols;
  fetch(c_first, first);
  __syncthreads();
  const Selection sel = select_largest<kDoubleKeys>(sc, images, C, n_sel, &scratch);
  for (int w = threadIdx.x; w < (C >> 3); w += kSelectThreads) {
    uint32_t m = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) m |= sel.has(sc[8 * w + i], 8 * w + i) ? 0xFu << (4 * i) : 0u;
    nib[w] = m;
  }
  if (mask_out && blockIdx.x == 0)
    for (int i = threadIdx.x; i < C; i += kSelectThreads) mask_out[i] = sel.has(sc[i], i) ? 1 : 0;
  __syncthreads();
  for (int c = c_first; c < per_row; c += kSelectThreads) {
    const uint4 m = reinterpret_cast<const uint4*>(nib)[c];
    if (c != c_first) fetch(c, first);
    for (int r0 = first; r0 < n_rows; r0 += 8 * step) {
      if (r0 != first) fetch(c, r0);
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (on >> u & 1) {
          v[u].x = (v[u].x & m.x) ^ flip; v[u].y = (v[u].y & m.y) ^ flip;
          v[u].z = (v[u].z & m.z) ^ flip; v[u].w = (v[u].w & m.w) ^ flip;
          reinterpret_cast<uint4*>(codes + (size_t)(r0 + u * step) * (C >> 1))[c] = v[u];
        }
    }
  }
}

template __global__ void select_mask_kernel<false>(uint8_t*, int, uint32_t, const int32_t*, const int32_t*, const unsigned long long*, int,
                                                   int, uint8_t*);
template __global__ void select_mask_kernel<true>(uint8_t*, int, uint32_t, const int32_t*, const int32_t*, const unsigned long long*, int,
                                                  int, uint8_t*);

// Weighted top-k combine: out[t, :] = sum over the token's slots, in slot order,
// of weight * y[row of (t, slot), :], accumulated in float32, rounded to bf16.
// One thread per (token, 8 columns); the block shape gives both without a division.  Row positions and weights, the
// routing's, are fetched while the projection in front still runs.  Bound by DRAM where the rows exceed L2
// (8192 tokens x 8 x 2048: 302 MB, 61 us) and by latency for few tokens: with 64-bit index divisions, and with the
// positions behind the wait, a layer of 256 tokens took 92.0 us (90.7 so), of one token 29.4 (28.9).
__global__ void __launch_bounds__(256)
combine_kernel(const uint16_t* __restrict__ y_pad, const int32_t* __restrict__ pos_pad,
               const float* __restrict__ wts, int T, int H, int topk, uint16_t* __restrict__ out,
               float* __restrict__ out_f32) {
  const int t = blockIdx.x * blockDim.y + threadIdx.y, c = blockIdx.y * blockDim.x + threadIdx.x;
  const bool mine = t < T && c < (H >> 3);
  float acc[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) acc[j] = 0.f;
  // eight slots at a time: all row positions first, then all row loads, so that the loads of a
  // token's rows are in flight together; the sum itself runs in slot order
  for (int s0 = 0; s0 < topk; s0 += 8) {
    int p[8];
    float w[8];
    uint4 v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const bool on = mine && s0 + j < topk;
      p[j] = on ? __ldg(pos_pad + t * topk + s0 + j) : -1;
      w[j] = on ? __ldg(wts + t * topk + s0 + j) : 0.f;
    }
    if (s0 == 0) {                                     // the routing's results are older than the kernel in front
      pdl_sync();
      if (!mine) return;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j)
      v[j] = p[j] >= 0 ? __ldcs(reinterpret_cast<const uint4*>(y_pad + (size_t)p[j] * H) + c) : make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (p[j] < 0) continue;
      float f[8];
      unpack8(v[j], f);
#pragma unroll
      for (int k = 0; k < 8; ++k) acc[k] = __fmaf_rn(w[j], f[k], acc[k]);
    }
  }
  if (out_f32) {                                       // partial sums of an expert-sharded call, unrounded
    float4* d = reinterpret_cast<float4*>(out_f32 + (size_t)t * H) + 2 * c;
    d[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
    d[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
  }
  if (out)
    reinterpret_cast<uint4*>(out + (size_t)t * H)[c] =
        make_uint4(f32x2_to_bf16x2(acc[0], acc[1]), f32x2_to_bf16x2(acc[2], acc[3]),
                   f32x2_to_bf16x2(acc[4], acc[5]), f32x2_to_bf16x2(acc[6], acc[7]));
}

// Export of padded dispatch-order buffers into linear dispatch order.
// One thread per (dispatched row, 16-channel block).
__global__ void __launch_bounds__(256)
export_site2_kernel(int A, const int32_t* __restrict__ n_rows_ptr, int I, const int32_t* __restrict__ perm,
                    const int32_t* __restrict__ pos_pad,
                    const uint8_t* __restrict__ hq_pad, const uint8_t* __restrict__ hsf_tiled,
                    const uint8_t* __restrict__ r2q_pad, const uint8_t* __restrict__ r2sf_tiled,
                    const uint8_t* __restrict__ mask2, uint8_t* __restrict__ hq, uint8_t* __restrict__ hsf, uint8_t* __restrict__ r2q,
                    uint8_t* __restrict__ r2sf) {
  pdl_sync();
  const int k16 = I >> 4;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)A * k16) return;
  const int row = (int)(i / k16), kb = (int)(i - (int64_t)row * k16);
  if (row >= *n_rows_ptr) return;          // an expert-sharded call dispatches only its own experts' rows
  const int p = pos_pad[perm[row]];
  const size_t so = sf_tiled_offset(p, kb, I >> 6);
  if (hq) *reinterpret_cast<uint2*>(hq + (size_t)row * (I >> 1) + kb * 8) =
      *reinterpret_cast<const uint2*>(hq_pad + (size_t)p * (I >> 1) + kb * 8);
  if (hsf) hsf[(size_t)row * k16 + kb] = hsf_tiled[so];
  if (r2q) {
    uint2 v = *reinterpret_cast<const uint2*>(r2q_pad + (size_t)p * (I >> 1) + kb * 8);
    // stored negated: flip the signs back, then clear the unselected channels again
    v.x = (v.x ^ 0x88888888u) & nibble_mask8(mask2 + kb * 16);
    v.y = (v.y ^ 0x88888888u) & nibble_mask8(mask2 + kb * 16 + 8);
    *reinterpret_cast<uint2*>(r2q + (size_t)row * (I >> 1) + kb * 8) = v;
  }
  if (r2sf) r2sf[(size_t)row * k16 + kb] = r2sf_tiled[so];
}


// ---------------------------------------------------------------------------
// Diagnostics of Eq. linear-mismatch: squared Frobenius norms of a - b, a and b for two bf16
// tensors of equal size (two versions of a layer output), accumulated in float64 in a fixed order
// (per-thread strided sums, warp tree, block tree, then the block partials in block order by
// whichever CTA finishes last), so the three numbers are reproducible bit for bit.
// `counter` must be zero on entry; out = {sum (a-b)^2, sum a^2, sum b^2}.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
mismatch_norms_kernel(const uint16_t* __restrict__ a, const uint16_t* __restrict__ b, int64_t n, double* __restrict__ partials,
                      unsigned int* __restrict__ counter, double* __restrict__ out) {
  pdl_sync();
  double s0 = 0.0, s1 = 0.0, s2 = 0.0;
  const int64_t n8 = n >> 3;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n8; i += stride) {
    const uint4 va = __ldcs(reinterpret_cast<const uint4*>(a) + i), vb = __ldcs(reinterpret_cast<const uint4*>(b) + i);
    float fa[8], fb[8];
    unpack8(va, fa);
    unpack8(vb, fb);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const double x = (double)fa[k], y = (double)fb[k], d = x - y;
      s0 = fma(d, d, s0); s1 = fma(x, x, s1); s2 = fma(y, y, s2);
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0)             // a tail that is not a multiple of 8 elements
    for (int64_t i = n8 << 3; i < n; ++i) {
      const double x = (double)bf16_bits_to_float(a[i]), y = (double)bf16_bits_to_float(b[i]), d = x - y;
      s0 = fma(d, d, s0); s1 = fma(x, x, s1); s2 = fma(y, y, s2);
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s0 += __shfl_xor_sync(0xFFFFFFFFu, s0, o);
    s1 += __shfl_xor_sync(0xFFFFFFFFu, s1, o);
    s2 += __shfl_xor_sync(0xFFFFFFFFu, s2, o);
  }
  __shared__ double red[3][8];
  __shared__ unsigned int last;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) { red[0][warp] = s0; red[1][warp] = s1; red[2][warp] = s2; }
  __syncthreads();
  if (threadIdx.x < 3) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[threadIdx.x][w];
    partials[(size_t)blockIdx.x * 3 + threadIdx.x] = t;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(counter, 1u);
  __syncthreads();
  if (last == gridDim.x - 1 && threadIdx.x < 3) {
    __threadfence();
    double t = 0.0;
    for (unsigned int g = 0; g < gridDim.x; ++g) t += __ldcg(partials + (size_t)g * 3 + threadIdx.x);
    out[threadIdx.x] = t;
  }
}

}  // namespace quads
