// Dense bf16 x bf16 GEMM on the 5th-generation tensor cores (tcgen05, kind::f16) for the
// one-sided rollout modes of the paper's ablations: out[T, N] = A[T, K] B[N, K]^T with float32
// accumulation in tensor memory, bf16 output.
//   W4A16: A = the activations as they are (bf16), B = the NVFP4 weights decoded to bf16;
//   W16A4: A = the decoded NVFP4 activations (Q_A then decode, bf16), B = the bf16 weights.
// The decoded operand is produced by the library's own decode / fake-quant kernels into the
// caller's workspace; this kernel is the contraction.
//
// Two kernels.  gemm_bf16_pair_kernel: persistent pairs of CTAs compute 256 x 256 tiles with cta_group::2 MMAs, each CTA
// holding its own 128 rows of A and half of B's -- 32 KB per CTA and stage.  gemm_bf16_wave_kernel: problems
// whose tiles of 128 x 128 fit the chip at once, K split over clusters.  (Single persistent CTAs with tiles of 128 x 64 to 256
// stood between the two; 48 KB per stage at 256 columns: 1024 x 4096 -> 4096 28.0 us, pairs 26.4, although only 64 of
// 74 have a tile; 64 x 4096 -> 4096 15.9, split 9.9; 512 x 4096 -> 4096 24.6, tiles of 128 x 128 17.0.)
//
// Pairs: 10 warps; warp 0 issues TMA tile loads (128-byte swizzle, 64 bf16 per
// row and stage) into a ring; warp 1 issues four K = 16 MMAs per stage and releases stages with
// tcgen05.commit; warps 2..9 drain one of TWO float32 accumulators (all 512 columns of tensor memory)
// while the MMAs of the next tile fill the other.  2048 x 4096 -> 4096: 45.8 us (1.50 PFLOP/s, 0.89 of the measured burst
// rate; 128 tiles on 74 pairs leave the second wave a quarter empty).
// Every wait is bounded; a wait that gives up records QUADS_ERR_TIMEOUT and all roles leave.  The status word is cleared by the
// first kernel of a call: the decode or the quantizer in front, or with nothing in front (`first`) the product itself, all
// of whose waits then begin behind the preceding kernel's end.  A kernel that did nothing else cost a call 1 to 1.4 us (replayed
// from a graph, W16A16 64 x 512 -> 512 5.4 us, 4.0 so; 64 x 4096 -> 4096 9.7, 8.9; 2048 x 2048 -> 2048 14.9, 13.9).
#include "kernels.cuh"
#include "split_k.cuh"
#include "tcgen05.cuh"

namespace quads {
namespace {

constexpr int kFStageK = 64;                         // bf16 elements per row per stage (128 bytes)
constexpr int kFBox = kBf16BoxRows;                  // rows of a TMA box
constexpr int kFTileA = 128 * 128;                   // 16 KB
constexpr int kFThreads = 320;
constexpr int kFEpiWarps = 8;
constexpr int kFStages = 6;
constexpr int kFTileN = 256;                         // columns of a pair's tile
constexpr int kFStageBytes = 2 * kFTileA;            // 128 rows of A, and of B the CTA's half of the tile
constexpr int kFBarOffset = kFStages * kFStageBytes;
constexpr int kFSmemBytes = kFBarOffset + 256 + 1024;

struct __align__(8) FBarriers {
  uint64_t full[kFStages];
  uint64_t empty[kFStages];
  uint64_t tmem_full[2];
  uint64_t tmem_empty[2];
  uint32_t tmem_base;
  int abort_flag;
};

template <int CG>
__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate) {
  if (CG == 1) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
  }
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kFThreads, 1)
gemm_bf16_pair_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b, int T, int N, int K,
                      int first, uint16_t* __restrict__ out, int32_t* __restrict__ status) {
  extern __shared__ uint8_t smem_dyn[];
  const uint32_t smem_base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_dyn + (smem_base - smem_u32(smem_dyn));
  FBarriers* bars = reinterpret_cast<FBarriers*>(smem_gen + kFBarOffset);
  const uint32_t bar_full = smem_u32(&bars->full[0]), bar_empty = smem_u32(&bars->empty[0]);
  const uint32_t bar_tfull = smem_u32(&bars->tmem_full[0]), bar_tempty = smem_u32(&bars->tmem_empty[0]);
  volatile int* abort_flag = &bars->abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();           // position inside the CTA pair
  const bool leader = rank == 0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kFStages; ++s) { mbar_init(bar_full + 8 * s, leader ? 2 : 1); mbar_init(bar_empty + 8 * s, 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(bar_tfull + 8 * b, 1); mbar_init(bar_tempty + 8 * b, kFEpiWarps * 2); }
    bars->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    prefetch_tmap(&tm_a);
    prefetch_tmap(&tm_b);
  }
  if (warp == 1) tmem_alloc<2>(smem_u32(&bars->tmem_base), 512);
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                   // both CTAs' barriers exist before any remote arrive
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;
  pdl_sync();                                        // the decoded operand comes from the preceding kernel
  if (first && blockIdx.x == 0 && threadIdx.x == 0) *status = 0;

  const int m_tiles = (T + 255) / 256, n_tiles = (N + kFTileN - 1) / kFTileN;
  const int total = m_tiles * n_tiles;
  const int k_stages = K / kFStageK;
  const int first_tile = blockIdx.x / 2, tile_step = gridDim.x / 2;

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    const bool issuer = elect_one();
    uint32_t stage = 0, phase = 0;
    bool ok = true;
    const uint32_t leader_full = map_to_cta(bar_full, 0);
    for (int tile = first_tile; tile < total && ok; tile += tile_step) {
      const int mt = tile / n_tiles, nt = tile - mt * n_tiles;
      const int arow = (mt * 2 + (int)rank) * 128;
      const int brow = nt * kFTileN + (int)rank * (kFTileN / 2);
      const int boxes_b = max(0, min(kFTileN / 2, N - brow)) / kFBox;   // boxes of weight rows that exist (N % 128 == 0)
      for (int ks = 0; ks < k_stages; ++ks) {
        ok = mbar_wait(bar_empty + 8 * stage, phase ^ 1u, abort_flag, status);
        if (!ok) break;
        if (issuer) {
          const uint32_t sb = smem_base + stage * kFStageBytes;
          const uint32_t bytes = (uint32_t)(kFTileA + boxes_b * kFBox * 128);
          const uint32_t full = leader_full + 8 * stage;          // both CTAs' loads credit the leader's barrier
          mbar_expect_tx_cluster(full, bytes);
          for (int b = 0; b < 128 / kFBox; ++b) tma_load_2d_pair(sb + b * kFBox * 128, &tm_a, ks * kFStageK, arow + b * kFBox, full);
          for (int b = 0; b < boxes_b; ++b) tma_load_2d_pair(sb + kFTileA + b * kFBox * 128, &tm_b, ks * kFStageK, brow + b * kFBox, full);
        }
        __syncwarp();
        if (++stage == kFStages) { stage = 0; phase ^= 1u; }
      }
    }
    for (int s = 0; s < kFStages && ok; ++s) {            // drain: every armed stage lands and is consumed
      ok = mbar_wait(bar_empty + 8 * stage, phase ^ 1u, abort_flag, status);
      if (++stage == kFStages) { stage = 0; phase ^= 1u; }
    }
  } else if (warp == 1 && !leader) {
    // the leader CTA issues the MMAs of the pair
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    const bool issuer = elect_one();
    uint32_t stage = 0, phase = 0;
    int it = 0;
    bool ok = true;
    // bf16 x bf16 -> float32, both operands K-major, M = 128 per CTA, N = 256
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kFTileN >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
    constexpr uint32_t kSwHi = (uint32_t)((8 * 128) >> 4) | (1u << 14) | (2u << 29);
    for (int tile = first_tile; tile < total && ok; tile += tile_step, ++it) {
      const int buf = it & 1;
      const uint32_t acc = tmem + (uint32_t)(buf * 256);
      const uint32_t tparity = (uint32_t)((it >> 1) & 1) ^ 1u;
      ok = mbar_wait_cluster(bar_tempty + 8 * buf, tparity, abort_flag, status);
      if (!ok) break;
      tc_fence_after();
      for (int ks = 0; ks < k_stages; ++ks) {
        ok = mbar_wait_cluster(bar_full + 8 * stage, phase, abort_flag, status);
        if (!ok) break;
        tc_fence_after();
        if (issuer) {
          const uint32_t sb = smem_base + stage * kFStageBytes;
          const uint32_t a_lo = ((sb & 0x3FFFFu) >> 4) | (1u << 16);
          const uint32_t b_lo = (((sb + kFTileA) & 0x3FFFFu) >> 4) | (1u << 16);
#pragma unroll
          for (int j = 0; j < 4; ++j)                    // 16 bf16 = 32 bytes along K per MMA
            tc_mma_bf16<2>(acc, ((uint64_t)kSwHi << 32) | (a_lo + 2 * j), ((uint64_t)kSwHi << 32) | (b_lo + 2 * j), idesc,
                            (ks > 0 || j > 0) ? 1u : 0u);
          tc_commit<2>(bar_empty + 8 * stage);
        }
        __syncwarp();
        if (++stage == kFStages) { stage = 0; phase ^= 1u; }
      }
      if (ok && issuer) tc_commit<2>(bar_tfull + 8 * buf);
      __syncwarp();
    }
  } else {
    // ------------------------------------------------------------ epilogue: thread = row, the two warps of a quadrant
    // take alternate groups of 64 columns (each stored as whole lines, see store_y_rows)
    const int q = warp & 3, ch = (warp - 2) >> 2;
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    const uint32_t tempty_addr = map_to_cta(bar_tempty, 0);
    const bool wide = (reinterpret_cast<size_t>(out) & 31) == 0;     // the caller's output may be aligned to 16 bytes only
    int it = 0;
    bool ok = true;
    for (int tile = first_tile; tile < total && ok; tile += tile_step, ++it) {
      const int mt = tile / n_tiles, nt = tile - mt * n_tiles;
      const int buf = it & 1;
      const int row0 = (mt * 2 + (int)rank) * 128 + q * 32;
      ok = mbar_wait(bar_tfull + 8 * buf, (uint32_t)((it >> 1) & 1), abort_flag, status);
      if (!ok) break;
      tc_fence_after();
#pragma unroll 1
      for (int c = ch * 64; c < kFTileN; c += 128) {
        const int n0 = nt * kFTileN + c;
        float v[64];
        tmem_ld32(lane_addr + buf * 256 + c, v);
        tmem_ld32(lane_addr + buf * 256 + c + 32, v + 32);
        tmem_ld_wait();
        if (n0 < N) {
          if (wide) store_y_rows(v, 1.0f, out + (size_t)row0 * N + n0, N, T - row0, lane);
          else store_y_rows<true>(v, 1.0f, out + (size_t)row0 * N + n0, N, T - row0, lane);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_remote_relaxed(tempty_addr + 8 * buf);        // this accumulator is free again
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) settle_if_abandoned(abort_flag);
  cluster_sync_all();                   // the peer may still be signalling this CTA's barriers
  tc_fence_after();
  if (warp == 1) tmem_dealloc<2>(tmem, 512);
}

// ---------------------------------------------------------------------------
// Problems whose tiles of 128 x 128 fit the chip at once: one tile per cluster of S CTAs, K split over them, whose partial
// tiles are added up over distributed shared memory in the order of the ranks (every CTA owns 128 / S columns and
// is sent them by the others, into the idle ring).  One CTA needs 0.185 us for a stage, mostly latency: 64 x 4096 ->
// 4096 used 64 SMs for all of K and took 16 us for 5 us of DRAM traffic.
// Warp 0 loads A, warp 10 B; the operand that is older than the preceding kernel is loaded without waiting for it.
// ---------------------------------------------------------------------------
constexpr int kWThreads = 352;
constexpr int kWLoadB = 10;

constexpr int kWTile = 128 * 128;                              // 128 rows of either operand
template <int BN>
struct WCfg {
  static constexpr int kStages = BN == 128 ? 7 : 4;
  static constexpr int kStageBytes = (1 + BN / 128) * kWTile;
  static constexpr int kBarOffset = kStages * kStageBytes;
  static constexpr int kSmemBytes = kBarOffset + 256 + 1024;
  static_assert(128 * 4 * (BN + 4 * kSplitMax) <= kBarOffset, "the exchange fits the ring");
  static_assert(kSmemBytes <= 232448, "shared memory");
};

struct __align__(8) WBarriers {
  uint64_t full[8];
  uint64_t empty[8];
  uint64_t done;
  uint32_t tmem_base;
  int abort_flag;
};

template <int BN>
__global__ void __launch_bounds__(kWThreads, 1)
gemm_bf16_wave_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b, int T, int N, int K, int split_log2,
                      int a_early, int b_early, uint16_t* __restrict__ out, int32_t* __restrict__ status) {
  using C = WCfg<BN>;
  constexpr int kWStages = C::kStages;
  extern __shared__ uint8_t smem_dyn[];
  const uint32_t smem_base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_dyn + (smem_base - smem_u32(smem_dyn));
  WBarriers* bars = reinterpret_cast<WBarriers*>(smem_gen + C::kBarOffset);
  const uint32_t bar_full = smem_u32(&bars->full[0]), bar_empty = smem_u32(&bars->empty[0]), bar_done = smem_u32(&bars->done);
  volatile int* abort_flag = &bars->abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int split = 1 << split_log2, part = (int)cluster_ctarank();      // share of K
  if (threadIdx.x == 0) {
    for (int s = 0; s < kWStages; ++s) { mbar_init(bar_full + 8 * s, 2); mbar_init(bar_empty + 8 * s, 1); }
    mbar_init(bar_done, 1);
    bars->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    prefetch_tmap(&tm_a);
    prefetch_tmap(&tm_b);
  }
  if (warp == 1) tmem_alloc<1>(smem_u32(&bars->tmem_base), BN);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;

  const int tile = (int)blockIdx.x >> split_log2, n_tiles = (N + BN - 1) / BN;
  const int mt = tile / n_tiles, nt = tile - mt * n_tiles;
  const int k_stages = K / kFStageK;
  const int ks0 = (part * k_stages) >> split_log2, ks1 = ((part + 1) * k_stages) >> split_log2;      // never empty: split <= k_stages
  const int row0 = mt * 128;
  // Behind a kernel of this call, which waited for its own predecessor before this one could start, the loader of the older operand goes
  // ahead, and with the weights (W16A4) the MMA warp too; behind somebody else's kernel (`first`: W16A16), which may run for
  // longer than a wait is allowed to take, nobody does.
  const bool first = !(a_early | b_early);
  const bool early = (warp == 0 && a_early) || ((warp == 1 || warp == kWLoadB) && b_early);
  // When the following kernel may start (it waits for this one's end itself).  Let go at once, the decode of a next W4A16 call gathers on
  // the SMs that this product leaves free, several CTAs to an SM, and the clusters of a next W16A16 product find too few free
  // SMs side by side (replayed from a graph, us, at once / behind the wait: W4A16 78 x 1024 -> 3968 10.0 / 9.3, 1045 x 640 -> 1408 8.2 / 7.7,
  // 132 x 1152 -> 3968 11.5 / 10.8, 173 x 768 -> 640 7.2 / 7.3; W16A16 235 x 2944 -> 640, 40 CTAs, 9.3 / 8.6, 366 x 2560 -> 512, 48 CTAs,
  // 8.9 / 8.4, 68 x 3968 -> 512, 32 CTAs, 7.0 / 7.2, 70 x 1408 -> 512, 16 CTAs, 5.7 / 5.9, 64 x 512 -> 512, no split, 3.85 / 4.0).
  const bool at_once = b_early || (first && (split == 1 || gridDim.x <= 32));
  if (warp == 1 && at_once) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (!early) pdl_sync();
  if (first && blockIdx.x == 0 && threadIdx.x == 64) *status = 0;

  if (warp == 0 || warp == kWLoadB) {
    // ------------------------------------------------------------ loaders
    const bool issuer = elect_one(), loads_b = warp == kWLoadB;
    const CUtensorMap* map = loads_b ? &tm_b : &tm_a;
    const int row = loads_b ? nt * BN : row0, boxes = (loads_b ? min(BN, N - row) : 128) / kFBox;      // (N % 128 == 0)
    uint32_t stage = 0, phase = 0;
    for (int ks = ks0; ks < ks1; ++ks) {
      if (!mbar_wait(bar_empty + 8 * stage, phase ^ 1u, abort_flag, status)) break;
      if (issuer) {
        const uint32_t dst = smem_base + stage * C::kStageBytes + (loads_b ? kWTile : 0), full = bar_full + 8 * stage;
        mbar_expect_tx(full, (uint32_t)(boxes * kFBox * 128));
        for (int b = 0; b < boxes; ++b) tma_load_2d(dst + b * kFBox * 128, map, ks * kFStageK, row + b * kFBox, full);
      }
      __syncwarp();
      if (++stage == kWStages) { stage = 0; phase ^= 1u; }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    const bool issuer = elect_one();
    uint32_t stage = 0, phase = 0;
    bool ok = true;
    constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    constexpr uint32_t kSwHi = (uint32_t)((8 * 128) >> 4) | (1u << 14) | (2u << 29);
    for (int ks = ks0; ks < ks1; ++ks) {
      ok = mbar_wait(bar_full + 8 * stage, phase, abort_flag, status);
      if (!ok) break;
      tc_fence_after();
      if (issuer) {
        const uint32_t sb = smem_base + stage * C::kStageBytes;
        const uint32_t a_lo = ((sb & 0x3FFFFu) >> 4) | (1u << 16);
        const uint32_t b_lo = (((sb + kWTile) & 0x3FFFFu) >> 4) | (1u << 16);
#pragma unroll
        for (int j = 0; j < 4; ++j)
          tc_mma_bf16<1>(tmem, ((uint64_t)kSwHi << 32) | (a_lo + 2 * j), ((uint64_t)kSwHi << 32) | (b_lo + 2 * j), idesc,
                          (ks > ks0 || j > 0) ? 1u : 0u);
        tc_commit<1>(bar_empty + 8 * stage);
      }
      __syncwarp();
      if (++stage == kWStages) { stage = 0; phase ^= 1u; }
    }
    if (ok && issuer) tc_commit<1>(bar_done);
    __syncwarp();
  }
  // ------------------------------------------------------------ epilogue.  The cluster's barriers are met by every warp, also
  // when a wait was abandoned.
  const bool epi = warp >= 2 && warp < kWLoadB;
  const int q = warp & 3, row = q * 32 + lane, rows_valid = min(128, T - row0);
  const int w_log2 = (BN == 128 ? 7 : 8) - split_log2, w = 1 << w_log2, ld = w + 4;      // columns a CTA owns, their row pitch
  if (epi) {
    mbar_wait(bar_done, 0u, abort_flag, status);       // all MMAs are done, so every stage of the ring has been read
    tc_fence_after();
  }
  if (split > 1) cluster_sync_all();              // ... in the whole cluster
  if (epi) {
    const bool wide = (reinterpret_cast<size_t>(out) & 31) == 0;                     // the caller's output may be aligned to 16 bytes only
#pragma unroll 1
    for (int c0 = ((warp - 2) >> 2) * 64; c0 < BN; c0 += 128) {
      float v[64];
      tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + c0, v);
      tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + c0 + 32, v + 32);
      tmem_ld_wait();
      if (split == 1) {
        const int n0 = nt * BN + c0;
        if (n0 >= N) continue;                         // (the missing half of a last tile)
        uint16_t* dst = out + (size_t)(row0 + q * 32) * N + n0;
        if (wide) store_y_rows(v, 1.0f, dst, N, rows_valid - q * 32, lane);
        else store_y_rows<true>(v, 1.0f, dst, N, rows_valid - q * 32, lane);
      } else if (row < rows_valid) {
        const uint32_t own = smem_base + (uint32_t)((part * 128 + row) * ld) * 4u;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int c = c0 + 4 * i;
          st_cluster_f4(map_to_cta(own + (uint32_t)(c & (w - 1)) * 4u, (uint32_t)(c >> w_log2)), v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        }
      }
    }
  }
  tc_fence_before();
  if (split > 1) cluster_sync_all(); else __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc<1>(tmem, BN);
  if (warp == 0) settle_if_abandoned(abort_flag);
  const int n0 = nt * BN + part * w;
  if (!epi || split == 1 || n0 >= N) return;           // (w <= 128: a CTA's columns are all there or all missing)
  const float* sums = reinterpret_cast<const float*>(smem_gen);
  const int r_log2 = w_log2 - 3;                       // a thread takes eight columns of a row
  for (int i = threadIdx.x - 64; i < rows_valid << r_log2; i += 256) {
    const int r = i >> r_log2, c = (i & ((1 << r_log2) - 1)) * 8;
    float4 lo, hi;
    sum_parts(sums + r * ld + c, 128 * ld, split, lo, hi);
    *reinterpret_cast<uint4*>(out + (size_t)(row0 + r) * N + n0 + c) =
        make_uint4(f32x2_to_bf16x2(lo.x, lo.y), f32x2_to_bf16x2(lo.z, lo.w), f32x2_to_bf16x2(hi.x, hi.y), f32x2_to_bf16x2(hi.z, hi.w));
  }
}

template <int BN>
quads_status launch_wave(const CUtensorMap& tm_a, const CUtensorMap& tm_b, int T, int N, int K, int split_log2, bool a_early, bool b_early,
                         uint16_t* out, int32_t* status, cudaStream_t stream) {
  const int ctas = ((T + 127) / 128) * ((N + BN - 1) / BN) << split_log2;
  QUADS_CUDA_OK(set_max_dynamic_smem<gemm_bf16_wave_kernel<BN>>(WCfg<BN>::kSmemBytes));
  if (split_log2 == 0)
    QUADS_CUDA_OK(launch_kernel(gemm_bf16_wave_kernel<BN>, dim3(ctas), dim3(kWThreads), (size_t)WCfg<BN>::kSmemBytes, stream, tm_a, tm_b, T, N, K,
                                split_log2, a_early ? 1 : 0, b_early ? 1 : 0, out, status));
  else
    QUADS_CUDA_OK(launch_clusters(gemm_bf16_wave_kernel<BN>, ctas, 1 << split_log2, kWThreads, (size_t)WCfg<BN>::kSmemBytes, stream, tm_a, tm_b, T, N,
                                  K, split_log2, a_early ? 1 : 0, b_early ? 1 : 0, out, status));
  return QUADS_OK;
}

// The split of K (log2) of a problem of one wave, or -1.  Fitted in us (replayed from a graph, 4096 -> 512, S = 1 / 2 / 4 / 8: 64 rows
// 15.6 / 11.1 / 8.6 / 8.0, 128 rows 15.8 / 12.3 / 10.5 / 11.0; 2048 -> 2048, 256 rows 10.1 / 9.7 / 10.7).  Clusters of four and eight do
// not fill every SM (see plan_split); from 17 clusters of four on two calls' do not fit side by side, which costs 1 to 2 us (S = 1 /
// 2 / 4: 30 tiles, W16A16 661 x 2176 -> 640 9.2 / 8.5 / 9.6, W4A16 11.7 / 10.8 / 13.6; 31 tiles, 93 x 2944 -> 3968 11.9 / 9.7 / 10.3; 32,
// 64 x 4096 -> 4096 15.2 / 11.1 / 10.8; 17, W4A16 84 x 1408 -> 2176 9.8 / 9.4 / 10.5; against 12, 366 x 2560 -> 512 10.2 / 8.8 / 8.4).
int plan_wave(int T, int N, int K, int n_sms) {
  return plan_split((int64_t)((T + 127) / 128) * (N / 128), T, K / kFStageK, 0.185, 1.25, 1.3, n_sms);
}

}  // namespace

quads_status launch_gemm_bf16(const CUtensorMap& tm_a, const CUtensorMap& tm_b, int T, int N, int K, bool a_early, bool b_early, uint16_t* out,
                              int32_t* status, int n_sms, cudaStream_t stream) {
  // Tiles of 128 x 128 in one wave; else of 128 x 256 in one wave while K is short (us per call, so / pairs: 700 x 1024 -> 4096 10.1 / 10.5,
  // 1024 x 2048 -> 4096 15.2 / 15.7, 9000 x 2048 -> 384 16.0 / 16.4; 1024 x 4096 -> 4096 28.0 / 26.4); else pairs.
  const int split_log2 = plan_wave(T, N, K, n_sms);
  if (split_log2 >= 0) return launch_wave<128>(tm_a, tm_b, T, N, K, split_log2, a_early, b_early, out, status, stream);
  if (K <= 2048 && (int64_t)((T + 127) / 128) * ((N + 255) / 256) <= n_sms)
    return launch_wave<256>(tm_a, tm_b, T, N, K, 0, a_early, b_early, out, status, stream);
  QUADS_CUDA_OK(set_max_dynamic_smem<gemm_bf16_pair_kernel>(kFSmemBytes));
  QUADS_CUDA_OK(launch_kernel(gemm_bf16_pair_kernel, dim3(n_sms / 2 * 2), dim3(kFThreads), (size_t)kFSmemBytes, stream, tm_a,
                              tm_b, T, N, K, a_early || b_early ? 0 : 1, out, status));
  return QUADS_OK;
}

}  // namespace quads
