// Dense bf16 x bf16 GEMM on the 5th-generation tensor cores (tcgen05, kind::f16) for the
// one-sided rollout modes of the paper's ablations: out[T, N] = A[T, K] B[N, K]^T with float32
// accumulation in tensor memory, bf16 output.
//   W4A16: A = the activations as they are (bf16), B = the NVFP4 weights decoded to bf16;
//   W16A4: A = the decoded NVFP4 activations (Q_A then decode, bf16), B = the bf16 weights.
// The decoded operand is produced by the library's own decode / fake-quant kernels into the
// caller's workspace; this kernel is the contraction.
//
// One persistent CTA per SM, 10 warps: warp 0 issues TMA tile loads (128-byte swizzle, 64 bf16 per
// row and stage) into a ring; warp 1 issues four K = 16 MMAs per stage and releases stages with
// tcgen05.commit; warps 2..9 drain one of TWO float32 accumulators (all 512 columns of tensor memory)
// while the MMAs of the next tile fill the other.  Every wait is bounded; a wait that gives up records
// QUADS_ERR_TIMEOUT and all roles leave.
//
// Two forms.  CG = 2: pairs of CTAs compute 256 x 256 tiles with cta_group::2 MMAs, each holding its own 128
// rows of A and half of B's -- 32 instead of 48 KB per CTA and stage, hence six stages instead of four and a third
// less traffic out of L2 and shared memory, which in a loop is what the power limit is spent on.  CG = 1:
// tiles of 128 x 64, 128 or 256 for problems that have no wave of pairs; the narrower ones spread a small
// problem over the chip.  2048 x 4096 -> 4096: 51.5 us single CTAs, 45.8 pairs (1.50 PFLOP/s, 0.89 of the measured burst
// rate; 128 tiles on 74 pairs leave the second wave a quarter empty).
#include "kernels.cuh"
#include "tcgen05.cuh"

namespace quads {
namespace {

constexpr int kFStageK = 64;                         // bf16 elements per row per stage (128 bytes)
constexpr int kFBox = kBf16BoxRows;                  // rows of a TMA box
constexpr int kFTileA = 128 * 128;                   // 16 KB
constexpr int kFThreads = 320;
constexpr int kFEpiWarps = 8;
constexpr int kFMaxStages = 6;

template <int CG>
struct FCfg {
  static constexpr int kStages = CG == 2 ? 6 : 4;
  static constexpr int kTileB = 256 * 128 / CG;
  static constexpr int kStageBytes = kFTileA + kTileB;
  static constexpr int kBarOffset = kStages * kStageBytes;
  static constexpr int kSmemBytes = kBarOffset + 256 + 1024;
};

struct __align__(8) FBarriers {
  uint64_t full[kFMaxStages];
  uint64_t empty[kFMaxStages];
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

template <int CG>
__device__ __forceinline__ void gemm_bf16_body(const CUtensorMap* tm_a, const CUtensorMap* tm_b, int T, int N, int K, int n_tile,
                                               uint16_t* __restrict__ out, int32_t* __restrict__ status) {
  using C = FCfg<CG>;
  constexpr int kStages = C::kStages;
  extern __shared__ uint8_t smem_dyn[];
  const uint32_t smem_base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_dyn + (smem_base - smem_u32(smem_dyn));
  FBarriers* bars = reinterpret_cast<FBarriers*>(smem_gen + C::kBarOffset);
  const uint32_t bar_full = smem_u32(&bars->full[0]), bar_empty = smem_u32(&bars->empty[0]);
  const uint32_t bar_tfull = smem_u32(&bars->tmem_full[0]), bar_tempty = smem_u32(&bars->tmem_empty[0]);
  volatile int* abort_flag = &bars->abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = CG == 1 ? 0u : cluster_ctarank();      // position inside the CTA pair
  const bool leader = rank == 0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) { mbar_init(bar_full + 8 * s, leader ? CG : 1); mbar_init(bar_empty + 8 * s, 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(bar_tfull + 8 * b, 1); mbar_init(bar_tempty + 8 * b, kFEpiWarps * CG); }
    bars->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    prefetch_tmap(tm_a);
    prefetch_tmap(tm_b);
  }
  if (warp == 1) tmem_alloc<CG>(smem_u32(&bars->tmem_base), 512);
  tc_fence_before();
  __syncthreads();
  if (CG == 2) cluster_sync_all();                   // both CTAs' barriers exist before any remote arrive
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;
  pdl_sync();                                        // the decoded operand comes from the preceding kernel

  const int m_tiles = (T + 128 * CG - 1) / (128 * CG), n_tiles = (N + n_tile - 1) / n_tile;
  const int total = m_tiles * n_tiles;
  const int k_stages = K / kFStageK;
  const int first_tile = blockIdx.x / CG, tile_step = gridDim.x / CG;

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    const bool issuer = elect_one();
    uint32_t stage = 0, phase = 0;
    bool ok = true;
    const uint32_t leader_full = CG == 2 ? map_to_cta(bar_full, 0) : bar_full;
    for (int tile = first_tile; tile < total && ok; tile += tile_step) {
      const int mt = tile / n_tiles, nt = tile - mt * n_tiles;
      const int arow = (mt * CG + (int)rank) * 128;
      const int brow = nt * n_tile + (int)rank * (n_tile / CG);
      const int boxes_b = max(0, min(n_tile / CG, N - brow)) / kFBox;   // boxes of weight rows that exist (N % 128 == 0)
      for (int ks = 0; ks < k_stages; ++ks) {
        ok = mbar_wait(bar_empty + 8 * stage, phase ^ 1u, abort_flag, status);
        if (!ok) break;
        if (issuer) {
          const uint32_t sb = smem_base + stage * C::kStageBytes;
          const uint32_t bytes = (uint32_t)(kFTileA + boxes_b * kFBox * 128);
          if (CG == 1) {
            const uint32_t full = bar_full + 8 * stage;
            mbar_expect_tx(full, bytes);
            for (int b = 0; b < 128 / kFBox; ++b) tma_load_2d(sb + b * kFBox * 128, tm_a, ks * kFStageK, arow + b * kFBox, full);
            for (int b = 0; b < boxes_b; ++b) tma_load_2d(sb + kFTileA + b * kFBox * 128, tm_b, ks * kFStageK, brow + b * kFBox, full);
          } else {
            const uint32_t full = leader_full + 8 * stage;        // both CTAs' loads credit the leader's barrier
            mbar_expect_tx_cluster(full, bytes);
            for (int b = 0; b < 128 / kFBox; ++b) tma_load_2d_pair(sb + b * kFBox * 128, tm_a, ks * kFStageK, arow + b * kFBox, full);
            for (int b = 0; b < boxes_b; ++b) tma_load_2d_pair(sb + kFTileA + b * kFBox * 128, tm_b, ks * kFStageK, brow + b * kFBox, full);
          }
        }
        __syncwarp();
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
      }
    }
    for (int s = 0; s < kStages && ok; ++s) {            // drain: every armed stage lands and is consumed
      ok = mbar_wait(bar_empty + 8 * stage, phase ^ 1u, abort_flag, status);
      if (++stage == kStages) { stage = 0; phase ^= 1u; }
    }
  } else if (warp == 1 && !leader) {
    // the leader CTA issues the MMAs of the pair
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    const bool issuer = elect_one();
    uint32_t stage = 0, phase = 0;
    int it = 0;
    bool ok = true;
    // bf16 x bf16 -> float32, both operands K-major, M = 128 per CTA of the group, N = n_tile
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n_tile >> 3) << 17) | ((uint32_t)((128 * CG) >> 4) << 24);
    constexpr uint32_t kSwHi = (uint32_t)((8 * 128) >> 4) | (1u << 14) | (2u << 29);
    for (int tile = first_tile; tile < total && ok; tile += tile_step, ++it) {
      const int buf = it & 1;
      const uint32_t acc = tmem + (uint32_t)(buf * 256);
      const uint32_t tparity = (uint32_t)((it >> 1) & 1) ^ 1u;
      ok = CG == 1 ? mbar_wait(bar_tempty + 8 * buf, tparity, abort_flag, status)
                   : mbar_wait_cluster(bar_tempty + 8 * buf, tparity, abort_flag, status);
      if (!ok) break;
      tc_fence_after();
      for (int ks = 0; ks < k_stages; ++ks) {
        ok = CG == 1 ? mbar_wait(bar_full + 8 * stage, phase, abort_flag, status)
                     : mbar_wait_cluster(bar_full + 8 * stage, phase, abort_flag, status);
        if (!ok) break;
        tc_fence_after();
        if (issuer) {
          const uint32_t sb = smem_base + stage * C::kStageBytes;
          const uint32_t a_lo = ((sb & 0x3FFFFu) >> 4) | (1u << 16);
          const uint32_t b_lo = (((sb + kFTileA) & 0x3FFFFu) >> 4) | (1u << 16);
#pragma unroll
          for (int j = 0; j < 4; ++j)                    // 16 bf16 = 32 bytes along K per MMA
            tc_mma_bf16<CG>(acc, ((uint64_t)kSwHi << 32) | (a_lo + 2 * j), ((uint64_t)kSwHi << 32) | (b_lo + 2 * j), idesc,
                            (ks > 0 || j > 0) ? 1u : 0u);
          tc_commit<CG>(bar_empty + 8 * stage);
        }
        __syncwarp();
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
      }
      if (ok && issuer) tc_commit<CG>(bar_tfull + 8 * buf);
      __syncwarp();
    }
  } else {
    // ------------------------------------------------------------ epilogue: thread = row, the two warps of a quadrant
    // take alternate groups of 64 columns (each stored as whole lines, see store_y_rows)
    const int q = warp & 3, ch = (warp - 2) >> 2;
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    const uint32_t tempty_addr = CG == 1 ? bar_tempty : map_to_cta(bar_tempty, 0);
    const bool wide = (reinterpret_cast<size_t>(out) & 31) == 0;     // the caller's output may be aligned to 16 bytes only
    int it = 0;
    bool ok = true;
    for (int tile = first_tile; tile < total && ok; tile += tile_step, ++it) {
      const int mt = tile / n_tiles, nt = tile - mt * n_tiles;
      const int buf = it & 1;
      const int row0 = (mt * CG + (int)rank) * 128 + q * 32;
      ok = mbar_wait(bar_tfull + 8 * buf, (uint32_t)((it >> 1) & 1), abort_flag, status);
      if (!ok) break;
      tc_fence_after();
#pragma unroll 1
      for (int c = ch * 64; c < n_tile; c += 128) {
        const int n0 = nt * n_tile + c;
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
      if (lane == 0) {                                    // this accumulator is free again
        if (CG == 1) mbar_arrive(bar_tempty + 8 * buf);
        else mbar_arrive_remote_relaxed(tempty_addr + 8 * buf);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (CG == 2) cluster_sync_all();                   // the peer may still be signalling this CTA's barriers
  tc_fence_after();
  if (warp == 1) tmem_dealloc<CG>(tmem, 512);
}

__global__ void __launch_bounds__(kFThreads, 1)
gemm_bf16_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b, int T, int N, int K, int n_tile,
                 uint16_t* __restrict__ out, int32_t* __restrict__ status) {
  gemm_bf16_body<1>(&tm_a, &tm_b, T, N, K, n_tile, out, status);
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kFThreads, 1)
gemm_bf16_pair_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b, int T, int N, int K,
                      uint16_t* __restrict__ out, int32_t* __restrict__ status) {
  gemm_bf16_body<2>(&tm_a, &tm_b, T, N, K, 256, out, status);
}

}  // namespace

quads_status launch_gemm_bf16(const CUtensorMap& tm_a, const CUtensorMap& tm_b, int T, int N, int K, uint16_t* out,
                              int32_t* status, int n_sms, cudaStream_t stream) {
  const int pair_tiles = ((T + 255) / 256) * ((N + 255) / 256);
  // From one wave of pairs on, however full the last one is (us, pairs / best single-CTA width: 2304 x 4096 -> 2304, 81 tiles, 44.6 /
  // 45.3; 2560 x 4096 -> 2560, 100 tiles, 44.4 / 50.1; 8192 x 2048 -> 640 25.0 / 25.3; 8192 x 4096 -> 4096 201 / 213; the one
  // form it loses at is a single column tile, half of it missing: 18945 x 2048 -> 128 23.4 / 17.8).
  if (pair_tiles >= n_sms / 2) {
    QUADS_CUDA_OK(set_max_dynamic_smem<gemm_bf16_pair_kernel>(FCfg<2>::kSmemBytes));
    QUADS_CUDA_OK(launch_kernel(gemm_bf16_pair_kernel, dim3(n_sms / 2 * 2), dim3(kFThreads), (size_t)FCfg<2>::kSmemBytes, stream, tm_a,
                                tm_b, T, N, K, out, status));
    return QUADS_OK;
  }
  // the tile width with the least (waves x time of a tile); a K step costs a tile about as much as 64 columns on top
  int n_tile = 256, best = 0;
  for (int n = 256; n >= 64; n /= 2) {
    const int tiles = ((T + 127) / 128) * ((N + n - 1) / n), cost = (tiles + n_sms - 1) / n_sms * (n + 64);
    if (n == 256 || cost < best) { best = cost; n_tile = n; }
  }
  QUADS_CUDA_OK(set_max_dynamic_smem<gemm_bf16_kernel>(FCfg<1>::kSmemBytes));
  const int tiles = ((T + 127) / 128) * ((N + n_tile - 1) / n_tile);
  const int grid = tiles < n_sms ? (tiles > 0 ? tiles : 1) : n_sms;
  QUADS_CUDA_OK(launch_kernel(gemm_bf16_kernel, dim3(grid), dim3(kFThreads), (size_t)FCfg<1>::kSmemBytes, stream, tm_a, tm_b, T, N, K,
                              n_tile, out, status));
  return QUADS_OK;
}

}  // namespace quads
