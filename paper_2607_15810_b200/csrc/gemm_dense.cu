// Dense NVFP4 x NVFP4 projection with few output tiles (see gemm.cu for the product, its operands and descriptors).
//
// A projection of a few hundred rows has fewer tiles of 128 x 256 than the chip has SMs, and each of them pulls in
// its operands over all of K at what one SM can take (about 100 GB/s): 16 CTAs took 12 us for one row of a
// 4096 x 4096 projection, whose weights are 2 us of DRAM time.  Here K is split as well: a cluster of S CTAs
// computes one tile of 128 x BN, each CTA over its share of K, and adds the partial tiles up over distributed shared
// memory -- every CTA sends each other one the columns that one owns and adds its own columns in the order
// of the ranks, so the result does not depend on timing.  The ring of operand stages is the exchange buffer:
// it is idle by then.
//
// One tile per CTA.  Warp 0 loads weights and their scales, which are older than the preceding kernel, without waiting
// for it; warp 10 loads the activation side behind it; warp 1 issues the MMAs; warps 2..9 are the epilogue.
// Every wait is bounded (status word, as in gemm.cu).
#include "kernels.cuh"
#include "split_k.cuh"
#include "tcgen05.cuh"

namespace quads {

namespace {

constexpr int kSteps = kGemmKSteps;                  // K = 64 MMAs per stage
constexpr int kRowBytes = kGemmStageKBytes;          // packed bytes of a row and stage
static_assert(kSteps == 4 && kRowBytes == 128, "laid out for 256-element K stages");
constexpr int kTileRows = 128 * kRowBytes;           // 128 rows of one operand
constexpr int kSfAtoms = kSteps * 512;               // their scales
constexpr int kEpiWarps = 8;
constexpr int kActWarp = 2 + kEpiWarps;
constexpr int kThreads = 32 * (kActWarp + 1);
constexpr int kTmemCols = 512;
constexpr int kTmemSfBase = 256;                     // accumulator: columns 0 .. BN - 1
constexpr int kTmemSfPerBuf = 64;                    // SFA 4/step | SFR 4/step | SFB 8/step, double buffered

template <int BN>
struct DCfg {
  static constexpr int kHalves = BN / 128;
  static constexpr int kOffR = kTileRows, kOffB = 2 * kTileRows;
  static constexpr int kOffSfA = kOffB + kHalves * kTileRows, kOffSfR = kOffSfA + kSfAtoms, kOffSfB = kOffSfR + kSfAtoms;
  static constexpr int kStageBytes = kOffSfB + kHalves * kSfAtoms;      // 55296 / 73728
  static constexpr int kStages = BN == 128 ? 4 : 3;
  static constexpr int kBarOffset = kStages * kStageBytes;
  static constexpr int kSmemBytes = kBarOffset + 256 + 1024;
  static_assert(128 * 4 * (BN + 4 * kSplitMax) <= kBarOffset, "the exchange fits the ring");
};

struct __align__(8) DBarriers {
  uint64_t full[4];
  uint64_t empty[4];
  uint64_t done;
  uint32_t tmem_base;
  int abort_flag;
};

template <int BN>
__global__ void __launch_bounds__(kThreads, 1)
gemm_dense_kernel(const GemmParams p, int split_log2, const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_r,
                  const __grid_constant__ CUtensorMap tm_b) {
  using C = DCfg<BN>;
  extern __shared__ uint8_t smem_dyn[];
  const uint32_t smem_base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_dyn + (smem_base - smem_u32(smem_dyn));
  DBarriers* bars = reinterpret_cast<DBarriers*>(smem_gen + C::kBarOffset);
  const uint32_t bar_full = smem_u32(&bars->full[0]), bar_empty = smem_u32(&bars->empty[0]), bar_done = smem_u32(&bars->done);
  volatile int* abort_flag = &bars->abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::kStages; ++s) { mbar_init(bar_full + 8 * s, 2); mbar_init(bar_empty + 8 * s, 1); }
    mbar_init(bar_done, 1);
    bars->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    prefetch_tmap(&tm_a);
    prefetch_tmap(&tm_b);
    if (p.has_resid) prefetch_tmap(&tm_r);
  }
  if (warp == 1) tmem_alloc<1>(smem_u32(&bars->tmem_base), kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;

  const int split = 1 << split_log2, rank = (int)cluster_ctarank(), tile = (int)blockIdx.x >> split_log2;
  const int mt = tile / p.n_tiles_n, nt = tile - mt * p.n_tiles_n;
  const int kt_count = p.K >> 6, k_stages = (kt_count + kSteps - 1) / kSteps;
  const int ks0 = (rank * k_stages) >> split_log2, ks1 = ((rank + 1) * k_stages) >> split_log2;      // never empty: split <= k_stages
  const bool resid = p.has_resid != 0;
  // the weight loader and the MMA warp read nothing that the preceding kernel wrote
  if (warp < 2) asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); else pdl_sync();

  if (warp == 0 || warp == kActWarp) {
    // ------------------------------------------------------------ loaders
    const bool issuer = elect_one(), weights = warp == 0;
    const int rt = nt * C::kHalves;                                  // 128-row tiles of the weight
    const bool half1 = C::kHalves == 2 && nt * BN + 128 < p.n_out;
    const uint8_t* sf0 = weights ? p.b_sf + (size_t)rt * kt_count * 512u : p.a_sf + (size_t)mt * kt_count * 512u;
    const uint8_t* sf1 = weights ? sf0 + (size_t)kt_count * 512u : p.r_sf + (size_t)mt * kt_count * 512u;
    const bool second = weights ? half1 : resid;
    const CUtensorMap *map0 = weights ? &tm_b : &tm_a, *map1 = weights ? &tm_b : &tm_r;
    const int row0 = weights ? rt * 128 : mt * 128, row1 = weights ? row0 + 128 : row0;
    const uint32_t dst0 = weights ? C::kOffB : 0, dst1 = dst0 + kTileRows;
    const uint32_t dsf0 = weights ? C::kOffSfB : C::kOffSfA, dsf1 = dsf0 + kSfAtoms;
    uint32_t stage = 0, phase = 0;
    for (int ks = ks0; ks < ks1; ++ks) {
      if (!mbar_wait(bar_empty + 8 * stage, phase ^ 1u, abort_flag, p.status)) break;
      if (issuer) {
        const uint32_t sb = smem_base + stage * C::kStageBytes, full = bar_full + 8 * stage;
        const uint32_t sf_bytes = (uint32_t)min(kSteps, kt_count - ks * kSteps) * 512u;
        const size_t sf_off = (size_t)ks * kSfAtoms;
        mbar_expect_tx(full, (kTileRows + sf_bytes) * (second ? 2u : 1u));
        tma_load_2d(sb + dst0, map0, ks * kRowBytes, row0, full);
        if (second) tma_load_2d(sb + dst1, map1, ks * kRowBytes, row1, full);
        bulk_load(sb + dsf0, sf0 + sf_off, sf_bytes, full);
        if (second) bulk_load(sb + dsf1, sf1 + sf_off, sf_bytes, full);
      }
      __syncwarp();
      if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    const bool issuer = elect_one();
    uint32_t stage = 0, phase = 0;
    bool ok = true;
    constexpr uint32_t idesc = (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    constexpr uint32_t kSwHi = (uint32_t)((8 * kRowBytes) >> 4) | (1u << 14) | (2u << 29);
    constexpr uint32_t kSfHi = (uint32_t)(128 >> 4) | (1u << 14);
    for (int ks = ks0; ks < ks1; ++ks) {
      ok = mbar_wait(bar_full + 8 * stage, phase, abort_flag, p.status);
      if (!ok) break;
      tc_fence_after();
      if (issuer) {
        const int atoms = min(kSteps, kt_count - ks * kSteps);
        const uint32_t sb = smem_base + stage * C::kStageBytes;
        const uint32_t sfcol = tmem + kTmemSfBase + ((uint32_t)ks & 1u) * kTmemSfPerBuf;
        const uint32_t a_lo = ((sb & 0x3FFFFu) >> 4) | (1u << 16);
        const uint32_t r_lo = (((sb + C::kOffR) & 0x3FFFFu) >> 4) | (1u << 16);
        const uint32_t b_lo = (((sb + C::kOffB) & 0x3FFFFu) >> 4) | (1u << 16);
        const uint32_t sfa_lo = ((sb + C::kOffSfA) & 0x3FFFFu) >> 4;
        const uint32_t sfr_lo = ((sb + C::kOffSfR) & 0x3FFFFu) >> 4;
        const uint32_t sfb_lo = ((sb + C::kOffSfB) & 0x3FFFFu) >> 4;
        auto copy_sf = [&](int j) {
          tc_cp_sf<1>(sfcol + 4 * j, ((uint64_t)kSfHi << 32) | (sfa_lo + 32 * j));
          if (resid) tc_cp_sf<1>(sfcol + 4 * kSteps + 4 * j, ((uint64_t)kSfHi << 32) | (sfr_lo + 32 * j));
          tc_cp_sf<1>(sfcol + 8 * kSteps + 8 * j, ((uint64_t)kSfHi << 32) | (sfb_lo + 32 * j));
          if (C::kHalves == 2) tc_cp_sf<1>(sfcol + 8 * kSteps + 8 * j + 4, ((uint64_t)kSfHi << 32) | (sfb_lo + (kSfAtoms >> 4) + 32 * j));
        };
        copy_sf(0);
#pragma unroll
        for (int j = 0; j < kSteps; ++j) {
          if (j + 1 < atoms) copy_sf(j + 1);
          if (j < atoms) {
            const uint64_t bdesc = ((uint64_t)kSwHi << 32) | (b_lo + 2 * j);
            tc_mma_nvf4<1>(tmem, ((uint64_t)kSwHi << 32) | (a_lo + 2 * j), bdesc, idesc, sfcol + 4 * j, sfcol + 8 * kSteps + 8 * j,
                           (ks > ks0 || j > 0) ? 1u : 0u);
            if (resid)
              tc_mma_nvf4<1>(tmem, ((uint64_t)kSwHi << 32) | (r_lo + 2 * j), bdesc, idesc, sfcol + 4 * kSteps + 4 * j,
                             sfcol + 8 * kSteps + 8 * j, 1u);
          }
        }
        tc_commit<1>(bar_empty + 8 * stage);
      }
      __syncwarp();
      if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
    }
    if (ok && issuer) tc_commit<1>(bar_done);
    __syncwarp();
  }
  // ------------------------------------------------------------ epilogue.  The cluster's barriers are met by every warp, also when
  // a wait was abandoned.
  const bool epi = warp >= 2 && warp < kActWarp;
  const int q = warp & 3;                              // tensor-memory lanes of this warp
  const int row = q * 32 + lane, rows_valid = min(128, p.dense_rows - mt * 128);
  const int w_log2 = (BN == 128 ? 7 : 8) - split_log2, w = 1 << w_log2;      // columns a CTA owns
  const int ld = w + 4;                                // row pitch (a pad of 16 bytes spreads the banks)
  const float scale = !epi ? 0.f : __fmul_rn(p.a_gs ? p.a_gs[0] : gs_from_amax_bits(p.a_amax_bits[0]), p.b_gs[0]);
  if (epi) {
    mbar_wait(bar_done, 0u, abort_flag, p.status);     // all MMAs are done, so every stage of the ring has been read
    tc_fence_after();
  }
  if (split > 1) cluster_sync_all();                   // ... in the whole cluster
  if (epi) {
    const bool wide = (reinterpret_cast<size_t>(p.out_bf16) & 31) == 0;
#pragma unroll 1
    for (int c0 = ((warp - 2) >> 2) * 64; c0 < BN; c0 += 128) {
      float v[64];
      tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + c0, v);
      tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + c0 + 32, v + 32);
      tmem_ld_wait();
      if (split == 1) {
        const int n0 = nt * BN + c0;
        uint16_t* dst = p.out_bf16 + (size_t)(mt * 128 + q * 32) * p.n_out + n0;
        if (n0 >= p.n_out) continue;                   // (the missing half of a last tile)
        if (wide) store_y_rows(v, scale, dst, p.n_out, rows_valid - q * 32, lane);
        else store_y_rows<true>(v, scale, dst, p.n_out, rows_valid - q * 32, lane);
      } else if (row < rows_valid) {
        const uint32_t own = smem_base + (uint32_t)((rank * 128 + row) * ld) * 4u;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int c = c0 + 4 * i;
          st_cluster_f4(map_to_cta(own + (uint32_t)(c & (w - 1)) * 4u, (uint32_t)(c >> w_log2)), v[4 * i], v[4 * i + 1], v[4 * i + 2],
                        v[4 * i + 3]);
        }
      }
    }
  }
  tc_fence_before();
  if (split > 1) cluster_sync_all(); else __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc<1>(tmem, kTmemCols);
  if (warp == 0) settle_if_abandoned(abort_flag);
  const int n0 = nt * BN + rank * w;
  if (!epi || split == 1 || n0 >= p.n_out) return;     // (w <= 128: a CTA's columns are all there or all missing)
  const float* part = reinterpret_cast<const float*>(smem_gen);
  const int r_log2 = w_log2 - 3;                       // a thread takes eight columns of a row
  for (int i = threadIdx.x - 64; i < rows_valid << r_log2; i += 32 * kEpiWarps) {
    const int r = i >> r_log2, c = (i & ((1 << r_log2) - 1)) * 8;
    float4 lo, hi;
    sum_parts(part + r * ld + c, 128 * ld, split, lo, hi);
    *reinterpret_cast<uint4*>(p.out_bf16 + (size_t)(mt * 128 + r) * p.n_out + n0 + c) =
        make_uint4(f32x2_to_bf16x2(lo.x * scale, lo.y * scale), f32x2_to_bf16x2(lo.z * scale, lo.w * scale),
                   f32x2_to_bf16x2(hi.x * scale, hi.y * scale), f32x2_to_bf16x2(hi.z * scale, hi.w * scale));
  }
}

template <int BN>
quads_status launch_bn(GemmParams p, int split_log2, const GemmMaps& m, cudaStream_t stream) {
  p.n_tiles_n = (p.n_out + BN - 1) / BN;
  const int tiles = (p.dense_rows + 127) / 128 * p.n_tiles_n;
  QUADS_CUDA_OK(set_max_dynamic_smem<gemm_dense_kernel<BN>>(DCfg<BN>::kSmemBytes));
  constexpr size_t kSmem = DCfg<BN>::kSmemBytes;
  if (split_log2 == 0)
    QUADS_CUDA_OK(launch_kernel(gemm_dense_kernel<BN>, dim3(tiles), dim3(kThreads), kSmem, stream, p, split_log2, m.a, m.r, m.b));
  else
    QUADS_CUDA_OK(launch_clusters(gemm_dense_kernel<BN>, tiles << split_log2, 1 << split_log2, kThreads, kSmem, stream, p, split_log2, m.a, m.r, m.b));
  return QUADS_OK;
}

// Tile width and split of K (log2) of a dense projection; split_log2 = -1 where the persistent kernels take it (more tiles than SMs).
// Tiles of 128 columns if they fit one wave, else of 256 (700 x 4096 -> 4096 32.5 us per call with the persistent kernel, 31.2 so; where
// both fit, 128 are ahead: 512 x 2048 -> 2048 24.4 / 22.4).  A stage of K takes a CTA 0.39 us, the exchange about 1 + log2(S) us with 128
// rows (4096 -> 1024, S = 1 / 2 / 4 / 8: one row 20.9 / 17.9 / 16.4 / 15.6, 64 rows 22.0 / 20.0 / 18.9 / 19.1, 128 rows 24.4 / 23.4 / 22.9 /
// 23.8; 2048 -> 2048, 128 rows 16.6 / 17.2 / 17.8; one row, 2048 -> 2048: 12.7 with 64 CTAs in clusters of four, 15.9 with 128 in clusters
// of eight).
struct DensePlan { int bn, split_log2; };
DensePlan plan_dense(int rows, int K, int N, int n_sms) {
  const int k_stages = (K + 64 * kSteps - 1) / (64 * kSteps), m_tiles = (rows + 127) / 128;
  const int lg = plan_split((int64_t)m_tiles * (N / 128), rows, k_stages, 0.39, 1.0, 0.0, n_sms);
  if (lg >= 0) return DensePlan{128, lg};
  return DensePlan{256, m_tiles * (int64_t)((N + 255) / 256) <= n_sms ? 0 : -1};
}

}  // namespace

bool gemm_dense_ok(int rows, int K, int N, int n_sms) { return plan_dense(rows, K, N, n_sms).split_log2 >= 0; }

// From 1024 rows on, where the persistent CTA pairs are the other form: ahead of them in one wave, but for a long K without residual
// in tiles of 256 columns, which the pairs' deeper ring suits better (replayed from a graph, us, pairs / so: 1024 x 512 -> 1024 10.3 / 7.9,
// with residual 18.5 / 15.9; 1500 x 2048 -> 512 13.7 / 11.7, 25.6 / 22.1; 4000 x 2048 -> 1024 17.0 / 17.1, 31.4 / 29.8; 2000 x 4096 -> 1024
// 19.5 / 17.6, 36.3 / 31.3; 8192 x 4096 -> 256 36.9 / 35.0, 62.3 / 58.0; 2000 x 4096 -> 2048 19.9 / 21.1, 37.6 / 36.0; beyond one wave 3000 x
// 2048 -> 2048 19.1 / 20.2).
bool gemm_dense_ahead_of_pairs(int rows, int K, int N, bool resid, int n_sms) {
  const DensePlan d = plan_dense(rows, K, N, n_sms);
  return d.split_log2 >= 0 && (d.bn == 128 || resid || K <= 2048);
}

quads_status launch_gemm_dense(const GemmParams& p, const GemmMaps& m, int n_sms, cudaStream_t stream) {
  const DensePlan d = plan_dense(p.dense_rows, p.K, p.n_out, n_sms);
  return d.bn == 128 ? launch_bn<128>(p, d.split_log2, m, stream) : launch_bn<256>(p, d.split_log2, m, stream);
}

}  // namespace quads
