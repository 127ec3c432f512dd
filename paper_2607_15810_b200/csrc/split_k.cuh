// The rule by which products whose tiles fit the chip at once split K over clusters (gemm_dense.cu, gemm_bf16.cu).
#pragma once
#include <algorithm>
#include <cstdint>

namespace quads {
namespace {

constexpr int kSplitMax = 8;                          // CTAs of a cluster

// The split of K (log2 S) with the least time, or -1 where the tiles don't fit the chip at once.  A CTA takes t_stage (us) per K stage;
// the exchange of partial tiles t_exchange * (1 + log2 S) with 128 rows in a tile, and in proportion with fewer.  The clusters have
// to be resident together: those of four fill 128 SMs, those of eight find room for 15 or 16, of which half are used.  t_crowd:
// what clusters of four cost on top from the 17th on, where those of two calls don't fit side by side.
inline int plan_split(int64_t tiles, int rows, int k_stages, double t_stage, double t_exchange, double t_crowd, int n_sms) {
  int best = -1;
  double cost = 1e30;
  for (int lg = 0; 1 << lg <= kSplitMax && 1 << lg <= k_stages; ++lg) {
    if (tiles << lg > (lg == 0 ? n_sms : lg == 1 ? n_sms / 2 * 2 : lg == 2 ? 128 : 64)) continue;
    const double c = ((k_stages + (1 << lg) - 1) >> lg) * t_stage + (lg ? std::min(rows, 128) / 128.0 * t_exchange * (1 + lg) + 0.05 * lg : 0.0) +
                     (lg == 2 && tiles > 16 ? t_crowd : 0.0);
    if (c < cost) { cost = c; best = lg; }
  }
  return best;
}

}  // namespace
}  // namespace quads
