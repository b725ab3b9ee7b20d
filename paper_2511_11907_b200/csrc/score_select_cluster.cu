// Host side of the one-cluster predictor (score_select_cluster.cuh): which shapes take it, and the launch.
#include <algorithm>
#include <cmath>

#include "score_select_cluster.cuh"

namespace kvswap {
namespace {

struct Plan {
  int g_shift, tile_rows, tiles, n_sub, n_rests, cluster, depth;
  bool whole_sm;                                         // a CTA's shared memory leaves no room for a second one
};

size_t cta_smem(const Problem& p, bool power_of_two, int depth) {
  auto by_group = [&](auto m, auto r) {
    constexpr int META = decltype(m)::value, R = decltype(r)::value;
    return power_of_two ? score_select_smem<META, R, 0>(depth, p.NG) : score_select_smem<META, R, -1>(depth, p.NG);
  };
  using F16 = std::integral_constant<int, KVSWAP_F16>;
  using F32 = std::integral_constant<int, KVSWAP_F32>;
  using R16 = std::integral_constant<int, 16>;
  using R32 = std::integral_constant<int, 32>;
  using R64 = std::integral_constant<int, 64>;
  if (p.meta_dtype == KVSWAP_E4M3) return score_select_smem<KVSWAP_E4M3, 32, 0>(depth, p.NG);
  if (p.meta_dtype == KVSWAP_F16) return p.r == 16 ? by_group(F16(), R16()) : p.r == 32 ? by_group(F16(), R32()) : by_group(F16(), R64());
  return p.r == 16 ? by_group(F32(), R16()) : p.r == 32 ? by_group(F32(), R32()) : by_group(F32(), R64());
}

bool plan(const Problem& p, Plan* pl) {
  if (p.NG < 1 || p.NG > kClusterMaxKeys || (p.flags & KVSWAP_SCORE_SOFTMAX) || !score_stream_rows(p) || p.meta_sn != p.r ||
      multi_term(p) || (p.d != 32 && p.d != 64 && p.d != 128))
    return false;
  if (p.scope == KVSWAP_SCOPE_ALL_HEADS && p.Hkv > kQueryCols) return false;      // the queries are built in one round
  const int elem = p.meta_dtype == KVSWAP_F32 ? 4 : p.meta_dtype == KVSWAP_F16 ? 2 : 1;
  int g_shift = -1;
  for (int s = 0; s <= 5; ++s) if ((1 << s) == p.G) g_shift = s;
  if (g_shift < 0 && p.meta_dtype == KVSWAP_E4M3) return false;
  const int fit = score_stage_rows(g_shift < 0, p.r * elem);
  pl->g_shift = g_shift;
  pl->tile_rows = g_shift >= 0 ? fit : fit / p.G * p.G;
  if (pl->tile_rows < p.G) return false;                 // a group does not fit a stage
  pl->tiles = int((int64_t(p.NG) * p.G + pl->tile_rows - 1) / pl->tile_rows);
  const int ns = (p.Hm == 1) ? std::min(kQueryCols, p.S) : 1;
  pl->n_sub = (p.Hm == 1) ? (p.S + kQueryCols - 1) / kQueryCols : 1;
  const int64_t n_rests = int64_t(p.B) * scored_heads(p) * pl->n_sub;
  if (n_rests > 2 * kNumSMs) return false;
  pl->n_rests = int(n_rests);
  // CTAs per row set: one for each scope to select for, then doubled while there is more than a tile per warp;
  // more than 8 only where few clusters are wanted (a GPC holds one cluster of 16, two of 8).
  int c = 1;
  while (c < ns) c *= 2;
  while (c < (n_rests <= 2 ? 16 : 8) && pl->tiles > c * kClusterWarps && n_rests * 2 * c <= 120) c *= 2;
  pl->cluster = c;
  // A second stage per warp makes a CTA fill an SM's shared memory; only where there are SMs to spare.  So do many
  // keys (fp16 rows of rank 32: 6784).  All clusters have to be resident at once: two CTAs per SM, or, with a CTA's
  // shared memory above half of an SM's, two clusters of 8 per GPC.  (At B = 18, 8 heads, N = 8192, G = 1, rank 32, which
  // do not fit so, predictor and attention 42.0 us in clusters, 29.5 with the two kernels.)
  const int64_t ctas = n_rests * c;
  pl->depth = pl->tiles > c * kClusterWarps && ctas <= 100 && cta_smem(p, g_shift >= 0, 2) <= 227 * 1024 ? 2 : 1;
  pl->whole_sm = cta_smem(p, g_shift >= 0, pl->depth) > 113 * 1024;
  // Beyond two tiles per warp the streaming kernels on all SMs are the faster: at B = 4, N = 32768 (r = 32, G = 8,
  // four tiles per warp) 14.5 us of both against 12 to 18 for clusters, at B = 1, N = 65536 13.4 against 16.
  return ctas <= (pl->whole_sm ? 132 : 264) && pl->tiles <= 2 * c * kClusterWarps;
}

}  // namespace

bool score_select_cluster_supported(const Problem& p) { Plan pl; return plan(p, &pl); }
bool score_select_cluster_grid(const Problem& p, ClusterGrid* g) {
  Plan pl;
  if (!plan(p, &pl)) return false;
  *g = ClusterGrid{pl.n_rests, pl.cluster, pl.whole_sm};
  return true;
}

// On its own, not beside an attention, a cluster that selects for one scope of per-head metadata pays while every warp
// has one tile: at B = 1, 8 heads, N = 16384 (two) 10.2 us against 9.5 of the two kernels, at N = 4096 7.0 against
// 9.2.  With joint metadata it pays throughout, or nearly: one sequence of 4 heads at N = 25000 11.2 us against 10.6, but
// two at N = 20000 9.8 against 13.4, and fp32 rows of rank 64 at N = 5690, one scope, 10.0 against 13.1.
bool score_select_cluster_pays_alone(const Problem& p) {
  Plan pl;
  return plan(p, &pl) && (p.Hm == 1 || pl.tiles <= pl.cluster * kClusterWarps);
}

cudaError_t launch_score_select_cluster(const Problem& p, const void* q, const float* proj, const void* meta, float* scores,
                                        int32_t* group_idx, int32_t* n_selected, uint32_t* err, cudaStream_t st) {
  Plan pl;
  if (!plan(p, &pl)) return cudaErrorInvalidValue;
  ClusterArgs a;
  a.q = q; a.proj = proj; a.meta = static_cast<const unsigned char*>(meta); a.scores = scores;
  a.group_idx = group_idx; a.n_selected = n_selected;
  a.tile_rows = pl.tile_rows; a.tiles = pl.tiles; a.n_sub = pl.n_sub;
  a.depth = pl.depth;
  a.meta_scale = exp2f(float(p.meta_exp));
  a.err = err;
  switch (p.meta_dtype) {
    case KVSWAP_F16:
      return p.r == 16   ? launch_score_select_rows<KVSWAP_F16, 16>(p, a, pl.g_shift, pl.cluster, pl.n_rests, st)
             : p.r == 32 ? launch_score_select_rows<KVSWAP_F16, 32>(p, a, pl.g_shift, pl.cluster, pl.n_rests, st)
                         : launch_score_select_rows<KVSWAP_F16, 64>(p, a, pl.g_shift, pl.cluster, pl.n_rests, st);
    case KVSWAP_E4M3: return launch_score_select_rows<KVSWAP_E4M3, 32>(p, a, pl.g_shift, pl.cluster, pl.n_rests, st);
    default:
      return p.r == 16   ? launch_score_select_rows<KVSWAP_F32, 16>(p, a, pl.g_shift, pl.cluster, pl.n_rests, st)
             : p.r == 32 ? launch_score_select_rows<KVSWAP_F32, 32>(p, a, pl.g_shift, pl.cluster, pl.n_rests, st)
                         : launch_score_select_rows<KVSWAP_F32, 64>(p, a, pl.g_shift, pl.cluster, pl.n_rests, st);
  }
}

}  // namespace kvswap
