// Host side of the streaming scorer (score_stream.cuh): which shapes take it, its work split, the launch.
#include <algorithm>
#include <cmath>

#include "score_stream.cuh"

namespace kvswap {
namespace {

constexpr int kMaxRowsPerCta = 65535;                     // keeps a 16-bit counter from overflowing (G = 1)

struct Plan {
  int g_shift;                                            // log2 G, or -1: any G, through the warps' buffers
  int tile_rows, tiles_per_row, n_sub, n_rests;
  int ctas, vset_items, ctas_per_vset, base, rem;
  bool fused;
  bool counts;
};

// Launch geometry of the streaming scorer for `p`; false when the shape does not take it.
bool plan(const Problem& p, Plan* pl) {
  if (p.NG < 1 || !score_stream_rows(p) || p.meta_sn != p.r) return false;
  const int elem = p.meta_dtype == KVSWAP_F32 ? 4 : p.meta_dtype == KVSWAP_F16 ? 2 : 1;
  int g_shift = -1;
  for (int s = 0; s <= 5; ++s) if ((1 << s) == p.G) g_shift = s;
  if (multi_term(p)) g_shift = -1;
  // E4M3 metadata is offered for groups of a power of two and one term per score only
  if (g_shift < 0 && p.meta_dtype == KVSWAP_E4M3) return false;
  const int fit = score_stage_rows(g_shift < 0, p.r * elem);
  const int tile_rows = g_shift >= 0 ? fit : fit / p.G * p.G;
  if (tile_rows < p.G) return false;                      // a group does not fit a stage
  const int64_t rows_total = int64_t(p.NG) * p.G;
  const int64_t tiles_per_row = (rows_total + tile_rows - 1) / tile_rows;
  const int n_sub = (p.Hm == 1) ? (p.S + kScoreCols - 1) / kScoreCols : 1;
  const int64_t n_rests = int64_t(p.B) * scored_heads(p) * n_sub;
  const int64_t items = n_rests * tiles_per_row;
  if (items >= (int64_t(1) << 30)) return false;
  pl->g_shift = g_shift;
  pl->tile_rows = tile_rows;
  pl->tiles_per_row = int(tiles_per_row); pl->n_sub = n_sub; pl->n_rests = int(n_rests);
  // One CTA per SM.  When the row sets divide the SMs (almost) evenly every row set gets its own CTAs,
  // so that no CTA works for two of them; otherwise all CTAs share the items as one contiguous range.
  const int per_set = int(kNumSMs / std::max<int64_t>(1, n_rests));
  if (n_rests <= kNumSMs && n_rests * per_set * 20 >= int64_t(kNumSMs) * 19 && tiles_per_row >= int64_t(per_set) * kScoreWarps) {
    pl->vset_items = int(tiles_per_row);
    pl->ctas_per_vset = per_set;
    pl->ctas = int(n_rests) * per_set;
  } else {
    pl->vset_items = int(items);
    pl->ctas_per_vset = int(std::max<int64_t>(1, std::min<int64_t>(kNumSMs, (items + kScoreWarps - 1) / kScoreWarps)));
    pl->ctas = pl->ctas_per_vset;
  }
  const int warps = pl->ctas_per_vset * kScoreWarps;
  pl->base = pl->vset_items / warps;
  pl->rem = pl->vset_items % warps;
  // The CTA builds the low-rank queries itself when it touches few row sets and the adapter has the
  // layout build_queries() reads (d a multiple of 32 up to 128; at most eight terms per score).
  const int64_t cta_items = int64_t(pl->base + 1) * kScoreWarps;
  const int64_t sets_touched = (cta_items + tiles_per_row - 1) / tiles_per_row + 1;
  pl->fused = (p.d == 32 || p.d == 64 || p.d == 128) && sets_touched <= kMaxSets && (!multi_term(p) || p.Hkv <= kScoreCols);
  pl->counts = cta_items * tile_rows <= kMaxRowsPerCta;   // a CTA's counts stay below 2^16 per counter
  return true;
}

}  // namespace

bool score_stream_rows(const Problem& p) {
  switch (p.meta_dtype) {
    case KVSWAP_F16: return p.r == 16 || p.r == 32 || p.r == 64;
    case KVSWAP_E4M3: return p.r == 32;
    default: return p.r == 16 || p.r == 32 || p.r == 64;
  }
}
bool score_stream_supported(const Problem& p) { Plan pl; return plan(p, &pl); }
bool score_stream_fuses_query(const Problem& p) { Plan pl; return plan(p, &pl) && pl.fused; }
bool score_stream_counts_top_digit(const Problem& p) { Plan pl; return plan(p, &pl) && pl.counts; }
// CTAs of the scorer that neither forms queries nor counts (kDeep, queries found in memory), where it leaves half of an SM's
// registers: 512 threads of 47 to 60 for fp16 rows of 16 or 32 and groups of 2 to 32, 52 to 60 for 8-bit rows and groups
// of 8 to 32 (fp16 rows of 64, fp32 rows, groups of one or of other lengths: 67 to 127).  Else 0.
int score_stream_light_ctas(const Problem& p) {
  Plan pl;
  if (!plan(p, &pl) || !pl.fused) return 0;
  const bool light = p.meta_dtype == KVSWAP_F16 ? p.r <= 32 && pl.g_shift >= 1 : p.meta_dtype == KVSWAP_E4M3 && pl.g_shift >= 3;
  return light ? pl.ctas : 0;
}
void score_stream_row_sets(const Problem& p, int* n_rests, int* n_sub) {
  Plan pl;
  const bool ok = plan(p, &pl);
  *n_rests = ok ? pl.n_rests : 0;
  *n_sub = ok ? pl.n_sub : 1;
}

cudaError_t launch_score_stream(const Problem& p, const void* q, const float* proj, const float* uq, const void* meta,
                                float* scores, uint32_t* top_hist, uint32_t* err, cudaStream_t st) {
  Plan pl;
  if (!plan(p, &pl)) return cudaErrorInvalidValue;
  if (top_hist != nullptr && !pl.counts) return cudaErrorInvalidValue;
  // With q == NULL the queries come from `uq` even where the kernel could build them.
  if (q == nullptr) pl.fused = false;
  if (pl.fused ? (proj == nullptr) : (uq == nullptr)) return cudaErrorInvalidValue;
  StreamArgs a;
  a.q = q; a.proj = proj; a.uq = uq; a.meta = static_cast<const unsigned char*>(meta); a.scores = scores;
  a.top_hist = top_hist;
  a.tile_rows = pl.tile_rows;
  a.tiles_per_row = pl.tiles_per_row; a.n_sub = pl.n_sub; a.n_rests = pl.n_rests;
  a.vset_items = pl.vset_items; a.ctas_per_vset = pl.ctas_per_vset; a.base = pl.base; a.rem = pl.rem;
  a.meta_scale = exp2f(float(p.meta_exp));
  a.err = err;
  switch (p.meta_dtype) {
    case KVSWAP_F16:
      return p.r == 16   ? launch_score_stream_rows<KVSWAP_F16, 16>(p, a, pl.g_shift, pl.fused, pl.ctas, st)
             : p.r == 32 ? launch_score_stream_rows<KVSWAP_F16, 32>(p, a, pl.g_shift, pl.fused, pl.ctas, st)
                         : launch_score_stream_rows<KVSWAP_F16, 64>(p, a, pl.g_shift, pl.fused, pl.ctas, st);
    case KVSWAP_E4M3: return launch_score_stream_rows<KVSWAP_E4M3, 32>(p, a, pl.g_shift, pl.fused, pl.ctas, st);
    default:
      return p.r == 16   ? launch_score_stream_rows<KVSWAP_F32, 16>(p, a, pl.g_shift, pl.fused, pl.ctas, st)
             : p.r == 32 ? launch_score_stream_rows<KVSWAP_F32, 32>(p, a, pl.g_shift, pl.fused, pl.ctas, st)
                         : launch_score_stream_rows<KVSWAP_F32, 64>(p, a, pl.g_shift, pl.fused, pl.ctas, st);
  }
}

}  // namespace kvswap
