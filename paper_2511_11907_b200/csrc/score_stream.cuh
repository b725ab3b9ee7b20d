// K2, streaming tensor-core scorer: low-rank query (Eq. 1), token scoring, head aggregation and group
// ReduceMax (Sec. 4.3) for metadata rows that are dense in memory: fp16 of rank 16, 32 or 64, E4M3 of rank
// 32, fp32 of rank 16, 32 or 64 (there with groups of up to 16).  The arithmetic of a block of rows is in score_tile.cuh.
//
// One persistent CTA per SM, 16 warps.  Work item = (sequence b, metadata head hm, block of 8 scopes, tile
// of up to 4 KB of rows); items are numbered with the tile fastest, a "row set" is the items of one
// (b, hm, scope block).  Every warp takes an equal contiguous share of tiles and pulls them into its own
// ring of shared-memory stages with bulk asynchronous copies (cp.async.bulk + mbarrier, bounded waits),
// kDepth tiles in flight per warp; where the inputs are settled the first tiles are requested before the dependency wait.
//
// With G a power of two up to 32 (template GS = log2 G) a finished group score leaves the registers at
// once.  Every other G that fits a tile (GS = -1) goes through a small shared-memory buffer of the warp,
// [scope][token]; so do scores that sum a term on every metadata head (per-head
// metadata under the all-heads scope): there a warp runs through the heads of up to kMultiTiles tiles,
// adding each head's products to the buffer, before it takes the maxima.
//
// Ranks 16 and 64, fp32 rows, other group sizes and several terms used to take a general fp32-pipe kernel, a
// kernel for the queries and a TopK of one CTA per list.  One layer at B = 2, N = 32768, r = 64, all-heads
// scope: 22 us scorer and 5 us TopK before, 10 and 4 us now; 26 layers of B = 12, N = 3830, r = 64,
// G = 4: 1572 -> 909 us; 24 layers of B = 5, N = 2244, fp32 r = 32: 584 -> 338 us.
//
// The CTA computes the summed low-rank queries of its row sets itself where it can (`fused`):
//     u[b, row, :] = sum over the KV heads g of the row's scope of (sum_{h: g(h) = g} q[b, h, :]) A_g
// which removes the separate low-rank query kernel and its launch dependency from the call.
//
// While it scores, the CTA counts the leading 12 bits of every group score's key in a
// shared-memory histogram (16-bit counters, 8 columns = the scopes of its first row set) and adds
// the non-zero counters to the global histograms at the end, four counters per 64-bit atomic (the
// global histograms have the same packed layout; a row has at most 65535 groups on this path).
// Scores of row sets that do not fit the 8 columns are counted in global memory directly.  The
// global histograms are zero on entry and left zero by the TopK kernel that starts from them
// (topk_select.cu; kvswap_workspace_init clears them once).
#pragma once

#include "async_copy.cuh"
#include "common.cuh"
#include "lowrank_query.cuh"
#include "score_tile.cuh"
#include "topk_keys.cuh"

namespace kvswap {

constexpr int kScoreWarps = kQueryWarps;                  // 16
constexpr int kScoreThreads = kScoreWarps * 32;
constexpr int kScoreDepth = 2;
constexpr int kScoreCols = kQueryCols;                    // scores per metadata row and instruction
constexpr int kHistWords = kScoreCols * kKeyTopBins / 2;  // two 16-bit counters per word
constexpr int kMaxSets = 4;                               // row sets one CTA may touch when it builds the queries itself
constexpr int kMultiTiles = 8;                            // tiles whose scores a warp sums over the heads together

// How a CTA works: kForms builds the low-rank queries and counts leading digits, kCounts finds the queries in memory, kDeep
// finds them too, does not count and has a third stage in the counters' place (a decode step whose select does without:
// topk_beside.cuh).  It flushes nothing, and with three stages a warp has nearly all of its 3.5 tiles in flight before its
// dependency wait: 14.7 -> 11.8 us as a launch of its own at B = 4, N = 131072.
enum ScoreMode { kForms, kCounts, kDeep };

template <int META, int R, int GS, ScoreMode MODE>
struct ScoreSmem {
  static constexpr int kDepth = MODE == kDeep ? kScoreDepth + 1 : kScoreDepth;
  unsigned char tiles[kScoreWarps * kDepth * ScoreStage<META, R, GS>::kBytes];   // 128 KB of stages, or 96; kDeep: 192 or 144
  uint32_t hist[MODE == kDeep ? 4 : kHistWords];          // 64 KB
  unsigned long long full[kScoreWarps * kDepth];
  float urow[MODE == kForms ? kMaxSets : 1][MODE == kForms ? kScoreCols * R : 4];   // summed low-rank queries per row set of the CTA
  static constexpr int kScratch = MODE == kForms ? kQuerySumFloats + kQueryPartFloats : 4;
  // scratch of build_queries (qsum, then upart), afterwards the warps' score buffers
  static constexpr int kBuffers = GS >= 0 ? 0 : kScoreWarps * kScoreCols * generic_pitch(ScoreStage<META, R, GS>::kRows);
  float sc[kBuffers > kScratch ? kBuffers : kScratch];
};

struct StreamArgs {
  const void* q;            // fused: [B, H_q, d] q_dtype
  const float* proj;        // fused: [H_kv, d, r]
  const float* uq;          // not fused: [B, Su, r] from the low-rank query kernel
  const unsigned char* meta;
  float* scores;
  uint32_t* top_hist;       // NULL, or [B * S, 4096] 16-bit counters, two per word
  int tile_rows;            // rows of a whole tile: ScoreStage::kRows, GS = -1: the multiple of G that fits
  int tiles_per_row, n_sub, n_rests;
  int vset_items, ctas_per_vset;   // work split: virtual sets of vset_items items, each shared by ctas_per_vset CTAs
  int base, rem;            // tiles per warp within a virtual set: base, +1 for the first rem warps
  float meta_scale;         // 2^meta_exp (1 unless the metadata is 8-bit)
  uint32_t* err;
};

template <int META, int R, int GS, ScoreMode MODE>   // GS = log2(G), 0..5, or -1
__global__ void __launch_bounds__(kScoreThreads, 1)
score_stream_kernel(Problem p, StreamArgs a) {
  constexpr uint32_t kFull = 0xffffffffu;
  constexpr bool FUSED = MODE == kForms;
  using Smem = ScoreSmem<META, R, GS, MODE>;
  constexpr int kRowBytes = MetaRows<META, R>::kRowBytes, kElem = MetaRows<META, R>::kElem;
  constexpr int kStageBytes = ScoreStage<META, R, GS>::kBytes, kStageRows = ScoreStage<META, R, GS>::kRows;
  constexpr int kDepth = Smem::kDepth, kWarps = kScoreWarps, kThreads = kScoreThreads, kCols = kScoreCols;
  extern __shared__ __align__(128) unsigned char dyn[];
  auto* sm = reinterpret_cast<Smem*>(dyn);
  const bool counts = MODE != kDeep && a.top_hist != nullptr;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rq = lane >> 2, qt = lane & 3;
  if (lane == 0) {                                  // every warp sets up its own stages
    for (int s = 0; s < kDepth; ++s) mbar_init(smem_addr(&sm->full[warp * kDepth + s]), 1);
    mbar_init_fence();
  }
  if (counts) {
    uint4* H = reinterpret_cast<uint4*>(sm->hist);
    for (int i = threadIdx.x; i < kHistWords / 4; i += kThreads) H[i] = make_uint4(0u, 0u, 0u, 0u);
  }
  __syncwarp();

  // ---- this warp's contiguous share of the work items -----------------------------------------------------
  const int tile_rows = GS >= 0 ? kStageRows : a.tile_rows;
  const bool multi = GS < 0 && multi_term(p);
  const int n_terms = multi ? p.Hkv : 1;            // stages of one tile
  const int rows_total = p.NG * p.G;
  const int hm_count = scored_heads(p);
  const int vset = blockIdx.x / a.ctas_per_vset, cta_in = blockIdx.x - vset * a.ctas_per_vset;
  auto share_first = [&](int w) { return vset * a.vset_items + w * a.base + min(w, a.rem); };
  const int wi = cta_in * kWarps + warp;
  const int first = share_first(wi);
  const int my_tiles = a.base + (wi < a.rem ? 1 : 0);
  const int my_stages = my_tiles * n_terms;
  const int cta_first = share_first(cta_in * kWarps), cta_last = share_first((cta_in + 1) * kWarps);   // [first, last) of the CTA
  const int rest0 = cta_first / a.tiles_per_row;                                  // the CTA's first row set
  const int n_sets = (cta_last > cta_first) ? (cta_last - 1) / a.tiles_per_row - rest0 + 1 : 0;
  const int ns_cols = (p.Hm == 1) ? min(kCols, p.S) : 1;                          // histogram columns per row set

  // Cursor over the warp's stages: tile by tile; with several terms per score, block after block of at most
  // kMultiTiles tiles of one row set, head by head inside a block.
  struct Cursor { int tile, rest, left, block, term, in; };   // left: tiles from the block's first one on; in: tile within the block
  auto block_len = [&](const Cursor& c) { return multi ? min(min(kMultiTiles, c.left), a.tiles_per_row - c.tile) : 1; };
  auto start = [&](Cursor& c) {
    c.tile = first % a.tiles_per_row; c.rest = first / a.tiles_per_row; c.left = my_tiles; c.term = 0; c.in = 0;
    c.block = block_len(c);
  };
  auto advance = [&](Cursor& c) {
    if (multi) {
      if (++c.in < c.block) return;
      c.in = 0;
      if (++c.term < n_terms) return;
      c.term = 0;
    }
    c.tile += c.block; c.left -= c.block;
    if (c.tile == a.tiles_per_row) { c.tile = 0; ++c.rest; }
    c.block = block_len(c);
  };
  Cursor f, c;                                      // next stage to request, next stage to consume
  start(f);
  c = f;

  const uint32_t ring = smem_addr(sm->tiles) + uint32_t(warp) * kDepth * kStageBytes;
  const unsigned char* f_base = nullptr;            // metadata of the fill cursor's (sequence, head)
  int f_base_rest = -1;
  auto fill = [&](int stage) {
    if (lane == 0) {
      if (f.rest != f_base_rest) {                  // divisions only when the cursor enters a new row set
        f_base_rest = f.rest;
        const int bh = f.rest / a.n_sub;
        f_base = a.meta + (int64_t(bh / hm_count) * p.meta_sb + int64_t(bh % hm_count) * p.meta_sh) * kElem;
      }
      const int tile = f.tile + f.in;
      const int rows = min(tile_rows, rows_total - tile * tile_rows);
      const uint32_t bar = smem_addr(&sm->full[warp * kDepth + stage]);
      const unsigned char* src = f_base + int64_t(tile) * tile_rows * kRowBytes;
      if (multi) src += int64_t(f.term) * p.meta_sh * kElem;
      mbar_arrive_expect_tx(bar, uint32_t(rows) * kRowBytes);
      bulk_g2s(ring + uint32_t(stage) * kStageBytes, src, uint32_t(rows) * kRowBytes, bar);
    }
    advance(f);
  };

  // ---- dependency wait, first tiles and the summed low-rank queries --------------------------------------
  // Without KVSWAP_INPUTS_SETTLED any input may be the previous kernel's output: wait first.  With it, only this
  // kernel's writes (scores and histograms, which the previous call's TopK may still read) have to wait, so the
  // queries are built while that kernel finishes.  Queries found in memory (not FUSED) are the previous kernel's in
  // either case, but that kernel let this one start when all before it was complete, or the metadata is settled:
  // its first tiles go out ahead of the wait.
  const bool settled = (p.flags & KVSWAP_INPUTS_SETTLED) != 0;
  if (FUSED && !settled) pdl_wait();
  for (int k = 0; k < kDepth && k < my_stages; ++k) fill(k);
  if constexpr (FUSED) {
    for (int s = 0; s < n_sets; ++s)
      build_queries<0, R>(p, a.q, a.proj, row_set(p, rest0 + s, a.n_sub), sm->sc, sm->sc + kQuerySumFloats, sm->urow[s]);
  }
  if (!FUSED || settled) pdl_wait();
  pdl_trigger();
  if constexpr (!FUSED) __syncthreads();             // the histogram is cleared (the fused path has synchronised)

  ScoreQuery<META, R> query;
  query.inv = 1.f;
  int cur_rest = -1, cur_term = -1;
  float* my_row = a.scores;                         // scores row of this lane's scope (scope rq of the current block)
  uint32_t* my_hist = nullptr;                      // its global histogram
  int my_col = -1;                                  // its column of the shared-memory histogram, or -1
  bool scope_ok = false;                            // the lane's scope exists
  float* const sc = sm->sc + (GS >= 0 ? 0 : warp * kCols * generic_pitch(kStageRows));
  int stage = 0;
  uint32_t phase = 0;
  bool timed_out = false;
  // A finished group score leaves the registers at once: to the score row and, as one count, to the
  // histogram of its key's leading digit.
  auto publish = [&](float* dst, float x) {
    x += 0.f;                                       // -0 becomes +0: the TopK that follows relies on it
    *dst = x;
    if (counts) {
      const uint32_t bin = score_key_top(x);
      if (my_col >= 0) {
        atomicAdd(&sm->hist[(my_col * kKeyTopBins + int(bin)) >> 1], 1u << ((bin & 1u) << 4));
      } else {
        atomicAdd(my_hist + (bin >> 1), 1u << ((bin & 1u) << 4));
      }
    }
  };
  for (int k = 0; k < my_stages; ++k) {
    const int tile = c.tile + c.in;
    if (c.rest != cur_rest || c.term != cur_term) { // new row set or term: rebuild the row operand
      const RowSet rs = row_set(p, c.rest, a.n_sub);
      // this lane supplies the query of row rq: scope sub * 8 + rq (joint), head hm or term (row 0 only)
      if constexpr (FUSED) {
        const float* u = sm->urow[c.rest - rest0] + qt * (R / 4);
        if (!multi) {
          query.set(u + rq * R, a.meta_scale);
        } else {
          float v[R / 4];
#pragma unroll
          for (int i = 0; i < R / 4; ++i) v[i] = (rq == 0) ? u[c.term * R + i] : 0.f;
          query.set(v, a.meta_scale);
        }
      } else {
        const int urow = (p.Hm == 1) ? rs.sub * kCols + rq : multi ? c.term : rs.hm;
        const bool have = (p.Hm == 1) ? (urow < p.S) : (rq == 0);
        const float4* ur = reinterpret_cast<const float4*>(a.uq + (int64_t(rs.b) * p.Su + urow) * R + qt * (R / 4));
        float v[R / 4];
#pragma unroll
        for (int i = 0; i < R / 16; ++i) {
          const float4 x = have ? ur[i] : make_float4(0.f, 0.f, 0.f, 0.f);
          v[4 * i] = x.x; v[4 * i + 1] = x.y; v[4 * i + 2] = x.z; v[4 * i + 3] = x.w;
        }
        query.set(v, a.meta_scale);
      }
      cur_term = c.term;
      if (c.rest != cur_rest) {
        cur_rest = c.rest;
        const int s0 = (p.Hm == 1) ? rs.sub * kCols : rs.hm;
        const int ns_cur = (p.Hm == 1) ? min(kCols, p.S - s0) : 1;
        scope_ok = rq < ns_cur;
        const int64_t prob = int64_t(rs.b) * p.S + s0 + (scope_ok ? rq : 0);
        my_row = a.scores + prob * p.score_pitch;
        if (counts) {
          my_hist = a.top_hist + prob * (kKeyTopBins / 2);
          const int col = (c.rest - rest0) * ns_cols + (multi ? 0 : rq);
          my_col = ((scope_ok || multi) && col < kCols) ? col : -1;
        }
      }
    }
    if (!__all_sync(kFull, mbar_wait(smem_addr(&sm->full[warp * kDepth + stage]), phase))) { timed_out = true; break; }
    const int rows = min(tile_rows, rows_total - tile * tile_rows);   // a multiple of G: groups never straddle tiles
    const uint32_t base = ring + uint32_t(stage) * kStageBytes + score_lane_offset<META, R>(lane);
    if (!multi) {
      float* dst = my_row + (GS >= 0 ? (tile * tile_rows) >> GS : tile * (tile_rows / p.G));   // first group of the tile
      score_tile_groups<META, R, GS, kStageRows>(base, rows, lane, query, p.G, scope_ok, sc,
                                                 [&](int gi, float x) { publish(dst + gi, x); });
    } else if constexpr (GS < 0) {
      // the one scope's token scores of the whole block of tiles, summed over the terms
      float* s = sc + c.in * tile_rows;
      for (int it = 0; it * 8 < rows; ++it) {
        float x0, x1;
        score_rows8<META, R>(base + uint32_t(it) * 8u * kRowBytes, query, &x0, &x1);
        const int i = it * 8 + 2 * qt;                           // (a tile's rows need not be whole reads)
        if (rq == 0 && i < rows) s[i] = (c.term == 0 ? 0.f : s[i]) + x0 * query.inv;
        if (rq == 0 && i + 1 < rows) s[i + 1] = (c.term == 0 ? 0.f : s[i + 1]) + x1 * query.inv;
      }
      if (c.term == n_terms - 1 && c.in == c.block - 1) {         // the block's sums are complete
        __syncwarp();
        const int n_groups = (min((c.tile + c.block) * tile_rows, rows_total) - c.tile * tile_rows) / p.G;
        float* dst = my_row + c.tile * (tile_rows / p.G);
        for (int gi = lane; gi < n_groups; gi += 32) {
          const float* t = sc + gi * p.G;
          float m = t[0];
          for (int i = 1; i < p.G; ++i) m = fmaxf(m, t[i]);
          publish(dst + gi, m);
        }
      }
    }
    __syncwarp();                                   // every lane has read the stage (and the buffer)
    advance(c);
    if (k + kDepth < my_stages) fill(stage);
    if (++stage == kDepth) { stage = 0; phase ^= 1u; }
  }
  if (timed_out) {
    if (lane == 0 && a.err) atomicExch(a.err, kDevTimeoutFull);
    for (int s = 0; s < kDepth; ++s) {              // bounded chance for copies in flight to land
      mbar_wait(smem_addr(&sm->full[warp * kDepth + s]), 0);
      mbar_wait(smem_addr(&sm->full[warp * kDepth + s]), 1);
    }
  }

  // ---- the CTA's counts join the global histograms --------------------------------------------------------
  if (counts) {
    __syncthreads();
    for (int i = threadIdx.x; i < kHistWords / 4; i += kThreads) {
      const uint4 v = reinterpret_cast<const uint4*>(sm->hist)[i];
      if ((v.x | v.y | v.z | v.w) == 0u) continue;
      const int col = (i * 8) / kKeyTopBins;                                      // 8 counters per vector
      const int rest = rest0 + col / ns_cols, in_set = col % ns_cols;
      if (rest >= a.n_rests) continue;
      const RowSet rs = row_set(p, rest, a.n_sub);
      const int s = (p.Hm == 1) ? rs.sub * kCols + in_set : rs.hm;
      if (s >= p.S) continue;
      unsigned long long* H = reinterpret_cast<unsigned long long*>(
          a.top_hist + (int64_t(rs.b) * p.S + s) * (kKeyTopBins / 2) + ((i * 4) % (kKeyTopBins / 2)));
      const unsigned long long lo = (unsigned long long)v.x | ((unsigned long long)v.y << 32);
      const unsigned long long hi = (unsigned long long)v.z | ((unsigned long long)v.w << 32);
      if (lo != 0ull) atomicAdd(H, lo);
      if (hi != 0ull) atomicAdd(H + 1, hi);
    }
  }
}

// One launch of the kernel for a stored type and rank; `g_shift` = log2 G or -1.  Instantiated one pair per
// translation unit (score_stream_*.cu).
template <int META, int R>
cudaError_t launch_score_stream_rows(const Problem& p, const StreamArgs& a, int g_shift, bool fused, int ctas, cudaStream_t st);

template <> cudaError_t launch_score_stream_rows<KVSWAP_F16, 16>(const Problem&, const StreamArgs&, int, bool, int, cudaStream_t);
template <> cudaError_t launch_score_stream_rows<KVSWAP_F16, 32>(const Problem&, const StreamArgs&, int, bool, int, cudaStream_t);
template <> cudaError_t launch_score_stream_rows<KVSWAP_F16, 64>(const Problem&, const StreamArgs&, int, bool, int, cudaStream_t);
template <> cudaError_t launch_score_stream_rows<KVSWAP_E4M3, 32>(const Problem&, const StreamArgs&, int, bool, int, cudaStream_t);
template <> cudaError_t launch_score_stream_rows<KVSWAP_F32, 16>(const Problem&, const StreamArgs&, int, bool, int, cudaStream_t);
template <> cudaError_t launch_score_stream_rows<KVSWAP_F32, 32>(const Problem&, const StreamArgs&, int, bool, int, cudaStream_t);
template <> cudaError_t launch_score_stream_rows<KVSWAP_F32, 64>(const Problem&, const StreamArgs&, int, bool, int, cudaStream_t);

template <int META, int R, int GS>
cudaError_t launch_score_stream_gs(const Problem& p, const StreamArgs& a, bool fused, int ctas, cudaStream_t st) {
  auto go = [&](auto kern, auto mode) -> cudaError_t {
    using Smem = ScoreSmem<META, R, GS, decltype(mode)::value>;
    static_assert(sizeof(Smem) + 128 <= 227 * 1024, "shared memory of one CTA");
    const size_t smem = sizeof(Smem) + 128;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
    return launch_pdl(kern, dim3(ctas), dim3(kScoreThreads), smem, st, p, a);
  };
  return fused                   ? go(score_stream_kernel<META, R, GS, kForms>, std::integral_constant<ScoreMode, kForms>())
         : a.top_hist != nullptr ? go(score_stream_kernel<META, R, GS, kCounts>, std::integral_constant<ScoreMode, kCounts>())
                                 : go(score_stream_kernel<META, R, GS, kDeep>, std::integral_constant<ScoreMode, kDeep>());
}

#define KVSWAP_SCORE_STREAM_ROWS(META, R)                                                                            \
  template <>                                                                                                        \
  cudaError_t launch_score_stream_rows<META, R>(const Problem& p, const StreamArgs& a, int g_shift, bool fused,      \
                                                int ctas, cudaStream_t st) {                                         \
    switch (g_shift) {                                                                                               \
      case 0: return launch_score_stream_gs<META, R, 0>(p, a, fused, ctas, st);                                      \
      case 1: return launch_score_stream_gs<META, R, 1>(p, a, fused, ctas, st);                                      \
      case 2: return launch_score_stream_gs<META, R, 2>(p, a, fused, ctas, st);                                      \
      case 3: return launch_score_stream_gs<META, R, 3>(p, a, fused, ctas, st);                                      \
      case 4: return launch_score_stream_gs<META, R, 4>(p, a, fused, ctas, st);                                      \
      case 5: return launch_score_stream_gs<META, R, 5>(p, a, fused, ctas, st);                                      \
      default:                                                                                                       \
        if constexpr (META == KVSWAP_E4M3) return cudaErrorInvalidValue;                                              \
        else return launch_score_stream_gs<META, R, -1>(p, a, fused, ctas, st);                                      \
    }                                                                                                                \
  }

}  // namespace kvswap
