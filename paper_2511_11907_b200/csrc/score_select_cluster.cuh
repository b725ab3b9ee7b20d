// The predictor of a short context in one kernel: low-rank query, token scores, group ReduceMax and TopK of
// one row set -- (sequence, metadata head, block of 8 scopes) -- by one cluster of CTAs (Sec. 4.3).
//
// The streaming scorer and the TopK behind it (score_stream.cuh, topk_parts.cuh) are built for bandwidth: with
// a megabyte of metadata per layer each takes 5 us, nearly all of it launch, dependency wait, clearing and
// flushing of histograms and barriers.  Here a cluster scores the row set's tiles (the arithmetic of
// score_tile.cuh, the same bits), every finished group score goes as a key straight into the shared memory of
// the CTA that will select for its scope (scope i of the set: rank i), and after one cluster barrier that CTA
// selects from its shared memory (topk_smem.cuh).  Scores, histograms and their clearing never touch memory.
// The cluster also shares the build of the low-rank queries: a warp takes a 32-channel piece of one head and
// sends its partial products to every CTA, so each adapter row is read once per cluster instead of once per CTA.
// Bound by latency: launch, the queries, one round of loads, two cluster barriers, the select's phases.  A call
// at 8 KV heads, r = 32, G = 8: 7.5 us against 11.6 of the two kernels at B = 1, N = 4096, 9.6 against 12.1 at
// N = 16384, 9.3 against 13.7 at B = 16, N = 4096; 0.5 of it is the wait ahead of the first request.
//
// CTA = 16 warps.  Tiles are dealt to the cluster's warps in contiguous shares, each pulled through the warp's
// own ring of `depth` stages with bulk asynchronous copies (bounded waits).
#pragma once

#include "async_copy.cuh"
#include "cluster.cuh"
#include "common.cuh"
#include "lowrank_query.cuh"
#include "score_tile.cuh"
#include "topk_smem.cuh"

namespace kvswap {

constexpr int kClusterWarps = 16;
constexpr int kClusterThreads = kClusterWarps * 32;
static_assert(kClusterThreads == kSelectThreads && kClusterThreads == kQueryThreads, "one CTA does all three");

struct ClusterArgs {
  const void* q;            // [B, H_q, d] q_dtype
  const float* proj;        // [H_kv, d, r]
  const unsigned char* meta;
  float* scores;            // NULL, or the caller's [B, S, NG]
  int32_t* group_idx;
  int32_t* n_selected;
  int tile_rows, tiles, n_sub;
  int depth;                // stages per warp
  float meta_scale;
  uint32_t* err;
};

// Shared memory of a CTA: fixed part, then depth stages per warp, then the keys of one scope.
template <int META, int R, int GS>
struct ClusterSmem {
  SelectScratch select;
  float upart[(R + 31) / 32][kQueryPartFloats];           // partial products of the queries, per 32 columns
  float urow[kQueryCols * R];
  uint32_t key_min, key_max;                              // of the scope this CTA selects for
  unsigned long long full[kClusterWarps * 2];
  float sc[GS >= 0 ? 4 : kClusterWarps * kQueryCols * generic_pitch(ScoreStage<META, R, GS>::kRows)];
};

template <int META, int R, int GS>
__global__ void __launch_bounds__(kClusterThreads, 2)
score_select_cluster_kernel(Problem p, ClusterArgs a) {
  constexpr uint32_t kAll = 0xffffffffu;
  constexpr int kRowBytes = MetaRows<META, R>::kRowBytes, kElem = MetaRows<META, R>::kElem;
  constexpr int kStageBytes = ScoreStage<META, R, GS>::kBytes, kStageRows = ScoreStage<META, R, GS>::kRows;
  extern __shared__ __align__(128) unsigned char dyn[];
  using Smem = ClusterSmem<META, R, GS>;
  auto* sm = reinterpret_cast<Smem*>(dyn);
  constexpr uint32_t kFixed = (uint32_t(sizeof(Smem)) + 127u) & ~127u;
  unsigned char* stages = dyn + kFixed;
  uint32_t* keys = reinterpret_cast<uint32_t*>(stages + size_t(kClusterWarps) * a.depth * kStageBytes);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rq = lane >> 2, qt = lane & 3;
  const int rank = int(cluster_rank()), n_ctas = int(cluster_size());
  const int rest = blockIdx.x / n_ctas;
  const RowSet rs = row_set(p, rest, a.n_sub);
  if (threadIdx.x == 0) { sm->key_min = 0xffffffffu; sm->key_max = 0u; }
  cluster_arrive();                                     // peers may be written to once all have started
  if (lane == 0) {
    for (int s = 0; s < a.depth; ++s) mbar_init(smem_addr(&sm->full[warp * 2 + s]), 1);
    mbar_init_fence();
  }
  for (int i = threadIdx.x; i < kKeyTopBins; i += kClusterThreads) sm->select.hist[i] = 0;
  __syncwarp();
  // Without KVSWAP_INPUTS_SETTLED any input -- query, adapter, metadata -- may be the previous kernel's output.
  const bool settled = (p.flags & KVSWAP_INPUTS_SETTLED) != 0;
  if (!settled) { pdl_wait(); pdl_trigger(); }

  // ---- this warp's contiguous share of the tiles; the first ones are requested at once -------------------------
  const int tile_rows = GS >= 0 ? kStageRows : a.tile_rows;
  const int rows_total = p.NG * p.G;
  const int n_warps = n_ctas * kClusterWarps, wi = rank * kClusterWarps + warp;
  const int base_tiles = a.tiles / n_warps, rem = a.tiles - base_tiles * n_warps;
  const int first = wi * base_tiles + min(wi, rem), my_tiles = base_tiles + (wi < rem ? 1 : 0);
  const unsigned char* src = a.meta + (int64_t(rs.b) * p.meta_sb + int64_t(rs.hm) * p.meta_sh) * kElem;
  const uint32_t ring = smem_addr(stages) + uint32_t(warp) * a.depth * kStageBytes;
  auto fill = [&](int k, int stage) {
    if (lane == 0) {
      const int tile = first + k;
      const int rows = min(tile_rows, rows_total - tile * tile_rows);
      const uint32_t bar = smem_addr(&sm->full[warp * 2 + stage]);
      mbar_arrive_expect_tx(bar, uint32_t(rows) * kRowBytes);
      bulk_g2s(ring + uint32_t(stage) * kStageBytes, src + int64_t(tile) * tile_rows * kRowBytes,
               uint32_t(rows) * kRowBytes, bar);
    }
  };
  for (int k = 0; k < a.depth && k < my_tiles; ++k) fill(k, k);

  // ---- this warp's pieces of the queries: item = (32 columns, KV head, 32 channels) ---------------------------
  // The adapter's rows are requested ahead of the cluster barrier.  The products are added in the order of
  // build_queries (lowrank_query.cuh): the same bits.
  constexpr int kPasses = (R + 31) / 32, kLoads = (R == 16) ? 16 : 32;
  const QueryTerms terms = query_terms(p, rs);
  const int ch_shift = query_chunk_shift(p), n_items = terms.n_terms << ch_shift;
  const int ch0 = (R == 16) ? (lane >> 4) : 0, step = (R == 16) ? 2 : 1, col = (R == 16) ? (lane & 15) : lane;
  float adapter[kLoads];
  auto request = [&](int item) {
    const int it = item % n_items, pass = item / n_items;
    const int64_t row = int64_t(terms.head0 + (it >> ch_shift)) * p.d + (it & ((1 << ch_shift) - 1)) * 32 + ch0;
    const float* P = a.proj + row * R + pass * 32 + col;
#pragma unroll
    for (int cc = 0; cc < kLoads; ++cc) adapter[cc] = P[cc * step * R];
  };
  int item = rank + n_ctas * warp;
  if (item < n_items * kPasses) request(item);
  cluster_wait();                                       // every CTA of the cluster has started
  for (; item < n_items * kPasses; item += n_ctas * kClusterWarps) {
    const int it = item % n_items, pass = item / n_items;
    const float qs = query_sum(p, a.q, rs.b, terms.head0 + (it >> ch_shift), (it & ((1 << ch_shift) - 1)) * 32 + lane);
    float acc = 0.f;
#pragma unroll
    for (int cc = 0; cc < kLoads; ++cc) acc = fmaf(__shfl_sync(kAll, qs, cc * step + ch0), adapter[cc], acc);
    if constexpr (R == 16) acc += __shfl_xor_sync(kAll, acc, 16);
    const uint32_t dst = smem_addr(&sm->upart[pass][it * 32 + lane]);
    for (int r = 0; r < n_ctas; ++r) cluster_store(cluster_map(dst, uint32_t(r)), __float_as_uint(acc));
    if (item + n_ctas * kClusterWarps < n_items * kPasses) request(item + n_ctas * kClusterWarps);
  }
  cluster_arrive();
  cluster_wait();                                       // the partial products have arrived
  for (int i = threadIdx.x; i < kQueryCols * R; i += kClusterThreads)
    sm->urow[i] = query_entry(sm->upart[(i % R) / 32], i / R, i % R, terms.n_terms, ch_shift, terms.row_per_term, 0.f);
  __syncthreads();
  if (settled) { pdl_wait(); pdl_trigger(); }

  // ---- scores: each key to the CTA that selects for its scope ----------------------------------------------------
  const int s0 = (p.Hm == 1) ? rs.sub * kQueryCols : rs.hm;
  const int ns = (p.Hm == 1) ? min(kQueryCols, p.S - s0) : 1;
  const bool scope_ok = rq < ns;
  ScoreQuery<META, R> query;
  query.set(sm->urow + rq * R + qt * (R / 4), a.meta_scale);
  const uint32_t owner = uint32_t(scope_ok ? rq : 0);
  const uint32_t dst_keys = cluster_map(smem_addr(keys), owner);
  uint32_t key_min = 0xffffffffu, key_max = 0u;
  float* const out_row = a.scores ? a.scores + (int64_t(rs.b) * p.S + s0 + (scope_ok ? rq : 0)) * p.NG : nullptr;
  float* const sc = sm->sc + (GS >= 0 ? 0 : warp * kQueryCols * generic_pitch(kStageRows));
  bool timed_out = false;
  int stage = 0;
  uint32_t phase = 0;
  for (int k = 0; k < my_tiles; ++k) {
    if (!__all_sync(kAll, mbar_wait(smem_addr(&sm->full[warp * 2 + stage]), phase))) { timed_out = true; break; }
    const int tile = first + k;
    const int rows = min(tile_rows, rows_total - tile * tile_rows);
    const int g0 = GS >= 0 ? (tile * tile_rows) >> (GS >= 0 ? GS : 0) : tile * (tile_rows / p.G);
    score_tile_groups<META, R, GS, kStageRows>(
        ring + uint32_t(stage) * kStageBytes + score_lane_offset<META, R>(lane), rows, lane, query, p.G, scope_ok, sc,
        [&](int gi, float x) {
          x += 0.f;                                     // -0 and +0 are the same score
          const int32_t u = __float_as_int(x);
          const uint32_t key = uint32_t(u) ^ (uint32_t(u >> 31) | 0x80000000u);
          key_min = min(key_min, key);
          key_max = max(key_max, key);
          cluster_store(dst_keys + uint32_t(g0 + gi) * 4u, key);
          if (out_row != nullptr) out_row[g0 + gi] = x;
        });
    __syncwarp();
    if (k + a.depth < my_tiles) fill(k + a.depth, stage);
    if (++stage == a.depth) { stage = 0; phase ^= 1u; }
  }
#pragma unroll
  for (int off = 1; off <= 2; off <<= 1) {              // the four lanes of a scope
    key_min = min(key_min, __shfl_xor_sync(kAll, key_min, off));
    key_max = max(key_max, __shfl_xor_sync(kAll, key_max, off));
  }
  if (scope_ok && qt == 0 && my_tiles > 0) {
    cluster_min(cluster_map(smem_addr(&sm->key_min), owner), key_min);
    cluster_max(cluster_map(smem_addr(&sm->key_max), owner), key_max);
  }
  if (timed_out) {
    if (lane == 0 && a.err) atomicExch(a.err, kDevTimeoutFull);
    for (int s = 0; s < a.depth; ++s) {                 // bounded chance for copies in flight to land
      mbar_wait(smem_addr(&sm->full[warp * 2 + s]), 0);
      mbar_wait(smem_addr(&sm->full[warp * 2 + s]), 1);
    }
  }
  cluster_arrive();
  cluster_wait();                                       // every key is in place (and the histogram cleared)

  // ---- the select of scope s0 + rank ------------------------------------------------------------------------------
  if (rank >= ns) return;
  const int64_t prob = int64_t(rs.b) * p.S + s0 + rank;
  int32_t* out = a.group_idx + prob * p.M;
  if (threadIdx.x == 0) a.n_selected[prob] = p.Mp;
  for (int i = p.Mp + threadIdx.x; i < p.M; i += kClusterThreads) out[i] = -1;
  if (p.Mp == p.NG) {                                   // everything is selected
    for (int i = threadIdx.x; i < p.NG; i += kClusterThreads) out[i] = i;
    return;
  }
  select_from_smem(keys, p.NG, p.Mp, sm->key_min, sm->key_max, out, sm->select);
}

// Fixed and per-stage shared memory of the kernel, and its launch, for a stored type and rank; `g_shift` =
// log2 G or -1.  Instantiated in score_select_cluster_*.cu.
template <int META, int R>
cudaError_t launch_score_select_rows(const Problem& p, const ClusterArgs& a, int g_shift, int cluster, int n_rests,
                                     cudaStream_t st);
template <> cudaError_t launch_score_select_rows<KVSWAP_F16, 16>(const Problem&, const ClusterArgs&, int, int, int, cudaStream_t);
template <> cudaError_t launch_score_select_rows<KVSWAP_F16, 32>(const Problem&, const ClusterArgs&, int, int, int, cudaStream_t);
template <> cudaError_t launch_score_select_rows<KVSWAP_F16, 64>(const Problem&, const ClusterArgs&, int, int, int, cudaStream_t);
template <> cudaError_t launch_score_select_rows<KVSWAP_E4M3, 32>(const Problem&, const ClusterArgs&, int, int, int, cudaStream_t);
template <> cudaError_t launch_score_select_rows<KVSWAP_F32, 16>(const Problem&, const ClusterArgs&, int, int, int, cudaStream_t);
template <> cudaError_t launch_score_select_rows<KVSWAP_F32, 32>(const Problem&, const ClusterArgs&, int, int, int, cudaStream_t);
template <> cudaError_t launch_score_select_rows<KVSWAP_F32, 64>(const Problem&, const ClusterArgs&, int, int, int, cudaStream_t);

// Keys of one scope in the selecting CTA's shared memory.  With more, one CTA takes longer to select from them than the
// TopK in parts: scorer and select at B = 1, 8 heads, r = 32, G = 1 14.0 us against 14.9 of the two kernels for 6000
// groups, 15.3 against 14.9 for 8192, 22.5 against 16.5 for 16384; at B = 16 19.8 against 24.4, 30.9 against 20.0 and
// 48.1 against 38.7.
constexpr int kClusterMaxKeys = 6144;

// Shared memory of a CTA with `depth` stages per warp and NG keys; GS counts only as a power of two (>= 0) or not.
template <int META, int R, int GS>
constexpr size_t score_select_smem(int depth, int NG) {
  constexpr size_t kFixed = (sizeof(ClusterSmem<META, R, GS>) + 127) & ~size_t(127);
  constexpr size_t kStages = size_t(kClusterWarps) * ScoreStage<META, R, GS>::kBytes;
  static_assert(kFixed + kStages + 4 * kClusterMaxKeys <= 227 * 1024, "at least one stage per warp fits");
  return kFixed + size_t(depth) * kStages + 4 * size_t((NG + 3) & ~3);
}

template <int META, int R, int GS>
cudaError_t launch_score_select_gs(const Problem& p, const ClusterArgs& args, int cluster, int n_rests, cudaStream_t st) {
  const size_t smem = score_select_smem<META, R, GS>(args.depth, p.NG);
  auto kern = score_select_cluster_kernel<META, R, GS>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  if (e != cudaSuccess) return e;
  if (cluster > 8 && (e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess) return e;
  return launch_pdl_cluster(kern, cluster, dim3(n_rests * cluster), dim3(kClusterThreads), smem, st, p, args);
}

#define KVSWAP_SCORE_SELECT_ROWS(META, R)                                                                            \
  template <>                                                                                                        \
  cudaError_t launch_score_select_rows<META, R>(const Problem& p, const ClusterArgs& a, int g_shift, int cluster,    \
                                                int n_rests, cudaStream_t st) {                                      \
    switch (g_shift) {                                                                                               \
      case 0: return launch_score_select_gs<META, R, 0>(p, a, cluster, n_rests, st);                                 \
      case 1: return launch_score_select_gs<META, R, 1>(p, a, cluster, n_rests, st);                                 \
      case 2: return launch_score_select_gs<META, R, 2>(p, a, cluster, n_rests, st);                                 \
      case 3: return launch_score_select_gs<META, R, 3>(p, a, cluster, n_rests, st);                                 \
      case 4: return launch_score_select_gs<META, R, 4>(p, a, cluster, n_rests, st);                                 \
      case 5: return launch_score_select_gs<META, R, 5>(p, a, cluster, n_rests, st);                                 \
      default:                                                                                                       \
        if constexpr (META == KVSWAP_E4M3) return cudaErrorInvalidValue;                                             \
        else return launch_score_select_gs<META, R, -1>(p, a, cluster, n_rests, st);                                 \
    }                                                                                                                \
  }

}  // namespace kvswap
