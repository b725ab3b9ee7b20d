// Host side of the tensor-core softmax scorer (score_softmax_tc.cuh): which shapes take it, its plan, the launches.
#include <algorithm>

#include "score_softmax_tc.cuh"

namespace kvswap {
namespace {

constexpr size_t kMaxSmem = 227 * 1024;

template <typename F>
auto by_rows(const Problem& p, F&& f) {
  if (p.meta_dtype == KVSWAP_F16) {
    if (p.r == 16) return f(std::integral_constant<int, KVSWAP_F16>(), std::integral_constant<int, 16>());
    if (p.r == 32) return f(std::integral_constant<int, KVSWAP_F16>(), std::integral_constant<int, 32>());
    return f(std::integral_constant<int, KVSWAP_F16>(), std::integral_constant<int, 64>());
  }
  if (p.r == 16) return f(std::integral_constant<int, KVSWAP_F32>(), std::integral_constant<int, 16>());
  if (p.r == 32) return f(std::integral_constant<int, KVSWAP_F32>(), std::integral_constant<int, 32>());
  return f(std::integral_constant<int, KVSWAP_F32>(), std::integral_constant<int, 64>());
}

// Launch plans of the statistics (pool = false) and the pooling kernel; false: the shape is not taken.
bool plan(const Problem& p, bool pool, bool counts, SoftmaxArgs* a, int* n_sets) {
  if (p.NG < 1 || p.meta_dtype == KVSWAP_E4M3 || !score_stream_rows(p) || p.meta_sn != p.r) return false;
  const int row_bytes = p.r * (p.meta_dtype == KVSWAP_F32 ? 4 : 2);
  const int fit = std::min(kSoftmaxMaxRows, 3072 / row_bytes / 8 * 8);
  const int64_t rows_total = int64_t(p.NG) * p.G;
  a->atomic = p.G > fit && (p.G > kSoftmaxMaxRows || p.G * row_bytes > 4096);
  a->tile_rows = !pool || a->atomic ? fit : p.G > fit ? p.G : fit / p.G * p.G;
  const bool scoped = p.Hm == 1 && p.scope == KVSWAP_SCOPE_KV_HEAD;
  a->n_sub = scoped ? (p.S + kSoftmaxScopes - 1) / kSoftmaxScopes : 1;
  const int64_t sets = int64_t(p.B) * (pool ? scored_heads(p) * a->n_sub : p.Hm);
  if (sets > (1 << 20)) return false;
  // Where a warp gets few tiles, shorter ones even the warps out: a tile costs its rows and some eight rows' worth of
  // hand-over.  (B = 4, N = 40001: three tiles of 24 rows instead of two of 48 in the longest share.)
  if (p.G <= a->tile_rows && !a->atomic) {
    const int64_t warps = std::max<int64_t>(1, kNumSMs / sets) * kSoftmaxWarps;
    int best = a->tile_rows;
    auto cost = [&](int rows) { return ((rows_total + rows - 1) / rows + warps - 1) / warps * (rows + 8); };
    const int step = pool ? p.G : 8;
    for (int rows = a->tile_rows - step; rows >= 16; rows -= step) if (cost(rows) < cost(best)) best = rows;
    a->tile_rows = best;
  }
  if ((rows_total + a->tile_rows - 1) / a->tile_rows > (1 << 28)) return false;
  a->tiles = int((rows_total + a->tile_rows - 1) / a->tile_rows);
  a->stage_bytes = (a->tile_rows + 7) / 8 * 8 * row_bytes;
  a->pitch = (a->tile_rows + 7) / 8 * 8 + 8;
  a->p_shift = 3;
  if (!pool) {
    a->units = 1;
    a->kb = ((p.Hm == 1 ? p.Hq : p.rho) + 7) / 8;
  } else if (scoped && p.rho <= 8) {
    a->p_shift = p.rho <= 1 ? 0 : p.rho <= 2 ? 1 : p.rho <= 4 ? 2 : 3;
    a->kb = 1;
    const int per_unit = 8 >> a->p_shift;
    a->units = (std::min(kSoftmaxScopes, p.S) + per_unit - 1) / per_unit;
  } else {
    a->kb = ((p.Hm == 1 && !scoped ? p.Hq : p.rho) + 7) / 8;
    a->units = scoped ? std::min(kSoftmaxScopes, p.S) : multi_term(p) ? p.Hkv : 1;
  }
  a->n_blocks = a->units * a->kb;
  *n_sets = int(sets);
  a->ctas_per_set = int(std::max<int64_t>(1, std::min<int64_t>({kNumSMs / sets, (a->tiles + kSoftmaxWarps - 1) / kSoftmaxWarps,
                                                                int64_t(score_softmax_chunks(p))})));
  if (counts && ((a->tiles + a->ctas_per_set - 1) / a->ctas_per_set + kSoftmaxWarps) * int64_t(a->tile_rows) / p.G > 65535) return false;
  for (a->depth = 2; a->depth >= 1; --a->depth)
    if (by_rows(p, [&](auto m, auto r) { return softmax_tc_smem<decltype(m)::value, decltype(r)::value>(*a, pool, counts); }) <= kMaxSmem) return true;
  return false;
}

}  // namespace

bool score_softmax_tc_supported(const Problem& p) {
  SoftmaxArgs a = {};
  int n;
  return plan(p, false, false, &a, &n) && plan(p, true, false, &a, &n);
}
// ... and the pooling kernel counts the leading digits of its scores' keys.
bool score_softmax_tc_counts(const Problem& p) {
  SoftmaxArgs a = {};
  int n;
  return plan(p, false, false, &a, &n) && plan(p, true, true, &a, &n) && !a.atomic;
}

cudaError_t launch_score_softmax_tc(const Problem& p, const void* meta, const float* u, float* stats, float* scores,
                                    uint32_t* top_hist, uint32_t* err, cudaStream_t st) {
  SoftmaxArgs s = {}, w = {};
  int n_stats = 0, n_pool = 0;
  if (!plan(p, false, false, &s, &n_stats) || !plan(p, true, top_hist != nullptr, &w, &n_pool)) return cudaErrorInvalidValue;
  for (SoftmaxArgs* a : {&s, &w}) {
    a->u = u; a->meta = static_cast<const unsigned char*>(meta); a->stats = stats; a->scores = scores;
    a->top_hist = top_hist; a->err = err;
    a->stat_pitch = score_softmax_chunks(p);
    a->stat_parts = s.ctas_per_set;
  }
  return by_rows(p, [&](auto m, auto r) {
    constexpr int META = decltype(m)::value, R = decltype(r)::value;
    const size_t smem_s = softmax_tc_smem<META, R>(s, false, false),
                 smem_w = softmax_tc_smem<META, R>(w, true, top_hist != nullptr);
    auto ks = softmax_tc_stats_kernel<META, R>;
    auto kw = softmax_tc_pool_kernel<META, R>;
    cudaError_t e = cudaFuncSetAttribute(ks, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem_s));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kw, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem_w));
    if (e == cudaSuccess) e = launch_pdl(ks, dim3(n_stats * s.ctas_per_set), dim3(kSoftmaxThreads), smem_s, st, p, s);
    if (e == cudaSuccess) e = launch_pdl(kw, dim3(n_pool * w.ctas_per_set), dim3(kSoftmaxThreads), smem_w, st, p, w);
    return e;
  });
}

}  // namespace kvswap
