// The select of a decode step that runs beside a gather: launch and kernel (topk_beside.cuh has the body).
#include <algorithm>

#include "async_copy.cuh"
#include "combine.cuh"
#include "common.cuh"
#include "lowrank_query.cuh"
#include "topk_beside.cuh"

namespace kvswap {
namespace {

struct AheadArgs {
  const void* q;            // NULL: no queries
  const float* proj;
  float* uq;
  int n_rests, n_sub;
};

// Rows of partials a CTA merges at a time, D threads and one named barrier each.
template <int D> constexpr int kMergeRows = kBesideThreads / D;

template <int D>
struct AheadSmem {
  float qsum[kQuerySumFloats], upart[kQueryPartFloats], urow[kQueryCols * 32];
  float w[kMergeRows<D>][kMaxSplits], norm[kMergeRows<D>][2];
};

// The first CTAs merge split partials of an earlier layer's gather and form the summed low-rank queries of a later layer, the
// others select, a problem each.  What the first CTAs read was complete before this kernel was let in (step.cu), so they do
// not wait: they run beside the scorer whose scores the others wait for.  The queries are stored where the later layer's
// scorer looks for them, with that scorer's own build_queries() (the same bits): it starts on its tiles at once.
template <int P, int D>
__global__ void __launch_bounds__(kBesideThreads, 2)
select_beside_kernel(Problem p, const float* __restrict__ scores, int32_t* __restrict__ group_idx,
                     int32_t* __restrict__ n_selected, CombineJob job, int n_first, AheadArgs a) {
  __shared__ union __align__(16) { BesideSmem select; AheadSmem<D> ahead; } sm;
  if (int(blockIdx.x) >= n_first) {
    topk_beside_body<P>(p, scores, group_idx, n_selected, int(blockIdx.x) - n_first, sm.select);
    return;
  }
  pdl_trigger();
  const int slot = int(threadIdx.x) / D;
  for (int row = blockIdx.x * kMergeRows<D>; row < job.rows; row += n_first * kMergeRows<D>) {
    combine_row<D, false>(job, row + slot, int(threadIdx.x) % D, sm.ahead.w[slot], sm.ahead.norm[slot], 1 + slot);
    __syncthreads();                                    // the weights are free for the next rows
  }
  if (a.q != nullptr) {
    for (int rest = blockIdx.x; rest < a.n_rests; rest += n_first) {
      const RowSet rs = row_set(p, rest, a.n_sub);
      auto form = [&](auto rank) {
        constexpr int R = decltype(rank)::value;
        build_queries<0, R, kQueryWarps, true>(p, a.q, a.proj, rs, sm.ahead.qsum, sm.ahead.upart, sm.ahead.urow);
        store_queries<R>(p, rs, sm.ahead.urow, a.uq);
      };
      if (p.r == 32) form(std::integral_constant<int, 32>());
      else form(std::integral_constant<int, 16>());
      __syncthreads();                                  // urow is free for the next row set
    }
  }
  pdl_wait();
}

}  // namespace

// CTAs that merge and form queries.  One CTA per SM where that is enough: a second one would keep the gather off its SM.
static int first_ctas(const Problem& p, int rows, int n_rests) {
  const int spare = std::max(kNumSMs - p.B * p.S, 16), rows_per_cta = kBesideThreads / p.d;
  return std::min(spare, std::max((rows + 4 * rows_per_cta - 1) / (4 * rows_per_cta), n_rests));
}

// Where the select of a step runs beside gather and scorer: its CTAs have to find room beside the scorer's, one to an SM.
// - A scorer that leaves less than half of the registers keeps it, and the queries of the next layer, off its SMs until it has
//   finished.  Six layers of 4 sequences, 8 heads, 65536 tokens, 5600 attended, us a layer without / with the select beside:
//   fp16 rows of 64 35.7 / 39.9, fp32 rows 35.9 / 40.6, groups of 12 34.0 / 38.1, softmax 66.2 / 71.6; fp16 rows of 32 31.9 / 29.4.
// - Where the scorer leaves SMs idle the CTAs gather there, two to an SM, whose share of the gather then waits; the more so when
//   they do not all find room: 128 scorer CTAs, 20 idle: fp16 rows of 32, 32768 tokens 28.6 / 26.7 with 40 CTAs; 8-bit
//   rows, 65536 tokens 31.8 / 28.4 with 20 CTAs, 31.9 / 32.0 with 40, 32.0 / 32.7 with 80.  (Four idle ones do not show:
//   12 layers of 3 sequences, 98301 tokens, 144 CTAs, 25.8 / 22.8.)
// - With one list for all heads there are few selects to hide, 29.6 / 29.7; with a compact cache per head the scorer takes
//   most of the layer, 48.1 / 48.5.
// - With selects on most SMs the gather is slowed down by as much: 16 sequences of 32768 tokens 40.6 / 40.0, 65536 tokens of three
//   query heads per list, groups of 16 68.7 / 68.4.
bool select_beside_supported(const Problem& p) {
  if (plan_topk_beside(p) == 0 || (p.d != 64 && p.d != 128)) return false;
  if (p.Hm != 1 || p.scope != KVSWAP_SCOPE_KV_HEAD || (p.flags & KVSWAP_SCORE_SOFTMAX) || 2 * p.B * p.S > kNumSMs) return false;
  int n_rests, n_sub;
  score_stream_row_sets(p, &n_rests, &n_sub);
  const int scorer = score_stream_light_ctas(p), idle = kNumSMs - scorer;
  return scorer > 0 && (idle <= 4 || p.B * p.S + first_ctas(p, p.B * p.Hq, n_rests) <= 2 * idle);
}

cudaError_t launch_select_beside(const Problem& p, const float* scores, int32_t* group_idx, int32_t* n_selected,
                                 const CombineJob& job, const void* q_ahead, const float* proj_ahead, float* uq_ahead,
                                 cudaStream_t st) {
  if (!select_beside_supported(p)) return cudaErrorInvalidValue;
  AheadArgs a{q_ahead, proj_ahead, uq_ahead, 0, 1};
  if (q_ahead != nullptr) {
    if (proj_ahead == nullptr || uq_ahead == nullptr) return cudaErrorInvalidValue;
    score_stream_row_sets(p, &a.n_rests, &a.n_sub);            // the scorer's row sets
  }
  const int n_probs = p.B * p.S, n_first = first_ctas(p, job.rows, a.n_rests);
  auto go = [&](auto kern) {
    // The SM is shared with a gather, which needs the largest carve-out of shared memory: with another one the SM would
    // have to drain first.
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    return e != cudaSuccess ? e
                            : launch_pdl(kern, dim3(n_first + n_probs), dim3(kBesideThreads), 0, st, p, scores, group_idx,
                                         n_selected, job, n_first, a);
  };
  const int P = plan_topk_beside(p);
  if (p.d == 128)
    return P == 1 ? go(select_beside_kernel<1, 128>) : P == 2 ? go(select_beside_kernel<2, 128>) : go(select_beside_kernel<4, 128>);
  return P == 1 ? go(select_beside_kernel<1, 64>) : P == 2 ? go(select_beside_kernel<2, 64>) : go(select_beside_kernel<4, 64>);
}

}  // namespace kvswap
