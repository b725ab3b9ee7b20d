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
  float qsum[kQuerySumFloats], upart[kQueryPartFloats], urow[kQueryCols * 64];
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
      else if (p.r == 16) form(std::integral_constant<int, 16>());
      else form(std::integral_constant<int, 64>());
      __syncthreads();                                  // urow is free for the next row set
    }
  }
  pdl_wait();
}

}  // namespace

bool select_beside_supported(const Problem& p) { return plan_topk_beside(p) > 0 && (p.d == 64 || p.d == 128); }

cudaError_t launch_select_beside(const Problem& p, const float* scores, int32_t* group_idx, int32_t* n_selected,
                                 const CombineJob& job, const void* q_ahead, const float* proj_ahead, float* uq_ahead,
                                 cudaStream_t st) {
  if (!select_beside_supported(p)) return cudaErrorInvalidValue;
  // Query sets of the launch: the scorer's row sets, except that the KV heads of per-head metadata are taken eight at a
  // time like the scopes of joint metadata (a row's sum is the same).
  AheadArgs a{q_ahead, proj_ahead, uq_ahead, 0, 1};
  Problem pq = p;
  if (q_ahead != nullptr) {
    if (!score_stream_fuses_query(p) || proj_ahead == nullptr || uq_ahead == nullptr) return cudaErrorInvalidValue;
    score_stream_row_sets(p, &a.n_rests, &a.n_sub);
    if (p.Hm != 1 && p.scope == KVSWAP_SCOPE_KV_HEAD) {
      pq.Hm = 1;
      a.n_sub = (p.Hkv + kQueryCols - 1) / kQueryCols;
      a.n_rests = p.B * a.n_sub;
    }
  }
  // One CTA per SM where that is enough: a second one would keep the gather off its SM.
  const int n_probs = p.B * p.S, spare = std::max(kNumSMs - n_probs, 16), rows = kBesideThreads / p.d;
  const int n_first = std::min(spare, std::max((job.rows + 4 * rows - 1) / (4 * rows), a.n_rests));
  auto go = [&](auto kern) {
    // The SM is shared with a gather, which needs the largest carve-out of shared memory: with another one the SM would
    // have to drain first.
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    return e != cudaSuccess ? e
                            : launch_pdl(kern, dim3(n_first + n_probs), dim3(kBesideThreads), 0, st, pq, scores, group_idx,
                                         n_selected, job, n_first, a);
  };
  const int P = plan_topk_beside(p);
  if (p.d == 128) return P == 1 ? go(select_beside_kernel<1, 128>) : P == 2 ? go(select_beside_kernel<2, 128>) : go(select_beside_kernel<4, 128>);
  return P == 1 ? go(select_beside_kernel<1, 64>) : P == 2 ? go(select_beside_kernel<2, 64>) : go(select_beside_kernel<4, 64>);
}

}  // namespace kvswap
