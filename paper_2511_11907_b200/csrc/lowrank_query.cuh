// Summed low-rank queries (Eq. 1, the query side): u = sum over heads h of q_h A_g(h), one row per
// selection scope.  The device code is shared by the streaming scorer, which builds the queries of
// its own row sets (score_stream.cuh), and by the kernel that builds them one layer ahead beside the
// split-K combine (topk_select.cu): both therefore produce the same bits.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "common.cuh"

namespace kvswap {

constexpr int kQueryThreads = 512;                        // threads that call build_queries together
constexpr int kQueryWarps = kQueryThreads / 32;
constexpr int kQueryCols = 8;                             // query rows (scopes) per row set
constexpr int kQuerySumFloats = 8 * 128;                  // shared scratch: summed queries of up to 8 KV heads
constexpr int kQueryPartFloats = 32 * 32;                 // shared scratch: partial products, [item][column]

__device__ __forceinline__ float load_q(const void* q, int dtype, int64_t i) {
  if (dtype == KVSWAP_F32) return static_cast<const float*>(q)[i];
  if (dtype == KVSWAP_BF16) return __bfloat162float(static_cast<const __nv_bfloat16*>(q)[i]);
  return __half2float(static_cast<const __half*>(q)[i]);
}

// Metadata heads that are scored on their own: one when a score sums over all of them.
__host__ __device__ __forceinline__ int scored_heads(const Problem& p) {
  return (p.Hm == 1 || p.scope == KVSWAP_SCOPE_ALL_HEADS) ? 1 : p.Hkv;
}
// A score that sums terms on several metadata heads (per-head metadata, all-heads scope).
__host__ __device__ __forceinline__ bool multi_term(const Problem& p) { return p.Hm != 1 && p.scope == KVSWAP_SCOPE_ALL_HEADS; }

// (sequence, metadata head, scope block) of a row set.
struct RowSet { int b, hm, sub; };
__device__ __forceinline__ RowSet row_set(const Problem& p, int rest, int n_sub) {
  const int hm_count = scored_heads(p);
  const int bh = rest / n_sub;
  return RowSet{bh / hm_count, bh % hm_count, rest % n_sub};
}

// The terms that feed the rows of a row set: term t adds to row t (or 0) and reads KV head head0 + t.
struct QueryTerms { int n_terms, head0; bool row_per_term; };
__device__ __forceinline__ QueryTerms query_terms(const Problem& p, RowSet rs) {
  const bool joint = p.Hm == 1;
  const bool all_heads = joint && p.scope == KVSWAP_SCOPE_ALL_HEADS;
  const bool multi = multi_term(p);
  return QueryTerms{(all_heads || multi) ? p.Hkv : joint ? min(kQueryCols, p.S - rs.sub * kQueryCols) : 1,
                    (all_heads || multi) ? 0 : joint ? rs.sub * kQueryCols : rs.hm, (joint && !all_heads) || multi};
}
// log2 of the 32-channel pieces of a head: 4, 2 or 1
__device__ __forceinline__ int query_chunk_shift(const Problem& p) { return (p.d == 128) ? 2 : (p.d == 64) ? 1 : 0; }

// Sum over a KV head's query heads of channel c: the loads of four heads go out together.
__device__ __forceinline__ float query_sum(const Problem& p, const void* q, int b, int head, int c) {
  const int64_t at = (int64_t(b) * p.Hq + int64_t(head) * p.rho) * p.d + c;
  float s = 0.f;
  for (int h0 = 0; h0 < p.rho; h0 += 4) {
    float v[4];
#pragma unroll
    for (int hh = 0; hh < 4; ++hh) v[hh] = (h0 + hh < p.rho) ? load_q(q, p.q_dtype, at + int64_t(h0 + hh) * p.d) : 0.f;
    s += (v[0] + v[1]) + (v[2] + v[3]);
  }
  return s;
}

// Entry (row, j) of the summed queries of up to eight terms from the partial products upart[item][32] of
// column block j / 32, added in a fixed order; s: the sum over the terms before these.
__device__ __forceinline__ float query_entry(const float* upart, int row, int j, int nt, int ch_shift, bool row_per_term, float s) {
  const int chunks = 1 << ch_shift;
  if (row_per_term) {                                                  // the items of term `row`
    if (row < nt)
      for (int ch = 0; ch < chunks; ++ch) s += upart[((row << ch_shift) + ch) * 32 + (j & 31)];
  } else if (row == 0) {
    for (int it = 0; it < (nt << ch_shift); ++it) s += upart[it * 32 + (j & 31)];
  }
  return s;
}

// Summed low-rank queries of one row set into urow[8][R], R = p.r = 16, 32 or 64 (rows beyond the set's
// scopes are zero).  The KV heads that feed the rows are taken eight at a time, 32 columns at a time.  An
// item is 32 channels of one head: a warp multiplies the head's summed query by the adapter rows (coalesced
// 128-byte reads of A_g; at R = 16 a read covers two channels); it requests the adapter rows of its
// items first, then the CTA sums the query heads into shared memory, so that both loads share one
// round trip.  The partial products are added in a fixed order, whatever the number of warps.  Threads 0 ..
// 32 NW - 1 of the CTA call (NW = 16: at most two items per warp, LEAN: one after the other, or NW = 32: one; both take half
// the registers), and
// meet at barrier BAR (0: the CTA has exactly that many threads).  qsum [kQuerySumFloats] and upart
// [kQueryPartFloats] are shared-memory scratch, urow [8 * R] receives the result.
template <int BAR, int R, int NW = kQueryWarps, bool LEAN = false>
__device__ void build_queries(const Problem& p, const void* q, const float* __restrict__ proj, RowSet rs,
                              float* qsum, float* upart, float* urow) {
  auto sync = [] {
    if constexpr (BAR == 0) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"n"(BAR), "n"(32 * NW) : "memory");
  };
  static_assert(NW == 16 || NW == 32, "warps for the (at most) 32 items");
  constexpr int kLoads = (R == 16) ? 16 : 32;                             // adapter reads per item
  constexpr int kPasses = (R + 31) / 32;                                  // blocks of 32 columns
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const QueryTerms qt = query_terms(p, rs);
  const int n_terms = qt.n_terms, head0 = qt.head0, ch_shift = query_chunk_shift(p);
  const int chunks = 1 << ch_shift;
  const int d_shift = ch_shift + 5;
  // channel and column of load cc of an item: R = 16 takes channels 2 cc and 2 cc + 1 at once
  const int ch0 = (R == 16) ? (lane >> 4) : 0, step = (R == 16) ? 2 : 1, col = (R == 16) ? (lane & 15) : lane;
  for (int t0 = 0; t0 < n_terms; t0 += 8) {
    const int nt = min(8, n_terms - t0);
    const int n_items = nt << ch_shift;                            // <= 32: items warp and (NW = 16) warp + 16
    const int it0 = warp, it1 = warp + NW;
#pragma unroll 1
    for (int pass = 0; pass < kPasses; ++pass) {
      constexpr bool kSecond = NW == 16 && !LEAN;
      float a0[kLoads], a1[kSecond ? kLoads : 1];
      auto request = [&](int it, float* a) {
        const int64_t at = int64_t(head0 + t0 + (it >> ch_shift)) * p.d + (it & (chunks - 1)) * 32 + ch0;
        const float* P = proj + at * R + pass * 32 + col;
#pragma unroll
        for (int cc = 0; cc < kLoads; ++cc) a[cc] = (it < n_items) ? P[cc * step * R] : 0.f;
      };
      request(it0, a0);
      if constexpr (kSecond) request(it1, a1);
      if (pass == 0) {
        for (int i = tid; i < (nt << d_shift); i += 32 * NW) {
          const int tt = i >> d_shift, c = i & (p.d - 1);
          qsum[tt * 128 + c] = query_sum(p, q, rs.b, head0 + t0 + tt, c);
        }
        sync();
      }
      auto multiply = [&](int it, const float (&a)[kLoads]) {
        if (it >= n_items) return;
        const float* qs = qsum + (it >> ch_shift) * 128 + (it & (chunks - 1)) * 32 + ch0;
        float acc = 0.f;
#pragma unroll
        for (int cc = 0; cc < kLoads; ++cc) acc = fmaf(qs[cc * step], a[cc], acc);
        if constexpr (R == 16) acc += __shfl_xor_sync(0xffffffffu, acc, 16);
        upart[it * 32 + lane] = acc;
      };
      multiply(it0, a0);
      if constexpr (kSecond) {
        multiply(it1, a1);
      } else if constexpr (NW == 16) {
        request(it1, a0);
        multiply(it1, a0);
      }
      sync();
      if (tid < kQueryCols * 32) {
        const int row = tid >> 5, j = tid & 31, at = row * R + pass * 32 + j;
        if (pass * 32 + j < R) {
          urow[at] = query_entry(upart, row, j, nt, ch_shift, qt.row_per_term, (t0 == 0) ? 0.f : urow[at]);
        }
      }
      sync();
    }
  }
}

// Rows of urow[8][R] (build_queries) to the query buffer uq [B, Su, r] that the scorer reads
// when it does not build the queries itself: row i of a joint row set is scope sub * 8 + i, of a set of
// per-head terms head i, the one row of a per-head row set is head hm.  Threads 0 .. 255 of the callers store.
template <int R>
__device__ __forceinline__ void store_queries(const Problem& p, RowSet rs, const float* urow, float* __restrict__ uq) {
  if (threadIdx.x >= kQueryCols * 32) return;
  const bool multi = multi_term(p);
  for (int i = threadIdx.x; i < kQueryCols * R; i += kQueryCols * 32) {
    const int row = i / R, j = i % R;
    const int dst = (p.Hm == 1) ? rs.sub * kQueryCols + row : multi ? row : rs.hm;
    const bool have = (p.Hm == 1 || multi) ? (dst < p.Su) : (row == 0);
    if (have) uq[(int64_t(rs.b) * p.Su + dst) * p.r + j] = urow[i];
  }
}

}  // namespace kvswap
