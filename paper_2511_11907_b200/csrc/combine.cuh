// Merge of the split-K partials of one (sequence, head) row: the body shared by the stand-alone
// combine kernel (sparse_decode.cu) and the kernel that runs it beside a TopK (topk_select.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace kvswap {

constexpr int kMaxSplits = 256;
constexpr int kGatherWarps = 8;   // warps per CTA of the gathers

// Partials [rows, slots, D + 2] = (m, l, acc[D]) of a gather whose lists (heads_per_list rows each) were dealt to
// warps_per_list consecutive warps, kGatherWarps to a CTA: of a row's slots as many are filled as CTAs took part in its list,
// all of them where lists have CTAs to themselves (`whole`).
struct CombineJob {
  const float* partial;
  float* out;              // [rows, D]
  float* lse;              // NULL or [rows]
  int rows, slots, heads_per_list, warps_per_list;

  __host__ __device__ __forceinline__ bool whole() const { return warps_per_list % kGatherWarps == 0; }
  __device__ __forceinline__ int filled(int row) const {
    const int first = row / heads_per_list * warps_per_list;
    return (first + warps_per_list - 1) / kGatherWarps - first / kGatherWarps + 1;
  }
};

inline CombineJob combine_job(const Problem& p, const Workspace& w, const float* partial, float* out, float* lse) {
  return CombineJob{partial, out, lse, p.B * p.Hq, w.splits, w.heads_per_cta, w.warps_per_list};
}

// D threads (c = 0..D-1) merge row `row` of `job`.  Every load of the row's first splits is issued before anything is
// computed (one memory round trip; the loads bypass L1, as the partials need not be those of the kernel waited for); the
// split weights are formed once by the first warp of the D threads and shared through w_s [kMaxSplits] and norm_s [2].  The
// D threads meet at named barrier `barrier` (0 = the CTA-wide one: then the CTA has exactly D threads).  Without a row
// (row >= job.rows) the threads only keep the barrier company.
// WHOLE: every slot is filled (job.whole()).  The kernels that only meet such jobs are built without the division, whose
// instructions alone took 0.9 us of a call with a separate combine (45.1 -> 44.2 us for a score_select and a sparse_decode
// of 92 MB, 4 sequences).
template <int D, bool WHOLE>
__device__ __forceinline__ void combine_row(const CombineJob& job, int row, int c, float* w_s, float* norm_s, int barrier) {
  constexpr float kLn2 = 0.6931471805599453f;
  constexpr int kUnroll = 16;
  const bool live = row < job.rows;
  const int splits = WHOLE ? job.slots : job.filled(row);
  const float* src = job.partial + int64_t(row) * job.slots * (D + 2);
  float a_first[kUnroll], m_first = -INFINITY, l_first = 0.f;
#pragma unroll
  for (int s = 0; s < kUnroll; ++s) a_first[s] = (live && s < splits) ? __ldcg(src + s * (D + 2) + 2 + c) : 0.f;
  if (live && c < 32 && c < splits) { m_first = __ldcg(src + c * (D + 2)); l_first = __ldcg(src + c * (D + 2) + 1); }
  if (live && c < 32) {
    // weights: lane s handles splits s, s + 32, ...
    float mx = m_first;
    for (int s = c + 32; s < splits; s += 32) mx = fmaxf(mx, __ldcg(src + s * (D + 2)));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    const float w_first = (mx > -INFINITY) ? exp2f(m_first - mx) : 0.f;
    w_s[c] = w_first;                                    // (lanes beyond the splits: not read)
    float lsum = l_first * w_first;
    for (int s = c + 32; s < splits; s += 32) {
      const float w = (mx > -INFINITY) ? exp2f(__ldcg(src + s * (D + 2)) - mx) : 0.f;
      w_s[s] = w;
      lsum = fmaf(__ldcg(src + s * (D + 2) + 1), w, lsum);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, off);
    if (c == 0) {
      norm_s[0] = (lsum > 0.f) ? 1.f / lsum : 0.f;
      norm_s[1] = (lsum > 0.f) ? (mx + log2f(lsum)) * kLn2 : -INFINITY;
    }
  }
  if (barrier == 0) __syncthreads();
  else asm volatile("bar.sync %0, %1;" ::"r"(barrier), "r"(D) : "memory");
  if (!live) return;
  float a = 0.f;
#pragma unroll
  for (int s = 0; s < kUnroll; ++s) if (s < splits) a = fmaf(a_first[s], w_s[s], a);
  for (int s = kUnroll; s < splits; ++s) a = fmaf(__ldcg(src + s * (D + 2) + 2 + c), w_s[s], a);
  job.out[int64_t(row) * D + c] = a * norm_s[0];
  if (job.lse != nullptr && c == 0) job.lse[row] = norm_s[1];
}

}  // namespace kvswap
