// TopK of one list whose keys lie in the CTA's shared memory (Sec. 4.3): the select of the kernel that scores
// and selects in one cluster (score_select_cluster.cuh).
#pragma once

#include "topk_keys.cuh"

namespace kvswap {

constexpr int kSelectThreads = 512;
constexpr int kSelectWarps = kSelectThreads / 32;
constexpr int kSelectRanked = 256;                    // keys sharing a bin that are ranked pairwise

struct SelectScratch {
  int hist[kKeyTopBins];
  uint32_t few[kSelectRanked];
  int warp_tot[kSelectWarps];
  uint32_t warp_cnt[kSelectWarps];
  int bin, want, cnt, n_few;
};

// Bin of the candidate of descending rank `want` (1-based) in scratch.hist[0 .. kKeyTopBins): thread t holds
// eight bins counted from the top.  Publishes (bin, rank inside it, its population); ends with a barrier.
__device__ __forceinline__ void select_find_bin(SelectScratch& s, int want) {
  constexpr uint32_t kAll = 0xffffffffu;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int base = kKeyTopBins - 8 * (tid + 1);
  const int4 lo = *reinterpret_cast<const int4*>(&s.hist[base]), hi = *reinterpret_cast<const int4*>(&s.hist[base + 4]);
  const int c[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
  const int local = ((c[0] + c[1]) + (c[2] + c[3])) + ((c[4] + c[5]) + (c[6] + c[7]));
  const int wsum = __reduce_add_sync(kAll, local);
  if (lane == 0) s.warp_tot[warp] = wsum;
  __syncthreads();
  const int w = (lane < kSelectWarps) ? s.warp_tot[lane] : 0;
  int incl = w;
#pragma unroll
  for (int off = 1; off < kSelectWarps; off <<= 1) {
    const int t = __shfl_up_sync(kAll, incl, off);
    if (lane >= off) incl += t;
  }
  const uint32_t reached = __ballot_sync(kAll, lane < kSelectWarps && incl >= want);
  if (reached != 0u && warp == __ffs(reached) - 1) {          // this warp holds the rank
    int acc = __shfl_sync(kAll, incl - w, warp);
    int mine = local;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int t = __shfl_up_sync(kAll, mine, off);
      if (lane >= off) mine += t;
    }
    acc += mine - local;
    if (acc < want && acc + local >= want) {
#pragma unroll
      for (int i = 7; i >= 0; --i) {
        if (acc < want && acc + c[i] >= want) { s.bin = base + i; s.want = want - acc; s.cnt = c[i]; }
        acc += c[i];
      }
    }
  }
  __syncthreads();
}

// Score of a key.
__device__ __forceinline__ float key_score(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// The Mp largest of keys[0 .. NG) (larger key = larger score), lower index first among equal ones, as
// ascending indices in out[0 .. Mp); 0 < Mp < NG.  key_min, key_max: the extremes of the keys.  All
// kSelectThreads threads of the CTA call; keys are complete, scratch.hist is zero and a barrier lies behind both.
//
// Bound by its chain of barrier-separated phases, so there are few.  The scores are counted in 4096 bins of
// equal width over their range (a monotonic map, so a bin holds consecutive ranks), which leaves a few keys
// in the bin of the Mp-th and spreads the counting over many addresses; the leading 12 bits of the keys put
// 2048 scores into some thirty bins, and counting and ranking them took 2.5 us longer.  The bin's keys are
// gathered, each is ranked against all by one thread, and the selected indices are written by ballot, a
// contiguous segment per warp.  A bin of more than kSelectRanked keys (far outliers, many equal scores) is
// resolved by the digits of the keys instead.
__device__ __forceinline__ void select_from_smem(const uint32_t* keys, int NG, int Mp, uint32_t key_min, uint32_t key_max,
                                                 int32_t* __restrict__ out, SelectScratch& s) {
  constexpr uint32_t kAll = 0xffffffffu;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float low = key_score(key_min), range = key_score(key_max) - low;
  const float scale = (range > 0.f && range < INFINITY) ? float(kKeyTopBins - 1) / range : 0.f;
  auto bin_of = [&](uint32_t k) { return min(max(int((key_score(k) - low) * scale), 0), kKeyTopBins - 1); };
  for (int i = tid; i < NG; i += kSelectThreads) atomicAdd(&s.hist[bin_of(keys[i])], 1);
  if (tid == 0) s.n_few = 0;
  __syncthreads();
  select_find_bin(s, Mp);
  const int bin = s.bin, want = s.want, cnt = s.cnt;
  uint32_t kth;                                        // keys > kth are selected, plus need_eq keys == kth
  int need_eq;
  if (cnt > kSelectRanked) {
    uint32_t prefix = 0u, known = 0u;                  // known high bits of the Mp-th key
    int left = Mp;
    for (int shift = 20; shift >= -4; shift -= 12) {   // digits of 12, 12 and 8 bits
      const int low_bit = max(shift, 0);
      const uint32_t digit = shift >= 0 ? 0xfffu : 0xffu;
      __syncthreads();
      for (int i = tid; i < kKeyTopBins; i += kSelectThreads) s.hist[i] = 0;
      __syncthreads();
      for (int i = tid; i < NG; i += kSelectThreads)
        if ((keys[i] & known) == prefix) atomicAdd(&s.hist[(keys[i] >> low_bit) & digit], 1);
      __syncthreads();
      select_find_bin(s, left);
      prefix |= uint32_t(s.bin) << low_bit;
      known |= digit << low_bit;
      left = s.want;
    }
    kth = prefix;
    need_eq = left;
  } else {
    const int n_rows = (NG + kSelectThreads - 1) / kSelectThreads;
    for (int r = 0; r < n_rows; ++r) {
      const int i = r * kSelectThreads + tid;
      const uint32_t k = (i < NG) ? keys[i] : 0u;
      const bool in = i < NG && bin_of(k) == bin;
      const uint32_t m = __ballot_sync(kAll, in);
      if (m != 0u) {
        int at = 0;
        if (lane == 0) at = atomicAdd(&s.n_few, __popc(m));
        at = __shfl_sync(kAll, at, 0) + __popc(m & ((1u << lane) - 1u));
        if (in && at < kSelectRanked) s.few[at] = k;
      }
    }
    if (tid < 4 && cnt + tid < kSelectRanked) s.few[cnt + tid] = 0u;   // pad to a whole vector, below every key
    __syncthreads();
    for (int i = tid; i < cnt; i += kSelectThreads) {
      const uint32_t v = s.few[i];
      int gt = 0, eq = 0;
      for (int j = 0; j < cnt; j += 4) {
        const uint4 o = *reinterpret_cast<const uint4*>(&s.few[j]);
        gt += int(o.x > v) + int(o.y > v) + int(o.z > v) + int(o.w > v);
        eq += int(o.x == v) + int(o.y == v) + int(o.z == v) + int(o.w == v);
      }
      if (gt < want && want <= gt + eq) { s.bin = int(v); s.cnt = want - gt; }     // equal keys write the same
    }
    __syncthreads();
    kth = uint32_t(s.bin);
    need_eq = s.cnt;
  }

  // ---- selected indices in order: warp w takes keys [w seg, (w + 1) seg) --------------------------------------
  const int seg = ((NG + kSelectThreads - 1) / kSelectThreads) * 32;
  const int i0 = warp * seg, i1 = min(NG, i0 + seg);
  uint32_t counts = 0u;                                // (> kth) << 16 | (== kth)
  for (int i = i0; i < i1; i += 32) {
    const uint32_t k = (i + lane < i1) ? keys[i + lane] : 0u;
    counts += (uint32_t(__popc(__ballot_sync(kAll, k > kth))) << 16) + uint32_t(__popc(__ballot_sync(kAll, k == kth)));
  }
  if (lane == 0) s.warp_cnt[warp] = counts;
  __syncthreads();
  const uint32_t before = __reduce_add_sync(kAll, (lane < warp) ? s.warp_cnt[lane] : 0u);      // kSelectWarps <= 32
  int eq_seen = int(before & 0xffffu);
  int pos = int(before >> 16) + min(eq_seen, need_eq);
  for (int i = i0; i < i1; i += 32) {
    const uint32_t k = (i + lane < i1) ? keys[i + lane] : 0u;
    const uint32_t m_eq = __ballot_sync(kAll, k == kth), below = (1u << lane) - 1u;
    const bool take = k > kth || (k == kth && eq_seen + __popc(m_eq & below) < need_eq);
    const uint32_t m = __ballot_sync(kAll, take);
    if (take) out[pos + __popc(m & below)] = i + lane;
    pos += __popc(m);
    eq_seen += __popc(m_eq);
  }
}

}  // namespace kvswap
