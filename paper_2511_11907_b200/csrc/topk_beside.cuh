// TopK over rows of group scores beside a gather: the per-CTA body of select_beside_kernel (select_beside.cu).
#pragma once

#include "async_copy.cuh"
#include "common.cuh"
#include "topk_keys.cuh"

namespace kvswap {

// ------------------------------------------------------------------------------------------
// One CTA of 512 threads per problem, which reads the row once.
//   1. Rows of more than kListKeys keys: a bound from an even sample of the row, the 22 leading bits of its key of a rank
//      some 3.5 deviations below the M'-th key's share.
//   2. The keys that reach the bound (all keys of a short row) are listed: some 1.5 M' of them.
//   3. A histogram of the list over 1024 equal intervals of the keys finds the interval of the M'-th key; the few keys in
//      that are ranked by one warp (while they are many, it is cut in turn, down to single keys).
//   4. The selected ones are bits of a map, four keys per lane of a part of 128, from which the positions follow: population
//      counts, one scan over the parts.
// Where the list does not come out as expected (more than its room, or fewer than M': scores that run with the position of
// their groups, or long ties) the digits are counted over the whole row instead, which is exact for every input.
//
// It runs beside the gather of the layer before, in what that leaves of an SM: half of the registers and some 30 KB of
// shared memory.  Unlike topk_parts.cuh it needs no counts of the scorer, whose flush would lie between the two gathers,
// and one CTA does with a row.  A histogram of all keys in place of the sample kept the SM's shared memory busy (many keys
// share a bin) and held up the gather beside it.  Bound by latency, and by the gather's share of the issue slots: loads,
// sample, list, histogram, ranking, scan, writes; 13.2 us for 16384 groups as a launch of its own (B = 4, 8 heads), where the
// kernel that starts from the scorer's counts takes 9.4 with four CTAs per row.
// ------------------------------------------------------------------------------------------
constexpr int kBesideThreads = 512;
constexpr int kBesideWarps = kBesideThreads / 32;
constexpr int kBesidePart = 128;               // keys of a part
constexpr int kBesideParts = 256;               // of a row
constexpr int kListKeys = 2048;              // room of the list
constexpr int kDigit = 1024;                 // bins of the second and third digit
constexpr int kBesideFew = 32;                 // candidates that one warp ranks directly instead of by another digit

// Even sample of a row: one key of every NG / 2^bits, and the rank in it that the M'-th key's share falls behind.
struct BesideSample {
  int bits, rank;
  // Whether the list has room for the keys that reach a sampled key of that rank, 3.5 deviations allowed for.
  __host__ __device__ __forceinline__ bool list_has_room(int at_rank, int NG) const {
    return (float(at_rank) + 3.5f * sqrtf(float(at_rank))) * float(NG) <= float(kListKeys << bits);
  }
};
__host__ __device__ __forceinline__ BesideSample beside_sample(int NG, int Mp) {
  BesideSample s;
  s.bits = NG > 8192 ? 11 : 10;
  const float share = float(Mp) * float(1 << s.bits) / float(NG);
  s.rank = int(share + 3.5f * sqrtf(share)) + 4;
  return s;
}

struct BesideSmem {
  uint32_t sel[4 * kBesideParts];               // selected keys: word 4 v + e, bit lane: key 128 v + 4 lane + e
  uint32_t hist[kKeyTopBins / 2];            // leading digit: two 16-bit counters a word; kDigit words otherwise; at last the
                                             // map of the keys equal to the threshold
  uint32_t list_key[kListKeys];
  uint16_t list_idx[kListKeys];
  uint32_t before[kBesideParts];                // selected << 16 | equal keys in the parts before
  uint32_t warp_tot[kBesideWarps];
  uint32_t key_max;                          // of the list
  int bin, want, cnt, n_list, n_few;
  uint16_t few[kBesideFew];
};
static_assert(kKeyTopBins / 2 >= kDigit && kDigit >= 4 * kBesideParts, "the histogram has room for all three");
static_assert(kBesideParts * kBesidePart <= 65535, "counters");

// Thread t holds the populations c[0 .. PER - 1] of bins base .. base + PER - 1, base = PER (kBesideThreads - t - 1): the
// CTA's threads cover a histogram from the top.  Finds the bin that holds the candidate of descending rank `want`
// (1-based) and writes it, the rank inside the bin and its population.  All threads call; a barrier must follow
// before the results are read, and one precede before sm.warp_tot is reused.
template <int PER>
__device__ __forceinline__ void beside_find_bin(const int (&c)[PER], int want, BesideSmem& sm) {
  constexpr uint32_t kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int base = PER * (kBesideThreads - int(threadIdx.x) - 1);
  int local = 0;
#pragma unroll
  for (int i = 0; i < PER; ++i) local += c[i];
  const int wsum = __reduce_add_sync(kAll, local);
  if (lane == 0) sm.warp_tot[warp] = uint32_t(wsum);
  __syncthreads();
  const int w = (lane < kBesideWarps) ? int(sm.warp_tot[lane]) : 0;
  int incl = w;
#pragma unroll
  for (int off = 1; off < kBesideWarps; off <<= 1) {
    const int t = __shfl_up_sync(kAll, incl, off);
    if (lane >= off) incl += t;
  }
  const uint32_t reached = __ballot_sync(kAll, incl >= want && lane < kBesideWarps);
  if (reached == 0u) return;                                   // fewer candidates than `want`: leave the defaults
  const int holder = __ffs(reached) - 1;
  if (warp != holder) return;
  int acc = __shfl_sync(kAll, incl - w, holder);               // candidates in the warps above this one
  int mine = local;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int t = __shfl_up_sync(kAll, mine, off);
    if (lane >= off) mine += t;
  }
  acc += mine - local;                                         // ... and in the threads above this one
  if (acc < want && acc + local >= want) {
#pragma unroll
    for (int i = PER - 1; i >= 0; --i) {
      if (acc < want && acc + c[i] >= want) { sm.bin = base + i; sm.want = want - acc; sm.cnt = c[i]; }
      acc += c[i];
    }
  }
}

__device__ __forceinline__ float beside_elem(const float4& x, int e) { return e == 0 ? x.x : e == 1 ? x.y : e == 2 ? x.z : x.w; }

// Body of the select of problem `prob`; all kBesideThreads threads of the CTA call.
template <int P>
__device__ __forceinline__ void topk_beside_body(const Problem& p, const float* __restrict__ scores,
                                                int32_t* __restrict__ group_idx, int32_t* __restrict__ n_selected,
                                                int prob, BesideSmem& sm) {
  constexpr uint32_t kAll = 0xffffffffu;
  const int NG = p.NG, Mp = p.Mp;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t below = (1u << lane) - 1u;
  const int n_parts = (NG + kBesidePart - 1) / kBesidePart;
  for (int i = tid; i < kKeyTopBins / 2; i += kBesideThreads) sm.hist[i] = 0u;
  for (int i = tid; i < 4 * n_parts; i += kBesideThreads) sm.sel[i] = 0u;
  if (tid == 0) { sm.bin = 0; sm.want = 1; sm.cnt = 0; sm.n_list = 0; sm.n_few = 0; sm.key_max = 0u; }
  pdl_trigger();
  pdl_wait();
  const float* R = scores + int64_t(prob) * p.score_pitch;
  int32_t* out = group_idx + int64_t(prob) * p.M;

  const bool vec = (p.score_pitch & 3) == 0;   // rows start 16-byte aligned and are padded to whole vectors
  auto load = [&](int v) -> float4 {           // the lane's keys of part v
    const int i = v * kBesidePart + 4 * lane;
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (v < n_parts) {
      if (vec) {
        if (i < NG) x = __ldcg(reinterpret_cast<const float4*>(R + i));
      } else {
        if (i < NG) x.x = __ldcg(R + i);
        if (i + 1 < NG) x.y = __ldcg(R + i + 1);
        if (i + 2 < NG) x.z = __ldcg(R + i + 2);
        if (i + 3 < NG) x.w = __ldcg(R + i + 3);
      }
    }
    return x;
  };

  if (tid == 0) n_selected[prob] = Mp;
  for (int i = Mp + tid; i < p.M; i += kBesideThreads) out[i] = -1;
  if (Mp == NG) {                              // everything is selected
    for (int i = tid; i < NG; i += kBesideThreads) out[i] = i;
    return;
  }
  auto set = [](uint32_t* map, int i) { atomicOr(&map[(i / kBesidePart) * 4 + (i & 3)], 1u << ((i % kBesidePart) >> 2)); };
  auto count_top = [&](uint32_t key) {         // leading digit, two counters a word
    const uint32_t bin = key >> (32 - kKeyTopBits);
    atomicAdd(&sm.hist[bin >> 1], 1u << ((bin & 1u) << 4));
  };
  auto find_top = [&](int rank) {
    __syncthreads();
    const uint4 h = reinterpret_cast<const uint4*>(sm.hist)[kBesideThreads - 1 - tid];
    const int c[8] = {int(h.x & 0xffffu), int(h.x >> 16), int(h.y & 0xffffu), int(h.y >> 16),
                      int(h.z & 0xffffu), int(h.z >> 16), int(h.w & 0xffffu), int(h.w >> 16)};
    beside_find_bin(c, rank, sm);
    __syncthreads();
  };
  auto find_digit = [&](int rank) {
    __syncthreads();
    const uint2 hv = reinterpret_cast<const uint2*>(sm.hist)[kBesideThreads - 1 - tid];
    const int c[2] = {int(hv.x), int(hv.y)};
    beside_find_bin(c, rank, sm);
    __syncthreads();
  };
  auto clear_digit = [&] {
    for (int i = tid; i < kDigit; i += kBesideThreads) sm.hist[i] = 0u;
    __syncthreads();
  };

  // ---- the first round of keys, and a bound ------------------------------------------------------------------------
  constexpr int kSample = P == 4 ? 4 : 2;      // keys per thread, at most
  const BesideSample even = beside_sample(NG, Mp);
  const int bits = even.bits, rank = even.rank;
  const bool sampled = NG > kListKeys;
  bool exact = false;                          // the digits of the whole row are counted instead
  float sample[kSample];
#pragma unroll
  for (int k = 0; k < kSample; ++k)
    sample[k] = sampled && (k + 1) * kBesideThreads <= (1 << bits) ? __ldcg(R + (((tid + k * kBesideThreads) * NG) >> bits)) : 0.f;
  constexpr int kRound = kBesideWarps * P;       // parts of a round
  float4 x[P];
#pragma unroll
  for (int q = 0; q < P; ++q) x[q] = load(warp + kBesideWarps * q);
  uint32_t bound = 0u;                         // keys that reach it are listed
  __syncthreads();                             // the histogram and the map are cleared
  if (sampled) {
#pragma unroll
    for (int k = 0; k < kSample; ++k) if ((k + 1) * kBesideThreads <= (1 << bits)) count_top(score_key(sample[k]));
    find_top(rank);
    const uint32_t top = uint32_t(sm.bin);
    const int want = sm.want, reach = rank - want + sm.cnt;    // samples that reach the bin
    clear_digit();
    bound = top << 20;
    if (!even.list_has_room(reach, NG)) {                      // too coarse
#pragma unroll
      for (int k = 0; k < kSample; ++k) {
        const uint32_t key = score_key(sample[k]);
        if ((key >> 20) == top && (k + 1) * kBesideThreads <= (1 << bits)) atomicAdd(&sm.hist[(key >> 10) & (kDigit - 1)], 1u);
      }
      find_digit(want);
      bound |= uint32_t(sm.bin) << 10;
      clear_digit();
    }
  }

  // ---- the keys that reach the bound --------------------------------------------------------------------------------------
  int need_eq = 0;                             // keys of the map of equal keys (sm.hist) to take, lowest indices first
  uint32_t* const equal = sm.hist;
  if (!exact) {
    // scores are compared as floats; what is not below the bound and yet has a smaller key (a NaN) is left to the digits
    const float bound_score = __uint_as_float((bound & 0x80000000u) ? bound ^ 0x80000000u : ~bound);
    uint32_t key_max = 0u;
    bool odd = false;
    for (int v0 = 0; v0 < n_parts; v0 += kRound) {
      float4 next[P];                          // requested while this round is looked through
#pragma unroll
      for (int q = 0; q < P; ++q) next[q] = load(v0 + kRound + warp + kBesideWarps * q);
      const int i0 = (v0 + warp) * kBesidePart + 4 * lane;
      uint32_t hits = 0u;                      // bit 4 q + e
#pragma unroll
      for (int q = 0; q < P; ++q)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (!(beside_elem(x[q], e) < bound_score) && i0 + q * (kBesideWarps * kBesidePart) + e < NG) hits |= 1u << (4 * q + e);
      const int mine = __popc(hits);
      int incl = mine;                         // the lane's place in the warp's share of the list
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int t = __shfl_up_sync(kAll, incl, off);
        if (lane >= off) incl += t;
      }
      int slot = 0;
      if (lane == 31 && incl > 0) slot = atomicAdd(&sm.n_list, incl);
      slot = __shfl_sync(kAll, slot, 31) + incl - mine;
#pragma unroll
      for (int q = 0; q < P; ++q)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if ((hits >> (4 * q + e)) & 1u) {
            const uint32_t key = score_key(beside_elem(x[q], e));
            key_max = max(key_max, key);
            odd = odd || key < bound;
            if (slot < kListKeys) {
              sm.list_key[slot] = key;
              sm.list_idx[slot] = uint16_t(i0 + q * (kBesideWarps * kBesidePart) + e);
            }
            ++slot;
          }
#pragma unroll
      for (int q = 0; q < P; ++q) x[q] = next[q];
    }
    key_max = __reduce_max_sync(kAll, key_max);
    if (lane == 0) atomicMax(&sm.key_max, key_max);
    exact = __syncthreads_or(odd) || sm.n_list < Mp || sm.n_list > kListKeys;
  }
  if (!exact) {
    // ---- intervals of the list's keys, until few keys share the M'-th key's ------------------------------------------------
    const int n = sm.n_list;
    // `span` intervals of 2^shift keys from `low`, first over the whole list, then over the one interval found: the keys
    // above that are among the Mp - want that are selected already, and counted again they would raise the threshold.
    uint32_t low = bound, span = kDigit;
    int want = Mp, shift = max(0, 22 - __clz(int((sm.key_max - bound) | 1u)));
    while (true) {
      for (int j = tid; j < n; j += kBesideThreads) {
        const uint32_t k = sm.list_key[j];
        const uint32_t at = (k - low) >> shift;
        if (k >= low && at < span) atomicAdd(&sm.hist[at], 1u);
      }
      find_digit(want);
      low += uint32_t(sm.bin) << shift;
      want = sm.want;
      if (sm.cnt == want || sm.cnt <= kBesideFew || shift == 0) break;
      const int finer = max(0, shift - 10);
      span = 1u << (shift - finer);
      shift = finer;
      clear_digit();
    }
    const int cnt = sm.cnt;
    const bool whole = cnt == want, few = !whole && cnt <= kBesideFew, ties = !whole && !few;
    if (ties) {                                // shift = 0: equal keys, the lowest indices are taken
      need_eq = want;
      __syncthreads();
      clear_digit();
    }
    for (int j = tid; j < n; j += kBesideThreads) {
      const uint32_t k = sm.list_key[j];
      if (k < low) continue;
      if (whole || ((k - low) >> shift) != 0u) set(sm.sel, sm.list_idx[j]);
      else if (ties) set(equal, sm.list_idx[j]);
      else {
        const int at = atomicAdd(&sm.n_few, 1);
        if (at < kBesideFew) sm.few[at] = uint16_t(j);
      }
    }
    if (few) {                                 // one warp ranks them: larger key first, then the lower index
      __syncthreads();
      if (warp == 0) {
        const bool have = lane < min(sm.n_few, kBesideFew);
        const int j = have ? sm.few[lane] : 0;
        const uint32_t key = have ? sm.list_key[j] : 0u;
        const int idx = have ? int(sm.list_idx[j]) : 0x7fffffff;
        int rank = 0;
        for (int o = 0; o < cnt; ++o) {
          const uint32_t ko = __shfl_sync(kAll, key, o);
          const int io = __shfl_sync(kAll, idx, o);
          rank += (ko > key || (ko == key && io < idx)) ? 1 : 0;
        }
        if (have && rank < want) set(sm.sel, idx);
      }
    }
  } else {
    // ---- three digits over the whole row, read again ------------------------------------------------------------------------
    __syncthreads();
    for (int i = tid; i < kKeyTopBins / 2; i += kBesideThreads) sm.hist[i] = 0u;
    __syncthreads();
    auto count = [&](int known_shift, uint32_t known, int shift) {
      for (int i = tid; i < NG; i += kBesideThreads) {
        const uint32_t key = score_key(__ldcg(R + i));
        if ((key >> known_shift) == known) atomicAdd(&sm.hist[(key >> shift) & (kDigit - 1)], 1u);
      }
    };
    for (int i = tid; i < NG; i += kBesideThreads) count_top(score_key(__ldcg(R + i)));
    find_top(Mp);
    const uint32_t top = uint32_t(sm.bin);
    const int want = sm.want;
    clear_digit();
    count(20, top, 10);
    find_digit(want);
    const uint32_t prefix = (top << 10) | uint32_t(sm.bin);
    const int want2 = sm.want;
    clear_digit();
    count(10, prefix, 0);
    find_digit(want2);
    const uint32_t kth = (prefix << 10) | uint32_t(sm.bin);
    need_eq = sm.want;
    clear_digit();
    for (int v = warp; v < n_parts; v += kBesideWarps) {
      const float4 y = load(v);
      uint32_t gt_word = 0u, eq_word = 0u;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const bool have = v * kBesidePart + 4 * lane + e < NG;
        const uint32_t key = score_key(beside_elem(y, e));
        const uint32_t gt = __ballot_sync(kAll, have && key > kth), eq = __ballot_sync(kAll, have && key == kth);
        if (lane == e) { gt_word = gt; eq_word = eq; }
      }
      if (lane < 4) { sm.sel[4 * v + lane] = gt_word; equal[4 * v + lane] = eq_word; }
    }
  }
  __syncthreads();

  // ---- positions: an exclusive scan over the parts, selected and equal keys packed 16 + 16 bits --------------------------
  auto count4 = [](const uint4& m) { return uint32_t(__popc(m.x) + __popc(m.y) + __popc(m.z) + __popc(m.w)); };
  {
    uint32_t own = 0u;
    if (tid < n_parts) {
      own = count4(reinterpret_cast<const uint4*>(sm.sel)[tid]) << 16;
      if (need_eq > 0) own |= count4(reinterpret_cast<const uint4*>(equal)[tid]);
    }
    uint32_t incl = own;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t t = __shfl_up_sync(kAll, incl, off);
      if (lane >= off) incl += t;
    }
    if (lane == 31) sm.warp_tot[warp] = incl;
    __syncthreads();
    for (int w = 0; w < min(warp, kBesideParts / 32); ++w) incl += sm.warp_tot[w];
    if (tid < n_parts) sm.before[tid] = incl - own;
    __syncthreads();
  }
  if (!exact && need_eq == 0) {                // every selected key is on the list
    for (int j = tid; j < sm.n_list; j += kBesideThreads) {
      const int i = sm.list_idx[j], v = i / kBesidePart, e = i & 3;
      const uint32_t lanes = (1u << ((i % kBesidePart) >> 2)) - 1u, own = lanes + 1u;       // lanes below, the key's lane
      const uint4 m = reinterpret_cast<const uint4*>(sm.sel)[v];
      const uint32_t word = e == 0 ? m.x : e == 1 ? m.y : e == 2 ? m.z : m.w;
      if ((word & own) == 0u) continue;
      const uint32_t upto = lanes | own;       // words of the elements before e count the key's own lane too
      const int pos = int(sm.before[v] >> 16) + __popc(m.x & (e > 0 ? upto : lanes)) + __popc(m.y & (e > 1 ? upto : lanes)) +
                      __popc(m.z & (e > 2 ? upto : lanes)) + __popc(m.w & lanes);
      if (pos < p.M) out[pos] = i;
    }
    return;
  }
  for (int v = warp; v < n_parts; v += kBesideWarps) {
    const uint4 s = reinterpret_cast<const uint4*>(sm.sel)[v], q = reinterpret_cast<const uint4*>(equal)[v];
    const uint32_t before = sm.before[v];
    auto lower = [&](const uint4& m) { return __popc(m.x & below) + __popc(m.y & below) + __popc(m.z & below) + __popc(m.w & below); };
    int gt_before = int(before >> 16) + lower(s), eq_before = int(before & 0xffffu) + lower(q);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const uint32_t sw = e == 0 ? s.x : e == 1 ? s.y : e == 2 ? s.z : s.w, qw = e == 0 ? q.x : e == 1 ? q.y : e == 2 ? q.z : q.w;
      const bool gt = (sw >> lane) & 1u, eq = ((qw >> lane) & 1u) && eq_before < need_eq;
      const int pos = gt_before + min(eq_before, need_eq);
      if ((gt || eq) && pos < p.M) out[pos] = v * kBesidePart + 4 * lane + e;
      gt_before += gt;
      eq_before += (qw >> lane) & 1u;
    }
  }
}

// Parts per warp and round (1, 2 or 4); 0 when the row is too long for this select (or empty), or when so many are to be
// selected that the list has no room for what a sample lets through: counting the row's digits instead is exact, but
// slow (4 sequences, 16384 groups, M = 1400: 42.5 us a layer against 36.3 with the select behind the gather).
inline int plan_topk_beside(const Problem& p) {
  if (p.NG < 1 || p.NG > kBesideParts * kBesidePart) return 0;
  const BesideSample s = beside_sample(p.NG, p.Mp);
  if (p.NG > kListKeys && !s.list_has_room(s.rank, p.NG)) return 0;
  const int need = (p.NG + kBesidePart * kBesideWarps - 1) / (kBesidePart * kBesideWarps);
  return need <= 1 ? 1 : need <= 2 ? 2 : 4;
}

}  // namespace kvswap
