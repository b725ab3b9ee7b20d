// Softmax variant of the scorer on the tensor cores (KVSWAP_SCORE_SOFTMAX; what it computes: score_softmax.cu)
// for metadata rows that are dense in memory, fp16 or fp32 of rank 16, 32 or 64.
//
//   softmax_tc_stats_kernel  per head the running maximum and sum of 2^(logit - max) over a share of the tokens
//   softmax_tc_pool_kernel   the logits again (the rows now come from L2), weights, sum over the heads of a scope,
//                            maximum over the tokens of a group, leading-digit counts for the TopK
//
// Both walk the tiles as the streaming scorer does (score_stream.cuh): 16 warps per CTA, each with its own
// contiguous share of tiles and its own ring of stages filled by bulk asynchronous copies (bounded waits), the first
// ones requested ahead of the dependency wait: the query kernel in front of both lets its successor start only after its
// own wait, when all that came before it, the metadata's producer included, was complete.  A CTA belongs to one row set.  The logits of eight heads and
// eight tokens are one call of score_rows8() (score_tile.cuh: products exact, one rounding per accumulation);
// the row operands of all heads of the set, "blocks" of eight, lie ready as fragments in shared memory, so the
// number of heads is not limited by registers.
//
// Which heads share a block follows from what is summed.  Heads of one KV head are summed over lanes, so rho of
// up to eight is padded to a power of two P and a block holds 8 / P KV heads (one "unit" of kb = 1 blocks); a
// larger rho, or a sum over all heads, is a unit of kb blocks whose weights are added in the lanes first.
//
// Bound by instruction issue: per eight tokens and eight heads 2 to 4 matrix instructions, two exponentials per
// lane and up to eight shuffles, twice the logits; not by memory (the kernels it replaced read each row two bytes
// at a time per lane and took 14 + 19 us at B = 4, N = 40001, 16 heads, r = 32).
#pragma once

#include "async_copy.cuh"
#include "common.cuh"
#include "lowrank_query.cuh"
#include "score_tile.cuh"
#include "topk_keys.cuh"

namespace kvswap {

constexpr int kSoftmaxWarps = 16;
constexpr int kSoftmaxThreads = kSoftmaxWarps * 32;
constexpr int kSoftmaxMaxRows = 48;                       // token rows per tile
constexpr int kSoftmaxMultiTiles = 8;                     // tiles whose weights a warp sums over the metadata heads together
constexpr int kSoftmaxScopes = kQueryCols;                // scopes of a row set

struct SoftmaxArgs {
  const float* u;           // [B, H_q, r] per-head low-rank queries, scaled by log2(e) / sqrt(d)
  const unsigned char* meta;
  float* stats;             // [B, H_q, stat_pitch] pairs (max, sum), stat_parts of them valid
  float* scores;
  uint32_t* top_hist;       // NULL, or [B * S, 4096] 16-bit counters (score_stream.cuh)
  int stat_pitch, stat_parts;
  int tile_rows, tiles, stage_bytes, depth, ctas_per_set, n_sub;
  int units, kb, p_shift;   // pool: units of kb blocks, P = 1 << p_shift lanes per sum
  int n_blocks;
  int pitch;                // pool: floats between scopes of a warp's buffer
  bool atomic;              // pool: groups are longer than a tile: maxima meet in the score row (cleared by the stats kernel)
  uint32_t* err;
};

// Ready row operands of one block: lane-major vectors, so that a warp reads them without bank conflicts.
template <int META, int R>
struct SoftmaxBlock {
  static constexpr int KS = R / 16;
  uint4 a[KS][32];
  uint2 third[META == KVSWAP_F32 ? KS : 1][32];
  float inv[32];

  __device__ __forceinline__ void put(const ScoreQuery<META, R>& q, int lane) {
#pragma unroll
    for (int j = 0; j < KS; ++j) a[j][lane] = make_uint4(q.a[j][0], q.a[j][1], q.a[j][2], q.a[j][3]);
    if constexpr (META == KVSWAP_F32) {
#pragma unroll
      for (int j = 0; j < KS; ++j) third[j][lane] = make_uint2(q.third[j][0], q.third[j][1]);
    }
    inv[lane] = q.inv;
  }
  __device__ __forceinline__ void get(ScoreQuery<META, R>& q, int lane) const {
#pragma unroll
    for (int j = 0; j < KS; ++j) {
      const uint4 v = a[j][lane];
      q.a[j][0] = v.x; q.a[j][1] = v.y; q.a[j][2] = v.z; q.a[j][3] = v.w;
    }
    if constexpr (META == KVSWAP_F32) {
#pragma unroll
      for (int j = 0; j < KS; ++j) { const uint2 v = third[j][lane]; q.third[j][0] = v.x; q.third[j][1] = v.y; }
    }
    q.inv = inv[lane];
  }
};

// Row operand of the block whose row lane / 4 is head `head` (or nothing: -1) of sequence b.
template <int META, int R>
__device__ __forceinline__ void softmax_put_block(SoftmaxBlock<META, R>* blk, const Problem& p, const float* u, int b, int head,
                                                  int lane) {
  const float4* src = reinterpret_cast<const float4*>(u + (int64_t(b) * p.Hq + max(head, 0)) * R + (lane & 3) * (R / 4));
  float v[R / 4];
#pragma unroll
  for (int i = 0; i < R / 16; ++i) {
    const float4 x = head >= 0 ? __ldcg(src + i) : make_float4(0.f, 0.f, 0.f, 0.f);
    v[4 * i] = x.x; v[4 * i + 1] = x.y; v[4 * i + 2] = x.z; v[4 * i + 3] = x.w;
  }
  ScoreQuery<META, R> q;
  q.set(v, 1.f);
  blk->put(q, lane);
}

// A warp's ring of stages over one metadata array of a row set.
struct SoftmaxRing {
  uint32_t base, bars;      // shared-memory addresses
  const unsigned char* src; // tile 0
  int row_bytes, stage_bytes, tile_rows, rows_total, lane;

  __device__ __forceinline__ int rows(int tile) const { return min(tile_rows, rows_total - tile * tile_rows); }
  __device__ __forceinline__ void fill(int tile, int64_t offset, int stage) const {
    if (lane != 0) return;
    const uint32_t bytes = uint32_t(rows(tile)) * uint32_t(row_bytes), bar = bars + uint32_t(stage) * 8u;
    mbar_arrive_expect_tx(bar, bytes);
    bulk_g2s(base + uint32_t(stage * stage_bytes), src + offset + int64_t(tile) * tile_rows * row_bytes, bytes, bar);
  }
  __device__ __forceinline__ void init(int depth) const {
    if (lane == 0) {
      for (int s = 0; s < depth; ++s) mbar_init(bars + uint32_t(s) * 8u, 1);
      mbar_init_fence();
    }
    __syncwarp();
  }
  // After a wait that gave up: records it, and gives copies in flight a bounded chance to land.
  __device__ __forceinline__ void give_up(int depth, uint32_t* err) const {
    if (lane == 0 && err) atomicExch(err, kDevTimeoutFull);
    for (int s = 0; s < depth; ++s) { mbar_wait(bars + uint32_t(s) * 8u, 0); mbar_wait(bars + uint32_t(s) * 8u, 1); }
  }
};

// ------------------------------------------------------------------------------------------
// Statistics.  Row set = (sequence, metadata head): all heads that read it, eight per block.
// ------------------------------------------------------------------------------------------
template <int META, int R>
__global__ void __launch_bounds__(kSoftmaxThreads, 1)
softmax_tc_stats_kernel(Problem p, SoftmaxArgs a) {
  constexpr uint32_t kAll = 0xffffffffu;
  constexpr int kRowBytes = MetaRows<META, R>::kRowBytes, kElem = MetaRows<META, R>::kElem;
  constexpr int kReads = kSoftmaxMaxRows / 8;
  extern __shared__ __align__(128) unsigned char dyn[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rq = lane >> 2, qt = lane & 3;
  const int set = blockIdx.x / a.ctas_per_set, cta_in = blockIdx.x - set * a.ctas_per_set;
  const int b = set / p.Hm, hm = set - b * p.Hm;
  const int h0 = (p.Hm == 1) ? 0 : hm * p.rho, nh = (p.Hm == 1) ? p.Hq : p.rho, nb = (nh + 7) / 8;
  unsigned char* after = dyn + size_t(kSoftmaxWarps) * a.depth * a.stage_bytes;
  auto* blocks = reinterpret_cast<SoftmaxBlock<META, R>*>(after);
  float2* state = reinterpret_cast<float2*>(blocks + nb);                        // [warp][block][lane] (max, sum)
  unsigned long long* bars = reinterpret_cast<unsigned long long*>(state + kSoftmaxWarps * nb * 32);

  SoftmaxRing ring{smem_addr(dyn) + uint32_t(warp * a.depth * a.stage_bytes), smem_addr(bars + warp * 2),
                   a.meta + (int64_t(b) * p.meta_sb + int64_t(hm) * p.meta_sh) * kElem, kRowBytes, a.stage_bytes, a.tile_rows,
                   p.NG * p.G, lane};
  ring.init(a.depth);
  const int n_warps = a.ctas_per_set * kSoftmaxWarps, wi = cta_in * kSoftmaxWarps + warp;
  const int base_tiles = a.tiles / n_warps, rem = a.tiles - base_tiles * n_warps;
  const int first = wi * base_tiles + min(wi, rem), my_tiles = base_tiles + (wi < rem ? 1 : 0);
  for (int k = 0; k < a.depth && k < my_tiles; ++k) ring.fill(first + k, 0, k);
  for (int i = lane; i < nb * 32; i += 32) state[warp * nb * 32 + i] = make_float2(-INFINITY, 0.f);
  pdl_wait();
  pdl_trigger();
  if (a.atomic) {                                    // the pooling kernel takes maxima in this sequence's score rows
    const int64_t elems = int64_t(p.B) * p.S * p.score_pitch;
    for (int64_t i = int64_t(blockIdx.x) * kSoftmaxThreads + threadIdx.x; i < elems; i += int64_t(gridDim.x) * kSoftmaxThreads)
      a.scores[i] = 0.f;
  }
  for (int blk = warp; blk < nb; blk += kSoftmaxWarps) {
    const int h = blk * 8 + rq;
    softmax_put_block<META, R>(&blocks[blk], p, a.u, b, h < nh ? h0 + h : -1, lane);
  }
  __syncthreads();

  int stage = 0;
  uint32_t phase = 0;
  bool ok = true;
  for (int k = 0; k < my_tiles; ++k) {
    ok = __all_sync(kAll, mbar_wait(ring.bars + uint32_t(stage) * 8u, phase));
    if (!ok) break;
    const int rows = ring.rows(first + k);
    const uint32_t base = ring.base + uint32_t(stage * a.stage_bytes) + score_lane_offset<META, R>(lane);
    for (int blk = 0; blk < nb; ++blk) {
      ScoreQuery<META, R> q;
      blocks[blk].get(q, lane);
      float2 st = state[(warp * nb + blk) * 32 + lane];
      float x[2 * kReads], m = st.x;
#pragma unroll
      for (int it = 0; it < kReads; ++it) {
        x[2 * it] = x[2 * it + 1] = -INFINITY;
        if (it * 8 < rows) {
          float x0, x1;
          score_rows8<META, R>(base + uint32_t(it) * 8u * kRowBytes, q, &x0, &x1);
          if (it * 8 + 2 * qt < rows) x[2 * it] = x0 * q.inv;
          if (it * 8 + 2 * qt + 1 < rows) x[2 * it + 1] = x1 * q.inv;
          m = fmaxf(m, fmaxf(x[2 * it], x[2 * it + 1]));
        }
      }
      if (m > -INFINITY) {
        float l = st.y * exp2f(st.x - m);
#pragma unroll
        for (int i = 0; i < 2 * kReads; ++i) if ((i / 2) * 8 < rows) l += exp2f(x[i] - m);
        state[(warp * nb + blk) * 32 + lane] = make_float2(m, l);
      }
    }
    __syncwarp();
    if (k + a.depth < my_tiles) ring.fill(first + k + a.depth, 0, stage);
    if (++stage == a.depth) { stage = 0; phase ^= 1u; }
  }
  if (!ok) ring.give_up(a.depth, a.err);

  // ---- one (max, sum) per head: 64 partial states each, four heads per warp and round ------------------------------
  __syncthreads();
  for (int h8 = warp * 4; h8 < nb * 8; h8 += kSoftmaxWarps * 4) {
    const int h = h8 + (lane >> 3), part = lane & 7;
    float m = -INFINITY, l = 0.f;
    float2 v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int e = part + 8 * i;                    // warp e / 4, token lane e % 4
      v[i] = state[((e >> 2) * nb + h / 8) * 32 + (h & 7) * 4 + (e & 3)];
      m = fmaxf(m, v[i].x);
    }
#pragma unroll
    for (int off = 1; off <= 4; off <<= 1) m = fmaxf(m, __shfl_xor_sync(kAll, m, off));
#pragma unroll
    for (int i = 0; i < 8; ++i) l += (v[i].x > -INFINITY) ? v[i].y * exp2f(v[i].x - m) : 0.f;
#pragma unroll
    for (int off = 1; off <= 4; off <<= 1) l += __shfl_xor_sync(kAll, l, off);
    if (part == 0 && h < nh)
      reinterpret_cast<float2*>(a.stats)[(int64_t(b) * p.Hq + h0 + h) * a.stat_pitch + cta_in] = make_float2(m, l);
  }
}

// ------------------------------------------------------------------------------------------
// Weights, head sum, group maximum.
// ------------------------------------------------------------------------------------------
template <int META, int R>
__global__ void __launch_bounds__(kSoftmaxThreads, 1)
softmax_tc_pool_kernel(Problem p, SoftmaxArgs a) {
  constexpr uint32_t kAll = 0xffffffffu;
  constexpr int kRowBytes = MetaRows<META, R>::kRowBytes, kElem = MetaRows<META, R>::kElem;
  constexpr int kReads = kSoftmaxMaxRows / 8;
  constexpr int kCounters = kSoftmaxScopes * kKeyTopBins / 2;    // words of two 16-bit counters
  extern __shared__ __align__(128) unsigned char dyn[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rq = lane >> 2, qt = lane & 3;
  const int set = blockIdx.x / a.ctas_per_set, cta_in = blockIdx.x - set * a.ctas_per_set;
  const RowSet rs = row_set(p, set, a.n_sub);
  const bool multi = multi_term(p), scoped = p.Hm == 1 && p.scope == KVSWAP_SCOPE_KV_HEAD;
  const int s0 = scoped ? rs.sub * kSoftmaxScopes : (p.scope == KVSWAP_SCOPE_KV_HEAD ? rs.hm : 0);
  const int ns = scoped ? min(kSoftmaxScopes, p.S - s0) : 1;
  const int nb = a.n_blocks;
  unsigned char* after = dyn + size_t(kSoftmaxWarps) * a.depth * a.stage_bytes;
  uint32_t* hist = reinterpret_cast<uint32_t*>(after);
  if (a.top_hist != nullptr) after += kCounters * 4;
  auto* blocks = reinterpret_cast<SoftmaxBlock<META, R>*>(after);
  float2* norm = reinterpret_cast<float2*>(blocks + nb);                         // [block * 8 + row] (max, 1 / sum)
  float* sc = reinterpret_cast<float*>(norm + nb * 8) + warp * kSoftmaxScopes * a.pitch;
  unsigned long long* bars = reinterpret_cast<unsigned long long*>(reinterpret_cast<float*>(norm + nb * 8) +
                                                                   kSoftmaxWarps * kSoftmaxScopes * a.pitch);

  SoftmaxRing ring{smem_addr(dyn) + uint32_t(warp * a.depth * a.stage_bytes), smem_addr(bars + warp * 2),
                   a.meta + (int64_t(rs.b) * p.meta_sb + int64_t(rs.hm) * p.meta_sh) * kElem, kRowBytes, a.stage_bytes,
                   a.tile_rows, p.NG * p.G, lane};
  ring.init(a.depth);
  const int n_warps = a.ctas_per_set * kSoftmaxWarps, wi = cta_in * kSoftmaxWarps + warp;
  const int base_tiles = a.tiles / n_warps, rem = a.tiles - base_tiles * n_warps;
  const int first = wi * base_tiles + min(wi, rem), my_tiles = base_tiles + (wi < rem ? 1 : 0);

  // Stages in order: tile by tile; with several terms, block after block of at most kSoftmaxMultiTiles tiles, metadata
  // head by metadata head inside a block.
  const int n_terms = multi ? p.Hkv : 1, my_stages = my_tiles * n_terms;
  struct Cursor { int tile, block, term, in; };
  auto advance = [&](Cursor& c) {
    if (++c.in < c.block) return;
    c.in = 0;
    if (++c.term < n_terms) return;
    c.term = 0;
    c.tile += c.block;
    c.block = min(multi ? kSoftmaxMultiTiles : 1, max(1, my_tiles - c.tile));
  };
  Cursor f{0, min(multi ? kSoftmaxMultiTiles : 1, max(1, my_tiles)), 0, 0}, c = f;
  auto fill = [&](int stage) {
    ring.fill(first + f.tile + f.in, int64_t(f.term) * p.meta_sh * kElem, stage);
    advance(f);
  };
  for (int k = 0; k < a.depth && k < my_stages; ++k) fill(k);
  if (a.top_hist != nullptr)
    for (int i = threadIdx.x; i < ns * (kKeyTopBins / 8); i += kSoftmaxThreads) reinterpret_cast<uint4*>(hist)[i] = make_uint4(0u, 0u, 0u, 0u);
  pdl_wait();
  pdl_trigger();

  // ---- row operands and normalisers of the set's heads ---------------------------------------------------------------
  const int P = 1 << a.p_shift, per_unit = 8 >> a.p_shift;         // lanes per sum, KV heads per unit (kb = 1)
  auto head_of = [&](int slot) -> int {                            // head behind row slot % 8 of block slot / 8, or -1
    const int blk = slot >> 3, row = slot & 7, unit = blk / a.kb, k = blk - unit * a.kb;
    if (scoped) {
      const int kvh = (a.kb == 1) ? unit * per_unit + (row >> a.p_shift) : unit;
      const int j = (a.kb == 1) ? (row & (P - 1)) : k * 8 + row;
      return (kvh < ns && j < p.rho) ? (s0 + kvh) * p.rho + j : -1;
    }
    const int j = k * 8 + row;
    if (p.Hm == 1) return j < p.Hq ? j : -1;                       // all heads
    return j < p.rho ? (multi ? unit : rs.hm) * p.rho + j : -1;
  };
  for (int blk = warp; blk < nb; blk += kSoftmaxWarps)
    softmax_put_block<META, R>(&blocks[blk], p, a.u, rs.b, head_of(blk * 8 + rq), lane);
  for (int slot = warp; slot < nb * 8; slot += kSoftmaxWarps) {
    const int h = head_of(slot);
    float m = -INFINITY, l = 0.f;
    if (h >= 0) {                                                  // warp-uniform
      const float2* src = reinterpret_cast<const float2*>(a.stats) + (int64_t(rs.b) * p.Hq + h) * a.stat_pitch;
      constexpr int kParts = (kNumSMs + 31) / 32;                   // a set has at most one CTA per SM
      float2 v[kParts];
#pragma unroll
      for (int i = 0; i < kParts; ++i) {
        v[i] = (lane + 32 * i < a.stat_parts) ? __ldcg(src + lane + 32 * i) : make_float2(-INFINITY, 0.f);
        m = fmaxf(m, v[i].x);
      }
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) m = fmaxf(m, __shfl_xor_sync(kAll, m, off));
#pragma unroll
      for (int i = 0; i < kParts; ++i) if (v[i].x > -INFINITY) l += v[i].y * exp2f(v[i].x - m);
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) l += __shfl_xor_sync(kAll, l, off);
    }
    if (lane == 0) norm[slot] = (h >= 0) ? make_float2(m, 1.f / l) : make_float2(0.f, 0.f);   // l >= 1: the maximum itself
  }
  __syncthreads();

  auto sum_lanes = [&](float x) {                                  // over the heads of one sum
    if (P >= 2) x += __shfl_xor_sync(kAll, x, 4);
    if (P >= 4) x += __shfl_xor_sync(kAll, x, 8);
    if (P >= 8) x += __shfl_xor_sync(kAll, x, 16);
    return x;
  };
  auto publish = [&](int s, int g, float x) {                      // scope of the set, group
    const int64_t prob = int64_t(rs.b) * p.S + s0 + s;
    x += 0.f;
    if (a.atomic) { atomicMax(reinterpret_cast<int*>(a.scores + prob * p.score_pitch + g), __float_as_int(x)); return; }
    a.scores[prob * p.score_pitch + g] = x;
    if (a.top_hist != nullptr) {
      const uint32_t bin = score_key_top(x);
      atomicAdd(&hist[(s * kKeyTopBins + int(bin)) >> 1], 1u << ((bin & 1u) << 4));
    }
  };
  // Maxima over the groups of tokens [n0, n0 + rows), whose weights lie in sc[scope * pitch + token - n0].
  auto pool = [&](int n0, int rows, int scopes, int pitch) {
    const int g0 = n0 / p.G, n_groups = (n0 + rows - 1) / p.G - g0 + 1;
    for (int i = lane; i < scopes * n_groups; i += 32) {
      const int s = i / n_groups, g = g0 + i - s * n_groups;
      const int t0 = max(n0, g * p.G) - n0, t1 = min(n0 + rows, (g + 1) * p.G) - n0;
      const float* w = sc + s * pitch;
      float m = w[t0];
      for (int t = t0 + 1; t < t1; ++t) m = fmaxf(m, w[t]);
      publish(s, g, m);
    }
  };

  int stage = 0;
  uint32_t phase = 0;
  bool ok = true;
  for (int k = 0; k < my_stages; ++k) {
    ok = __all_sync(kAll, mbar_wait(ring.bars + uint32_t(stage) * 8u, phase));
    if (!ok) break;
    const int tile = first + c.tile + c.in, rows = ring.rows(tile);
    const uint32_t base = ring.base + uint32_t(stage * a.stage_bytes) + score_lane_offset<META, R>(lane);
    const int u0 = multi ? c.term : 0, u1 = multi ? c.term + 1 : a.units;
    for (int unit = u0; unit < u1; ++unit) {
      const int s = unit * per_unit + (rq >> a.p_shift);           // scope of this lane's sum
      const bool owner = multi ? rq == 0 : (rq & (P - 1)) == 0 && s < ns;
      float* dst = multi ? sc + c.in * a.tile_rows : sc + s * a.pitch;
      auto put = [&](int it, float x0, float x1) {
        x0 = sum_lanes(x0); x1 = sum_lanes(x1);
        const int t = it * 8 + 2 * qt;
        if (!owner) return;
        if (!multi) {
          *reinterpret_cast<float2*>(dst + t) = make_float2(x0, x1);
        } else {                                                   // (a tile's rows need not be whole reads)
          if (t < rows) dst[t] = (c.term == 0 ? 0.f : dst[t]) + x0;
          if (t + 1 < rows) dst[t + 1] = (c.term == 0 ? 0.f : dst[t + 1]) + x1;
        }
      };
      auto weights = [&](const ScoreQuery<META, R>& q, float2 n, int it, float* x0, float* x1) {
        score_rows8<META, R>(base + uint32_t(it) * 8u * kRowBytes, q, x0, x1);
        *x0 = exp2f(*x0 * q.inv - n.x) * n.y;
        *x1 = exp2f(*x1 * q.inv - n.x) * n.y;
      };
      ScoreQuery<META, R> q;
      if (a.kb == 1) {
        blocks[unit].get(q, lane);
        const float2 n = norm[unit * 8 + rq];
#pragma unroll
        for (int it = 0; it < kReads; ++it)
          if (it * 8 < rows) {
            float x0, x1;
            weights(q, n, it, &x0, &x1);
            put(it, x0, x1);
          }
      } else {
        float x[2 * kReads] = {};
        for (int kk = 0; kk < a.kb; ++kk) {
          blocks[unit * a.kb + kk].get(q, lane);
          const float2 n = norm[(unit * a.kb + kk) * 8 + rq];
#pragma unroll
          for (int it = 0; it < kReads; ++it)
            if (it * 8 < rows) {
              float x0, x1;
              weights(q, n, it, &x0, &x1);
              x[2 * it] += x0; x[2 * it + 1] += x1;
            }
        }
#pragma unroll
        for (int it = 0; it < kReads; ++it) if (it * 8 < rows) put(it, x[2 * it], x[2 * it + 1]);
      }
    }
    __syncwarp();
    if (!multi) {
      pool(tile * a.tile_rows, rows, ns, a.pitch);
    } else if (c.term == n_terms - 1 && c.in == c.block - 1) {     // the block's sums are complete
      const int t0 = first + c.tile;
      pool(t0 * a.tile_rows, min((t0 + c.block) * a.tile_rows, ring.rows_total) - t0 * a.tile_rows, 1, 0);
    }
    __syncwarp();                                                  // every lane is done with the stage and the buffer
    advance(c);
    if (k + a.depth < my_stages) fill(stage);
    if (++stage == a.depth) { stage = 0; phase ^= 1u; }
  }
  if (!ok) ring.give_up(a.depth, a.err);

  // ---- the CTA's counts join the global histograms ---------------------------------------------------------------------
  if (a.top_hist != nullptr) {
    __syncthreads();
    for (int i = threadIdx.x; i < ns * (kKeyTopBins / 8); i += kSoftmaxThreads) {
      const uint4 v = reinterpret_cast<const uint4*>(hist)[i];
      if ((v.x | v.y | v.z | v.w) == 0u) continue;
      const int col = (i * 8) / kKeyTopBins;                       // 8 counters per vector
      unsigned long long* H = reinterpret_cast<unsigned long long*>(
          a.top_hist + (int64_t(rs.b) * p.S + s0 + col) * (kKeyTopBins / 2) + ((i * 4) % (kKeyTopBins / 2)));
      const unsigned long long lo = (unsigned long long)v.x | ((unsigned long long)v.y << 32);
      const unsigned long long hi = (unsigned long long)v.z | ((unsigned long long)v.w << 32);
      if (lo != 0ull) atomicAdd(H, lo);
      if (hi != 0ull) atomicAdd(H + 1, hi);
    }
  }
}

// Host: shared memory of the two kernels, and their launches.  Instantiated in score_softmax_tc.cu.
template <int META, int R>
size_t softmax_tc_smem(const SoftmaxArgs& a, bool pool, bool counts) {
  const size_t ring = size_t(kSoftmaxWarps) * a.depth * a.stage_bytes;
  const size_t blocks = size_t(a.n_blocks) * sizeof(SoftmaxBlock<META, R>), bars = size_t(kSoftmaxWarps) * 16;
  if (!pool) return ring + blocks + size_t(kSoftmaxWarps) * a.n_blocks * 32 * sizeof(float2) + bars;
  return ring + blocks + (counts ? size_t(kSoftmaxScopes) * kKeyTopBins * 2 : 0) + size_t(a.n_blocks) * 8 * sizeof(float2) +
         size_t(kSoftmaxWarps) * kSoftmaxScopes * a.pitch * sizeof(float) + bars;
}

}  // namespace kvswap
