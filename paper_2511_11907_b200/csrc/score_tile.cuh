// Scores of eight metadata rows at a time on the tensor cores: the per-warp arithmetic of the streaming
// scorer (Eq. 1 and the head sum of Sec. 4.3), for metadata rows of R = 16, 32 or 64 entries in fp16,
// E4M3 (R = 32) or fp32.
//
// With joint metadata one row feeds up to 8 scores (the per-KV-head scopes): an [rows x R].[R x 8]
// contraction, which the fp32 pipes cannot sustain at HBM rate; it runs on mma.sync m16n8k16 with fp32
// accumulation and without rounding an input: scopes are the row operand, 8 tokens the column operand.
//   fp16, E4M3  (whose values convert to fp16 exactly): a query is scaled by a power of two and split into
//               an fp16 head (rows 0..7 of the row operand) and an fp16 remainder (rows 8..15), so one
//               instruction per k-step yields both partial products.
//   fp32        both operands are split into three bf16 pieces (8 + 8 + 8 mantissa bits); a k-step takes
//               the products u1 m1, u2 m1, u1 m2, u2 m2, u1 m3, u2 m3 and u3 m1, in four instructions: what
//               is left out is below 2^-24 of the product, the rounding of one fp32 multiplication.
//
// Operand layout.  Lane (g = lane / 4, t = lane % 4) reads the R / 4 consecutive entries t R/4 .. of row g of
// an 8-row block.  The contraction index may be permuted freely as long as both operands agree, so k-step
// j takes the lane's entries 4j .. 4j+3 as the four values it owes for token g (the column operand, 8 tokens
// wide), and the row operand holds the same entries of the query of scope g.  The accumulator then holds,
// in lane (g, t), the scores of scope g for tokens 2t and 2t+1.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "common.cuh"

namespace kvswap {

// One stage of staged metadata: the rows of kBytes bytes; META is a kvswap_dtype.
template <int META, int R>
struct MetaRows {
  static constexpr int kElem = META == KVSWAP_F32 ? 4 : META == KVSWAP_F16 ? 2 : 1;
  static constexpr int kRowBytes = R * kElem;
  static_assert(kRowBytes == 32 || kRowBytes == 64 || kRowBytes == 128 || kRowBytes == 256, "rows the tile reads are laid out for");
};

__device__ __forceinline__ void mma16816_f16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                             uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma16816_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                              uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t pack_half2(__half lo, __half hi) {
  return uint32_t(__half_as_ushort(lo)) | (uint32_t(__half_as_ushort(hi)) << 16);
}

// The row operand of one warp: lane (g, t) supplies entries t R/4 .. of the query of scope g.
template <int META, int R>
struct ScoreQuery {
  static constexpr int KS = R / 16, E = R / 4;
  uint32_t a[KS][4];                                 // a0, a2: rows 0..7, a1, a3: rows 8..15
  uint32_t third[META == KVSWAP_F32 ? KS : 1][2];    // fp32: the third piece (rows 0..7)
  float inv;                                         // undoes the scaling of this lane's scope

  // All lanes of the warp call.  meta_scale: the power of two the metadata is stored with.
  __device__ __forceinline__ void set(const float (&u)[E], float meta_scale) {
    if constexpr (META == KVSWAP_F32) {
      inv = meta_scale;
#pragma unroll
      for (int j = 0; j < KS; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t w[3];
          split3_bf16(u[4 * j + 2 * h], u[4 * j + 2 * h + 1], w);
          a[j][2 * h] = w[0]; a[j][2 * h + 1] = w[1]; third[j][h] = w[2];
        }
    } else {
      float mx = 0.f;
#pragma unroll
      for (int i = 0; i < E; ++i) mx = fmaxf(mx, fabsf(u[i]));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      // power of two that brings the largest entry into [2^14, 2^15)
      int sh = 0;
      if (mx > 0.f && mx < INFINITY) sh = min(120, max(-113, 14 - (int((__float_as_uint(mx) >> 23) & 0xffu) - 127)));
      const float scale = __uint_as_float(uint32_t(sh + 127) << 23);
      inv = __uint_as_float(uint32_t(127 - sh) << 23) * meta_scale;
      __half hi[E], lo[E];
#pragma unroll
      for (int i = 0; i < E; ++i) {
        const float us = u[i] * scale;
        hi[i] = __float2half_rn(us);
        lo[i] = __float2half_rn(us - __half2float(hi[i]));
      }
#pragma unroll
      for (int j = 0; j < KS; ++j) {
        a[j][0] = pack_half2(hi[4 * j], hi[4 * j + 1]); a[j][2] = pack_half2(hi[4 * j + 2], hi[4 * j + 3]);
        a[j][1] = pack_half2(lo[4 * j], lo[4 * j + 1]); a[j][3] = pack_half2(lo[4 * j + 2], lo[4 * j + 3]);
      }
    }
  }
  __device__ __forceinline__ void set(const float* u, float meta_scale) {       // E floats, 16-byte aligned
    float v[E];
#pragma unroll
    for (int i = 0; i < E / 4; ++i) {
      const float4 x = reinterpret_cast<const float4*>(u)[i];
      v[4 * i] = x.x; v[4 * i + 1] = x.y; v[4 * i + 2] = x.z; v[4 * i + 3] = x.w;
    }
    set(v, meta_scale);
  }
};

// Byte offset inside an 8-row block at which a lane starts reading (score_rows8 adds the rest).  Rows of 128
// bytes are read in two 16-byte pieces, the odd rows' in the other order, so that the eight lanes of a
// shared-memory phase fall into eight different bank groups; rows of 256 in four, the odd rows' halves swapped.
template <int META, int R>
__device__ __forceinline__ uint32_t score_lane_offset(int lane) {
  constexpr int kRowBytes = MetaRows<META, R>::kRowBytes;
  if constexpr (kRowBytes <= 64) return uint32_t(lane) * (kRowBytes / 4);
  else if constexpr (kRowBytes == 128) return uint32_t(lane >> 2) * 128u + uint32_t(lane & 3) * 32u + uint32_t((lane >> 2) & 1) * 16u;
  else return uint32_t(lane >> 2) * 256u + uint32_t(lane & 3) * 64u + uint32_t((lane >> 2) & 1) * 32u;
}

// Unscaled scores of scope g for tokens 2t and 2t + 1 of the 8-row block; `addr` = block + score_lane_offset().
template <int META, int R>
__device__ __forceinline__ void score_rows8(uint32_t addr, const ScoreQuery<META, R>& q, float* x0, float* x1) {
  constexpr int KS = R / 16, kRowBytes = MetaRows<META, R>::kRowBytes, kWords = kRowBytes / 16;
  uint32_t raw[kWords];                              // the lane's entries as stored
  if constexpr (kRowBytes == 32) {
    asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(raw[0]), "=r"(raw[1]) : "r"(addr));
  } else if constexpr (kRowBytes == 64) {
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(raw[0]), "=r"(raw[1]), "=r"(raw[2]), "=r"(raw[3]) : "r"(addr));
  } else if constexpr (kRowBytes == 256) {
    uint32_t x[16];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(x[4 * i]), "=r"(x[4 * i + 1]), "=r"(x[4 * i + 2]), "=r"(x[4 * i + 3])
                   : "r"(addr ^ uint32_t(i * 16)));
    const bool swapped = (addr & 32u) != 0u;         // blocks are 128-byte aligned
#pragma unroll
    for (int i = 0; i < 8; ++i) { raw[i] = swapped ? x[8 + i] : x[i]; raw[8 + i] = swapped ? x[i] : x[8 + i]; }
  } else {
    uint32_t x[4], y[4];
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]) : "r"(addr));
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(y[0]), "=r"(y[1]), "=r"(y[2]), "=r"(y[3]) : "r"(addr ^ 16u));
    const bool swapped = (addr & 16u) != 0u;         // blocks are 128-byte aligned
#pragma unroll
    for (int i = 0; i < 4; ++i) { raw[i] = swapped ? y[i] : x[i]; raw[4 + i] = swapped ? x[i] : y[i]; }
  }
  float d[4] = {0.f, 0.f, 0.f, 0.f};                 // d[0], d[1]: rows 0..7, d[2], d[3]: rows 8..15
  if constexpr (META == KVSWAP_F32) {
    uint32_t m[2 * KS][3];                           // the pieces of each pair of entries
#pragma unroll
    for (int i = 0; i < 2 * KS; ++i) split3_bf16(__uint_as_float(raw[2 * i]), __uint_as_float(raw[2 * i + 1]), m[i]);
#pragma unroll
    for (int j = 0; j < KS; ++j) {                   // small products first: the accumulator truncates
      mma16816_bf16(d, q.third[j][0], 0u, q.third[j][1], 0u, m[2 * j][0], m[2 * j + 1][0]);
      mma16816_bf16(d, q.a[j][0], q.a[j][1], q.a[j][2], q.a[j][3], m[2 * j][2], m[2 * j + 1][2]);
    }
#pragma unroll
    for (int k = 1; k >= 0; --k)
#pragma unroll
      for (int j = 0; j < KS; ++j) mma16816_bf16(d, q.a[j][0], q.a[j][1], q.a[j][2], q.a[j][3], m[2 * j][k], m[2 * j + 1][k]);
  } else {
    uint32_t w[2 * KS];                              // entries as fp16 pairs
    if constexpr (META == KVSWAP_E4M3) {
#pragma unroll
      for (int i = 0; i < 2 * KS; ++i) {
        const uint16_t pair = uint16_t(raw[i >> 1] >> ((i & 1) * 16));
        asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(w[i]) : "h"(pair));
      }
    } else {
#pragma unroll
      for (int i = 0; i < 2 * KS; ++i) w[i] = raw[i];
    }
#pragma unroll
    for (int j = 0; j < KS; ++j) mma16816_f16(d, q.a[j][0], q.a[j][1], q.a[j][2], q.a[j][3], w[2 * j], w[2 * j + 1]);
  }
  *x0 = d[0] + d[2];
  *x1 = d[1] + d[3];
}

// ReduceMax over the groups of one staged tile of `rows` rows (a multiple of G); `base` = stage +
// score_lane_offset().  Every finished group goes to publish(group within the tile, score) in exactly one lane,
// the lane of its scope (lane / 4), if `scope_ok`.  GS = log2 G: the maximum is a max over two registers and at
// most two shuffles.  GS = -1: any G, through the warp's buffer `sc` [8 scopes][generic_pitch(STAGE_ROWS)].
constexpr int kGenericRows = 48;                          // GS = -1: token rows per tile, at most
__host__ __device__ constexpr int generic_pitch(int rows) { return rows % 32 == 24 ? rows + 16 : rows + 8; }   // floats between scopes (bank spread)

template <int META, int R, int GS, int STAGE_ROWS, typename Publish>
__device__ __forceinline__ void score_tile_groups(uint32_t base, int rows, int lane, const ScoreQuery<META, R>& query,
                                                  int G, bool scope_ok, float* sc, const Publish& publish) {
  constexpr uint32_t kAll = 0xffffffffu;
  constexpr int kRowBytes = MetaRows<META, R>::kRowBytes;
  const int rq = lane >> 2, qt = lane & 3;
  if constexpr (GS >= 0) {
    const int ngt = rows >> GS;                       // groups in this tile
    float mine[(STAGE_ROWS + 31) / 32] = {};          // G = 8: the groups of reads qt, qt + 4, .. are this lane's to publish
    float run = -INFINITY;                            // running maximum of a 16- or 32-row group
#pragma unroll
    for (int it = 0; it < STAGE_ROWS / 8; ++it) {
      if (it * 8 < rows) {
        float x0, x1;
        score_rows8<META, R>(base + uint32_t(it) * 8u * kRowBytes, query, &x0, &x1);
        if constexpr (GS == 0) {                                   // tokens 2t and 2t+1 of this read are groups
          if (scope_ok && it * 8 + 2 * qt < rows) publish(it * 8 + 2 * qt, x0 * query.inv);
          if (scope_ok && it * 8 + 2 * qt + 1 < rows) publish(it * 8 + 2 * qt + 1, x1 * query.inv);
        } else {
          float m = fmaxf(x0, x1);
          if constexpr (GS >= 2) m = fmaxf(m, __shfl_xor_sync(kAll, m, 1));
          if constexpr (GS >= 3) m = fmaxf(m, __shfl_xor_sync(kAll, m, 2));
          // (a ragged last tile holds a whole number of groups, but not of 8-row reads when G < 8)
          if constexpr (GS == 1) { if (scope_ok && it * 4 + qt < ngt) publish(it * 4 + qt, m * query.inv); }
          else if constexpr (GS == 2) {
            if (scope_ok && (qt & 1) == 0 && it * 2 + (qt >> 1) < ngt) publish(it * 2 + (qt >> 1), m * query.inv);
          }
          else if constexpr (GS == 3) { if (qt == (it & 3)) mine[it >> 2] = m; }
          else {                                                   // G = 16 or 32: 2 or 4 reads per group
            run = fmaxf(run, m);
            if (((it + 1) & ((1 << (GS - 3)) - 1)) == 0) {
              const int gi = it >> (GS - 3);
              if (scope_ok && qt == (gi & 3)) publish(gi, run * query.inv);
              run = -INFINITY;
            }
          }
        }
      }
    }
    if constexpr (GS == 3) {
#pragma unroll
      for (int h = 0; h < (STAGE_ROWS + 31) / 32; ++h)
        if (scope_ok && (4 * h + qt) * 8 < rows) publish(4 * h + qt, mine[h] * query.inv);
    }
  } else {
#pragma unroll 2
    for (int it = 0; it * 8 < rows; ++it) {
      float x0, x1;
      score_rows8<META, R>(base + uint32_t(it) * 8u * kRowBytes, query, &x0, &x1);
      *reinterpret_cast<float2*>(sc + rq * generic_pitch(STAGE_ROWS) + it * 8 + 2 * qt) = make_float2(x0 * query.inv, x1 * query.inv);
    }
    __syncwarp();
    const int ngt = rows / G;
    if (scope_ok) {
      for (int gi = qt; gi < ngt; gi += 4) {
        const float* s = sc + rq * generic_pitch(STAGE_ROWS) + gi * G;
        float m = s[0];
        for (int i = 1; i < G; ++i) m = fmaxf(m, s[i]);
        publish(gi, m);
      }
    }
  }
}

// Rows of one stage: 4 KB where a finished score leaves the registers (the hand-over of a stage costs the
// same whatever its size: 4 KB x 2 stages measured 1.3 us per layer faster than 2 KB x 4 at B = 4,
// N = 131072); GS = -1 takes 3 KB, which leaves room for the warps' score buffers.  A stage is read eight rows at
// a time, whole: it holds a multiple of eight, which for rows of 256 bytes takes 4 KB; so do 32 rows of 128 bytes.
__host__ __device__ constexpr int score_stage_bytes(bool generic, int row_bytes) { return generic && row_bytes < 128 ? 3072 : 4096; }
__host__ __device__ constexpr int score_stage_rows(bool generic, int row_bytes) {
  const int fit = score_stage_bytes(generic, row_bytes) / row_bytes;
  return generic && fit > kGenericRows ? kGenericRows : fit;
}
template <int META, int R, int GS>
struct ScoreStage {
  static constexpr int kBytes = score_stage_bytes(GS < 0, MetaRows<META, R>::kRowBytes);
  static constexpr int kRows = score_stage_rows(GS < 0, MetaRows<META, R>::kRowBytes);
  static_assert(kRows % 8 == 0, "whole reads");
};

}  // namespace kvswap
