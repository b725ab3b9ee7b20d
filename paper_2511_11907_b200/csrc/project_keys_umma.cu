// K1 on the 5th-generation tensor cores: metadata build K_lr = Flatten(K) A (Sec. 4.2) with
// tcgen05.mma, accumulators in tensor memory and operands staged by TMA.
//
// Covers bf16 and fp16 K with d in {64, 128} and r in {16, 32, 64} (r = 32, d = 128 are the benchmark
// shapes); project_keys.cu keeps the warp-level path for everything else.
//
// The adapter stays fp32-exact: every entry is split into three pieces of K's type (fp16: scaled by a
// power of two per column, undone in the epilogue), laid out by a small preparation kernel as a K-major [3r x d] operand per KV head, so one instruction shape
// M = 128 tokens, N = 3r (48, 96 or 192) columns, K = 16 channels yields the three partial products
// side by side; the epilogue adds them in fp32.  The tensor core adds into its accumulator with
// truncation, so a chain inside tensor memory covers one KV head (d / 16 instructions); the sum
// over the heads of a joint row is kept in registers with round-to-nearest adds.
//
// CTA = 6 warps, persistent (one per SM):
//   warp 0   producer: per (token tile, KV head) d / 64 TMA boxes of K (128 rows x 64 channels,
//            128-byte swizzle) and as many of the split adapter into a ring of stages;
//   warp 1   issues the MMAs (one thread), owns the tensor-memory allocation (two accumulators);
//   warps 2-5 epilogue: tcgen05.ld of the finished accumulator (one token row per thread), sum of
//            the three pieces, running sum over heads, one rounding into the metadata type.
// fp16 K used to take the fp32-pipe kernel: a layer of 4 x 32768 tokens (8 heads of 128, r = 32) took 402 us, here
// 57 us, bf16 52 us.  (Prompts of a few thousand tokens: project_keys_short.cu.)  The launch overlaps the split of the adapter (programmatic
// dependent launch, K requested before the wait): four layers of 4 x 131072 bf16 tokens 879 -> 859 us.
// Stages and accumulators are handed over through mbarriers; every wait is bounded.
#include <algorithm>
#include <type_traits>

#include "async_copy.cuh"
#include "common.cuh"
#include "project_keys_short.cuh"
#include "tensor_map.cuh"
#include "umma.cuh"

namespace kvswap {
namespace {

constexpr int kTileM = 128;                                // tokens per tile
constexpr uint32_t kAHalf = kTileM * 128;                  // 128 rows x 128 bytes (64 channels of 16 bits)
constexpr int kThreadsUmma = 6 * 32;
constexpr size_t kMaxDynamicSmem = 227 * 1024;
constexpr int kMaxStages = 6;

// Sizes for head dimension D and rank R.
template <int D, int R>
struct Cfg {
  static constexpr int kD = D, kR = R;
  static constexpr int kNcols = 3 * R;                                   // accumulator columns: the three pieces side by side
  static constexpr int kHalves = D / 64;                                 // 128-byte-wide boxes per operand row
  static constexpr uint32_t kBHalf = uint32_t(kNcols) * 128;
  static constexpr uint32_t kStageBytes = kHalves * (kAHalf + kBHalf);   // d = 128, r = 32: 57344
  // as many stages as fit beside the 1 KB of alignment slack, six at most (d = 128: 4 at r = 32, 5 at r = 16, 2 at r = 64)
  static constexpr int kFit = int((kMaxDynamicSmem - 1024) / kStageBytes);
  static constexpr int kStages = kFit > kMaxStages ? kMaxStages : kFit;
  static_assert(kStages >= 2, "at least two stages");
  static constexpr uint32_t kAccStride = (kNcols <= 128) ? 128 : 256;    // tensor-memory columns between the two accumulators
  static constexpr uint32_t kTmemCols = 2 * kAccStride;
  static_assert((D == 64 || D == 128) && (R == 16 || R == 32 || R == 64), "shapes of the tcgen05 projection");
  static_assert(kNcols % 16 == 0 && kNcols <= 256, "N of a 128-row tcgen05.mma");
};

// ---- the adapter as three 16-bit pieces, [g][piece * r + j][c] (K-major rows of d channels) ----------
// bf16 pieces carry 8 + 8 + 8 mantissa bits at fp32's exponent range.  fp16 pieces carry 11 bits each but
// bottom out at 2^-24, so every column of a head (of a pair of heads that share an accumulator) is first
// multiplied by a power of two that brings its largest entry into [2^14, 2^15): what the three pieces
// then miss is below 2^-39 of that entry.  The epilogue multiplies by the inverse, `unscale` [block][r].
// One CTA per block of kD channels (one head, or a pair of 64-channel heads) and 16 columns: thread
// (part, j) holds 16 channels of column j, so all loads of the CTA go out together and a piece leaves as
// two 16-byte stores.  With the one thread per entry and 2-byte stores r channels apart that this
// replaces, the kernel took 2.8 us at 8 heads of 128, r = 32.
template <typename T>
__global__ void __launch_bounds__(128)
split_adapter_kernel(const float* __restrict__ proj, T* __restrict__ bsplit, float* __restrict__ unscale, int head_dim,
                     int block_dim, int r) {
  __shared__ float part_max[8][16];
  const int j = blockIdx.y * 16 + (threadIdx.x & 15), part = threadIdx.x >> 4;
  const int per = block_dim >> 3;                          // channels per thread: 16 or 8
  const int c0 = part * per;                               // within the block
  pdl_wait();                                              // the pieces may still be in use by the call before
  pdl_trigger();
  float v[16];
  const float* src = proj + (int64_t(blockIdx.x) * block_dim + c0) * r + j;
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = (i < per) ? src[int64_t(i) * r] : 0.f;
  float scale = 1.f;
  if constexpr (std::is_same<T, __half>::value) {
    float mx = 0.f;
#pragma unroll
    for (int i = 0; i < 16; ++i) mx = fmaxf(mx, fabsf(v[i]));
    part_max[part][threadIdx.x & 15] = mx;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; ++k) mx = fmaxf(mx, part_max[k][threadIdx.x & 15]);
    int sh = 0;
    if (mx > 0.f && mx < INFINITY) sh = min(120, max(-113, 14 - (int((__float_as_uint(mx) >> 23) & 0xffu) - 127)));
    scale = __uint_as_float(uint32_t(sh + 127) << 23);
    if (part == 0) unscale[int64_t(blockIdx.x) * r + j] = __uint_as_float(uint32_t(127 - sh) << 23);
  }
  __align__(16) T piece[3][16];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    float rest = v[i] * scale;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      piece[k][i] = T(rest);                               // round to nearest even
      rest -= float(piece[k][i]);
    }
  }
  const int g = (int64_t(blockIdx.x) * block_dim + c0) / head_dim, c = c0 % head_dim;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    uint4* dst = reinterpret_cast<uint4*>(bsplit + (int64_t(g) * 3 * r + k * r + j) * head_dim + c);
    dst[0] = reinterpret_cast<const uint4*>(piece[k])[0];
    if (per == 16) dst[1] = reinterpret_cast<const uint4*>(piece[k])[1];
  }
}

struct UmmaShared {
  unsigned long long full[kMaxStages];     // stage loaded (TMA bytes)
  unsigned long long empty[kMaxStages];    // stage consumed (MMA commit)
  unsigned long long acc_full[2];          // accumulator finished (MMA commit)
  unsigned long long acc_empty[2];         // accumulator read out (4 epilogue warps)
  uint32_t tmem_base;
  uint32_t abort;
};

// D = channels multiplied per stage.  PAIR (D = 128 with heads of 64 channels, joint metadata): a stage
// holds two KV heads, one per 64-channel half, so the chain inside tensor memory sums a pair of heads
// and there are half as many stages to hand over.
// KV_T: the type of K and of the adapter pieces (one tcgen05.mma takes both operands in one 16-bit type).
template <typename KV_T, int D, int R, typename META_T, bool PAIR>
__global__ void __launch_bounds__(kThreadsUmma, 1)
project_keys_umma_kernel(Problem p, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_b,
                         META_T* __restrict__ meta, const float* __restrict__ unscale, int n_begin, int n_end,
                         int tiles_per_row, uint32_t* __restrict__ err) {
  constexpr bool kScaled = std::is_same<KV_T, __half>::value;
  using C = Cfg<D, R>;
  constexpr int kD = D, kR = R, kNcols = C::kNcols, kStages = C::kStages, kHalves = C::kHalves;
  constexpr uint32_t kBHalf = C::kBHalf, kStageBytes = C::kStageBytes, kTmemCols = C::kTmemCols, kAccStride = C::kAccStride;
  constexpr int kChunk = (R < 32) ? R : 32;                // accumulator columns per tensor-memory load
  extern __shared__ unsigned char dyn_raw[];
  const uint32_t stage0 = (smem_addr(dyn_raw) + 1023u) & ~1023u;          // swizzled tiles need 1024-byte alignment
  __shared__ UmmaShared sh;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) { mbar_init(smem_addr(&sh.full[s]), 1); mbar_init(smem_addr(&sh.empty[s]), 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(smem_addr(&sh.acc_full[a]), 1); mbar_init(smem_addr(&sh.acc_empty[a]), 4); }
    sh.abort = 0;
    mbar_init_fence();
  }
  if (warp == 1) {
    tmem_alloc(smem_addr(&sh.tmem_base), kTmemCols);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sh.tmem_base;

  // Work: contiguous range of (sequence, metadata head, token tile) items; a step = (item, KV head).
  const int g_count = PAIR ? p.Hkv / 2 : (p.Hm == 1) ? p.Hkv : 1;      // stages per (token tile) item
  const int64_t items = int64_t(p.B) * p.Hm * tiles_per_row;
  const int64_t first = items * blockIdx.x / gridDim.x, last = items * (blockIdx.x + 1) / gridDim.x;
  const int n_steps = int(last - first) * g_count;

  // The kernel before this one splits the adapter, and let this one start once everything before it was
  // complete: K may be fetched at once, the pieces and their scales only after the wait.  No early trigger
  // here: the stages leave little of an SM's shared memory, so what follows would find no room before the end.
  if (warp == 0) {
    // ================================ producer ==============================================
    if (lane == 0) {
      auto place = [&](int s, int* n0, int* g, int* b) {                  // token, head and sequence of step s
        const int64_t item = first + s / g_count;
        const int tile = int(item % tiles_per_row), bh = int(item / tiles_per_row);
        const int hm = bh % p.Hm;
        *b = bh / p.Hm;
        *g = ((p.Hm == 1) ? 0 : hm) + (s % g_count) * (PAIR ? 2 : 1);
        *n0 = n_begin + tile * kTileM;
      };
      auto load_k = [&](int s) {
        const int stage = s % kStages;
        const uint32_t dst = stage0 + uint32_t(stage) * kStageBytes, bar = smem_addr(&sh.full[stage]);
        int n0, g, b;
        place(s, &n0, &g, &b);
        mbar_arrive_expect_tx(bar, kStageBytes);
#pragma unroll
        for (int h = 0; h < kHalves; ++h)                                  // channels and head of this half
          tma_load_4d(dst + uint32_t(h) * kAHalf, &map_k, bar, PAIR ? 0 : 64 * h, n0, PAIR ? g + h : g, b);
      };
      auto load_b = [&](int s) {
        const int stage = s % kStages;
        const uint32_t dst = stage0 + uint32_t(stage) * kStageBytes, bar = smem_addr(&sh.full[stage]);
        int n0, g, b;
        place(s, &n0, &g, &b);
#pragma unroll
        for (int h = 0; h < kHalves; ++h)
          tma_load_2d(dst + kHalves * kAHalf + uint32_t(h) * kBHalf, &map_b, bar, PAIR ? 0 : 64 * h, (PAIR ? g + h : g) * kNcols);
      };
      const int early = min(n_steps, kStages);
      for (int s = 0; s < early; ++s) load_k(s);
      pdl_wait();
      for (int s = 0; s < early; ++s) load_b(s);
      for (int s = early; s < n_steps; ++s) {
        const int stage = s % kStages, use = s / kStages;
        if (use > 0 && !mbar_wait(smem_addr(&sh.empty[stage]), uint32_t(use - 1) & 1u)) { sh.abort = 1; if (err) atomicExch(err, kDevTimeoutEmpty); break; }
        load_k(s);
        load_b(s);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ================================ MMA issuer ============================================
    if (lane == 0) {
      constexpr uint32_t idesc = umma_idesc(kScaled, kNcols);
      for (int s = 0; s < n_steps; ++s) {
        const int stage = s % kStages, use = s / kStages, buf = s & 1, acc_use = s >> 1;
        if (acc_use > 0 && !mbar_wait(smem_addr(&sh.acc_empty[buf]), uint32_t(acc_use - 1) & 1u)) { sh.abort = 1; if (err) atomicExch(err, kDevTimeoutEmpty); break; }
        if (!mbar_wait(smem_addr(&sh.full[stage]), uint32_t(use) & 1u)) { sh.abort = 1; if (err) atomicExch(err, kDevTimeoutFull); break; }
        tc_fence_after();
        const uint32_t a0 = stage0 + uint32_t(stage) * kStageBytes, b0 = a0 + kHalves * kAHalf;
#pragma unroll
        for (int k = 0; k < kD / 16; ++k) {
          const uint32_t half = k >> 2, koff = uint32_t(k & 3) * 32u;     // 16 channels = 32 bytes inside the swizzle row
          umma_16bit(tmem + uint32_t(buf) * kAccStride, umma_desc(a0 + half * kAHalf + koff), umma_desc(b0 + half * kBHalf + koff),
                    idesc, k > 0 ? 1u : 0u);
        }
        umma_commit(smem_addr(&sh.empty[stage]));         // the stage may be refilled once these MMAs have read it
        umma_commit(smem_addr(&sh.acc_full[buf]));        // ... and the accumulator is complete
      }
    }
    __syncwarp();
  } else {
    // ================================ epilogue ==============================================
    const int quarter = warp & 3;                          // tensor-memory lanes 32 * quarter .. + 31
    const int row = quarter * 32 + lane;                   // token row of the tile owned by this thread
    float acc[kR];
#pragma unroll
    for (int j = 0; j < kR; ++j) acc[j] = 0.f;
    bool ok = true;
    if constexpr (kScaled) pdl_wait();                     // the scales are the split kernel's
    for (int s = 0; s < n_steps && ok; ++s) {
      const int buf = s & 1, acc_use = s >> 1;
      ok = __all_sync(0xffffffffu, mbar_wait(smem_addr(&sh.acc_full[buf]), uint32_t(acc_use) & 1u));
      if (!ok) { if (lane == 0) { sh.abort = 1; if (err) atomicExch(err, kDevTimeoutFull); } break; }
      tc_fence_after();
      const uint32_t taddr = tmem + (uint32_t(quarter * 32) << 16) + uint32_t(buf) * kAccStride;
      const float* us = nullptr;                           // scales of this step's head, or pair of heads
      if constexpr (kScaled) us = unscale + int64_t(((p.Hm == 1) ? 0 : int((first + s / g_count) / tiles_per_row) % p.Hm) + s % g_count) * kR;
#pragma unroll
      for (int c0 = 0; c0 < kR; c0 += kChunk) {            // the pieces of columns c0 .. c0 + kChunk - 1 sit kR columns apart
        float hi[kChunk], mid[kChunk], lo[kChunk];
        tmem_ld_cols(taddr + c0, hi);
        tmem_ld_cols(taddr + kR + c0, mid);
        tmem_ld_cols(taddr + 2 * kR + c0, lo);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < kChunk; ++j) {
          const float sum = (lo[j] + mid[j]) + hi[j];
          if constexpr (kScaled) acc[c0 + j] = fmaf(sum, us[c0 + j], acc[c0 + j]);      // a power of two: exact
          else acc[c0 + j] += sum;
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_addr(&sh.acc_empty[buf]));
      if ((s + 1) % g_count == 0) {                        // last head of the item: one rounding, one row out
        const int64_t item = first + s / g_count;
        const int tile = int(item % tiles_per_row), bh = int(item / tiles_per_row);
        const int hm = bh % p.Hm, b = bh / p.Hm;
        const int n = n_begin + tile * kTileM + row;
        if (n < n_end) {
          META_T* dst = meta + int64_t(b) * p.meta_sb + int64_t(hm) * p.meta_sh + int64_t(n) * p.meta_sn;
          if constexpr (sizeof(META_T) == 1) {             // E4M3: the row is kR bytes
            const float sc = meta_store_scale(p);
            uint32_t w[kR / 4];
#pragma unroll
            for (int j = 0; j < kR / 4; ++j)
              w[j] = uint32_t(to_e4m3x2(acc[4 * j] * sc, acc[4 * j + 1] * sc)) |
                     (uint32_t(to_e4m3x2(acc[4 * j + 2] * sc, acc[4 * j + 3] * sc)) << 16);
#pragma unroll
            for (int j = 0; j < kR / 16; ++j)
              reinterpret_cast<uint4*>(dst)[j] = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
            static_assert(kR % 16 == 0, "whole 16-byte vectors per row");
          } else if constexpr (sizeof(META_T) == 2) {
            uint32_t w[kR / 2];
#pragma unroll
            for (int j = 0; j < kR / 2; ++j) {
              const __half2 h = __floats2half2_rn(acc[2 * j], acc[2 * j + 1]);
              w[j] = *reinterpret_cast<const uint32_t*>(&h);
            }
#pragma unroll
            for (int j = 0; j < kR / 8; ++j)
              reinterpret_cast<uint4*>(dst)[j] = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
          } else {
#pragma unroll
            for (int j = 0; j < kR / 4; ++j)
              reinterpret_cast<float4*>(dst)[j] = make_float4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]);
          }
        }
#pragma unroll
        for (int j = 0; j < kR; ++j) acc[j] = 0.f;
      }
    }
  }

  // ---- teardown: every loop above is bounded, so every warp arrives ------------------------------------
  tc_fence_before();
  __syncthreads();
  if (sh.abort && threadIdx.x == 0) {
    // a wait gave up: give copies that may still be in flight a bounded chance to land
    for (int s = 0; s < kStages; ++s) { mbar_wait(smem_addr(&sh.full[s]), 0); mbar_wait(smem_addr(&sh.full[s]), 1); }
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_free(tmem, kTmemCols);
  }
}

}  // namespace

static bool umma_shape(const Problem& p) {
  return p.kv_dtype != KVSWAP_F32 && (p.d == 64 || p.d == 128) && (p.r == 16 || p.r == 32 || p.r == 64);
}

size_t project_keys_umma_scratch_bytes(const Problem& p) {
  if (!umma_shape(p)) return 0;
  // the pieces of the adapter, and (fp16) one scale per head and column
  return size_t(p.Hkv) * 3 * p.r * p.d * sizeof(__nv_bfloat16) + size_t(p.Hkv) * p.r * sizeof(float);
}

namespace {

template <typename KV_T, int D, int R, bool PAIR>
cudaError_t launch_umma(const Problem& p, const CUtensorMap& map_k, const CUtensorMap& map_b, void* meta,
                        const float* unscale, int n_begin, int n_end, uint32_t* err, cudaStream_t st) {
  using C = Cfg<D, R>;
  const int tiles_per_row = (n_end - n_begin + kTileM - 1) / kTileM;
  const int64_t items = int64_t(p.B) * p.Hm * tiles_per_row;
  const int ctas = int(std::max<int64_t>(1, std::min<int64_t>(kNumSMs, items)));
  const size_t smem = size_t(C::kStages) * C::kStageBytes + 1024;
  auto go = [&](auto kern, auto* meta_t) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
    return launch_pdl(kern, dim3(ctas), dim3(kThreadsUmma), smem, st, p, map_k, map_b, meta_t, unscale, n_begin, n_end,
                      tiles_per_row, err);
  };
  if constexpr (R == 32) {                                 // 8-bit metadata exists for r = 32 only
    if (p.meta_dtype == KVSWAP_E4M3) return go(project_keys_umma_kernel<KV_T, D, R, e4m3_t, PAIR>, static_cast<e4m3_t*>(meta));
  }
  if (p.meta_dtype == KVSWAP_E4M3) return cudaErrorInvalidValue;
  if (p.meta_dtype == KVSWAP_F16) return go(project_keys_umma_kernel<KV_T, D, R, __half, PAIR>, static_cast<__half*>(meta));
  return go(project_keys_umma_kernel<KV_T, D, R, float, PAIR>, static_cast<float*>(meta));
}

}  // namespace

// Returns true (and sets *result) when this path took the problem.
bool try_launch_project_keys_umma(const Problem& p, const void* K, const float* proj, void* meta, int n_begin,
                                  int n_end, void* scratch, uint32_t* err, cudaStream_t st, cudaError_t* result) {
  if (!umma_shape(p) || (p.meta_dtype == KVSWAP_E4M3 && p.r != 32)) return false;
  if (p.kv_sn != p.d && (p.kv_sn * 2) % 16 != 0) return false;
  EncodeTiledFn enc = tensor_map_encoder();
  if (enc == nullptr) return false;
  ShortPlan sp;
  const bool is_short = plan_project_keys_short(p, n_begin, n_end, &sp);        // needs no scratch
  // Heads of 64 channels are multiplied in pairs where one metadata row sums all heads; alone they
  // leave each stage half as much to do, and at r = 16 the warp-level kernel is the faster one.
  const bool pair = p.d == 64 && p.Hm == 1 && p.Hkv % 2 == 0;
  if (!is_short && (scratch == nullptr || (p.d == 64 && !pair && p.r == 16))) return false;
  const int ncols = 3 * p.r;
  const bool bf16 = p.kv_dtype == KVSWAP_BF16;
  CUtensorMap map_k, map_b;
  if (!make_rows_tensor_map(&map_k, K, 2, bf16, p.d, p.N, p.Hkv, p.B, p.kv_sn, p.kv_sh, p.kv_sb, kTileM)) return false;
  if (is_short) {
    *result = launch_project_keys_short(p, sp, map_k, proj, meta, n_begin, n_end, err, st);
    return true;
  }
  {
    const cuuint64_t dims[2] = {cuuint64_t(p.d), cuuint64_t(p.Hkv) * ncols};
    const cuuint64_t strides[1] = {cuuint64_t(p.d) * 2};
    const cuuint32_t box[2] = {64, cuuint32_t(ncols)}, estr[2] = {1, 1};
    if (enc(&map_b, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, scratch, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return false;
  }
  float* unscale = reinterpret_cast<float*>(static_cast<char*>(scratch) + size_t(p.Hkv) * ncols * p.d * 2);
  const int block_dim = pair ? 2 * p.d : p.d;
  const dim3 split_grid(p.Hkv * p.d / block_dim, p.r / 16);
  *result = bf16 ? launch_pdl(split_adapter_kernel<__nv_bfloat16>, split_grid, dim3(128), 0, st, proj,
                              static_cast<__nv_bfloat16*>(scratch), unscale, p.d, block_dim, p.r)
                 : launch_pdl(split_adapter_kernel<__half>, split_grid, dim3(128), 0, st, proj,
                              static_cast<__half*>(scratch), unscale, p.d, block_dim, p.r);
  if (*result != cudaSuccess) return true;
  auto by_type = [&](auto d_tag, auto r_tag, auto pair_tag) {
    constexpr int D = decltype(d_tag)::value, R = decltype(r_tag)::value;
    constexpr bool P = decltype(pair_tag)::value;
    return bf16 ? launch_umma<__nv_bfloat16, D, R, P>(p, map_k, map_b, meta, unscale, n_begin, n_end, err, st)
                : launch_umma<__half, D, R, P>(p, map_k, map_b, meta, unscale, n_begin, n_end, err, st);
  };
  auto by_rank = [&](auto d_tag, auto pair_tag) {
    return p.r == 16   ? by_type(d_tag, std::integral_constant<int, 16>(), pair_tag)
           : p.r == 32 ? by_type(d_tag, std::integral_constant<int, 32>(), pair_tag)
                       : by_type(d_tag, std::integral_constant<int, 64>(), pair_tag);
  };
  using D128 = std::integral_constant<int, 128>;
  using D64 = std::integral_constant<int, 64>;
  *result = pair         ? by_rank(D128(), std::true_type())
            : p.d == 128 ? by_rank(D128(), std::false_type())
                         : by_rank(D64(), std::false_type());
  return true;
}

}  // namespace kvswap
