// K1 for short prompts: the projection of project_keys_umma.cu (same arithmetic: adapter in three 16-bit pieces, one
// chain inside tensor memory per KV head or pair of 64-channel heads) as one launch in which every CTA has its
// operands to itself.
//
// The persistent kernel is built for bandwidth: a launch splits the adapter, then a CTA per SM walks its token tiles
// head by head.  A prompt of 5000 tokens is 40 tiles, i.e. 40 CTAs that take eight steps each behind that launch.
// Here a CTA takes the `hpc` heads of one tile that are its share, splits their adapter rows itself straight into the
// swizzled operand layout, and the CTAs of a tile, a cluster, add their accumulators through distributed shared memory,
// each writing a share of the rows.  Nothing is handed over twice: all loads go out at once, every head has its own
// accumulator.  Bound by latency: launch, the trip of K and the adapter, the split, one chain, the cluster barrier.
#include <algorithm>
#include <type_traits>

#include "async_copy.cuh"
#include "cluster.cuh"
#include "common.cuh"
#include "project_keys_short.cuh"
#include "tensor_map.cuh"
#include "umma.cuh"

namespace kvswap {
namespace {

constexpr int kRows = 128;                                 // tokens per tile
constexpr int kThreads = 256;
constexpr int kIssuer = 128;                               // thread that requests K and issues the MMAs (warp 4)
constexpr int kMaxHeads = 4;                               // heads (or pairs) per CTA
constexpr int kMaxCluster = 8;
constexpr size_t kMaxSmem = 220 * 1024;
__host__ __device__ constexpr int short_ctas_per_sm(int r) { return r <= 32 ? 3 : 2; }      // by registers

template <int D, int R>
struct ShortCfg {                                          // D channels per accumulator: a head, or a pair of 64-channel heads
  static constexpr int kNcols = 3 * R, kHalves = D / 64;
  static constexpr uint32_t kAHalf = kRows * 128, kBHalf = uint32_t(kNcols) * 128;
  static constexpr uint32_t kHeadBytes = kHalves * (kAHalf + kBHalf);    // operands: K rows, then adapter pieces
  static constexpr uint32_t kAccStride = (kNcols <= 64) ? 64 : (kNcols <= 128) ? 128 : 256;
};

__device__ __forceinline__ float4 cluster_load4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}

// Four consecutive entries of a metadata row.
__device__ __forceinline__ void store_meta4(const Problem& p, void* meta, int64_t at, float4 v) {
  if (p.meta_dtype == KVSWAP_F16) {
    const __half2 a = __floats2half2_rn(v.x, v.y), b = __floats2half2_rn(v.z, v.w);
    *reinterpret_cast<uint2*>(static_cast<__half*>(meta) + at) =
        make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
  } else if (p.meta_dtype == KVSWAP_F32) {
    *reinterpret_cast<float4*>(static_cast<float*>(meta) + at) = v;
  } else {
    const float s = meta_store_scale(p);
    *reinterpret_cast<uint32_t*>(static_cast<uint8_t*>(meta) + at) =
        uint32_t(to_e4m3x2(v.x * s, v.y * s)) | (uint32_t(to_e4m3x2(v.z * s, v.w * s)) << 16);
  }
}

template <typename KV_T, int D, int R, bool PAIR>
__global__ void __launch_bounds__(kThreads, short_ctas_per_sm(R))
project_keys_short_kernel(Problem p, const __grid_constant__ CUtensorMap map_k, const float* __restrict__ proj, void* meta,
                          int n_begin, int n_end, int tiles_per_row, int hpc, uint32_t tmem_cols,
                          uint32_t* __restrict__ err) {
  using C = ShortCfg<D, R>;
  constexpr bool kScaled = std::is_same<KV_T, __half>::value;
  extern __shared__ unsigned char dyn_raw[];
  const uint32_t stage0 = (smem_addr(dyn_raw) + 1023u) & ~1023u;       // swizzled operands need 1024-byte alignment
  unsigned char* stage_ptr = dyn_raw + (stage0 - smem_addr(dyn_raw));
  __shared__ unsigned long long full[kMaxHeads], done[kMaxHeads];
  __shared__ uint32_t tmem_base;
  __shared__ uint32_t col_max[R];
  __shared__ float unscale[kMaxHeads][R];

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = int(cluster_rank()), n_ctas = int(cluster_size());
  const int item = blockIdx.x / n_ctas, tile = item % tiles_per_row, bh = item / tiles_per_row;
  const int hm = bh % p.Hm, b = bh / p.Hm;
  const int n0 = n_begin + tile * kRows;
  const int blk0 = ((p.Hm == 1) ? 0 : hm) + rank * hpc;                // first head, or pair, of this CTA
  if (tid == kIssuer) {
    for (int s = 0; s < hpc; ++s) { mbar_init(smem_addr(&full[s]), 1); mbar_init(smem_addr(&done[s]), 1); }
    mbar_init_fence();
  }
  pdl_wait();                                                          // K and the adapter may be the previous kernel's output
  // The next launch may set itself up beside this one: 28 layers of a prompt of 5003 fp16 tokens 256 -> 252 us.  It waits before
  // it reads the rows written here; only a call whose inputs are settled does not, and rows that work enqueued before it still
  // writes are not (KVSWAP_INPUTS_SETTLED asks for a full dependency in between).
  pdl_trigger();
  if (tid == kIssuer) {
    for (int s = 0; s < hpc; ++s) {
      const uint32_t dst = stage0 + uint32_t(s) * C::kHeadBytes, bar = smem_addr(&full[s]);
      mbar_arrive_expect_tx(bar, C::kHalves * C::kAHalf);
#pragma unroll
      for (int h = 0; h < C::kHalves; ++h)
        tma_load_4d(dst + uint32_t(h) * C::kAHalf, &map_k, bar, PAIR ? 0 : 64 * h, n0, PAIR ? 2 * (blk0 + s) + h : blk0 + s, b);
    }
  }
  if (warp == kIssuer / 32) { __syncwarp(); tmem_alloc(smem_addr(&tmem_base), tmem_cols); }

  // ---- the adapter's pieces, straight into the operand layout ----------------------------------------------------------
  // Task = (column j, eight channels); the loads of a head go out together.  fp16 pieces are scaled per column as split_adapter_kernel does it.
  constexpr int kTasks = R * (D / 8), kPer = (kTasks + kThreads - 1) / kThreads;
  for (int s = 0; s < hpc; ++s) {
    const float* src = proj + int64_t(blk0 + s) * D * R;
    float v[kPer][8];
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int t = tid + u * kThreads, j = t % R, c0 = (t / R) * 8;
#pragma unroll
      for (int i = 0; i < 8; ++i) v[u][i] = (t < kTasks) ? src[int64_t(c0 + i) * R + j] : 0.f;
    }
    if constexpr (kScaled) {
      __syncthreads();                                                 // (the maxima of the head before are read)
      if (tid < R) col_max[tid] = 0u;
      __syncthreads();
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        const int t = tid + u * kThreads;
        float mx = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) mx = fmaxf(mx, fabsf(v[u][i]));
        if (t < kTasks) atomicMax(&col_max[t % R], __float_as_uint(mx));
      }
      __syncthreads();
    }
    unsigned char* B = stage_ptr + size_t(s) * C::kHeadBytes + C::kHalves * C::kAHalf;
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int t = tid + u * kThreads, j = t % R, c0 = (t / R) * 8;
      if (t >= kTasks) continue;
      float scale = 1.f;
      if constexpr (kScaled) {
        const float mx = __uint_as_float(col_max[j]);
        int sh = 0;
        if (mx > 0.f && mx < INFINITY) sh = min(120, max(-113, 14 - (int((__float_as_uint(mx) >> 23) & 0xffu) - 127)));
        scale = __uint_as_float(uint32_t(sh + 127) << 23);
        if (c0 == 0) unscale[s][j] = __uint_as_float(uint32_t(127 - sh) << 23);
      }
      __align__(16) KV_T piece[3][8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        float rest = v[u][i] * scale;
#pragma unroll
        for (int k = 0; k < 3; ++k) { piece[k][i] = KV_T(rest); rest -= float(piece[k][i]); }
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int row = k * R + j, in_half = (c0 & 63) >> 3;           // 16-byte piece of the 128-byte row, swizzled
        *reinterpret_cast<uint4*>(B + (c0 >> 6) * C::kBHalf + row * 128 + ((in_half ^ (row & 7)) << 4)) =
            *reinterpret_cast<const uint4*>(piece[k]);
      }
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");         // written by threads, read by the tensor core
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;

  // ---- multiply ----------------------------------------------------------------------------------------------------------
  if (tid == kIssuer) {
    constexpr uint32_t idesc = umma_idesc(kScaled, C::kNcols);
    for (int s = 0; s < hpc; ++s) {
      if (!mbar_wait(smem_addr(&full[s]), 0u) && !mbar_wait(smem_addr(&full[s]), 0u) && err) atomicExch(err, kDevTimeoutFull);
      tc_fence_after();
      const uint32_t a0 = stage0 + uint32_t(s) * C::kHeadBytes, b0 = a0 + C::kHalves * C::kAHalf;
#pragma unroll
      for (int k = 0; k < D / 16; ++k) {
        const uint32_t half = k >> 2, koff = uint32_t(k & 3) * 32u;    // 16 channels = 32 bytes inside the swizzle row
        umma_16bit(tmem + uint32_t(s) * C::kAccStride, umma_desc(a0 + half * C::kAHalf + koff),
                   umma_desc(b0 + half * C::kBHalf + koff), idesc, k > 0 ? 1u : 0u);
      }
      umma_commit(smem_addr(&done[s]));
    }
  }
  __syncwarp();

  // ---- sum of the pieces and of this CTA's heads: one token row per thread of the first four warps ----------------------------
  float* const red = reinterpret_cast<float*>(stage_ptr);              // [kRows][R + 4]: the operands are read by then
  constexpr int kPitch = R + 4;
  if (warp < 4) {                                                      // tensor-memory lanes 32 * warp .. + 31
    constexpr int kChunk = 16;                                         // (few registers: several CTAs share an SM)
    float acc[R];
#pragma unroll
    for (int j = 0; j < R; ++j) acc[j] = 0.f;
    for (int s = 0; s < hpc; ++s) {
      const bool ok = __all_sync(0xffffffffu, mbar_wait(smem_addr(&done[s]), 0u) || mbar_wait(smem_addr(&done[s]), 0u));
      if (!ok && lane == 0 && err) atomicExch(err, kDevTimeoutFull);
      tc_fence_after();
      const uint32_t taddr = tmem + (uint32_t(warp * 32) << 16) + uint32_t(s) * C::kAccStride;
#pragma unroll
      for (int c0 = 0; c0 < R; c0 += kChunk) {
        float hi[kChunk], mid[kChunk], lo[kChunk];
        tmem_ld_cols(taddr + c0, hi);
        tmem_ld_cols(taddr + R + c0, mid);
        tmem_ld_cols(taddr + 2 * R + c0, lo);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < kChunk; ++j) {
          const float sum = (lo[j] + mid[j]) + hi[j];
          if constexpr (kScaled) acc[c0 + j] = fmaf(sum, unscale[s][c0 + j], acc[c0 + j]);      // a power of two: exact
          else acc[c0 + j] += sum;
        }
      }
    }
    tc_fence_before();
    float4* dst = reinterpret_cast<float4*>(red + (warp * 32 + lane) * kPitch);
#pragma unroll
    for (int j = 0; j < R / 4; ++j) dst[j] = make_float4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]);
  }
  __syncthreads();
  if (warp == kIssuer / 32) { tc_fence_after(); tmem_free(tmem, tmem_cols); }
  if (n_ctas > 1) { cluster_arrive(); cluster_wait(); }                // every CTA's sums are in place

  // ---- this CTA's share of the rows: sum over the cluster in rank order, one rounding ------------------------------------------
  const int share = kRows / n_ctas, r0 = rank * share;
  for (int e = tid; e < share * (R / 4); e += kThreads) {
    const int row = r0 + e / (R / 4), c4 = e % (R / 4);
    const uint32_t at = stage0 + uint32_t(row * kPitch + 4 * c4) * 4u;
    float4 x[kMaxCluster], sum = make_float4(0.f, 0.f, 0.f, 0.f);      // all loads out at once: one trip, not one per CTA
#pragma unroll
    for (int r = 0; r < kMaxCluster; ++r)
      if (r < n_ctas) x[r] = cluster_load4(cluster_map(at, uint32_t(r)));
#pragma unroll
    for (int r = 0; r < kMaxCluster; ++r)
      if (r < n_ctas) { sum.x += x[r].x; sum.y += x[r].y; sum.z += x[r].z; sum.w += x[r].w; }
    const int n = n0 + row;
    if (n < n_end)
      store_meta4(p, meta, int64_t(b) * p.meta_sb + int64_t(hm) * p.meta_sh + int64_t(n) * p.meta_sn + 4 * c4, sum);
  }
  if (n_ctas > 1) { cluster_arrive(); cluster_wait(); }                // no CTA leaves while a peer may still read its sums
}

template <typename KV_T, int D, int R, bool PAIR>
cudaError_t launch_short(const Problem& p, const ShortPlan& pl, const CUtensorMap& map_k, const float* proj, void* meta,
                         int n_begin, int n_end, uint32_t* err, cudaStream_t st) {
  using C = ShortCfg<D, R>;
  uint32_t cols = 32;
  while (cols < uint32_t(pl.hpc) * C::kAccStride) cols *= 2;
  const size_t smem = std::max(size_t(pl.hpc) * C::kHeadBytes, size_t(kRows) * (R + 4) * sizeof(float)) + 1024;
  auto kern = project_keys_short_kernel<KV_T, D, R, PAIR>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  if (e != cudaSuccess) return e;
  return launch_pdl_cluster(kern, pl.cluster, dim3(unsigned(pl.items * pl.cluster)), dim3(kThreads), smem, st, p, map_k, proj,
                            meta, n_begin, n_end, pl.tiles, pl.hpc, cols, err);
}

}  // namespace

// Work split for a shape of project_keys_umma.cu; false when the persistent kernel is to take it.
bool plan_project_keys_short(const Problem& p, int n_begin, int n_end, ShortPlan* pl) {
  if (p.meta_dtype == KVSWAP_E4M3 && p.r != 32) return false;
  pl->pair = p.d == 64 && p.Hm == 1 && p.Hkv % 2 == 0;
  const int heads = pl->pair ? p.Hkv / 2 : (p.Hm == 1) ? p.Hkv : 1;    // accumulators per tile
  const size_t head_bytes = size_t(p.d == 128 || pl->pair ? 2 : 1) * 128 * (kRows + 3 * p.r);
  const int stride = 3 * p.r <= 64 ? 64 : 3 * p.r <= 128 ? 128 : 256;
  pl->tiles = (n_end - n_begin + kRows - 1) / kRows;
  pl->items = int64_t(p.B) * p.Hm * pl->tiles;
  // All CTAs are resident at once (shared memory, tensor memory, registers), with as few heads one after the other as
  // that allows.  8 heads of 128, r = 32: B = 1, N = 1500 5.7 us against 10.3 of the persistent kernel and its adapter
  // launch, N = 5003 (three CTAs per SM) 8.9 against 10.3; at N = 9000, where a second wave would start, 20 against
  // 10.4.  Two tiles per CTA, sharing the split adapter, took 17 us there, and operands from an adapter launch 10.3.
  for (int cluster = kMaxCluster; cluster >= 1; cluster /= 2) {
    const int hpc = heads / cluster;
    const size_t smem = hpc * head_bytes + 2048;
    if (heads % cluster != 0 || hpc > kMaxHeads || hpc * stride > 512 || smem > kMaxSmem) continue;
    const int per_sm = std::min({int((227 * 1024) / smem), 512 / (hpc * stride), short_ctas_per_sm(p.r)});
    if (pl->items * cluster > int64_t(kNumSMs) * per_sm) continue;
    pl->cluster = cluster; pl->hpc = hpc;
    return true;
  }
  return false;
}

cudaError_t launch_project_keys_short(const Problem& p, const ShortPlan& pl, const CUtensorMap& map_k, const float* proj,
                                      void* meta, int n_begin, int n_end, uint32_t* err, cudaStream_t st) {
  auto go = [&](auto d_tag, auto r_tag, auto pair_tag) {
    constexpr int D = decltype(d_tag)::value, R = decltype(r_tag)::value;
    constexpr bool P = decltype(pair_tag)::value;
    return p.kv_dtype == KVSWAP_BF16 ? launch_short<__nv_bfloat16, D, R, P>(p, pl, map_k, proj, meta, n_begin, n_end, err, st)
                                     : launch_short<__half, D, R, P>(p, pl, map_k, proj, meta, n_begin, n_end, err, st);
  };
  auto by_rank = [&](auto d_tag, auto pair_tag) {
    return p.r == 16   ? go(d_tag, std::integral_constant<int, 16>(), pair_tag)
           : p.r == 32 ? go(d_tag, std::integral_constant<int, 32>(), pair_tag)
                       : go(d_tag, std::integral_constant<int, 64>(), pair_tag);
  };
  using D128 = std::integral_constant<int, 128>;
  using D64 = std::integral_constant<int, 64>;
  return pl.pair ? by_rank(D128(), std::true_type()) : p.d == 128 ? by_rank(D128(), std::false_type()) : by_rank(D64(), std::false_type());
}

}  // namespace kvswap
