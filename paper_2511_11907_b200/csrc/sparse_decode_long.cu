// K4 for long gathers: the split-K gather of sparse_decode.cu (virtual token list, self-fed warps, swizzled stages; read that
// file's head first) with the warps of the whole GPU dealt to the lists instead of whole CTAs, stages of 16 tokens and one CTA
// per SM, in half of an SM's registers, so that a decode step runs the next layer's select beside it (topk_beside.cuh, step.cu).
//
// Bound by HBM: 134 MB (B = 4, 8 KV heads, 8192 tokens attended) in 28.1 us as a launch of its own, as the sixteen warps per SM
// of sparse_decode.cu.  What made eight warps keep up: 16 tokens per stage (half the softmax bookkeeping, P.V with k = 16), two chains of
// products per block of logits, the sum of the weights left to the lanes until the end, one address per block of eight rows where
// G is a multiple of 8.
#include <algorithm>
#include <cstdint>

#include "async_copy.cuh"
#include "combine.cuh"
#include "common.cuh"
#include "gather.cuh"

namespace kvswap {
namespace {

constexpr int kTok = 16;                        // tokens per stage
constexpr int kWarps = kGatherWarps;            // warps per CTA
constexpr int kThreads = kWarps * 32;
constexpr int kMaxDepth = 8;                    // stages per warp, at most

// Control block at the start of dynamic shared memory.
struct Control {
  uint32_t mask[kWarps * kMaxDepth];            // bit t: token slot t of the stage holds a row
};
constexpr int kControlBytes = (sizeof(Control) + 255) & ~255;

template <typename KV_T>
__device__ __forceinline__ void mma_k16_full(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  if constexpr (std::is_same<KV_T, __nv_bfloat16>::value) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
  } else {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
  }
}
// The tensor-core engine of sparse_decode.cu on two blocks of eight tokens at a time.
template <typename KV_T, int D, int RH>
struct LongEngine {
  static constexpr int kBlocks = kTok / 8;
  static_assert(sizeof(KV_T) == 2, "16-bit K/V and q of one type");
  static constexpr uint32_t ROWB = D * sizeof(KV_T);
  static constexpr uint32_t kFull = 0xffffffffu;
  static constexpr int KS = D / 16;          // k-steps of the logits = 16-channel blocks of the output
  uint32_t qa[KS][2];                        // A fragments of Q (rows 0..7 of each k-step)
  float oacc[KS][4];                         // out^T: [block][0,1] channel 16*blk+g, heads 2t,2t+1; [2,3] channel +8
  float m_run, l_run;                        // of head g = lane / 4: the maximum, and the sum over the lane's tokens
  float scale;
  int lane, g, t;
  uint32_t ld_row, ld_piece;                 // ldmatrix: row this lane addresses, piece within a 64-byte span

  __device__ __forceinline__ void init(const KV_T* q0, int lane_) {
    lane = lane_; g = lane >> 2; t = lane & 3;
    scale = kLog2e * rsqrtf(float(D));
    ld_row = uint32_t(lane & 7); ld_piece = uint32_t(lane >> 3);
    const uint32_t* qrow = reinterpret_cast<const uint32_t*>(q0 + (g < RH ? g : 0) * D);   // 2 channels per word
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
      qa[ks][0] = (g < RH) ? qrow[8 * ks + t] : 0u;            // channels 16ks + 2t, +1
      qa[ks][1] = (g < RH) ? qrow[8 * ks + 4 + t] : 0u;        // channels 16ks + 8 + 2t, +1
    }
#pragma unroll
    for (int i = 0; i < KS; ++i) { oacc[i][0] = oacc[i][1] = oacc[i][2] = oacc[i][3] = 0.f; }
    m_run = -INFINITY; l_run = 0.f;
  }

  __device__ __forceinline__ void chunk(uint32_t kstage, uint32_t vstage, uint32_t mask) {
    // ---- logits of head g for tokens 2t, 2t+1 of each block; two chains of products per block ------------
    const bool head_ok = g < RH;
    float s0[kBlocks], s1[kBlocks], cmax = -INFINITY;
#pragma unroll
    for (int n = 0; n < kBlocks; ++n) {
      float even[4] = {0.f, 0.f, 0.f, 0.f}, odd[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int kk = 0; kk < D / 32; ++kk) {
        uint32_t r[4];                                                                // channels 32kk .. 32kk+31
        ldsm_x4(kstage + swz<ROWB>(8 * n + ld_row, (uint32_t(4 * kk) + ld_piece) << 4), r);
        mma_k16<KV_T>(even, qa[2 * kk][0], qa[2 * kk][1], r[0], r[1]);
        mma_k16<KV_T>(odd, qa[2 * kk + 1][0], qa[2 * kk + 1][1], r[2], r[3]);
      }
      s0[n] = (head_ok && ((mask >> (8 * n + 2 * t)) & 1u)) ? (even[0] + odd[0]) * scale : -INFINITY;
      s1[n] = (head_ok && ((mask >> (8 * n + 2 * t + 1)) & 1u)) ? (even[1] + odd[1]) * scale : -INFINITY;
      cmax = fmaxf(cmax, fmaxf(s0[n], s1[n]));
    }
    // ---- online softmax of head g over the four lanes that share it ----------------------------------
    cmax = fmaxf(cmax, __shfl_xor_sync(kFull, cmax, 1));
    cmax = fmaxf(cmax, __shfl_xor_sync(kFull, cmax, 2));
    const float m_new = fmaxf(m_run, cmax);
    const float m_safe = (m_new == -INFINITY) ? 0.f : m_new;
    float p0[kBlocks], p1[kBlocks], psum = 0.f;                // 0 for absent tokens / heads
#pragma unroll
    for (int n = 0; n < kBlocks; ++n) {
      p0[n] = ex2(s0[n] - m_safe);
      p1[n] = ex2(s1[n] - m_safe);
      psum += p0[n] + p1[n];
    }
    const float cr = ex2(m_run - m_safe);                      // 0 while nothing has been seen yet
    l_run = fmaf(l_run, cr, psum);                             // of this lane's tokens: the lanes are added in store()
    m_run = m_new;
    if (__any_sync(kFull, head_ok && cr != 1.f)) {
      // accumulator columns of this lane are heads 2t and 2t+1: their factors live in lanes 8t, 8t+4
      const float c0 = __shfl_sync(kFull, cr, (8 * t) & 31), c1 = __shfl_sync(kFull, cr, (8 * t + 4) & 31);
#pragma unroll
      for (int i = 0; i < KS; ++i) { oacc[i][0] *= c0; oacc[i][1] *= c1; oacc[i][2] *= c0; oacc[i][3] *= c1; }
    }
    // ---- out^T += V^T P, P = head + remainder -----------------------------------------------------------
    uint32_t phi[kBlocks], plo[kBlocks];
#pragma unroll
    for (int n = 0; n < kBlocks; ++n) split_pair<KV_T>(p0[n], p1[n], phi[n], plo[n]);
    const uint32_t row = ld_row + 8u * (ld_piece >> 1), piece = ld_piece & 1u;   // matrices: token block, then 8 channels
#pragma unroll
    for (int i = 0; i < KS; ++i) {
      uint32_t r[4];
      ldsm_x4_trans(vstage + swz<ROWB>(row, (uint32_t(2 * i) + piece) << 4), r);          // V^T, channels 16i .. 16i+15
      mma_k16_full<KV_T>(oacc[i], r, phi[0], phi[1]);
      mma_k16_full<KV_T>(oacc[i], r, plo[0], plo[1]);
    }
  }

  __device__ __forceinline__ void store(float* sm_m, float* sm_l, float* sm_acc) const {
    float l = l_run + __shfl_xor_sync(kFull, l_run, 1);
    l += __shfl_xor_sync(kFull, l, 2);
    if (t == 0) { sm_m[g] = m_run; sm_l[g] = l; }            // g = 0..7: one slot per possible head
#pragma unroll
    for (int i = 0; i < KS; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int head = 2 * t + (e & 1), ch = 16 * i + g + ((e & 2) ? 8 : 0);
        if (head < RH) sm_acc[head * D + ch] = oacc[i][e];
      }
  }
};

// Where the attended tokens of one CTA come from.
struct TokenSource {
  const int32_t* idx;      // selection row
  int NG, G, g_shift;      // g_shift = log2(G) when G is a power of two, else -1
  int sel_tokens, tail0;   // M * G, NG * G
  int v_begin, v_end;      // this warp's range of the virtual token list

  // Group ordinal of virtual token v (v < sel_tokens).
  __device__ __forceinline__ int group_of(int v) const { return g_shift >= 0 ? (v >> g_shift) : (v / G); }
};

// How the lists -- (sequence, KV head, RH of its query heads) -- are dealt to the warps of the grid.
struct SplitGrid {
  int lists, warps_per_list;
  int slots;               // CTAs a list is spread over, at most: the partials [lists * RH, slots, D + 2] have room for them
};

template <typename KV_T, int D, int RH>
__global__ void __launch_bounds__(kThreads, 2)           // (two: no more than 128 registers)
sparse_decode_long_kernel(Problem p, const KV_T* __restrict__ q, const KV_T* __restrict__ K,
                            const KV_T* __restrict__ V, const int32_t* __restrict__ group_idx,
                            const int32_t* __restrict__ n_selected, float* __restrict__ partial, SplitGrid sg, int depth,
                            int g_shift, uint32_t* __restrict__ err) {
  constexpr uint32_t ROWB = D * sizeof(KV_T);                  // bytes of one K or V row
  constexpr uint32_t HALFB = kTok * ROWB;                      // K (or V) part of a stage
  constexpr uint32_t kPieces = ROWB / 16;                      // 16-byte pieces per row
  constexpr uint32_t STAGEB = 2 * HALFB;
  constexpr uint32_t kFull = 0xffffffffu;

  extern __shared__ unsigned char smem_raw[];
  Control* ctl = reinterpret_cast<Control*>(smem_raw);
  // Stage ring, aligned to 128 bytes (the swizzle works on row-relative offsets).
  const uint32_t ring = (smem_addr(smem_raw) + kControlBytes + 127u) & ~127u;
  unsigned char* ring_ptr = smem_raw + (ring - smem_addr(smem_raw));

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Warps are numbered through the grid; warps_per_list consecutive ones share a list, whose chunks are dealt to them in
  // contiguous, (almost) equal ranges.  Where that is no multiple of kWarps a CTA serves the end of one list and the start
  // of the next: each of its warps works for one list.
  const int list = (blockIdx.x * kWarps + warp) / sg.warps_per_list;
  const int share = blockIdx.x * kWarps + warp - list * sg.warps_per_list;
  const bool live = list < sg.lists;                           // (the last CTA may have warps to spare)
  const int chunks = p.rho / RH;                               // lists of one KV head
  const int bg = (live ? list : 0) / chunks;
  const int g = bg % p.Hkv, b = bg / p.Hkv;
  const int srow = (p.scope == KVSWAP_SCOPE_KV_HEAD) ? g : 0;

  // Everything below may depend on the previous kernel in the stream -- unless the caller has
  // promised that q and the selection are settled: then only this kernel's writes (the partials,
  // which the previous launch's combine may still be reading) have to wait for it.
  const bool settled = (p.flags & KVSWAP_INPUTS_SETTLED) != 0;
  const bool wait_late = settled && (p.flags & kFlagWaitLate) != 0;
  if (!settled) pdl_wait();
  pdl_trigger();

  // The virtual token list is laid out for M selected groups, whatever n_selected says (slots of
  // groups beyond n_selected are simply absent), so that the split of the list does not wait for a
  // global read: n_selected is fetched together with the first group indices.
  TokenSource src;
  src.idx = group_idx + (int64_t(b) * p.S + srow) * p.M;
  src.NG = p.NG; src.G = p.G; src.g_shift = g_shift;
  src.tail0 = p.NG * p.G;
  src.sel_tokens = p.M * p.G;
  int my_chunks;                                               // of this warp
  {
    const int total = src.sel_tokens + (p.N - src.tail0);
    const int n_chunks = (total + kTok - 1) / kTok, base = n_chunks / sg.warps_per_list, rem = n_chunks % sg.warps_per_list;
    my_chunks = live ? base + (share < rem ? 1 : 0) : 0;
    src.v_begin = (share * base + min(share, rem)) * kTok;
    src.v_end = min(total, src.v_begin + my_chunks * kTok);
  }
  const int n_sel_given = n_selected[int64_t(b) * p.S + srow];
  const int n_sel = max(0, min(n_sel_given, p.M));
  // KVSWAP_CHECK_INDICES: the first warp of each list looks it over once, ahead of the loop (which skips what
  // is out of range either way), and records what it finds.  (No wait in this kernel can run out: err serves this only.)
  if ((p.flags & KVSWAP_CHECK_INDICES) != 0 && err != nullptr && live && share == 0) {
    bool bad = n_sel != n_sel_given;
    for (int i = lane; i < n_sel; i += 32) {
      const int j = src.idx[i];
      bad = bad || (j != -1 && (j < 0 || j >= p.NG));
    }
    if (bad) atomicExch(err, kDevBadIndex);
  }

  const unsigned char* Kg = reinterpret_cast<const unsigned char*>(K + int64_t(b) * p.kv_sb + int64_t(g) * p.kv_sh);
  const unsigned char* Vg = reinterpret_cast<const unsigned char*>(V + int64_t(b) * p.kv_sb + int64_t(g) * p.kv_sh);
  const bool blocks = kPieces <= 32 && p.G % 8 == 0 && p.kv_sn * int64_t(sizeof(KV_T)) < (int64_t(1) << 28);
  const int64_t row_pitch = p.kv_sn * int64_t(sizeof(KV_T));   // bytes between token rows in global memory

  // Entry of the selection row behind token slot `lane` of this warp's k-th chunk, or -1: the one dependent
  // global read of the fill path, issued early so that its latency hides behind a chunk's compute.  (It does not wait for
  // n_selected: the row has M entries whatever that says.)
  auto fetch_group = [&](int k) -> int {
    const int v = src.v_begin + k * kTok + lane;
    if (lane < kTok && k < my_chunks && v < src.v_end && v < src.sel_tokens) {
      return src.idx[src.group_of(v)];
    }
    return -1;
  };
  // Fill: bring chunk k into `stage` (one commit group).  `j` is fetch_group(k).  All lanes call.
  auto fill = [&](int k, int j, int stage) {
    if (k < my_chunks) {
      const int v = src.v_begin + k * kTok + lane;
      int n = -1;                                              // token row behind slot `lane` (lanes beyond kTok: none)
      if (lane < kTok && v < src.v_end) {
        if (v < src.sel_tokens) {
          const int go = src.group_of(v);
          if (j >= 0 && j < src.NG && go < n_sel) n = j * src.G + (v - go * src.G);
        } else {
          n = src.tail0 + (v - src.sel_tokens);
        }
      }
      const uint32_t vmask = __ballot_sync(kFull, n >= 0);
      if (lane == 0) ctl->mask[stage] = vmask;
      const uint32_t kdst = ring + uint32_t(stage) * STAGEB;
      if (blocks) {
        // G a multiple of 8: the rows of a block of 8 slots follow each other, those that are absent last
        constexpr uint32_t kRows = 32 / kPieces < 1 ? 1 : 32 / kPieces;   // rows a read of the warp covers
        static_assert(kPieces <= 32, "a row is one read at most");
        const uint32_t r0 = uint32_t(lane) / kPieces, c = uint32_t(lane) % kPieces;
        const uint32_t step = uint32_t(kRows) * uint32_t(row_pitch);
#pragma unroll
        for (int blk = 0; blk < kTok / 8; ++blk) {
          const int n0 = max(__shfl_sync(kFull, n, 8 * blk), 0);
          const int64_t off = (int64_t(n0) + r0) * row_pitch + int64_t(c) * 16;
          const unsigned char* ks = Kg + off;
          const unsigned char* vs = Vg + off;
          const uint32_t have = vmask >> (8 * blk);
#pragma unroll
          for (uint32_t i = 0; i < 8 / kRows; ++i) {
            const uint32_t bytes = (have >> (i * kRows + r0)) & 1u ? 16u : 0u;
            const uint32_t d = kdst + swz<ROWB>(8 * blk + i * kRows + r0, c << 4);
            cp_async16(d, ks, bytes);
            cp_async16(d + HALFB, vs, bytes);
            ks += step;
            vs += step;
          }
        }
      } else {
#pragma unroll
        for (uint32_t i = 0; i < kTok * kPieces / 32; ++i) {
          const uint32_t e = i * 32 + uint32_t(lane);
          const uint32_t r = e / kPieces, c = e % kPieces;
          const int n_r = __shfl_sync(kFull, n, int(r));
          const int64_t off = int64_t(n_r < 0 ? 0 : n_r) * row_pitch + int64_t(c) * 16;
          const uint32_t bytes = n_r < 0 ? 0u : 16u;
          const uint32_t d = kdst + swz<ROWB>(r, c << 4);
          cp_async16(d, Kg + off, bytes);
          cp_async16(d + HALFB, Vg + off, bytes);
        }
      }
    }
    cp_async_commit();                                         // an empty group keeps the count uniform
  };

  // ---- prologue: fill the first `depth` stages ---------------------------------------------------
  {
#pragma unroll 1
    for (int k0 = 0; k0 < depth; k0 += 4) {                    // four index reads at a time
      int j0[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) j0[k] = (k0 + k < depth) ? fetch_group(k0 + k) : -1;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (k0 + k < depth) fill(k0 + k, j0[k], warp + kWarps * (k0 + k));
    }
  }
  LongEngine<KV_T, D, RH> eng;
  eng.init(q + int64_t(live ? list : 0) * RH * D, lane);       // a list's RH query rows are consecutive, list after list
  int slot = 0;
  for (int k = 0; k < my_chunks; ++k) {
    const int stage = warp + kWarps * slot;
    const int j_next = fetch_group(k + depth);     // consumed by the refill at the end of the iteration
    // `depth` groups are in flight and the oldest is chunk k's: wait until depth - 1 remain.
    switch (depth) {
      case 2: cp_async_wait<1>(); break;
      case 3: cp_async_wait<2>(); break;
      case 4: cp_async_wait<3>(); break;
      case 5: cp_async_wait<4>(); break;
      case 6: cp_async_wait<5>(); break;
      case 7: cp_async_wait<6>(); break;
      default: cp_async_wait<7>(); break;
    }
    __syncwarp();                                  // every lane's pieces of the chunk have landed
    const uint32_t mask = ctl->mask[stage];
    if (mask != 0u) {
      const uint32_t kstage = ring + uint32_t(stage) * STAGEB;
      eng.chunk(kstage, kstage + HALFB, mask);
    }
    __syncwarp();                                  // all lanes are done with the stage
    fill(k + depth, j_next, stage);
    if (++slot == depth) slot = 0;
  }
  cp_async_wait<0>();

  // ---- merge the warps of the CTA ------------------------------------------------------------------
  __syncthreads();
  // The ring is idle now (every copy was waited for); reuse it for the merge.
  float* sm_m = reinterpret_cast<float*>(ring_ptr);                 // [kWarps][8]
  float* sm_l = sm_m + kWarps * 8;                                  // [kWarps][8]
  float* sm_acc = sm_l + kWarps * 8;                                // [kWarps][RH][D]
  eng.store(sm_m + warp * 8, sm_l + warp * 8, sm_acc + warp * RH * D);
  __syncthreads();
  if (settled && !wait_late) pdl_wait();
  // partial [RH][D + 2] = (m, l, acc[D]) of each list in the CTA
  const int list0 = int(blockIdx.x) * kWarps / sg.warps_per_list;
  const int n_lists = min((int(blockIdx.x) * kWarps + kWarps - 1) / sg.warps_per_list, sg.lists - 1) - list0 + 1;
  for (int i = threadIdx.x; i < n_lists * RH * D; i += kThreads) {
    const int ls = i / (RH * D), hh = i / D - ls * RH, c = i % D;
    const int w_at = (list0 + ls) * sg.warps_per_list - int(blockIdx.x) * kWarps;   // its first warp, counted from the CTA's first
    const int w0 = max(0, w_at), w1 = min(kWarps, w_at + sg.warps_per_list);
    float mx = -INFINITY;
#pragma unroll
    for (int k = 0; k < kWarps; ++k) if (k >= w0 && k < w1) mx = fmaxf(mx, sm_m[k * 8 + hh]);
    float lsum = 0.f, a = 0.f;
    if (mx > -INFINITY) {
#pragma unroll
      for (int k = 0; k < kWarps; ++k) {
        if (k < w0 || k >= w1) continue;
        const float w = ex2(sm_m[k * 8 + hh] - mx);
        lsum = fmaf(sm_l[k * 8 + hh], w, lsum);
        a = fmaf(sm_acc[(k * RH + hh) * D + c], w, a);
      }
    }
    const int slot0 = (list0 + ls) * sg.warps_per_list / kWarps;                     // the list's first CTA
    float* dst = partial + ((int64_t(list0 + ls) * RH + hh) * sg.slots + (int(blockIdx.x) - slot0)) * (D + 2);
    if (c == 0) { dst[0] = mx; dst[1] = lsum; }
    dst[2 + c] = a;
  }
  if (wait_late) pdl_wait();
}

template <typename KV_T, int D, int RH>
cudaError_t launch_rows(const Problem& p, const Workspace& w, const void* q, const void* K, const void* V, const int32_t* group_idx,
                        const int32_t* n_selected, float* partial, uint32_t* err, cudaStream_t st) {
  const size_t smem = kControlBytes + 128 + size_t(kWarps) * w.depth * 2 * kTok * D * sizeof(KV_T);
  int g_shift = -1;
  for (int sft = 0; sft < 31; ++sft) if ((1 << sft) == p.G) g_shift = sft;
  const SplitGrid sg{p.B * p.Hkv * (p.rho / RH), w.warps_per_list, w.splits};
  auto kern = sparse_decode_long_kernel<KV_T, D, RH>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3((sg.lists * sg.warps_per_list + kWarps - 1) / kWarps), dim3(kThreads), smem, st, p,
                    static_cast<const KV_T*>(q), static_cast<const KV_T*>(K), static_cast<const KV_T*>(V), group_idx, n_selected,
                    partial, sg, w.depth, g_shift, err);
}

template <typename KV_T, int D>
cudaError_t launch_heads(const Problem& p, const Workspace& w, const void* q, const void* K, const void* V, const int32_t* gi,
                         const int32_t* ns, float* partial, uint32_t* err, cudaStream_t st) {
  switch (w.heads_per_cta) {
    case 8: return launch_rows<KV_T, D, 8>(p, w, q, K, V, gi, ns, partial, err, st);
    case 7: return launch_rows<KV_T, D, 7>(p, w, q, K, V, gi, ns, partial, err, st);
    case 6: return launch_rows<KV_T, D, 6>(p, w, q, K, V, gi, ns, partial, err, st);
    case 5: return launch_rows<KV_T, D, 5>(p, w, q, K, V, gi, ns, partial, err, st);
    case 4: return launch_rows<KV_T, D, 4>(p, w, q, K, V, gi, ns, partial, err, st);
    case 3: return launch_rows<KV_T, D, 3>(p, w, q, K, V, gi, ns, partial, err, st);
    case 2: return launch_rows<KV_T, D, 2>(p, w, q, K, V, gi, ns, partial, err, st);
    default: return launch_rows<KV_T, D, 1>(p, w, q, K, V, gi, ns, partial, err, st);
  }
}

}  // namespace

void plan_long_gather(const Problem& p, Workspace* w) {
  const int64_t problems = int64_t(p.B) * p.Hkv * (p.rho / w->heads_per_cta), best = w->splits;
  const int64_t tokens = int64_t(p.M) * p.G + (p.N - int64_t(p.NG) * p.G);
  const size_t row = size_t(p.d) * 2;
  // A long gather of the tensor-core engine deals the warps of the whole GPU to the lists, not whole CTAs, with stages of 16
  // tokens and one CTA per SM: it leaves half of the registers to the next layer's select, which a decode step then runs
  // beside it (step.cu), and takes as long as two CTAs of half the stages or a little longer (a score_select and a
  // sparse_decode of 92 MB, 4 sequences, 8 heads: 42.6 against 42.0 us; 8 sequences, heads of 64 channels 44.0 against 45.1).
  // The select takes longer the more groups there are, and the scorer behind waits for both: not where the gather is over
  // long before.  us a layer with the other plan / with this one and no bound on the lookahead / bounded to one layer:
  //   4 sequences,  32768 tokens   50 MB 24.1 / 20.9 / 22.5    80 MB 28.6 / 26.7 / 28.4    110 MB 33.7 / 32.2 / 33.7
  //   4 sequences,  65536 tokens   50 MB 25.6 / 23.3 / 25.3    80 MB 30.1 / 27.7 / 30.0    110 MB 35.1 / 32.4 / 34.5
  //   8 sequences,  65536 tokens   50 MB 31.3 / 27.7 / 30.1    80 MB 36.2 / 32.0 / 35.0    110 MB 40.8 / 36.2 / 39.3
  //   4 sequences, 131072 tokens   60 MB 32.5 / 30.5 / 32.8    80 MB 35.7 / 34.1 / 37.1    110 MB 40.7 / 38.2 / 41.5
  // (groups of 8; 2 sequences of 50003 tokens, 26 MB: 25.4 / 26.2 unbounded).  134 MB of the last row gain again,
  // 43.2 / 38.8 / 41.9.
  const int64_t bytes = problems * tokens * int64_t(2 * row);
  w->long_gather = p.kv_dtype != KVSWAP_F32 && p.q_dtype == p.kv_dtype && select_beside_supported(p) &&
                   bytes >= std::max<int64_t>(47 << 20, int64_t(p.NG) * 5000);
  if (!w->long_gather) return;
  const int64_t n_stages = (tokens + kTok - 1) / kTok;
  auto slots_of = [&](int64_t per_list) {                        // CTAs that a list is spread over, at most
    int64_t most = 1;
    for (int64_t l = 0; l < std::min<int64_t>(kWarps, problems); ++l)
      most = std::max(most, ((l + 1) * per_list - 1) / kWarps - l * per_list / kWarps + 1);
    return most;
  };
  auto cost = [&](int64_t per_list) {                // in half stages of the slowest warp; 4 for what a CTA costs by itself
    const int64_t ctas = (problems * per_list + kWarps - 1) / kWarps;
    return (ctas + kNumSMs - 1) / kNumSMs * ((n_stages + per_list - 1) / per_list * 2 + 4);
  };
  int64_t per_list = 1;
  const int64_t limit = std::max<int64_t>(kWarps, n_stages);
  for (int64_t waves = 1; waves <= 8; ++waves) {                 // as many as fit so many waves, then as few as do the same work
    int64_t k = std::min(limit, waves * kNumSMs * kWarps / problems);
    if (k < 1) continue;
    const int64_t each = (n_stages + k - 1) / k;
    k = (n_stages + each - 1) / each;
    // (never more than `best` CTAs: see splits_room)
    if (slots_of(k) > best) k = k >= kWarps ? k / kWarps * kWarps : k >= 4 ? 4 : k >= 2 ? 2 : 1;
    if (slots_of(k) <= best && cost(k) < cost(per_list)) per_list = k;
  }
  w->depth = int(std::min<size_t>(kMaxDepth, (192u << 10) / (kWarps * 2 * kTok * row)));
  w->warps_per_list = int(per_list);
  w->splits = int(slots_of(per_list));
}

cudaError_t launch_long_gather(const Problem& p, const Workspace& w, const void* q, const void* K, const void* V,
                               const int32_t* group_idx, const int32_t* n_selected, float* partial, uint32_t* err, cudaStream_t st) {
  if (p.kv_dtype == KVSWAP_BF16)
    return p.d == 128 ? launch_heads<__nv_bfloat16, 128>(p, w, q, K, V, group_idx, n_selected, partial, err, st)
                      : launch_heads<__nv_bfloat16, 64>(p, w, q, K, V, group_idx, n_selected, partial, err, st);
  return p.d == 128 ? launch_heads<__half, 128>(p, w, q, K, V, group_idx, n_selected, partial, err, st)
                    : launch_heads<__half, 64>(p, w, q, K, V, group_idx, n_selected, partial, err, st);
}

}  // namespace kvswap
