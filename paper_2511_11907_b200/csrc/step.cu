// C-ABI entry points that serve all layers of a model in one call: the decode step over
// HBM-resident stores (one stream, each layer predicted one layer ahead of its attention), the
// decode step over reuse buffers in front of a slow tier (its copies on two streams of their own)
// and the append steps.  The tiered step keeps those two streams and a set of events per device;
// nothing else here keeps state.
#include <algorithm>
#include <mutex>
#include <vector>

#include "api_internal.cuh"
#include "combine.cuh"
#include "common.cuh"

using namespace kvswap;

extern "C" {

int kvswap_append_step(const kvswap_shape* shape, const kvswap_layers* layers, const void* k_new, const void* v_new,
                       int32_t* flushed_opt, void* cuda_stream) {
  if (flushed_opt != nullptr) *flushed_opt = 0;
  Problem p;
  int st = resolve_grown(shape, &p);
  if (st != KVSWAP_OK) return st;
  if (layers == nullptr || layers->K == nullptr || layers->V == nullptr || layers->meta == nullptr ||
      layers->proj == nullptr || k_new == nullptr || v_new == nullptr)
    return KVSWAP_ERR_NULL;
  if (layers->n_layers < 1) return KVSWAP_ERR_SHAPE;
  if (misaligned(k_new) || misaligned(v_new)) return KVSWAP_ERR_ALIGN;
  for (int l = 0; l < layers->n_layers; ++l) {
    if (layers->K[l] == nullptr || layers->V[l] == nullptr || layers->meta[l] == nullptr || layers->proj[l] == nullptr)
      return KVSWAP_ERR_NULL;
    if (misaligned(layers->K[l]) || misaligned(layers->V[l]) || misaligned(layers->meta[l]) ||
        misaligned(layers->proj[l]))
      return KVSWAP_ERR_ALIGN;
  }
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  // The tables are declared const for the read-only calls; this one writes the stores.
  void* const* Ks = const_cast<void* const*>(layers->K);
  void* const* Vs = const_cast<void* const*>(layers->V);
  if (launch_append_rows(p, k_new, v_new, Ks, Vs, layers->n_layers, p.N - 1, stream) != cudaSuccess)
    return KVSWAP_ERR_CUDA;
  if (p.N % p.G == 0) {
    if (launch_project_keys_layers(p, layers->K, layers->proj, const_cast<void* const*>(layers->meta),
                                   layers->n_layers, p.N - p.G, p.N, stream) != cudaSuccess)
      return KVSWAP_ERR_CUDA;
    if (flushed_opt != nullptr) *flushed_opt = 1;
  }
  return KVSWAP_OK;
}

static int check_layers(const kvswap_layers* layers, bool need_kv = true) {
  if (layers == nullptr || layers->meta == nullptr || layers->proj == nullptr) return KVSWAP_ERR_NULL;
  if (need_kv && (layers->K == nullptr || layers->V == nullptr)) return KVSWAP_ERR_NULL;
  if (layers->n_layers < 1 || layers->max_lookahead < 0) return KVSWAP_ERR_SHAPE;
  return KVSWAP_OK;
}

// The shape under which kvswap_sparse_decode sees a reuse store: n_slots groups followed by the
// rolling-buffer rows, dense [B, H_kv, (n_slots + 1) G, d].
static kvswap_shape reuse_store_shape(const kvswap_shape& s, int32_t n_slots) {
  kvswap_shape r = s;
  const int64_t R = int64_t(n_slots + 1) * s.group_size;
  r.n_ctx = n_slots * s.group_size + s.n_ctx % s.group_size;
  r.kv_stride_n = s.head_dim;
  r.kv_stride_h = R * s.head_dim;
  r.kv_stride_b = int64_t(s.n_kv_heads) * R * s.head_dim;
  return r;
}

// Per-device resources of the tiered step: two streams for the slow tier's copies and two events per layer.  Created
// on first use, kept for the life of the process.
namespace {
struct StepResources {
  cudaStream_t fetch[2] = {nullptr, nullptr};   // layers take turns
  cudaEvent_t join = nullptr;
  std::vector<cudaEvent_t> selected;     // selected[l]: layer l's selection is written
  std::vector<cudaEvent_t> fetched;      // fetched[l]: layer l's selected groups are in its reuse store
};
constexpr int kMaxDevices = 64;
std::mutex g_step_mutex;
StepResources g_step[kMaxDevices];

cudaError_t grow(std::vector<cudaEvent_t>* evs, int n) {
  while (int(evs->size()) < n) {
    cudaEvent_t ev = nullptr;
    cudaError_t e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    if (e != cudaSuccess) return e;
    evs->push_back(ev);
  }
  return cudaSuccess;
}

// Must be called with g_step_mutex held.
cudaError_t step_resources(int n_layers, StepResources** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  StepResources& r = g_step[dev];
  for (cudaStream_t& f : r.fetch) {
    if (f != nullptr) continue;
    e = cudaStreamCreateWithFlags(&f, cudaStreamNonBlocking);
    if (e != cudaSuccess) { f = nullptr; return e; }
  }
  if (r.join == nullptr) {
    e = cudaEventCreateWithFlags(&r.join, cudaEventDisableTiming);
    if (e != cudaSuccess) { r.join = nullptr; return e; }
  }
  if ((e = grow(&r.selected, n_layers)) != cudaSuccess) return e;
  if ((e = grow(&r.fetched, n_layers)) != cudaSuccess) return e;
  *out = &r;
  return cudaSuccess;
}
}  // namespace

// One decode step over all layers; with `tiers` the attention is served from per-layer reuse buffers
// that the fetch streams keep filled from the slow tier.
static int decode_step_impl(const kvswap_shape* shape, const kvswap_layers* layers, const kvswap_tiers* tiers,
                            const void* q, float* out, float* lse_opt, int32_t* group_idx, int32_t* n_selected,
                            void* ws, size_t ws_bytes, const kvswap_probe* probe_opt, void* cuda_stream) {
  Problem p;
  int st = resolve(shape, &p);
  if (st != KVSWAP_OK) return st;
  st = check_layers(layers, tiers == nullptr);
  if (st != KVSWAP_OK) return st;
  if (q == nullptr || out == nullptr || group_idx == nullptr || n_selected == nullptr) return KVSWAP_ERR_NULL;
  // Tiered: the predictor uses the head of the workspace, the attention over the reuse stores
  // (another shape, another plan) the part behind it, since the two run on different streams.
  kvswap_shape shape_attn = *shape;
  void* ws_attn = ws;
  size_t ws_attn_bytes = ws_bytes;
  if (tiers != nullptr) {
    Problem pr;
    if (tiers->max_groups < 1) return KVSWAP_ERR_SHAPE;
    st = resolve_reuse(shape, tiers->n_slots, tiers->max_groups, &pr);
    if (st != KVSWAP_OK) return st;
    if (tiers->K_slow == nullptr || tiers->V_slow == nullptr || tiers->K_reuse == nullptr ||
        tiers->V_reuse == nullptr || tiers->state == nullptr || tiers->slot_idx == nullptr ||
        tiers->miss_group == nullptr || tiers->miss_slot == nullptr || tiers->n_miss == nullptr)
      return KVSWAP_ERR_NULL;
    if (tiers->state_bytes < sizeof(int32_t) * reuse_state_words(pr, tiers->n_slots, tiers->max_groups))
      return KVSWAP_ERR_WORKSPACE;
    for (int l = 0; l < layers->n_layers; ++l) {
      if (tiers->K_slow[l] == nullptr || tiers->V_slow[l] == nullptr || tiers->K_reuse[l] == nullptr ||
          tiers->V_reuse[l] == nullptr || tiers->state[l] == nullptr)
        return KVSWAP_ERR_NULL;
      if (misaligned(tiers->K_slow[l]) || misaligned(tiers->V_slow[l]) || misaligned(tiers->K_reuse[l]) ||
          misaligned(tiers->V_reuse[l]) || misaligned(tiers->state[l]))
        return KVSWAP_ERR_ALIGN;
    }
    shape_attn = reuse_store_shape(*shape, tiers->n_slots);
    const size_t head_bytes = (kvswap_workspace_bytes(shape) + 255) & ~size_t(255);
    if (ws == nullptr) return KVSWAP_ERR_NULL;
    if (ws_bytes < head_bytes + kvswap_workspace_bytes(&shape_attn)) return KVSWAP_ERR_WORKSPACE;
    ws_attn = static_cast<char*>(ws) + head_bytes;
    ws_attn_bytes = ws_bytes - head_bytes;
  }
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  const int L = layers->n_layers;
  const size_t q_bytes = size_t(p.B) * p.Hq * p.d * dtype_bytes(p.q_dtype);
  const size_t out_elems = size_t(p.B) * p.Hq * p.d;
  const size_t idx_elems = size_t(p.B) * p.S * p.M, nsel_elems = size_t(p.B) * p.S;
  Workspace w;
  st = check_score_select(shape, q, layers->proj[0], layers->meta[0], group_idx, n_selected, nullptr, ws, ws_bytes,
                          &p, &w);
  if (st != KVSWAP_OK) return st;
  for (int l = 0; l < L; ++l) {
    if (layers->proj[l] == nullptr || layers->meta[l] == nullptr) return KVSWAP_ERR_NULL;
    if (tiers == nullptr && (layers->K[l] == nullptr || layers->V[l] == nullptr)) return KVSWAP_ERR_NULL;
    if (tiers == nullptr && (misaligned(layers->K[l]) || misaligned(layers->V[l]))) return KVSWAP_ERR_ALIGN;
    if (misaligned(layers->proj[l]) || misaligned(layers->meta[l])) return KVSWAP_ERR_ALIGN;
  }

  if (tiers == nullptr) {
    if (misaligned(out) || (lse_opt && (reinterpret_cast<uintptr_t>(lse_opt) & 3u))) return KVSWAP_ERR_ALIGN;
    // Schedule (Sec. 4.3, online prediction, and Sec. 4.4): layer l + 1 is scored ahead of layer l's
    // attention -- as early as a model allows whose layer-(l+1) prediction is formed from the input of
    // layer l, which exists once layer l - 1 has been attended -- and its TopK follows that attention.
    // All on the caller's stream, every kernel a programmatic dependent launch, so each kernel's
    // set-up and first fetches overlap its predecessor's tail:
    //   score(0) select(0) | score(1) attention(0) select(1) | score(2) attention(1) select(2) | ...
    // The scorer streams the compact cache at HBM rate and the attention gathers at HBM rate; neither
    // leaves the other room on an SM, so they run one after the other, and what the order hides is
    // the latency-bound part: the TopK of layer l + 1 is not needed before attention l + 1, and the
    // gather of layer l starts fetching while the scorer of layer l + 1 drains.
    // Settled inputs: the first layer's predictor waits for whatever wrote the step's inputs (unless the caller
    // has promised that they are settled), so they are complete before any later kernel of the step starts; a selection
    // is complete before the scorer that precedes its attention passes its own dependency wait.
    Problem p_settled = p;
    p_settled.flags |= KVSWAP_INPUTS_SETTLED;
    Problem p_wait = p;                             // the last attention: its selection may be the launch before it
    p_wait.flags &= ~KVSWAP_INPUTS_SETTLED;
    kvswap_shape shape_settled = *shape;
    shape_settled.flags |= KVSWAP_INPUTS_SETTLED;
    auto ev = [&](void* e) { if (e != nullptr) cudaEventRecord(static_cast<cudaEvent_t>(e), stream); };
    auto probed = [&](int l) { return probe_opt != nullptr && probe_opt->layer == l; };
    // Where the kernel that merges layer l's partials and selects for layer l + 1 can also form the
    // summed low-rank queries of layer l + 2 (its combine CTAs idle until the gather has finished),
    // that layer's scorer finds them in the workspace and goes straight to its tiles.  The workspace
    // has two query buffers: the scorer of layer l + 1 may still be reading its own.
    const bool ahead = query_ahead_supported(p);
    const bool merges = select_merges_with_combine(p) && (p.d == 64 || p.d == 128) && w.splits <= kMaxSplits;
    int formed_for = -1;                            // the layer whose queries the last merged launch formed
    auto score = [&](int l) -> int {
      if (probed(l)) ev(probe_opt->ev_begin);
      const void* ql = static_cast<const char*>(q) + size_t(l) * q_bytes;
      return score_launch(l == 0 ? p : p_settled, w, ql, layers->proj[l], layers->meta[l], nullptr, ws, stream,
                          formed_for == l ? (l & 1) : -1) == cudaSuccess
                 ? KVSWAP_OK : KVSWAP_ERR_CUDA;
    };
    auto select = [&](int l) -> int {
      const cudaError_t e = select_launch(p_settled, w, group_idx + size_t(l) * idx_elems,
                                          n_selected + size_t(l) * nsel_elems, nullptr, ws, stream);
      if (probed(l)) ev(probe_opt->ev_mid);
      return e == cudaSuccess ? KVSWAP_OK : KVSWAP_ERR_CUDA;
    };
    // The attention of layer l and the TopK of layer l + 1: the split-K gather, then one kernel that
    // merges its partials and selects (where the select has that form), else the two one after the other.
    float* partial = reinterpret_cast<float*>(static_cast<char*>(ws) + w.off_partial);
    auto attend_then_select = [&](int l) -> int {
      const void* ql = static_cast<const char*>(q) + size_t(l) * q_bytes;
      float* out_l = out + size_t(l) * out_elems;
      float* lse_l = lse_opt ? lse_opt + size_t(l) * p.B * p.Hq : nullptr;
      const int32_t* idx_l = group_idx + size_t(l) * idx_elems;
      const int32_t* nsel_l = n_selected + size_t(l) * nsel_elems;
      const bool next = l + 1 < L;
      // (the last layer's attention follows its own TopK directly: that selection is not settled)
      // Where the merged launch follows, the gather waits for the scorer before it as soon as its
      // first fills are out and lets that launch start only then: its TopK, whose inputs that scorer
      // wrote, need not wait for the gather.
      Problem p_early = p_settled;
      p_early.flags |= kFlagWaitEarly;
      const Problem& pa = !next ? p_wait : merges ? p_early : p_settled;
      if (launch_sparse_decode(pa, w, ql, layers->K[l], layers->V[l], idx_l, nsel_l, partial, out_l, lse_l,
                               static_cast<uint32_t*>(ws), stream, /*combine=*/false) != cudaSuccess)
        return KVSWAP_ERR_CUDA;
      cudaError_t e = cudaSuccess;
      const bool form = ahead && l + 2 < L;
      const void* q_ahead = form ? static_cast<const char*>(q) + size_t(l + 2) * q_bytes : nullptr;
      Problem p_two_back = p_settled;
      p_two_back.flags |= kFlagInputsTwoBack;
      const bool merged = next && merges &&
                          select_with_combine_launch(p_two_back, w, group_idx + size_t(l + 1) * idx_elems,
                                                     n_selected + size_t(l + 1) * nsel_elems, ws,
                                                     combine_job(p, w, partial, out_l, lse_l), p.d, stream, &e, q_ahead,
                                                     form ? layers->proj[l + 2] : nullptr, (l + 2) & 1);
      if (merged && form && e == cudaSuccess) formed_for = l + 2;
      if (!merged) {
        e = launch_combine(p, combine_job(p, w, partial, out_l, lse_l), CombineJob{}, stream);
      }
      if (probed(l)) ev(probe_opt->ev_end);
      if (e != cudaSuccess) return KVSWAP_ERR_CUDA;
      if (next && !merged) return select(l + 1);
      if (next && probed(l + 1)) ev(probe_opt->ev_mid);
      return KVSWAP_OK;
    };
    // Short contexts: the predictor of a layer is one launch of clusters and so is its attention (the splits
    // merge in the cluster), and the two run side by side:
    //   predict(0) | predict(1) attention(0) | predict(2) attention(1) | ..
    // predict(l + 1) waits for attention(l - 1) and only then lets attention(l) start, which finds the selection
    // of predict(l) complete: attention(l - 1) waited for it before it wrote its results.  Two launches a layer
    // instead of three, and neither waits for the other: 36 layers of B = 1, N = 16384, 8 KV heads, M = 256 through
    // host memory 539 -> 425 us; at B = 1, N = 4096 a layer takes 8.5 us against 12.9.
    // Where the splits do not merge in clusters a combine follows each gather.
    if (score_select_cluster_supported(p) && (w.merge_in_cluster || w.beside)) {
      auto predict = [&](int l) -> int {
        if (probed(l)) ev(probe_opt->ev_begin);
        const cudaError_t e = launch_score_select_cluster(
            l == 0 ? p : p_settled, static_cast<const char*>(q) + size_t(l) * q_bytes, layers->proj[l], layers->meta[l], nullptr,
            group_idx + size_t(l) * idx_elems, n_selected + size_t(l) * nsel_elems, static_cast<uint32_t*>(ws), stream);
        if (probed(l)) ev(probe_opt->ev_mid);
        return e == cudaSuccess ? KVSWAP_OK : KVSWAP_ERR_CUDA;
      };
      // predict(l + 1) had waited for all that came before it when attention(l) was let in: that one waits last.
      Problem p_late = p_settled;
      p_late.flags |= kFlagWaitLate;
      float* partial = w.merge_in_cluster ? nullptr : reinterpret_cast<float*>(static_cast<char*>(ws) + w.off_partial);
      int status = predict(0);
      for (int l = 0; l < L && status == KVSWAP_OK; ++l) {
        if (l + 1 < L) status = predict(l + 1);
        if (status != KVSWAP_OK) break;
        // (the last layer's attention follows an attention directly: its selection is complete when that one is)
        const cudaError_t e = launch_sparse_decode(
            l + 1 < L ? p_late : p_wait, w, static_cast<const char*>(q) + size_t(l) * q_bytes, layers->K[l], layers->V[l],
            group_idx + size_t(l) * idx_elems, n_selected + size_t(l) * nsel_elems, partial, out + size_t(l) * out_elems,
            lse_opt ? lse_opt + size_t(l) * p.B * p.Hq : nullptr, static_cast<uint32_t*>(ws), stream);
        if (probed(l)) ev(probe_opt->ev_end);
        if (e != cudaSuccess) status = KVSWAP_ERR_CUDA;
      }
      return status;
    }
    // Long gathers: the select of a layer runs beside the gather of the layer before, which takes one CTA per SM and half of its
    // registers, instead of behind it:
    //   score(0) select(0) | score(1) select(1) attention(0) | score(2) select(2) attention(1) | ...
    // The launch of select(l + 1) also forms the queries of layer l + 2, beside score(l + 1); the scorer does not count leading
    // digits.  With a lookahead of one layer a combine follows each gather, and score(l + 1) waits for that of layer l - 1, whose
    // outputs the input of layer l + 1 is made from.  Otherwise the launch of select(l + 1) merges the partials of
    // attention(l - 1) too, beside score(l + 1).
    // What each kernel waits for: score(l + 1) for attention(l - 1) or its combine and all before it, and lets select(l + 1)
    // start only then; select(l + 1) lets attention(l) start when its own CTAs have, so the selection of layer l is complete by
    // then; it waits for score(l + 1); attention(l) waits for select(l + 1): with one buffer of partials before it writes them,
    // as the merge may still read those of layer l - 1, with two (layers take turns) at its end.  So up to three kernels are in
    // flight: a scorer's successor starts only when all before the scorer is complete, and every kernel waits before it ends.
    // 12 layers of B = 4, N = 131072, M = 1024: 518 us with the select behind the gather, 466 with it beside that, 503 with a
    // lookahead of one layer; eight tokens over 12 layers of B = 8, N = 32760, one layer: 3239, 3114.
    if (w.long_gather) {
      const bool merge_first = layers->max_lookahead == 1;
      const bool two = 2 * w.splits <= w.splits_room;
      auto partial_of = [&](int l) { return two && (l & 1) ? partial + size_t(p.B) * p.Hq * w.splits * (p.d + 2) : partial; };
      Problem p_late = p_settled;
      p_late.flags |= kFlagWaitLate;
      CombineJob pending = {};                      // gathered, not merged
      cudaError_t e = cudaSuccess;
      auto predict = [&](int l) {
        const void* ql = static_cast<const char*>(q) + size_t(l) * q_bytes;
        if (probed(l)) ev(probe_opt->ev_begin);
        e = score_launch(p_settled, w, ql, layers->proj[l], layers->meta[l], nullptr, ws, stream, formed_for == l ? (l & 1) : -1,
                         /*beside=*/true);
        const bool form = ahead && l + 1 < L;
        if (e == cudaSuccess)
          e = select_beside_launch(p_settled, w, group_idx + size_t(l) * idx_elems, n_selected + size_t(l) * nsel_elems, ws,
                                   pending, stream, form ? static_cast<const char*>(ql) + q_bytes : nullptr,
                                   form ? layers->proj[l + 1] : nullptr, (l + 1) & 1);
        if (form) formed_for = l + 1;
        pending = CombineJob{};
        if (probed(l)) ev(probe_opt->ev_mid);
      };
      int status = score(0);
      if (status == KVSWAP_OK) status = select(0);
      if (status != KVSWAP_OK) return status;
      for (int l = 0; l < L && e == cudaSuccess; ++l) {
        const bool last = l + 1 == L;
        if (!last) predict(l + 1);
        if (last && pending.rows > 0 && !two && e == cudaSuccess) {
          e = launch_combine(p, pending, CombineJob{}, stream);
          pending = CombineJob{};
        }
        // (the last layer's attention follows an attention, or its own selection)
        float* out_l = out + size_t(l) * out_elems;
        float* lse_l = lse_opt ? lse_opt + size_t(l) * p.B * p.Hq : nullptr;
        if (e == cudaSuccess)
          e = launch_sparse_decode(last ? p_wait : two ? p_late : p_settled, w, static_cast<const char*>(q) + size_t(l) * q_bytes,
                                   layers->K[l], layers->V[l], group_idx + size_t(l) * idx_elems,
                                   n_selected + size_t(l) * nsel_elems, partial_of(l), out_l, lse_l,
                                   static_cast<uint32_t*>(ws), stream, /*combine=*/false);
        const CombineJob job = combine_job(p, w, partial_of(l), out_l, lse_l);
        if (last || merge_first || probed(l)) {
          if (e == cudaSuccess) e = launch_combine(p, job, pending, stream);
          pending = CombineJob{};
          if (probed(l)) ev(probe_opt->ev_end);
        } else {
          pending = job;
        }
      }
      return e == cudaSuccess ? KVSWAP_OK : KVSWAP_ERR_CUDA;
    }
    int status = score(0);
    if (status == KVSWAP_OK) status = select(0);
    for (int l = 0; l < L && status == KVSWAP_OK; ++l) {
      if (l + 1 < L) status = score(l + 1);
      if (status == KVSWAP_OK) status = attend_then_select(l);
    }
    return status;
  }

  // Tiered schedule.  The caller's stream predicts and attends, one layer ahead as in kvswap_decode_step; the slow
  // tier's link is kept busy from two streams of its own:
  //   caller's stream:  predict(0) | predict(1) wait fetched[0] attend(0) | predict(2) wait fetched[1] attend(1) | ..
  //   fetch streams:    wait selected[l];  lookup and fill(l);  record fetched[l]        (two, layers take turns: the
  //                     lookup of a layer runs while the layer before it is still copied)
  // A layer's misses cross the link while the layer before it is attended and the next one predicted.  (With lookup
  // and fill behind each other on the predictor's stream the link idled during every prediction: 1580 us for four
  // steps of four layers, B = 1, N = 16384, M = 256, 8 KV heads of 128, of which the link needs 1184; now 1427.)
  // The first layer's predictor waits for the step's inputs (unless the caller has promised that they are settled), and
  // a slot list is awaited through its event: the inputs of the others are settled.
  kvswap_shape shape_settled = shape_attn;
  shape_settled.flags |= KVSWAP_INPUTS_SETTLED;
  Problem p_settled = p;
  p_settled.flags |= KVSWAP_INPUTS_SETTLED;
  std::lock_guard<std::mutex> lock(g_step_mutex);
  StepResources* res = nullptr;
  if (step_resources(L, &res) != cudaSuccess) return KVSWAP_ERR_CUDA;

  auto predict_and_fetch = [&](int l) -> int {
    const void* ql = static_cast<const char*>(q) + size_t(l) * q_bytes;
    int32_t* idx_l = group_idx + size_t(l) * idx_elems;
    int32_t* nsel_l = n_selected + size_t(l) * nsel_elems;
    if (score_select_launch(l == 0 ? p : p_settled, w, ql, layers->proj[l], layers->meta[l], idx_l, nsel_l, nullptr, ws, stream) != cudaSuccess ||
        cudaEventRecord(res->selected[l], stream) != cudaSuccess ||
        cudaStreamWaitEvent(res->fetch[l & 1], res->selected[l], 0) != cudaSuccess ||
        launch_reuse_fetch(p, tiers->n_slots, tiers->max_groups, idx_l, nsel_l, static_cast<int32_t*>(tiers->state[l]),
                           tiers->K_slow[l], tiers->V_slow[l], tiers->K_reuse[l], tiers->V_reuse[l],
                           tiers->slot_idx + size_t(l) * idx_elems, tiers->miss_group + size_t(l) * idx_elems,
                           tiers->miss_slot + size_t(l) * idx_elems, tiers->n_miss + size_t(l) * nsel_elems,
                           res->fetch[l & 1]) != cudaSuccess ||
        cudaEventRecord(res->fetched[l], res->fetch[l & 1]) != cudaSuccess)
      return KVSWAP_ERR_CUDA;
    return KVSWAP_OK;
  };
  int status = predict_and_fetch(0);
  for (int l = 0; l < L && status == KVSWAP_OK; ++l) {
    if (l + 1 < L) status = predict_and_fetch(l + 1);
    if (status != KVSWAP_OK) break;
    if (cudaStreamWaitEvent(stream, res->fetched[l], 0) != cudaSuccess) { status = KVSWAP_ERR_CUDA; break; }
    status = kvswap_sparse_decode(&shape_settled, static_cast<const char*>(q) + size_t(l) * q_bytes, tiers->K_reuse[l],
                                  tiers->V_reuse[l], tiers->slot_idx + size_t(l) * idx_elems,
                                  n_selected + size_t(l) * nsel_elems, out + size_t(l) * out_elems,
                                  lse_opt ? lse_opt + size_t(l) * p.B * p.Hq : nullptr, ws_attn, ws_attn_bytes, cuda_stream);
  }
  if (status != KVSWAP_OK) {
    // a launch failed: join whatever the fetch streams were given after their last awaited events
    for (cudaStream_t f : res->fetch)
      if (cudaEventRecord(res->join, f) != cudaSuccess || cudaStreamWaitEvent(stream, res->join, 0) != cudaSuccess)
        return KVSWAP_ERR_CUDA;
  }
  return status;
}

int kvswap_decode_step(const kvswap_shape* shape, const kvswap_layers* layers, const void* q, float* out,
                       float* lse_opt, int32_t* group_idx, int32_t* n_selected, void* ws, size_t ws_bytes,
                       const kvswap_probe* probe_opt, void* cuda_stream) {
  return decode_step_impl(shape, layers, nullptr, q, out, lse_opt, group_idx, n_selected, ws, ws_bytes, probe_opt,
                          cuda_stream);
}

size_t kvswap_tiered_workspace_bytes(const kvswap_shape* shape, int32_t n_slots) {
  Problem p;
  if (resolve_reuse(shape, n_slots, 0, &p) != KVSWAP_OK) return 0;
  const kvswap_shape r = reuse_store_shape(*shape, n_slots);
  const size_t tail = kvswap_workspace_bytes(&r);
  if (tail == 0) return 0;
  return ((kvswap_workspace_bytes(shape) + 255) & ~size_t(255)) + tail;
}

int kvswap_decode_step_tiered(const kvswap_shape* shape, const kvswap_layers* layers, const kvswap_tiers* tiers,
                              const void* q, float* out, float* lse_opt, int32_t* group_idx, int32_t* n_selected,
                              void* ws, size_t ws_bytes, void* cuda_stream) {
  if (tiers == nullptr) return KVSWAP_ERR_NULL;
  return decode_step_impl(shape, layers, tiers, q, out, lse_opt, group_idx, n_selected, ws, ws_bytes, nullptr,
                          cuda_stream);
}

int kvswap_append_step_tiered(const kvswap_shape* shape, const kvswap_layers* layers, const kvswap_tiers* tiers,
                              const void* k_new, const void* v_new, int32_t* flushed_opt, void* cuda_stream) {
  if (flushed_opt != nullptr) *flushed_opt = 0;
  Problem p;                                   // the grown context: N + 1 tokens, the slow tier's strides
  int st = resolve_grown(shape, &p);
  if (st != KVSWAP_OK) return st;
  st = check_layers(layers, false);
  if (st != KVSWAP_OK) return st;
  if (tiers == nullptr || tiers->K_slow == nullptr || tiers->V_slow == nullptr || tiers->K_reuse == nullptr ||
      tiers->V_reuse == nullptr || k_new == nullptr || v_new == nullptr)
    return KVSWAP_ERR_NULL;
  if (tiers->n_slots < 1) return KVSWAP_ERR_SHAPE;
  // the grown context must still fit the slot tables the next tiered step will use
  if (tiers->max_groups > 0 && p.NG > tiers->max_groups) return KVSWAP_ERR_SHAPE;
  if (misaligned(k_new) || misaligned(v_new)) return KVSWAP_ERR_ALIGN;
  const int L = layers->n_layers;
  for (int l = 0; l < L; ++l) {
    if (tiers->K_slow[l] == nullptr || tiers->V_slow[l] == nullptr || tiers->K_reuse[l] == nullptr ||
        tiers->V_reuse[l] == nullptr || layers->meta[l] == nullptr || layers->proj[l] == nullptr)
      return KVSWAP_ERR_NULL;
    if (misaligned(tiers->K_slow[l]) || misaligned(tiers->V_slow[l]) || misaligned(tiers->K_reuse[l]) ||
        misaligned(tiers->V_reuse[l]) || misaligned(layers->meta[l]) || misaligned(layers->proj[l]))
      return KVSWAP_ERR_ALIGN;
  }
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  // The new token joins the rolling-buffer rows of every layer's reuse store.
  const int64_t fast_rows = int64_t(tiers->n_slots + 1) * p.G;
  const int n = p.N - 1;                       // its position in the context
  Problem fast = p;
  fast.kv_sn = p.d;
  fast.kv_sh = fast_rows * p.d;
  fast.kv_sb = int64_t(p.Hkv) * fast.kv_sh;
  if (launch_append_rows(fast, k_new, v_new, tiers->K_reuse, tiers->V_reuse, L, tiers->n_slots * p.G + n % p.G,
                         stream) != cudaSuccess)
    return KVSWAP_ERR_CUDA;
  if (p.N % p.G == 0) {
    // The group is complete: its rows go to the slow tier, and its compact-cache rows are built
    // from there (the projection reads the rows it was just handed; same stream).
    if (launch_flush_rows(p, tiers->K_reuse, tiers->V_reuse, const_cast<void* const*>(tiers->K_slow),
                          const_cast<void* const*>(tiers->V_slow), L, fast_rows, int64_t(tiers->n_slots) * p.G,
                          p.N - p.G, stream) != cudaSuccess ||
        launch_project_keys_layers(p, tiers->K_slow, layers->proj, const_cast<void* const*>(layers->meta), L,
                                   p.N - p.G, p.N, stream) != cudaSuccess)
      return KVSWAP_ERR_CUDA;
    if (flushed_opt != nullptr) *flushed_opt = 1;
  }
  return KVSWAP_OK;
}

int kvswap_decode_step_host(const kvswap_shape* shape, const kvswap_layers* layers, const void* q_host,
                            float* out_host, void* q_dev, float* out_dev, int32_t* group_idx,
                            int32_t* n_selected, void* ws, size_t ws_bytes, void* cuda_stream) {
  Problem p;
  int st = resolve(shape, &p);
  if (st != KVSWAP_OK) return st;
  st = check_layers(layers);
  if (st != KVSWAP_OK) return st;
  if (q_host == nullptr || out_host == nullptr || q_dev == nullptr || out_dev == nullptr) return KVSWAP_ERR_NULL;
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  const size_t L = size_t(layers->n_layers);
  const size_t q_bytes = L * p.B * p.Hq * p.d * dtype_bytes(p.q_dtype);
  const size_t out_bytes = L * p.B * p.Hq * p.d * sizeof(float);
  if (cudaMemcpyAsync(q_dev, q_host, q_bytes, cudaMemcpyHostToDevice, stream) != cudaSuccess) return KVSWAP_ERR_CUDA;
  st = kvswap_decode_step(shape, layers, q_dev, out_dev, nullptr, group_idx, n_selected, ws, ws_bytes, nullptr,
                          cuda_stream);
  if (st != KVSWAP_OK) return st;
  if (cudaMemcpyAsync(out_host, out_dev, out_bytes, cudaMemcpyDeviceToHost, stream) != cudaSuccess)
    return KVSWAP_ERR_CUDA;
  return KVSWAP_OK;
}

}  // extern "C"
