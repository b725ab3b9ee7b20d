"""What is timed: the calls a user of this library makes while a model decodes and prefills.

A case names a kind of pass (below), the attention shape of a model, the length and number of its
sequences and the options of the method.  Inputs are seeded synthetic tensors drawn on the GPU: K, V
and q from N(0, 1), where `heavy` says so with that share of positions whose keys are aligned with the
query, an orthonormal adapter (what the right singular vectors of such keys are), and a compact cache
computed here in fp32, so that inputs depend on the seed alone.

kinds
  calls    per layer kvswap_score_select, then kvswap_sparse_decode: a model that runs its own layers
           between the calls
  step     kvswap_decode_step over all layers
  host     kvswap_decode_step_host: queries come from and outputs go to pinned host memory
  grow     `steps` generated tokens: kvswap_append_step, then kvswap_decode_step, each with the
           context one token longer; one of the tokens completes a group of the compact cache
  tiered   the K/V of the whole context in pinned host memory behind reuse buffers in HBM: `steps`
           kvswap_decode_step_tiered from empty buffers on, over a random walk of queries
  prefill  kvswap_project_keys over the whole prompt, layer by layer
"""
import math

import torch

from paper_2511_11907_b200 import binding as kv
from paper_2511_11907_b200 import runtime as rt

_TORCH = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16, "e4m3": torch.float8_e4m3fn}
_TAG = {"f32": kv.KVSWAP_F32, "bf16": kv.KVSWAP_BF16, "f16": kv.KVSWAP_F16, "e4m3": kv.KVSWAP_E4M3}
_SIZE = {"f32": 4, "bf16": 2, "f16": 2, "e4m3": 1}


def _case(kind, layers, batch, n_ctx, q_heads, kv_heads, head_dim, rank, group, top_k, kv_type="bf16", meta="f16",
          per_head=False, all_heads=False, softmax=False, heavy=0.0, steps=1):
    return dict(kind=kind, layers=layers, batch=batch, n_ctx=n_ctx, q_heads=q_heads, kv_heads=kv_heads,
                head_dim=head_dim, rank=rank, group=group, top_k=top_k, kv=kv_type, meta=meta, per_head=per_head,
                all_heads=all_heads, softmax=softmax, heavy=heavy, steps=steps)


def listed():
    """Shapes are those of the library's five benchmark configurations, with as many layers as fit a GPU three
    times over, and ragged, other-typed or other-optioned neighbours of them."""
    def named(name, *a, **k):
        return dict(_case(*a, **k), name=name)

    return [
        # the smallest use: one layer of a small fp32 model with a 2K context; launches and the host count
        named("calls_f32_2k", "calls", 1, 1, 2048, 8, 2, 64, 16, 4, 32, kv_type="f32", meta="f32"),
        # one user's chat with a 16K context, end to end through host memory: every layer is a small launch
        named("host_b1_16k", "host", 36, 1, 16384, 32, 8, 128, 32, 8, 256, heavy=0.01),
        # a server's batch that generates 8 tokens; the last one completes a group
        named("grow_b8_32k", "grow", 12, 8, 32760, 32, 8, 128, 32, 8, 400, steps=8),
        # many long sequences, three query heads per KV head, groups of 16
        named("step_b16_64k", "step", 6, 16, 65536, 24, 8, 128, 32, 16, 256, heavy=0.005),
        # few very long sequences: the benchmark's headline shape
        named("step_b4_128k", "step", 12, 4, 131072, 32, 8, 128, 32, 8, 1024),
        # one adapter per KV head (the more accurate, larger compact cache), fp16 model, ragged length
        named("step_per_head_f16", "step", 8, 2, 50003, 32, 8, 128, 32, 8, 400, kv_type="f16", per_head=True),
        # 8-bit compact cache, odd batch, ragged length
        named("step_e4m3_ragged", "step", 12, 3, 98301, 24, 8, 128, 32, 16, 300, meta="e4m3"),
        # the paper's selection (one per sequence, scores summed over all heads) at twice the rank, layer by layer
        named("calls_all_heads_r64", "calls", 8, 2, 32768, 32, 8, 128, 64, 8, 400, all_heads=True),
        # scores as attention weights (softmax per head before the head sum), heads of 64 channels
        named("step_softmax_d64", "step", 8, 4, 40001, 16, 4, 64, 32, 8, 400, softmax=True),
        # long-document prefill of four layers
        named("prefill_b4_128k", "prefill", 4, 4, 131072, 32, 8, 128, 32, 8, 1024),
        # a user's prompt of a few thousand tokens, fp16 model, all layers
        named("prefill_f16_5k", "prefill", 28, 1, 5003, 32, 8, 128, 32, 8, 256, kv_type="f16"),
        # cache in host memory: the step after prefill, which fetches everything, and three that reuse most of it
        named("tiered_b1_16k", "tiered", 4, 1, 16384, 32, 8, 128, 32, 8, 256, steps=4),
    ]


def draw(rng):
    """One more case of the same ranges."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choices(["step", "calls", "prefill", "host", "grow", "tiered"], [38, 22, 18, 10, 6, 6])[0]
    kv_type = rng.choices(["bf16", "f16", "f32"], [65, 22, 13])[0]
    head_dim = rng.choice([128, 128, 128, 64])
    kv_heads = rng.choice([2, 4, 8, 8, 8])
    rho = rng.choice([1, 2, 3, 4, 4, 4, 8])
    rank = rng.choices([16, 32, 64], [15, 65, 20])[0]
    per_head = rng.random() < 0.25
    all_heads = rng.random() < 0.2
    softmax = kind != "prefill" and rng.random() < 0.1
    group = rng.choices([4, 8, 16, 32, 12], [20, 40, 20, 10, 10])[0]
    meta = "f32" if kv_type == "f32" and rng.random() < 0.7 else "f16"
    # the 8-bit compact cache: rank 32, groups of a power of two, raw scores, one score term per row
    if meta == "f16" and rank == 32 and group != 12 and not softmax and not (per_head and all_heads) and rng.random() < 0.2:
        meta = "e4m3"
    n_ctx = log_int(1500, 131072)
    batch = log_int(1, 16)
    if kind == "tiered":
        n_ctx, batch = log_int(1500, 20000), rng.choice([1, 1, 2])
    top_k = min(log_int(32, 1024), max(16, n_ctx // group // 4))
    # a drawn case stays below the largest listed ones, in memory and in work
    row = kv_heads * head_dim * _SIZE[kv_type]
    most = {"tiered": 0.25e9, "prefill": 4e9 if kv_type == "bf16" else 1.5e9}.get(kind, 10e9)
    stores = 1 if kind == "prefill" else 2
    while stores * batch * n_ctx * row > most:
        if batch > 1:
            batch //= 2
        else:
            n_ctx = n_ctx * 2 // 3
    layers = max(1, min(rng.randint(1, 36), int(most / (stores * batch * n_ctx * row))))
    steps = {"grow": min(group, 8), "tiered": 3}.get(kind, 1)
    if kind == "grow":                                           # one of the tokens completes a group
        n_ctx = (n_ctx // group + 1) * group - rng.randint(1, steps)
    c = _case(kind, layers, batch, n_ctx, kv_heads * rho, kv_heads, head_dim, rank, group, top_k, kv_type, meta,
              per_head, all_heads, softmax, rng.choice([0.0, 0.005, 0.01]) if kind != "prefill" else 0.0, steps)
    while work(c)["bytes"] > 5e9 and c["layers"] > 1:
        c["layers"] -= 1
    return c


def _shape(c, n_ctx, rows):
    """The library's description of the case with n_ctx tokens in stores that have room for `rows`."""
    hm = c["kv_heads"] if c["per_head"] else 1
    d, r = c["head_dim"], c["rank"]
    return kv.make_shape(
        batch=c["batch"], n_ctx=n_ctx, n_q_heads=c["q_heads"], n_kv_heads=c["kv_heads"], head_dim=d, rank=r,
        meta_heads=hm, group_size=c["group"], top_k=c["top_k"], kv_dtype=_TAG[c["kv"]], meta_dtype=_TAG[c["meta"]],
        q_dtype=_TAG[c["kv"]], scope=kv.KVSWAP_SCOPE_ALL_HEADS if c["all_heads"] else kv.KVSWAP_SCOPE_KV_HEAD,
        kv_strides=(c["kv_heads"] * rows * d, rows * d, d), meta_strides=(hm * rows * r, rows * r, r),
        flags=kv.KVSWAP_SCORE_SOFTMAX if c["softmax"] else 0)


def _compact_cache(K, proj, per_head, out):
    """K_lr = Flatten(K) A in fp32, one rounding into the stored type."""
    for b in range(K.shape[0]):
        x = torch.bmm(K[b].float(), proj)                       # [H_kv, N, r]
        out[b] = (x if per_head else x.sum(0, keepdim=True)).to(out.dtype)


def _plant(K, q, share, gen):
    """Keys of cosine 0.8 with the mean query of their KV head, at the same positions in every head."""
    B, H, N, d = K.shape
    n = max(1, int(share * N))
    pos = torch.randperm(N, generator=gen, device=K.device)[:n]
    qh = q.float().view(B, H, -1, d).mean(2)
    qh = qh / qh.norm(dim=-1, keepdim=True)
    noise = torch.randn((B, H, n, d), generator=gen, device=K.device)
    noise -= (noise * qh[:, :, None]).sum(-1, keepdim=True) * qh[:, :, None]
    noise /= noise.norm(dim=-1, keepdim=True)
    K[:, :, pos] = (d ** 0.5 * (0.8 * qh[:, :, None] + 0.6 * noise)).to(K.dtype)


def prepare(case, seed):
    c = dict(case)
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    kind, L, B, N, H, d, r = c["kind"], c["layers"], c["batch"], c["n_ctx"], c["kv_heads"], c["head_dim"], c["rank"]
    hm = H if c["per_head"] else 1
    T = c["steps"]
    rows = N + (T if kind == "grow" else 0)
    tkv, tm = _TORCH[c["kv"]], _TORCH[c["meta"]]
    s = {"case": c, "shape": _shape(c, N, rows)}

    def normal(*size, dtype=tkv):
        return torch.empty(size, dtype=dtype, device=dev).normal_(generator=gen)

    # one orthonormal adapter over the flattened keys, or one per KV head
    if c["per_head"]:
        s["proj"] = [torch.linalg.qr(normal(H, d, r, dtype=torch.float32))[0].contiguous() for _ in range(L)]
    else:
        s["proj"] = [torch.linalg.qr(normal(H * d, r, dtype=torch.float32))[0].reshape(H, d, r).contiguous()
                     for _ in range(L)]
    if kind == "prefill":
        s["K"] = [normal(B, H, N, d) for _ in range(L)]
        s["meta"] = [torch.empty((B, hm, N, r), dtype=tm, device=dev) for _ in range(L)]
        s["ws"] = rt.alloc_workspace(s["shape"])
        return s

    # queries of consecutive tokens are correlated: a random walk with unit variance
    q = [normal(L, B, c["q_heads"], d, dtype=torch.float32)]
    for _ in range(T - 1):
        q.append(0.95 * q[-1] + (1 - 0.95 ** 2) ** 0.5 * normal(L, B, c["q_heads"], d, dtype=torch.float32))
    s["q"] = [x.to(tkv) for x in q]
    K, V, meta = [], [], []
    for l in range(L):
        k, v = normal(B, H, rows, d), normal(B, H, rows, d)
        if c["heavy"]:
            _plant(k, s["q"][0][l], c["heavy"], gen)
        m = torch.empty((B, hm, rows, r), dtype=tm, device=dev)
        _compact_cache(k, s["proj"][l], c["per_head"], m)
        if kind == "tiered":                                     # the store is in host memory
            k, v = (x.to("cpu").pin_memory() for x in (k, v))
        K.append(k), V.append(v), meta.append(m)
    s["meta"] = meta
    S = s["shape"].n_scopes
    outs = T if kind in ("grow", "tiered") else 1
    s["out"] = [torch.empty((L, B, c["q_heads"], d), dtype=torch.float32, device=dev) for _ in range(outs)]
    s["lse"] = [torch.empty((L, B, c["q_heads"]), dtype=torch.float32, device=dev) for _ in range(outs)]
    s["idx"] = [torch.empty((L, B, S, c["top_k"]), dtype=torch.int32, device=dev) for _ in range(outs)]
    s["nsel"] = [torch.empty((L, B, S), dtype=torch.int32, device=dev) for _ in range(outs)]
    if kind == "tiered":
        G, slots, groups = c["group"], 2 * c["top_k"], N // c["group"]
        s["slots"], s["groups"] = slots, groups
        kr = [torch.empty((B, H, (slots + 1) * G, d), dtype=tkv, device=dev) for _ in range(L)]
        vr = [torch.empty_like(x) for x in kr]
        for l in range(L):                                       # the rolling buffer lives in the reuse store
            kr[l][:, :, slots * G:slots * G + N % G] = K[l][:, :, groups * G:].to(dev)
            vr[l][:, :, slots * G:slots * G + N % G] = V[l][:, :, groups * G:].to(dev)
        n = kv.kvswap_reuse_state_bytes(s["shape"], slots, groups)
        s["state"] = [torch.empty(n // 4, dtype=torch.int32, device=dev) for _ in range(L)]
        s["slot_idx"], miss_group, miss_slot = (torch.empty_like(s["idx"][0]) for _ in range(3))
        s["n_miss"] = torch.empty_like(s["nsel"][0])
        s["tiers"] = kv.make_tiers(slots, groups, K, V, kr, vr, s["state"], s["slot_idx"], miss_group, miss_slot,
                                   s["n_miss"])
        s["layers"] = kv.make_layers(kr, vr, meta, s["proj"], 0)
        s["ws"] = torch.empty(kv.kvswap_tiered_workspace_bytes(s["shape"], slots), dtype=torch.uint8, device=dev)
        kv.kvswap_workspace_init(s["ws"])
        return s
    s["K"], s["V"] = K, V
    s["layers"] = kv.make_layers(K, V, meta, s["proj"], 1)
    s["shapes"] = [_shape(c, N + t, rows) for t in range(rows - N + 1)]
    s["ws"] = rt.alloc_workspace(s["shapes"][-1])
    if kind == "grow":
        s["k_new"], s["v_new"] = normal(T, L, B, H, d), normal(T, L, B, H, d)
    if kind == "host":
        s["q_host"] = s["q"][0].cpu().pin_memory()
        s["out_host"] = torch.empty(s["out"][0].shape, dtype=torch.float32).pin_memory()
    return s


def run(s):
    c, kind = s["case"], s["case"]["kind"]
    if kind == "prefill":
        for l in range(c["layers"]):
            kv.kvswap_project_keys(s["shape"], s["K"][l], s["proj"][l], s["meta"][l], 0, c["n_ctx"], s["ws"])
        return s["meta"]
    if kind == "calls":
        q, out, lse, idx, nsel = s["q"][0], s["out"][0], s["lse"][0], s["idx"][0], s["nsel"][0]
        for l in range(c["layers"]):
            kv.kvswap_score_select(s["shape"], q[l], s["proj"][l], s["meta"][l], idx[l], nsel[l], None, s["ws"])
            kv.kvswap_sparse_decode(s["shape"], q[l], s["K"][l], s["V"][l], idx[l], nsel[l], out[l], lse[l], s["ws"])
    elif kind == "step":
        kv.kvswap_decode_step(s["shape"], s["layers"], s["q"][0], s["out"][0], s["lse"][0], s["idx"][0], s["nsel"][0],
                              s["ws"])
    elif kind == "host":
        kv.kvswap_decode_step_host(s["shape"], s["layers"], s["q_host"], s["out_host"], s["q"][0], s["out"][0],
                                   s["idx"][0], s["nsel"][0], s["ws"])
        return {"out": s["out_host"], "idx": s["idx"], "nsel": s["nsel"]}
    elif kind == "grow":
        for t in range(c["steps"]):
            kv.kvswap_append_step(s["shapes"][t], s["layers"], s["k_new"][t], s["v_new"][t])
            kv.kvswap_decode_step(s["shapes"][t + 1], s["layers"], s["q"][t], s["out"][t], s["lse"][t], s["idx"][t],
                                  s["nsel"][t], s["ws"])
        # the written part of the stores: the appended rows, and the compact cache's rows of the completed group
        n, g0 = c["n_ctx"], c["n_ctx"] // c["group"] * c["group"]
        return {"out": s["out"], "lse": s["lse"], "idx": s["idx"], "nsel": s["nsel"],
                "k": [torch.stack([x[:, :, n:] for x in s["K"]]), torch.stack([x[:, :, n:] for x in s["V"]])],
                "meta": torch.stack([x[:, :, g0:g0 + c["group"]] for x in s["meta"]])}
    elif kind == "tiered":
        for l in range(c["layers"]):
            kv.kvswap_reuse_init(s["shape"], s["slots"], s["groups"], s["state"][l])
        for t in range(c["steps"]):
            kv.kvswap_decode_step_tiered(s["shape"], s["layers"], s["tiers"], s["q"][t], s["out"][t], s["lse"][t],
                                         s["idx"][t], s["nsel"][t], s["ws"])
        return {"out": s["out"], "lse": s["lse"], "idx": s["idx"], "nsel": s["nsel"], "slot": s["slot_idx"],
                "miss": s["n_miss"]}
    return {"out": s["out"], "lse": s["lse"], "idx": s["idx"], "nsel": s["nsel"]}


def work(c):
    L, B, N, H, d, r = c["layers"], c["batch"], c["n_ctx"], c["kv_heads"], c["head_dim"], c["rank"]
    hm = H if c["per_head"] else 1
    ekv, em = _SIZE[c["kv"]], _SIZE[c["meta"]]
    adapter = 4.0 * H * d * r
    if c["kind"] == "prefill":
        return {"bytes": L * (B * H * N * d * ekv + B * hm * N * r * em + adapter), "flops": L * 2.0 * B * N * H * d * r}
    G = c["group"]
    groups = N // G
    S = 1 if c["all_heads"] else H
    chosen = min(c["top_k"], groups)
    tokens = chosen * G + N % G
    scores = c["q_heads"] if c["softmax"] else H if c["per_head"] else S
    small = B * c["q_heads"] * d * (ekv + 4.0) + 4.0 * B * c["q_heads"] + 4.0 * B * S * (c["top_k"] + 1)
    step_bytes = B * hm * groups * G * r * em + adapter + 2.0 * B * H * tokens * d * ekv + small
    step_flops = 2.0 * B * c["q_heads"] * d * r + 2.0 * B * scores * N * r + 4.0 * B * c["q_heads"] * tokens * d
    if c["kind"] == "tiered":
        # what is fetched over the link (all of the first step's groups, about a quarter later) is read and written
        step_bytes += 2.0 * 2.0 * B * H * chosen * G * d * ekv * (1 + 0.25 * (c["steps"] - 1)) / c["steps"]
    if c["kind"] == "grow":
        step_bytes += 4.0 * B * H * d * ekv + B * (H * d * ekv + hm * r * em)
    return {"bytes": float(L * c["steps"] * step_bytes), "flops": float(L * c["steps"] * step_flops)}


# What storing the compact cache gives: measured against float64 sums rounded once, rel 1.8e-5 and one unit in
# the last place at 0.3 % of the fp16 values, rel 4.1e-7 and 3.2e-6 at most for fp32, and for the 8-bit type
# (steps of 1/8) the same sums falling on the other side of a rounding boundary; each times four.
_CACHE = {"f16": (7e-5, 4e-3), "f32": (1.6e-6, 1.3e-5), "e4m3": (5e-3, 0.5)}


def tolerance(c):
    rel, most = _CACHE[c["meta"]]
    if c["kind"] == "prefill":
        return {"rel": rel, "max": most}
    # Attention against float64 over the same selection, measured over these cases: rel up to 1.9e-6, 1.3e-5 at
    # most (16-bit K/V with fp32 sums); four times that.
    out = {"rel": 8e-6, "max": 6e-5, "differ": 0.0}
    if c["kind"] == "grow":
        out = {"rel": max(rel, out["rel"]), "max": max(most, out["max"]), "differ": 0.0}
    # Where many lists are selected, one may end in two groups whose scores agree to fp32 rounding: another order
    # of the sums may then keep the other one.  One such list: its later entries move up or down, and its heads
    # attend G other tokens.
    lists = c["layers"] * c["steps"] * c["batch"] * (1 if c["all_heads"] else c["kv_heads"])
    if lists >= 256:
        groups = c["n_ctx"] // c["group"]
        attended = min(c["top_k"], groups) * c["group"] + c["n_ctx"] % c["group"]
        out = {"rel": max(out["rel"], min(0.01, 1.5 * math.sqrt(2.0 * c["group"] / attended / lists))), "max": 0.9,
               "differ": 1.0 / lists}
    return out
