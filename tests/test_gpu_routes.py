"""Decode steps and calls on every schedule the library chooses from, each checked to have taken it: a step gives
exactly what the per-layer calls give, and a predictor what the oracle gives, on both sides of the lines between them."""
import dataclasses

import pytest
import torch

from paper_2511_11907_b200 import binding as kv
from paper_2511_11907_b200 import device_workload as DW
from paper_2511_11907_b200 import runtime as rt
from paper_2511_11907_b200 import workloads as W
from launches import launched
from test_gpu_decode_step import _run_case
from test_gpu_parity import run_layer_parity

pytestmark = pytest.mark.gpu

KV, ALL = W.SCOPE_KV_HEAD, W.SCOPE_ALL_HEADS

# kernels of a step of several layers
CHAIN = {"score_stream_kernel", "topk_parts_kernel", "sparse_decode_splitk_kernel", "combine_select_kernel", "combine_kernel"}
CLUSTERS = {"score_select_cluster_kernel", "sparse_decode_splitk_kernel"}      # the splits merge in clusters
BESIDE = CLUSTERS | {"combine_kernel"}


def _wl(**kw):
    base = dict(layers=4, batch=2, n_ctx=20011, top_k=40, calib_rows=1024)
    base.update(kw)
    if base.get("kv_dtype") == W.F32:
        base.update(meta_dtype=W.F32, q_dtype=W.F32)
    return dataclasses.replace(W.CONFIGS[5], name="routes", walk_steps=1, **base)


def _step_route(wl, meta_heads, scope, flags=0):
    dw = DW.build(wl, meta_heads, scope, walk_steps=1, reserve_bytes=1 << 30)
    shape = dw.shape.with_flags(flags)
    ws = rt.alloc_workspace(shape)
    for m in dw.meta:
        m.zero_()
    out = torch.empty((wl.layers, wl.batch, wl.n_q_heads, wl.head_dim), device="cuda")
    idx = torch.empty((wl.layers, wl.batch, shape.n_scopes, wl.top_k), dtype=torch.int32, device="cuda")
    nsel = torch.empty((wl.layers, wl.batch, shape.n_scopes), dtype=torch.int32, device="cuda")
    layers = dw.layer_tables()
    return launched(lambda: kv.kvswap_decode_step(shape, layers, dw.q_walk[0], out, None, idx, nsel, ws))


# The merged combine + TopK launch, which also forms the queries of the layer after next: 14 rows of partials per CTA at
# d = 64, every rank and type it takes, KV heads of per-head metadata eight at a time, several terms per score, lists
# of 2, 4 and 8 parts, more sequences than the launch of clusters takes.
@pytest.mark.parametrize("meta_heads,scope,kw", [
    ("joint", KV, dict(head_dim=64, batch=3, n_ctx=20019)),
    ("per_head", KV, dict(head_dim=64, n_ctx=18003)),
    ("joint", KV, dict(rank=16, batch=3, n_ctx=34003)),
    ("per_head", KV, dict(rank=16, head_dim=64, n_ctx=20003)),
    ("joint", KV, dict(rank=64, batch=3, n_ctx=9005)),
    ("joint", ALL, dict(rank=64, n_ctx=20005)),
    ("joint", KV, dict(kv_dtype=W.F32, batch=3, n_ctx=9001)),
    ("per_head", KV, dict(kv_dtype=W.F32, rank=16, n_ctx=9001)),
    ("joint", KV, dict(kv_dtype=W.F32, rank=64, group_size=4, batch=3, n_ctx=5001)),
    ("per_head", KV, dict(n_q_heads=24, n_kv_heads=12, n_ctx=9007)),
    ("joint", KV, dict(n_q_heads=24, n_kv_heads=12, n_ctx=17007)),
    ("per_head", ALL, dict(n_ctx=4099)),
    ("per_head", ALL, dict(head_dim=64, rank=16, n_ctx=9003)),
    ("joint", KV, dict(batch=40, n_ctx=1003)),
    ("joint", KV, dict(batch=1, n_ctx=50003)),                                 # 2 parts
    ("joint", KV, dict(batch=1, group_size=4, n_ctx=50003)),                   # 4 parts
    ("joint", KV, dict(batch=1, group_size=4, n_ctx=70003)),                   # 8 parts
    ("per_head", KV, dict(batch=1, group_size=4, head_dim=64, n_ctx=70003)),
])
def test_step_with_the_merged_combine_and_select(meta_heads, scope, kw):
    wl = _wl(**kw)
    assert set(_step_route(wl, 1 if meta_heads == "joint" else wl.n_kv_heads, scope)) == CHAIN
    _run_case(wl, meta_heads, scope)


@pytest.mark.parametrize("meta_heads,scope,kw", [
    ("joint", KV, dict(n_ctx=4101)),
    ("joint", KV, dict(head_dim=64, rank=16, n_q_heads=16, n_kv_heads=4, n_ctx=40001)),
    ("per_head", ALL, dict(n_ctx=4099)),
    ("per_head", KV, dict(kv_dtype=W.F32, rank=64, n_ctx=3001)),
])
def test_step_with_the_softmax_scorer(meta_heads, scope, kw):
    wl = _wl(**kw)
    route = (CHAIN - {"score_stream_kernel"}) | {"lowrank_query_heads_kernel", "softmax_tc_stats_kernel", "softmax_tc_pool_kernel"}
    assert set(_step_route(wl, 1 if meta_heads == "joint" else wl.n_kv_heads, scope, kv.KVSWAP_SCORE_SOFTMAX)) == route
    _run_case(wl, meta_heads, scope, flags=kv.KVSWAP_SCORE_SOFTMAX)


# Predictor and attention side by side: lists of one split, of up to 8 and of up to 16 (more than a portable cluster)
# merged in clusters, and longer ones by a combine kernel.
@pytest.mark.parametrize("meta_heads,kw,route", [
    ("joint", dict(batch=1, n_ctx=2048, top_k=8), CLUSTERS),                   # 1 split
    ("joint", dict(batch=1, n_ctx=4100, top_k=40), CLUSTERS),                  # 2
    ("per_head", dict(batch=1, n_ctx=4100, top_k=60), CLUSTERS),               # 3
    ("joint", dict(batch=2, n_ctx=4100, top_k=128), CLUSTERS),                 # 8
    ("joint", dict(batch=1, n_ctx=16384, top_k=150), CLUSTERS),                # 9
    ("joint", dict(batch=1, n_ctx=16384, top_k=256), CLUSTERS),                # 16
    ("joint", dict(batch=1, n_ctx=4096, top_k=256, kv_dtype=W.F32, head_dim=64), CLUSTERS),
    ("joint", dict(batch=1, n_ctx=4096, top_k=256, kv_dtype=W.F32), BESIDE),   # 16, but one CTA per SM
    ("joint", dict(batch=1, n_ctx=4096, top_k=256, kv_dtype=W.F32, n_q_heads=16, n_kv_heads=4), CLUSTERS),     # 16 SMs per list
    ("joint", dict(batch=1, n_ctx=4096, top_k=80, kv_dtype=W.F32), CLUSTERS),
    ("joint", dict(batch=1, n_ctx=16384, top_k=290), BESIDE),                  # 18
    ("joint", dict(batch=4, n_ctx=8003, top_k=400), BESIDE),
    ("per_head", dict(batch=1, n_ctx=16384, top_k=400), BESIDE),
])
def test_step_side_by_side(meta_heads, kw, route):
    wl = _wl(**kw)
    names = _step_route(wl, 1 if meta_heads == "joint" else wl.n_kv_heads, KV)
    assert set(names) == route
    assert len(names) == wl.layers * len(route)
    _run_case(wl, meta_heads, KV)


@pytest.mark.parametrize("batch,n_ctx,top_k,combine", [(1, 2048, 8, False), (2, 4100, 128, False), (1, 16384, 150, True), (1, 16384, 256, True)])
def test_attention_on_its_own(batch, n_ctx, top_k, combine):
    """A call merges up to 8 splits in clusters, where the step does, and more with a combine kernel."""
    wl = _wl(batch=batch, n_ctx=n_ctx, top_k=top_k)
    shape = rt.shape_for(wl, 1, KV)
    K = torch.zeros((batch, 8, n_ctx, 128), dtype=torch.bfloat16, device="cuda")
    q = torch.zeros((batch, 32, 128), dtype=torch.bfloat16, device="cuda")
    idx, nsel = rt.alloc_selection(shape)
    idx.copy_(torch.arange(top_k, dtype=torch.int32, device="cuda").expand_as(idx))
    nsel.fill_(top_k)
    (out, lse), ws = rt.alloc_output(shape), rt.alloc_workspace(shape)
    want = ["sparse_decode_splitk_kernel"] + (["combine_kernel"] if combine else [])
    assert launched(lambda: kv.kvswap_sparse_decode(shape, q, K, K, idx, nsel, out, lse, ws)) == want
    assert launched(lambda: kv.kvswap_sparse_decode_static(shape, q, K, K, idx, nsel, out, lse)) == want


# The lines between the launch of clusters and the streaming scorer, on both sides: 6144 groups, two tiles per warp.
@pytest.mark.parametrize("kw,name", [
    (dict(group_size=1, n_ctx=6144), "score_select_cluster_kernel"),
    (dict(group_size=1, n_ctx=6145), "score_stream_kernel"),
    (dict(group_size=1, n_ctx=6144, rank=64), "score_select_cluster_kernel"),
    (dict(group_size=3, n_ctx=3 * 6144 + 2), "score_select_cluster_kernel"),
    (dict(group_size=3, n_ctx=3 * 6145), "score_stream_kernel"),
    (dict(group_size=4, n_ctx=4 * 4112, n_kv_heads=2, n_q_heads=4), "score_select_cluster_kernel"),      # two tiles per warp
    (dict(group_size=8, n_ctx=8 * 4096), "score_select_cluster_kernel"),
    (dict(group_size=8, n_ctx=8 * 4097), "score_stream_kernel"),                                         # three
    (dict(group_size=1, n_ctx=5000, batch=20, rank=64, n_q_heads=8), "score_select_cluster_kernel"),     # two CTAs per SM
    (dict(group_size=1, n_ctx=6000, batch=20, rank=64, n_q_heads=8), "score_stream_kernel"),             # keys leave room for one
])
def test_predictor_on_both_sides_of_its_lines(kw, name):
    args = dict(layers=1, batch=1, n_q_heads=16, n_kv_heads=8, head_dim=64, top_k=70, calib_rows=600, heavy_frac=0.0)
    args.update(kw)
    wl = dataclasses.replace(W.CONFIGS[5], name="lines", walk_steps=1, **args)
    dl = run_layer_parity(W.make_layer(wl, 0, 1), KV)
    names = launched(lambda: kv.kvswap_score_select(dl.shape, dl.q, dl.proj, dl.meta, dl.idx, dl.nsel, None, dl.ws))
    assert names[0] == name
