"""Decode steps whose gather runs beside the next layer's select: bit for bit the per-layer calls, whose selection comes from
another kernel (topk_parts_kernel), over the shapes the gather takes and over scores that are awkward to select from."""
import dataclasses

import pytest
import torch

from paper_2511_11907_b200 import binding as kv
from paper_2511_11907_b200 import device_workload as DW
from paper_2511_11907_b200 import runtime as rt
from paper_2511_11907_b200 import workloads as W
from launches import launched
from test_gpu_decode_step import _run_case, _step_buffers

pytestmark = pytest.mark.gpu

KV, ALL = W.SCOPE_KV_HEAD, W.SCOPE_ALL_HEADS


def _wl(**kw):
    base = dict(layers=3, batch=4, n_ctx=20011, top_k=400, calib_rows=1024)
    base.update(kw)
    return dataclasses.replace(W.CONFIGS[5], name="long", walk_steps=1, **base)


def _route(wl, meta_heads, scope, flags=0, lookahead=0):
    dw = DW.build(wl, 1 if meta_heads == "joint" else wl.n_kv_heads, scope, walk_steps=1, reserve_bytes=1 << 30)
    shape = dw.shape.with_flags(flags)
    ws = rt.alloc_workspace(shape)
    for m in dw.meta:
        m.zero_()
    out, lse, idx, nsel = _step_buffers(dw)
    layers = dw.layer_tables(lookahead)
    return launched(lambda: kv.kvswap_decode_step(shape, layers, dw.q_walk[0], out, lse, idx, nsel, ws))


# A gather is long from 47 MiB on, and from 5000 bytes per group of the context; and only where the select has room beside the
# scorer (select_beside_supported).  Head counts that leave one to eight query heads per row, heads of 64 channels, groups whose
# rows do not fill blocks of eight, open groups of several lengths, one to four layers, lists of whole and of broken CTAs, both
# stored types and ranks.
@pytest.mark.parametrize("kw", [
    dict(),
    dict(layers=1),
    dict(layers=2, n_ctx=20015),
    dict(layers=4, n_q_heads=24, batch=3, top_k=300, group_size=16, n_ctx=33000 + 15),
    dict(kv_dtype=W.F16, q_dtype=W.F16, n_q_heads=64, n_ctx=20008),
    dict(n_q_heads=8, n_ctx=20009),
    dict(n_q_heads=88, n_ctx=20010),
    dict(head_dim=64, top_k=800),
    dict(group_size=4, top_k=800, n_ctx=20002),
    dict(group_size=2, batch=5, top_k=1400, n_ctx=20003),
    dict(group_size=32, top_k=100, n_ctx=20012),
    dict(rank=16, batch=5),
    dict(meta_dtype=W.E4M3, batch=5),
    dict(batch=8, top_k=200),
])
def test_step_with_a_long_gather(kw):
    wl = _wl(**kw)
    names = set(_route(wl, "joint", KV))
    assert "sparse_decode_long_kernel" in names and "sparse_decode_splitk_kernel" not in names
    assert ("select_beside_kernel" in names) == (wl.layers > 1)
    _run_case(wl, "joint", KV)


# Gathers as long whose select has no such room, or nothing to gain: the schedule of shorter ones
@pytest.mark.parametrize("meta_heads,scope,kw", [
    ("joint", KV, dict(rank=64, batch=5)),
    ("joint", KV, dict(rank=128)),
    ("joint", KV, dict(meta_dtype=W.F32)),
    ("joint", KV, dict(group_size=12, top_k=270)),
    ("joint", KV, dict(group_size=1, top_k=3200, n_ctx=10011)),
    ("joint", KV, dict(top_k=1900)),
    ("joint", KV, dict(batch=16, n_ctx=20003, top_k=200)),
    ("joint", KV, dict(batch=8, n_ctx=16005, top_k=200)),
    ("per_head", KV, dict(batch=3, top_k=550)),
    ("joint", ALL, dict(batch=6)),
    ("per_head", ALL, dict(batch=3, n_q_heads=32, n_kv_heads=16, top_k=300)),
])
def test_step_with_a_gather_as_long_and_no_room_beside_it(meta_heads, scope, kw):
    wl = _wl(**kw)
    names = set(_route(wl, meta_heads, scope))
    assert "sparse_decode_splitk_kernel" in names and not names & {"sparse_decode_long_kernel", "select_beside_kernel"}
    _run_case(wl, meta_heads, scope)


def test_step_with_a_gather_as_long_behind_the_softmax_scorer():
    wl = _wl()
    assert "sparse_decode_long_kernel" not in _route(wl, "joint", KV, kv.KVSWAP_SCORE_SOFTMAX)
    _run_case(wl, "joint", KV, flags=kv.KVSWAP_SCORE_SOFTMAX)


# four query heads per list, and one: eleven lists per KV head, whose partials have one buffer
@pytest.mark.parametrize("q_heads", [32, 88])
@pytest.mark.parametrize("lookahead", [0, 1, 2])
def test_lookahead_of_one_layer_merges_a_layer_before_the_next_but_one_is_scored(q_heads, lookahead):
    """... and another bound beside that, or ahead of the last gather where there is one buffer of partials."""
    wl = _wl(layers=4, n_q_heads=q_heads)
    predict, attend = ["score_stream_kernel", "select_beside_kernel"], ["sparse_decode_long_kernel"]
    if lookahead == 1:
        want = 3 * (predict + attend + ["combine_kernel"]) + attend + ["combine_kernel"]
    else:
        want = 3 * (predict + attend) + ["combine_kernel"] * (q_heads == 88) + attend + ["combine_kernel"]
    assert _route(wl, "joint", KV, lookahead=lookahead) == ["score_stream_kernel", "topk_parts_kernel"] + want
    _run_case(wl, "joint", KV, lookahead)


@pytest.mark.parametrize("layer", [0, 1, 2, 3])
@pytest.mark.parametrize("lookahead", [0, 1])
def test_probed_step_with_a_long_gather(layer, lookahead):
    wl = _wl(layers=4)
    dw = DW.build(wl, 1, KV, walk_steps=1, reserve_bytes=1 << 30)
    shape, q, ws = dw.shape, dw.q_walk[0], rt.alloc_workspace(dw.shape)
    for l in range(wl.layers):
        kv.kvswap_project_keys(shape, dw.K[l], dw.proj[l], dw.meta[l], 0, wl.n_ctx, ws)
    layers, plain, probed = dw.layer_tables(lookahead), _step_buffers(dw), _step_buffers(dw)
    kv.kvswap_decode_step(shape, layers, q, *plain, ws)
    events = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
    for e in events:
        e.record()                                           # (created on first use)
    kv.kvswap_decode_step(shape, layers, q, *probed, ws, kv.make_probe(layer, *events))
    torch.cuda.synchronize()
    assert events[0].elapsed_time(events[1]) > 0 and events[1].elapsed_time(events[2]) > 0
    assert all(torch.equal(a, b) for a, b in zip(plain, probed))
    assert kv.kvswap_read_device_status(ws) == 0


# Scores that the sampled bound, the list or its intervals do not fit: all equal, a few values (long ties at the threshold),
# rising with the position, a run of large ones, infinities; few, many and most groups selected.
@pytest.mark.parametrize("n_ctx,top_k", [(20011, 400), (70003, 512), (20011, 1500)])
@pytest.mark.parametrize("kind", ["equal", "few", "ramp", "run", "inf"])
def test_select_beside_on_awkward_scores(kind, n_ctx, top_k):
    wl = _wl(layers=2, n_ctx=n_ctx, top_k=top_k, batch=4 if n_ctx < 50000 else 3)
    dw = DW.build(wl, 1, KV, walk_steps=1, reserve_bytes=1 << 30)
    shape, q, ws = dw.shape, dw.q_walk[0], rt.alloc_workspace(dw.shape)
    for l in range(wl.layers):
        kv.kvswap_project_keys(shape, dw.K[l], dw.proj[l], dw.meta[l], 0, wl.n_ctx, ws)
        m = dw.meta[l]
        pos = torch.arange(wl.n_ctx, device="cuda", dtype=torch.float32)[None, None, :, None]
        if kind == "equal":
            m.copy_(m[:, :, :1].clone().expand_as(m))
        elif kind == "few":
            m.copy_(m[:, :, :1].clone().float() * (1 + (pos * 0.618).frac().mul(5).floor()))
        elif kind == "ramp":
            m.copy_(m[:, :, :1].clone().float() * (1 + pos / wl.n_ctx))
        elif kind == "run":
            m[:, :, 4096:4096 + 8 * top_k] *= 30
        else:
            m[:, :, ::97] = float("inf")
    out_a, lse_a, idx_a, nsel_a = _step_buffers(dw)
    for l in range(wl.layers):
        kv.kvswap_score_select(shape, q[l], dw.proj[l], dw.meta[l], idx_a[l], nsel_a[l], None, ws)
        kv.kvswap_sparse_decode(shape, q[l], dw.K[l], dw.V[l], idx_a[l], nsel_a[l], out_a[l], lse_a[l], ws)
    out_b, lse_b, idx_b, nsel_b = _step_buffers(dw)
    layers = dw.layer_tables()
    assert "select_beside_kernel" in launched(lambda: kv.kvswap_decode_step(shape, layers, q, out_b, lse_b, idx_b, nsel_b, ws))
    for buf in (out_b, lse_b, idx_b, nsel_b):
        buf.fill_(-7)
    kv.kvswap_decode_step(shape, layers, q, out_b, lse_b, idx_b, nsel_b, ws)
    torch.cuda.synchronize()
    assert kv.kvswap_read_device_status(ws) == 0
    assert torch.equal(nsel_a, nsel_b) and torch.equal(idx_a, idx_b)
    assert torch.equal(out_a, out_b) and torch.equal(lse_a, lse_b)


def _near_rows(kind, problems, groups, top_k, gen):
    """Rows of group scores [problems, groups] whose threshold lies among many equal or nearly equal scores."""
    def normal(*size):
        return torch.randn(size, generator=gen, dtype=torch.float64)

    def ulps(base, steps):
        return (torch.tensor(base, dtype=torch.float32).view(torch.int32) + steps.int()).view(torch.float32)

    if kind == "offset":                        # a common offset and a few outliers
        x = 1000 + (0.3 if groups > 8192 else 0.1) * normal(problems, groups)
        x[:, :20] += 5
    elif kind.startswith("ties"):               # so many equal scores across the threshold, among others spread widely
        n = int(kind[4:])
        x = (30 * normal(problems, groups)).float().sort(descending=True).values
        x[:, top_k - n // 2:top_k - n // 2 + n] = x[:, top_k:top_k + 1].clone()
    elif kind == "plateau":                     # more equal scores than the list has room for
        x = normal(problems, groups).float().sort(descending=True).values
        x[:, top_k - 100:top_k + 3000] = x[:, top_k:top_k + 1].clone()
    elif kind == "consecutive":                 # a hundred floats in a row, each many times
        x = ulps(1.0, torch.randint(0, 100, (problems, groups), generator=gen))
    else:                                       # "near": ties, with others up to 800 units in the last place above them
        x = torch.rand((problems, groups), generator=gen) * 0.5
        x[:, :top_k // 2] = 1.0
        x[:, top_k // 2:top_k + top_k // 2] = ulps(1.0, torch.randint(1, 800, (problems, top_k), generator=gen))
        x[:, top_k:top_k + top_k // 2] = 1.0
    x = x.float()
    return x.gather(1, torch.rand(x.shape, generator=gen).argsort(1))


# 24 to 40 rows per case, of whole and sampled lists; the selection is compared with the per-layer calls' and with a stable
# sort of the scores in float64.
@pytest.mark.parametrize("kind", ["offset", "ties33", "ties48", "ties128", "plateau", "consecutive", "near"])
@pytest.mark.parametrize("n_ctx,batch,top_k",
                         [(131072 + 3, 3, 1024), (32768 + 5, 5, 400), (16000 + 5, 5, 400), (32768 + 5, 5, 1400)])
def test_select_beside_among_nearly_equal_scores(kind, n_ctx, batch, top_k):
    wl = _wl(layers=2, n_ctx=n_ctx, top_k=top_k, batch=batch)
    groups, S = n_ctx // 8, wl.n_kv_heads
    if kind == "plateau" and groups < top_k + 3000:
        pytest.skip("no room for the plateau")
    dw = DW.build(wl, 1, KV, walk_steps=1, reserve_bytes=1 << 30)
    shape, q, ws = dw.shape, dw.q_walk[0], rt.alloc_workspace(dw.shape)
    # Columns s, s + 8 and s + 16 of the compact cache hold the scores of scope s in three fp16 pieces, 2^11 apart: its low-rank
    # query has 1, 2^-11 and 2^-22 there.
    q[..., 0] = 1 / wl.rho
    gen = torch.Generator().manual_seed(n_ctx + top_k)
    for l in range(wl.layers):
        dw.proj[l].zero_()
        dw.meta[l].zero_()
        x = _near_rows(kind, wl.batch * S, groups, top_k, gen).view(wl.batch, S, groups).cuda()
        for k in range(3):
            dw.proj[l][torch.arange(S), 0, torch.arange(S) + S * k] = 2.0 ** (-11 * k)
            piece = (x * 2.0 ** (11 * k)).half()
            x = x - piece.float() * 2.0 ** (-11 * k)
            dw.meta[l][:, 0, :groups * 8, S * k:S * (k + 1)] = piece.transpose(1, 2).repeat_interleave(8, 1)
    step = _step_buffers(dw)
    layers = dw.layer_tables()
    call = lambda: kv.kvswap_decode_step(shape, layers, q, *step, ws)
    names = launched(call)
    assert "select_beside_kernel" in names
    for buf in step:
        buf.fill_(-7)
    call()
    out, lse, idx, nsel = _step_buffers(dw)
    scores = torch.empty((wl.batch, S, groups), device="cuda")
    for l in range(wl.layers):
        kv.kvswap_score_select(shape, q[l], dw.proj[l], dw.meta[l], idx[l], nsel[l], scores, ws)
        kv.kvswap_sparse_decode(shape, q[l], dw.K[l], dw.V[l], idx[l], nsel[l], out[l], lse[l], ws)
        want = scores.double().sort(dim=-1, descending=True, stable=True).indices[..., :top_k].sort(-1).values
        assert torch.equal(idx[l].long(), want) and torch.equal(step[2][l].long(), want)
    assert kv.kvswap_read_device_status(ws) == 0
    assert torch.equal(step[3], nsel) and torch.equal(step[0], out) and torch.equal(step[1], lse)
