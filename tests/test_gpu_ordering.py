"""A call without KVSWAP_INPUTS_SETTLED may be enqueued right behind the kernel that writes any of its inputs.

The producer of these tests is kvswap_sparse_decode, whose kernels let their successor in the stream start while they
still run: its output buffer is the adapter, the metadata or the queries of the call behind it.  A call that read it
ahead of its dependency wait would see the buffer as it was before; results must be those for the finished buffer."""
import pytest
import torch

from paper_2511_11907_b200 import binding as kv
from paper_2511_11907_b200 import runtime as rt

pytestmark = pytest.mark.gpu


def _randn(*size, dtype=torch.float32, seed=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(size, device="cuda", generator=g).to(dtype)


class Producer:
    """An attention call of some 50 us over `rows` = B * 32 query rows of 128 channels, written into `target`."""

    def __init__(self, target):
        rows = target.numel() // 128
        assert rows % 32 == 0 and rows * 128 == target.numel()
        B = rows // 32
        tokens = max(1024, 65536 // B)                      # per KV head: a few hundred MB in all
        self.shape = kv.make_shape(batch=B, n_ctx=tokens, n_q_heads=32, n_kv_heads=8, head_dim=128, rank=32, meta_heads=1,
                                   group_size=8, top_k=tokens // 8, kv_dtype=kv.KVSWAP_BF16, meta_dtype=kv.KVSWAP_F16,
                                   q_dtype=kv.KVSWAP_BF16)
        self.K = _randn(B, 8, tokens, 128, dtype=torch.bfloat16, seed=1)
        self.V = _randn(B, 8, tokens, 128, dtype=torch.bfloat16, seed=2) * 64
        self.q = _randn(B, 32, 128, dtype=torch.bfloat16, seed=3)
        self.idx, self.nsel = rt.alloc_selection(self.shape)
        self.idx.copy_(torch.arange(tokens // 8, dtype=torch.int32, device="cuda").expand_as(self.idx))
        self.nsel.fill_(tokens // 8)
        self.ws = rt.alloc_workspace(self.shape)
        self.target = target

    def __call__(self):
        kv.kvswap_sparse_decode(self.shape, self.q, self.K, self.V, self.idx, self.nsel, self.target, None, self.ws)


def _check(target, consume, outputs):
    """`consume()` behind the producer gives what it gives once the producer has finished."""
    producer = Producer(target)
    producer()
    torch.cuda.synchronize()
    assert torch.isfinite(target).all() and target.std() > 0.1
    consume()
    torch.cuda.synchronize()
    want = [t.clone() for t in outputs]
    for _ in range(10):
        target.zero_()
        for t in outputs:
            t.zero_()
        torch.cuda.synchronize()
        torch.cuda._sleep(100000)                           # both calls are queued before the first one starts
        producer()
        consume()
        torch.cuda.synchronize()
        for got, ref in zip(outputs, want):
            assert torch.equal(got, ref)


def _select_args(N, G, H=8, d=128, r=32, top_k=64):
    shape = kv.make_shape(batch=1, n_ctx=N, n_q_heads=4 * H, n_kv_heads=H, head_dim=d, rank=r, meta_heads=1, group_size=G,
                          top_k=top_k, kv_dtype=kv.KVSWAP_F32, meta_dtype=kv.KVSWAP_F32, q_dtype=kv.KVSWAP_F32)
    return (shape, _randn(1, 4 * H, d, seed=4), _randn(H, d, r, seed=5) * 0.1, _randn(1, 1, N, r, seed=6),
            *rt.alloc_selection(shape), rt.alloc_workspace(shape))


# one launch of clusters; the streaming scorer with its TopK; a query kernel in front of the general scorer
ROUTES = [dict(N=2048, G=8), dict(N=32768, G=1, r=16), dict(N=4096, G=8, r=128)]


@pytest.mark.parametrize("what", ["adapter", "metadata", "query"])
@pytest.mark.parametrize("kw", ROUTES, ids=lambda kw: "N%d_G%d_r%d" % (kw["N"], kw["G"], kw.get("r", 32)))
@pytest.mark.parametrize("softmax", [False, True], ids=["logits", "softmax"])
def test_score_select_behind_the_producer_of_an_input(what, kw, softmax):
    shape, q, proj, meta, idx, nsel, ws = _select_args(**kw)
    if softmax:
        shape = shape.with_flags(kv.KVSWAP_SCORE_SOFTMAX)
        ws = rt.alloc_workspace(shape)
        proj, meta = proj * 0.1, meta * 0.1                 # logits of unit scale or so
    target = {"adapter": proj, "metadata": meta, "query": q}[what]
    if what == "query":                                      # 32 rows of 128 channels as they are
        assert target.numel() == 32 * 128
    _check(target, lambda: kv.kvswap_score_select(shape, q, proj, meta, idx, nsel, None, ws), [idx, nsel])


@pytest.mark.parametrize("N,per_head", [(1500, False), (700, True), (70000, False)])
@pytest.mark.parametrize("dtype", ["bf16", "f16", "f32"])
def test_project_keys_behind_the_producer_of_the_adapter(N, per_head, dtype):
    H, d, r = 8, 128, 32
    tag, t = {"bf16": (kv.KVSWAP_BF16, torch.bfloat16), "f16": (kv.KVSWAP_F16, torch.float16), "f32": (kv.KVSWAP_F32, torch.float32)}[dtype]
    hm = H if per_head else 1
    shape = kv.make_shape(batch=1, n_ctx=N, n_q_heads=4 * H, n_kv_heads=H, head_dim=d, rank=r, meta_heads=hm, group_size=8,
                          top_k=8, kv_dtype=tag, meta_dtype=kv.KVSWAP_F32, q_dtype=tag)
    K, proj = _randn(1, H, N, d, dtype=t, seed=7), _randn(H, d, r, seed=8)
    meta, ws = torch.empty((1, hm, N, r), device="cuda"), rt.alloc_workspace(shape)
    _check(proj, lambda: kv.kvswap_project_keys(shape, K, proj, meta, 0, N, ws), [meta])


# 2 layers of one sequence, 32 heads of 128 in fp32
@pytest.mark.parametrize("what", ["query", "adapter", "metadata"])
@pytest.mark.parametrize("N,G,r", [(2048, 8, 32), (32768, 1, 16), (4096, 8, 128)])
@pytest.mark.parametrize("kind", ["step", "tiered"])
def test_step_behind_the_producer_of_an_input(what, N, G, r, kind):
    L, H, d, M = 2, 8, 128, 64
    shape, _, _, _, _, _, _ = _select_args(N, G, r=r, top_k=M)
    q = _randn(L, 1, 4 * H, d, seed=9)
    proj = [_randn(H, d, r, seed=10 + l) * 0.1 for l in range(L)]
    meta = [_randn(1, 1, N, r, seed=20 + l) for l in range(L)]
    K, V = ([_randn(1, H, N, d, seed=30 + 10 * i + l) for l in range(L)] for i in range(2))
    out = torch.empty((L, 1, 4 * H, d), device="cuda")
    idx, nsel = torch.empty((L, 1, H, M), dtype=torch.int32, device="cuda"), torch.empty((L, 1, H), dtype=torch.int32, device="cuda")
    target = {"query": q, "adapter": proj[0], "metadata": meta[0]}[what]
    if kind == "step":
        layers, ws = kv.make_layers(K, V, meta, proj, 0), rt.alloc_workspace(shape)
        _check(target, lambda: kv.kvswap_decode_step(shape, layers, q, out, None, idx, nsel, ws), [out, idx, nsel])
        return
    slots, groups = 2 * M, N // G
    kr, vr = ([torch.zeros((1, H, (slots + 1) * G, d), device="cuda") for _ in range(L)] for _ in range(2))
    state = [torch.empty(kv.kvswap_reuse_state_bytes(shape, slots, groups) // 4, dtype=torch.int32, device="cuda") for _ in range(L)]
    lists, n_miss = [torch.empty_like(idx) for _ in range(3)], torch.empty_like(nsel)
    layers = kv.make_layers(kr, vr, meta, proj, 0)
    tiers = kv.make_tiers(slots, groups, K, V, kr, vr, state, *lists, n_miss)
    ws = torch.empty(kv.kvswap_tiered_workspace_bytes(shape, slots), dtype=torch.uint8, device="cuda")
    kv.kvswap_workspace_init(ws)
    for s in state:
        kv.kvswap_reuse_init(shape, slots, groups, s)
    _check(target, lambda: kv.kvswap_decode_step_tiered(shape, layers, tiers, q, out, None, idx, nsel, ws), [idx, nsel])


@pytest.mark.parametrize("layers_n", [1, 2, 3])
@pytest.mark.parametrize("N,M", [(2048, 64), (16384, 700), (70000, 96)])
def test_step_whose_inputs_are_settled_still_orders_its_own_kernels(layers_n, N, M):
    """KVSWAP_INPUTS_SETTLED on a step is about the step's inputs: the selections its attention reads are not among them."""
    L, H, d, r, G = layers_n, 8, 128, 32, 8
    shape = kv.make_shape(batch=1, n_ctx=N, n_q_heads=4 * H, n_kv_heads=H, head_dim=d, rank=r, meta_heads=1, group_size=G,
                          top_k=M, kv_dtype=kv.KVSWAP_BF16, meta_dtype=kv.KVSWAP_F16, q_dtype=kv.KVSWAP_BF16)
    bf = torch.bfloat16
    q = [_randn(L, 1, 4 * H, d, dtype=bf, seed=40 + i) for i in range(2)]
    K, V = ([_randn(1, H, N, d, dtype=bf, seed=50 + 10 * i + l) for l in range(L)] for i in range(2))
    meta = [_randn(1, 1, N, r, dtype=torch.float16, seed=70 + l) for l in range(L)]
    proj = [_randn(H, d, r, seed=80 + l) for l in range(L)]
    layers, ws = kv.make_layers(K, V, meta, proj, 0), rt.alloc_workspace(shape)
    out = torch.empty((L, 1, 4 * H, d), device="cuda")
    idx, nsel = torch.empty((L, 1, H, M), dtype=torch.int32, device="cuda"), torch.empty((L, 1, H), dtype=torch.int32, device="cuda")
    want = []
    for i in range(2):
        kv.kvswap_decode_step(shape, layers, q[i], out, None, idx, nsel, ws)
        want.append((out.clone(), idx.clone()))
    torch.cuda.synchronize()
    flagged = shape.with_flags(kv.KVSWAP_INPUTS_SETTLED)
    bad = torch.zeros((), dtype=torch.int64, device="cuda")
    for i in range(40):
        kv.kvswap_decode_step(flagged, layers, q[i % 2], out, None, idx, nsel, ws)
        bad += (~torch.isfinite(out)).any() | (out != want[i % 2][0]).any() | (idx != want[i % 2][1]).any()
    torch.cuda.synchronize()
    assert int(bad) == 0 and kv.kvswap_read_device_status(ws) == 0


# the short kernel, which lets its successor start early, the general one, and the tensor-core one of long prompts
@pytest.mark.parametrize("N,per_head,r", [(1500, False, 32), (3001, True, 32), (1500, False, 128), (70000, False, 32)])
@pytest.mark.parametrize("kind", ["call", "step"])
def test_scorer_behind_the_projection_of_its_metadata(N, per_head, r, kind):
    H, d, M = 8, 128, 64
    hm = H if per_head else 1
    shape = kv.make_shape(batch=1, n_ctx=N, n_q_heads=4 * H, n_kv_heads=H, head_dim=d, rank=r, meta_heads=hm, group_size=8,
                          top_k=M, kv_dtype=kv.KVSWAP_BF16, meta_dtype=kv.KVSWAP_F16, q_dtype=kv.KVSWAP_BF16)
    q, K = _randn(1, 1, 4 * H, d, dtype=torch.bfloat16, seed=90), _randn(1, H, N, d, dtype=torch.bfloat16, seed=91)
    proj = _randn(H, d, r, seed=92) * 0.1
    meta, ws = torch.empty((1, hm, N, r), dtype=torch.float16, device="cuda"), rt.alloc_workspace(shape)
    out = torch.empty((1, 1, 4 * H, d), device="cuda")
    idx = torch.empty((1, 1, H, M), dtype=torch.int32, device="cuda")
    nsel = torch.empty((1, 1, H), dtype=torch.int32, device="cuda")
    layers = kv.make_layers([K], [K], [meta], [proj], 0)

    def consume():
        if kind == "call":
            kv.kvswap_score_select(shape, q[0], proj, meta, idx[0], nsel[0], None, ws)
        else:
            kv.kvswap_decode_step(shape, layers, q, out, None, idx, nsel, ws)

    kv.kvswap_project_keys(shape, K, proj, meta, 0, N, ws)
    torch.cuda.synchronize()
    consume()
    torch.cuda.synchronize()
    want = idx.clone()
    for _ in range(10):
        meta.zero_()
        idx.fill_(-7)
        torch.cuda.synchronize()
        torch.cuda._sleep(100000)                           # both calls are queued before the first one starts
        kv.kvswap_project_keys(shape, K, proj, meta, 0, N, ws)
        consume()
        torch.cuda.synchronize()
        assert torch.equal(idx, want)
