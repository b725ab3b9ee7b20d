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
