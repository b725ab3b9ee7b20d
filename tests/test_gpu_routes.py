"""Calls on both sides of the lines between the kernels that the library chooses from, each checked to have taken the one
it should, against the oracle."""
import dataclasses

import pytest

from paper_2511_11907_b200 import binding as kv
from paper_2511_11907_b200 import workloads as W
from launches import launched
from test_gpu_parity import run_layer_parity

pytestmark = pytest.mark.gpu

KV = W.SCOPE_KV_HEAD


# The line at 6144 groups between the launch of clusters and the streaming scorer, on both sides of it, and the line
# at one tile per warp for fewer than eight scopes.
@pytest.mark.parametrize("kw,name", [
    (dict(group_size=1, n_ctx=6144), "score_select_cluster_kernel"),
    (dict(group_size=1, n_ctx=6145), "score_stream_kernel"),
    (dict(group_size=1, n_ctx=6144, rank=64), "score_select_cluster_kernel"),
    (dict(group_size=3, n_ctx=3 * 6144 + 2), "score_select_cluster_kernel"),
    (dict(group_size=3, n_ctx=3 * 6145), "score_stream_kernel"),
    (dict(group_size=4, n_ctx=4 * 4096, n_kv_heads=2, n_q_heads=4), "score_select_cluster_kernel"),
    (dict(group_size=4, n_ctx=4 * 4112, n_kv_heads=2, n_q_heads=4), "score_stream_kernel"),
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
