"""GPU parity of the float32 attention at the edges of its tiles: trees around 16 and 32 rows, prefixes around a tile of cache slots,
grouped heads, both head sizes, one and several splits."""
from dataclasses import replace

import pytest

import parity
from paper_2506_14158_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,L,B,Hq,Hkv,d", [(1, 1, 1, 1, 1, 64), (15, 17, 2, 4, 4, 64), (16, 16, 1, 4, 2, 128), (17, 31, 3, 4, 1, 64),
                                            (33, 32, 1, 2, 2, 128), (32, 95, 2, 4, 4, 128), (5, 1023, 1, 4, 4, 64), (128, 700, 1, 2, 1, 128)])
def test_f32_attention_edges(T, L, B, Hq, Hkv, d):
    cfg = replace(W.CONFIGS["c1"], name="t", config_id=170 + T % 7, B=B, T=T, L=L, Hq=Hq, Hkv=Hkv, d=d, tree="random", max_tree_depth=6)
    parent = W.make_trees(cfg)
    q, k, v = W.make_attention_inputs(cfg)
    got, ref, gst, rst = parity.attention_both(q, k, v, [L] * B, parent)
    parity.assert_attention_close(got, ref, gst, rst, parity.ATTN_TOL[cfg.dtype])
