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


@pytest.mark.parametrize("T,L,Hq,Hkv,d", [(15, 128, 4, 4, 64), (26, 37, 4, 2, 128), (64, 0, 2, 2, 64), (40, 600, 1, 1, 128)])
def test_another_branch_may_hold_anything(T, L, Hq, Hkv, d):
    # K and V of a node are read by the nodes below it only: NaN or Inf there must not reach a node on another branch (the slot is
    # not part of its sum, rather than entering it times zero)
    import numpy as np
    import torch

    from paper_2506_14158_b200 import s4c

    g = torch.Generator().manual_seed(T)
    C = L + T
    q = torch.randn(1, Hq, T, d, generator=g)
    k, v = (torch.randn(1, Hkv, C, d, generator=g) for _ in range(2))
    parent = W.random_tree(T, 6, np.random.default_rng(T))
    bad = [t for t in range(1, T) if t % 5 == 3]
    below = np.zeros(T, dtype=bool)
    for t in range(T):
        below[t] = t in bad or (t > 0 and below[parent[t]])
    assert below.any() and not below.all()
    dirty_k, dirty_v = k.clone(), v.clone()
    for n, t in enumerate(bad):
        dirty_k[:, :, L + t] = [float("nan"), float("inf"), 0.0][n % 3]
        dirty_v[:, :, L + t] = [float("inf"), float("nan"), float("-inf")][n % 3]
    out = {}
    for name, kk, vv in (("clean", k, v), ("dirty", dirty_k, dirty_v)):
        out[name] = s4c.tree_attention(q.cuda(), kk.cuda(), vv.cuda(), torch.tensor([L], dtype=torch.int32, device="cuda"),
                                       torch.tensor(np.asarray(parent)[None], dtype=torch.int32, device="cuda")).cpu()
    assert torch.isfinite(out["clean"]).all()
    assert torch.equal(out["dirty"][:, :, ~below], out["clean"][:, :, ~below])
