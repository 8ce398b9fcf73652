"""GPU parity at the edges of the sampling walk's pass (a vocabulary shorter than the CTAs' groups of 128, one that is no multiple of
4, the sizes where the kept values stop fitting beside the walk's state) and of the spread feature gather."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from paper_2506_14158_b200 import workloads as W
from parity import accept_both, assert_accept_equal, assert_compact_equal, compact_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [33, 129, 1023, 4100, 131072, 150001, 150004, 240001, 240004])
def test_sampling_walk_sizes(V):
    B, T = (16, 20) if V < 5000 else (3, 12)
    cfg = replace(W.CONFIGS["c2"], name="t", config_id=150 + V % 89, B=B, T=T, V=V, tree="random", logit_sigma=2.0, max_tree_depth=6)
    parent = W.make_trees(cfg)
    x = W.make_accept_inputs(cfg, parent, 0.9, token_mode="sampled")
    x["uniforms"][0, 1:] = 1.0 - 2.0 ** -24  # the first sequence rejects wherever it can: the longest chains
    got, ref = accept_both(x, parent, 0.9, max_depth=6)
    assert assert_accept_equal(got, ref, True) == 0


@pytest.mark.parametrize("B,Hkv,max_depth,hid,n_layers", [(1, 1, 0, 8, 1), (3, 1, 127, 4096, 1), (2, 8, 8, 4104, 2), (1, 32, 7, 4096, 1)])
def test_feature_gather_sizes(B, Hkv, max_depth, hid, n_layers):
    g = torch.Generator().manual_seed(hid + B)
    T, d, C, L = 128, 64, 200, 60
    k = [torch.randn(B, Hkv, C, d, generator=g).bfloat16() for _ in range(n_layers)]
    v = [torch.randn(B, Hkv, C, d, generator=g).bfloat16() for _ in range(n_layers)]
    feat = torch.randn(B, T, hid, generator=g).bfloat16()
    rng = np.random.default_rng(hid)
    a = rng.integers(0, max_depth + 1, B)
    a[0] = max_depth  # the whole path
    path = np.full((B, max_depth + 1), -1, dtype=np.int32)
    for b in range(B):
        path[b, : a[b] + 1] = np.concatenate([[0], np.sort(rng.choice(np.arange(1, T), a[b], replace=False))])
    old = np.full(B, L, dtype=np.int32)
    got, ref = compact_both(k, v, old, path, a, T, feat)
    assert_compact_equal(got, ref, old, T)
