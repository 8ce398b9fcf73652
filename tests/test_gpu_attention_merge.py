"""GPU parity of the attention launches whose end is a merge: turns, row copies and splits, at row counts around the tiles, with
padded trees (their rows are zero) and sequences that get no tile at all."""
import numpy as np
import pytest
import torch

from paper_2506_14158_b200 import workloads as W

from parity import ATTN_TOL, assert_attention_close, attention_both

pytestmark = pytest.mark.gpu


# unsplit: turns (65..128 rows), row copies in launches of one and of two CTAs per SM; split: turns of 8 splits (16 partials a row),
# copies fetched from the peers, two row tiles with an incomplete second one
@pytest.mark.parametrize("B,Hq,Hkv,T,L,d", [
    (16, 32, 8, 17, 530, 128), (19, 32, 8, 32, 600, 64), (16, 28, 4, 11, 1100, 128),
    (5, 32, 32, 1, 90, 128), (20, 8, 8, 33, 70, 64), (38, 8, 4, 31, 200, 128), (2, 2, 1, 1, 64, 128),
    (1, 4, 1, 26, 4300, 128), (1, 4, 2, 33, 4400, 64),
    (1, 16, 16, 1, 3000, 128), (1, 40, 40, 60, 2048, 64),
    (5, 32, 8, 33, 1500, 128), (4, 24, 8, 64, 1000, 64)])
def test_merges(B, Hq, Hkv, T, L, d):
    rng = np.random.default_rng(B * T)
    g = torch.Generator().manual_seed(L)
    lens = [int(x) for x in rng.integers(0, L + 1, B)]
    lens[0] = L
    if B > 1:
        lens[1] = 0  # the tree's own slots only: most splits have nothing to do
    nodes = [int(x) for x in rng.integers(1, T + 1, B)]
    nodes[0] = T
    q = torch.randn((B, Hq, T, d), generator=g).to(torch.bfloat16)
    k, v = (torch.randn((B, Hkv, L + T, d), generator=g).to(torch.bfloat16) for _ in range(2))
    parent = np.stack([W.random_tree(T, 8, rng) if T > 1 else np.full(1, -1, np.int32) for _ in range(B)])
    got, ref, gst, rst = attention_both(q, k, v, lens, parent, nodes)
    assert (rst == 0).all()
    assert_attention_close(got, ref, gst, rst, ATTN_TOL["bf16"])
