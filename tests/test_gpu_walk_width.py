"""GPU parity of the sampling walk where the number of its CTAs changes: vocabularies around 65536, few and many sequences, long chains of
rejections on a row."""
from dataclasses import replace

import pytest

from paper_2506_14158_b200 import workloads as W
from parity import accept_both, assert_accept_equal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [65535, 65536, 65537, 65540])
@pytest.mark.parametrize("B,T", [(1, 20), (12, 6)])
def test_walk_width(V, B, T):
    cfg = replace(W.CONFIGS["c2"], name="t", config_id=190 + V % 89, B=B, T=T, V=V, tree="random", logit_sigma=2.0, max_tree_depth=6)
    parent = W.make_trees(cfg)
    x = W.make_accept_inputs(cfg, parent, 0.9, token_mode="sampled")
    x["uniforms"][0, 1:] = 1.0 - 2.0 ** -24  # rejects wherever it can
    got, ref = accept_both(x, parent, 0.9, max_depth=6)
    assert assert_accept_equal(got, ref, True) == 0
