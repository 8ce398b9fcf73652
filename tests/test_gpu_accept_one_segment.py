"""GPU parity of the acceptance where a row becomes one segment and the walk one CTA: vocabularies around 4096, both modes, long chains
of rejections, padded trees."""
from dataclasses import replace

import numpy as np
import pytest

from paper_2506_14158_b200 import workloads as W
from parity import accept_both, assert_accept_equal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [33, 127, 1000, 4092, 4095, 4096, 4097])
@pytest.mark.parametrize("tau", [0.0, 0.7])
@pytest.mark.parametrize("B,T", [(1, 15), (9, 40)])
def test_one_segment(V, tau, B, T):
    cfg = replace(W.CONFIGS["c2"], name="t", config_id=210 + V % 89, B=B, T=T, V=V, tree="random", logit_sigma=1.5, max_tree_depth=8)
    parent = W.make_trees(cfg)
    x = W.make_accept_inputs(cfg, parent, tau, token_mode="sampled")
    if tau > 0:
        x["uniforms"][0, 1:] = 1.0 - 2.0 ** -24  # rejects wherever it can
    nodes = np.full(B, T, np.int32)
    nodes[-1] = max(1, T // 3)
    got, ref = accept_both(x, parent, tau, n_nodes=nodes, max_depth=8)
    assert assert_accept_equal(got, ref, tau > 0) == 0
