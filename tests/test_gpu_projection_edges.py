"""GPU parity of the projections' epilogues at their edges: rows around 32 and 128 (the rows of an epilogue warp, of a tile, of two
tiles), outputs whose last run of 32 columns is short, every combination of what follows the product."""
import numpy as np
import pytest
import torch

import test_gpu_linear as linear
import test_gpu_qkv_rope as qkv
from paper_2506_14158_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [1, 31, 32, 33, 127, 129, 161, 257])
@pytest.mark.parametrize("K,N", [(64, 40), (192, 1000), (2048, 264)])  # one tile; several; the K range shared out
def test_rows_and_short_runs(R, K, N):
    linear.test_linear_against_the_oracle(R, K, 0, N, R % 2 == 1, R % 3 != 0)


@pytest.mark.parametrize("R,K,N,res", [(1, 64, 24, True), (33, 320, 88, False), (129, 1024, 40, True), (257, 128, 1000, True)])
def test_gated_rows_and_short_runs(R, K, N, res):
    linear.test_gated_linear_against_the_oracle(R, K, N, res)


@pytest.mark.parametrize("B,T,Hq,Hkv,d", [(1, 1, 2, 1, 128), (1, 32, 4, 2, 64), (3, 11, 2, 2, 128), (2, 65, 4, 1, 64), (3, 43, 2, 1, 128)])
def test_qkv_rows(B, T, Hq, Hkv, d):
    rng = np.random.default_rng(B * T + d)
    H, C = 192, 300
    x = torch.from_numpy(rng.standard_normal((B, T, H)).astype(np.float32)).to(torch.bfloat16)
    w = torch.from_numpy((rng.standard_normal(((Hq + 2 * Hkv) * d, H)) / np.sqrt(H)).astype(np.float32)).to(torch.bfloat16)
    lens = rng.integers(0, C - T, B).astype(np.int32)
    parent = np.stack([W.random_tree(T, 8, rng) if T > 1 else np.full(1, -1, np.int32) for _ in range(B)])
    nodes = rng.integers(1, T + 1, B).astype(np.int32)
    got, ref, _ = qkv._run(x, w, lens, parent, Hq, Hkv, d, C, nodes)
    qkv._compare(got, ref, x, w, lens, nodes, T)
