"""The LM head's ranked choices at the edges of its epilogue: vocabularies around the runs of 32 columns that two warps take in turn,
rows around the 32 of a warp, many equal logits (exact small integers, so that the ranking is exact: greater logit, then lower token),
infinities and NaN."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,V", [(1, 1), (3, 31), (32, 33), (33, 64), (31, 95), (128, 97), (129, 160), (200, 257), (6, 14400), (40, 20001)])
@pytest.mark.parametrize("k", [1, 2, 4, 7])
def test_ranked_choices_with_many_ties(R, V, k):
    from paper_2506_14158_b200 import s4c

    H = 64
    rng = np.random.default_rng(R * V + k)
    w = rng.integers(-3, 4, (V, H)).astype(np.float32)
    x = np.zeros((R, H), np.float32)
    x[np.arange(R), rng.integers(0, H, R)] = 1.0  # a row's logits: one column of the weight
    if V > 40:
        w[rng.integers(0, V, 3), 5] = np.inf
        w[rng.integers(0, V, 3), 6] = -np.inf
        x[:, 5:7] = 0.0
        x[R // 2] = 0.0
        x[R // 2, 5] = 1.0
    logits = np.zeros((R, V))
    for r in range(R):
        with np.errstate(invalid="ignore"):
            logits[r] = (w.astype(np.float64) * x[r]).sum(axis=1)  # 0 * inf = NaN: never chosen
    t = s4c.lm_head_topk(torch.tensor(x).bfloat16().cuda(), torch.tensor(w).bfloat16().cuda(), k)
    got, val = t["token"].cpu().numpy().reshape(R, k), t["logit"].cpu().numpy().reshape(R, k)
    for r in range(R):
        ranked = [v for v in sorted(range(V), key=lambda v: (-logits[r, v], v) if logits[r, v] == logits[r, v] else (np.inf, v))
                  if logits[r, v] > -np.inf][:k]
        want = ranked + [-1] * (k - len(ranked))
        assert got[r].tolist() == want
        assert val[r, :len(ranked)].tolist() == logits[r, ranked].tolist()
