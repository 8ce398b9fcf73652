"""The native marshalling refuses what the library cannot take, before anything is launched (no GPU needed)."""
import pytest
import torch


def test_binding_refuses_cpu_tensors_wrong_shapes_and_types(s4c_lib):
    from paper_2506_14158_b200 import s4c

    q, kv = torch.zeros(1, 4, 8, 64), torch.zeros(1, 2, 128, 64)
    i = torch.zeros(1, dtype=torch.int32)
    par = torch.zeros(1, 8, dtype=torch.int32)
    with pytest.raises(ValueError, match="k_cache"):
        s4c.tree_attention(q, kv, torch.zeros(1, 2, 64, 64), i, par)
    with pytest.raises(TypeError, match="share one dtype"):
        s4c.tree_attention(q, kv.to(torch.bfloat16), kv, i, par)
    with pytest.raises(TypeError, match="float32 or bfloat16"):
        s4c.tree_attention(q.half(), kv.half(), kv.half(), i, par)
    with pytest.raises(TypeError, match="must be a tensor"):
        s4c.tree_attention(None, kv, kv, i, par)
    with pytest.raises(ValueError, match="no CPU path"):
        s4c.tree_attention(q, kv, kv, i, par, workspace=i, stream=type("S", (), {"cuda_stream": 0})())
    with pytest.raises(ValueError):
        s4c.tree_accept_tokens(i, par, par, 100)
