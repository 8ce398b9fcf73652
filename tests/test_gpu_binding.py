"""GPU: the native marshalling takes what `int()` and `float()` take, and raises torch's own exceptions."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _attention_inputs(B=1, H=4, T=8, d=64, C=128, dtype=torch.bfloat16):
    g = torch.Generator(device="cuda").manual_seed(3)
    q = torch.randn(B, H, T, d, generator=g, device="cuda").to(dtype)
    k, v = (torch.randn(B, H, C, d, generator=g, device="cuda").to(dtype) for _ in range(2))
    cl = torch.full((B,), 40, dtype=torch.int32, device="cuda")
    par = torch.arange(-1, T - 1, dtype=torch.int32, device="cuda").repeat(B, 1)
    return q, k, v, cl, par


def test_numbers_of_every_kind_are_taken():
    from paper_2506_14158_b200 import s4c

    q, k, v, cl, par = _attention_inputs()
    want = s4c.tree_attention(q, k, v, cl, par, scale=0.25, max_cache_len=64)
    for n, x in ((64.0, np.float32(0.25)), (np.int64(64), "0.25"), (torch.tensor(64), torch.tensor(0.25)), ("64", 0.25)):
        assert torch.equal(s4c.tree_attention(q, k, v, cl, par, scale=x, max_cache_len=n), want)
    tgt = tok = torch.zeros(1, 8, dtype=torch.int32, device="cuda")
    a = s4c.tree_accept_tokens(tgt, tok, par, 100, max_depth=7)
    b = s4c.tree_accept_tokens(tgt, tok, par, 100.0, max_depth=7.0)
    assert all(torch.equal(a[key], b[key]) for key in a)


def test_running_out_of_memory_raises_torchs_exception():
    from paper_2506_14158_b200 import s4c

    q, k, v, cl, par = _attention_inputs(B=256, H=32, T=64)  # an output of 64 MB
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    total = torch.cuda.get_device_properties(0).total_memory
    torch.cuda.set_per_process_memory_fraction(torch.cuda.memory_reserved() / total)
    try:
        with pytest.raises(torch.cuda.OutOfMemoryError):
            s4c.tree_attention(q, k, v, cl, par)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert s4c.tree_attention(q, k, v, cl, par).shape == q.shape
