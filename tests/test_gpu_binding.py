"""GPU: the native marshalling takes what `int()` and `float()` take, raises torch's own exceptions, and lets other threads run."""
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
    held = []
    try:
        with pytest.raises(torch.cuda.OutOfMemoryError):  # what room the pool still has goes first
            while len(held) < 1000:
                held.append(torch.empty_like(q))
        with pytest.raises(torch.cuda.OutOfMemoryError):
            s4c.tree_attention(q, k, v, cl, par)
    finally:
        held.clear()
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert s4c.tree_attention(q, k, v, cl, par).shape == q.shape


@pytest.mark.parametrize("call", ["attention", "accept", "compact", "lm_head", "accept_tokens"])
def test_other_threads_run_while_a_launch_waits_for_room_in_the_queue(call):
    # The stream is kept busy for some tenths of a second and launches are enqueued until one has to wait for room; another
    # thread notes the longest time for which it could not run meanwhile.
    import threading
    import time

    from paper_2506_14158_b200 import s4c

    q, k, v, cl, par = _attention_inputs()
    out = torch.empty_like(q)
    i32 = dict(dtype=torch.int32, device="cuda")
    status, one, tok = torch.zeros(1, **i32), torch.zeros(1, **i32), torch.zeros(1, 8, **i32)
    acc, nxt, path = torch.zeros(1, **i32), torch.zeros(1, **i32), torch.full((1, 8), -1, **i32)
    path[:, 0] = 0
    logits, tie = torch.zeros(1, 8, 64, device="cuda"), torch.zeros(1, 8, dtype=torch.uint8, device="cuda")
    hid, w = torch.ones(1, 64, dtype=torch.bfloat16, device="cuda"), torch.ones(128, 64, dtype=torch.bfloat16, device="cuda")
    logit = torch.zeros(1, device="cuda")
    run = {
        "attention": lambda: s4c.tree_attention(q, k, v, cl, par, out=out),
        "accept": lambda: s4c.tree_accept(logits, None, tok, par, 0.0, None, None, 7, acc, path, nxt, tie, status),
        "compact": lambda: s4c.kv_compact(None, None, 0, (1, 4, 128, 64), torch.bfloat16, one, path, acc, 8, status=status),
        "lm_head": lambda: s4c.lm_head_greedy(hid, w, nxt, logit, status),
        "accept_tokens": lambda: s4c.tree_accept_tokens(tok, tok, par, 64, None, 7, acc, path, nxt, status),
    }[call]
    run()
    torch.cuda.synchronize()
    gaps, done = [0.0], threading.Event()

    def tick():
        last = time.perf_counter()
        while not done.is_set():
            time.sleep(0.0005)
            now = time.perf_counter()
            gaps[0], last = max(gaps[0], now - last), now

    thread = threading.Thread(target=tick)
    thread.start()
    try:
        torch.cuda._sleep(800_000_000)  # about 0.4 s
        longest = 0.0
        for _ in range(20000):
            t0 = time.perf_counter()
            run()
            longest = max(longest, time.perf_counter() - t0)
            if longest > 0.1:
                break
    finally:
        done.set()
        thread.join()
        torch.cuda.synchronize()
    assert longest > 0.1, "no launch had to wait: the queue took them all"
    assert gaps[0] < 0.5 * longest, f"another thread stood still for {gaps[0]:.3f} s of a launch of {longest:.3f} s"
