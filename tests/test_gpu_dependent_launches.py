"""GPU: what a call may read ahead of its wait.  The calls are launched programmatically dependent, and a product requests tiles of
its weights while the call in front is still running; a weight that the call before that one wrote has to be complete all the same,
whichever call lies between."""
import pytest
import torch

pytestmark = pytest.mark.gpu

BETWEEN = ["embed_gather", "rmsnorm", "linear", "linear shared out", "linear_rmsnorm", "draft_level", "lm_head_greedy", "accept_tokens", "kv_compact",
           "qkv_rope", "qkv_rope_same_tree", "tree_attention"]


@pytest.mark.parametrize("consumer", ["linear", "qkv_rope_same_tree"])
@pytest.mark.parametrize("between", BETWEEN)
def test_a_weight_written_two_calls_earlier_is_complete(between, consumer):
    from paper_2506_14158_b200 import s4c

    g = torch.Generator(device="cuda").manual_seed(7)
    bf = lambda *s, std=1.0: (torch.randn(*s, generator=g, device="cuda") * std).bfloat16()
    ii = lambda *s, hi=8: torch.randint(0, hi, s, generator=g, device="cuda", dtype=torch.int32)
    H, T, C, d, heads = 8192, 8, 64, 128, 4
    N = 3 * heads * d
    # the weight's own product: several rounds of CTAs with an uneven last one, a tenth of a millisecond or more
    a, b = bf(N, H), bf(H, H, std=0.01)
    w = torch.empty(N, H, dtype=torch.bfloat16, device="cuda")
    assert s4c.linear_workspace_bytes(N, H, 0, H) == 0
    small, wide, narrow, norm = bf(4, H), bf(8192, H, std=0.01), bf(256, H, std=0.01), bf(256)
    few, w_few = bf(4, 256), bf(2048, 256, std=0.05)  # (four K slices: not shared out)
    ws = torch.empty(1 << 22, dtype=torch.uint8, device="cuda")
    tokens, cl, par = ii(1, T), torch.tensor([8], dtype=torch.int32, device="cuda"), torch.arange(-1, T - 1, dtype=torch.int32, device="cuda").view(1, T)
    q, k, v = torch.zeros(1, heads, T, d, dtype=torch.bfloat16, device="cuda"), bf(1, heads, C, d), bf(1, heads, C, d)
    x = bf(1, T, H)
    ws_qkv = torch.empty(s4c.qkv_rope_workspace_bytes(1, T, d), dtype=torch.uint8, device="cuda")
    w_qkv = bf(N, H, std=0.01)
    q2, k2, v2, att = q.clone(), k.clone(), v.clone(), q.clone()
    status, status2, length = (torch.zeros(1, dtype=torch.int32, device="cuda") for _ in range(3))
    s4c.qkv_rope(x, w_qkv, cl, par, q, k, v, status=status, workspace=ws_qkv)  # the tables of the consumer
    ws_qkv2, acc, path = ws_qkv.clone(), torch.zeros(1, dtype=torch.int32, device="cuda"), torch.full((1, T), -1, dtype=torch.int32, device="cuda")
    path[:, 0] = 0
    tree = dict(s4c.tree_build_topk(ii(1, 3, 2), [2], acc), n_nodes=torch.zeros(1, dtype=torch.int32, device="cuda"))
    topk_all, choice = ii(1, 3, 2), ii(1, 2)
    e_out, f_out, rows2 = bf(2, H), bf(2, H), [torch.zeros(2, dtype=torch.int32, device="cuda") for _ in range(2)]
    mid = {
        "embed_gather": lambda: s4c.embed_gather(wide, tokens),
        "rmsnorm": lambda: s4c.rmsnorm(small, wide[0].contiguous()),
        "linear": lambda: s4c.linear(few, w_few, workspace=ws),
        "linear shared out": lambda: s4c.linear(small, narrow, workspace=ws),
        "linear_rmsnorm": lambda: s4c.linear_rmsnorm(small, narrow, norm, workspace=ws),
        "draft_level": lambda: s4c.draft_level(choice, [2], ((0, 1), (1, 3)), topk_all, tree, acc, cl, wide, small[:1].contiguous(), e_out, f_out, *rows2),
        "lm_head_greedy": lambda: s4c.lm_head_greedy(small, wide),
        "accept_tokens": lambda: s4c.tree_accept_tokens(tokens, tokens, par, 8),
        "kv_compact": lambda: s4c.kv_compact(None, None, 0, (1, heads, C, d), torch.bfloat16, length, path, acc, T, status=status2),
        "qkv_rope": lambda: s4c.qkv_rope(x, w_qkv, cl, par, q2, k2, v2, workspace=ws_qkv2),
        "qkv_rope_same_tree": lambda: s4c.qkv_rope_same_tree(x, w_qkv, q2, k2, v2, ws_qkv2),
        "tree_attention": lambda: s4c.tree_attention(q2, k2, v2, cl, par, out=att),
    }[between]
    out = torch.empty(4, N, dtype=torch.bfloat16, device="cuda")

    def use():
        if consumer == "linear":
            return [s4c.linear(small, w, out=out, workspace=ws)]
        s4c.qkv_rope_same_tree(x, w, q, k, v, ws_qkv, status=status)
        return [q, k, v]

    assert s4c.linear_workspace_bytes(4, 256, 0, 2048) == 0 and 0 < s4c.linear_workspace_bytes(4, H, 0, 256) <= ws.numel()
    assert s4c.linear_workspace_bytes(4, H, 0, N) <= ws.numel()
    s4c.linear(a, b, out=w, workspace=ws)
    mid()
    torch.cuda.synchronize()
    want = [t.clone() for t in use()]
    assert all(torch.isfinite(t.float()).all() for t in want)
    for _ in range(5):
        w.fill_(float("nan"))
        length.zero_()
        torch.cuda.synchronize()
        s4c.linear(a, b, out=w, workspace=ws)
        mid()
        got = use()
        torch.cuda.synchronize()
        for x0, x1 in zip(want, got):
            assert torch.equal(x0, x1)
