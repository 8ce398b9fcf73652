"""GPU: s4c_draft_level against the calls that it stands for (s4c_tree_build_topk, row gathers), exactly: one sequence and several,
levels of one node, a tree that fills T and one that T cuts off, more choices than children, tokens outside the vocabulary, H of
one 16-byte word up to more words than threads, the last level (no next head)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,branching,k,H", [(1, 21, (2, 3, 1, 1), 3, 4096), (3, 16, (1, 1, 4), 4, 8), (5, 9, (4, 3), 6, 2056), (2, 128, (3, 4, 5, 2), 5, 64)])
def test_draft_level(B, T, branching, k, H):
    from paper_2506_14158_b200 import s4c

    g = torch.Generator().manual_seed(T)
    V = 50
    ri = lambda lo, hi, *s: torch.randint(lo, hi, s, generator=g, dtype=torch.int32).cuda()
    table = torch.randn(V, H, generator=g).bfloat16().cuda()
    root, pos = ri(0, V, B), ri(5, 99, B)
    topk = ri(0, V, B, T, k)
    topk_all = topk.clone()
    tree = {n: torch.full((B, T), -7, dtype=torch.int32, device="cuda") for n in ("tokens", "parent", "position")}
    tree["n_nodes"] = torch.zeros(B, dtype=torch.int32, device="cuda")
    ref = s4c.tree_build_topk(topk, branching, root, pos)
    n, par = int(ref["n_nodes"][0]), ref["parent"][0].tolist()
    depth = [0]
    for i in range(1, n):
        depth.append(depth[par[i]] + 1)
    levels = [(depth.index(j), len(depth) - depth[::-1].index(j)) for j in range(max(depth) + 1)] + [None]
    for (s, e), nxt in zip(levels[:-1], levels[1:]):
        choice = ri(-V // 2, V + V // 2, B * (e - s), k)
        topk[:, s:e] = choice.view(B, e - s, k)
        rows = 0 if nxt is None else nxt[1] - nxt[0]
        feats = torch.randn(B * (e - s), H, generator=g).bfloat16().cuda()
        eo, fo = (torch.full((B * rows, H), 9.0, dtype=torch.bfloat16, device="cuda") for _ in range(2))
        to, po = (torch.full((B * rows,), -7, dtype=torch.int32, device="cuda") for _ in range(2))
        if nxt is None:
            s4c.draft_level(choice, branching, ((s, e), None), topk_all, tree, root, pos)
        else:
            s4c.draft_level(choice, branching, ((s, e), nxt), topk_all, tree, root, pos, table, feats, eo, fo, to, po)
        ref = s4c.tree_build_topk(topk, branching, root, pos)
        assert torch.equal(topk_all, topk)
        for key in tree:
            assert torch.equal(tree[key], ref[key]), key
        if nxt is None:
            continue
        want = ref["tokens"][:, nxt[0]:nxt[1]].reshape(-1)
        assert torch.equal(to, want) and torch.equal(po, ref["position"][:, nxt[0]:nxt[1]].reshape(-1))
        assert torch.equal(eo, s4c.embed_gather(table, want.contiguous()))
        src = torch.tensor([b * (e - s) + par[i] - s for b in range(B) for i in range(*nxt)])
        assert torch.equal(fo, feats[src.cuda()])
