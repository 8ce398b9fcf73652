"""The work a serving program has this library do, as timed cases.

Five kinds of work, each through the package's public entry points:

  verify     the attention, acceptance and compaction of one verify step over all decoder layers (`VerifyStep`): the form in
             which a program that runs the projections itself uses the library.  Multi-layer steps are replayed as the CUDA
             graph the class captures; the one-layer step runs eagerly.
  target     the target model's whole verify pass (`TargetVerify`), weights resident, captured once in a CUDA graph.
  draft      one drafting round of three heads (`MultiHeadDrafter`), captured once in a CUDA graph.
  attention  a single attention call from a program's own decoder layer, eager (`s4c.tree_attention`).
  head       LM head with the greedy choice and the walk on the choices, eager (`s4c.lm_head_greedy`, `s4c.tree_accept_tokens`).

Model shapes are the ones the benchmark and the tests use (7B, 13B and 8B layers, and the small float32 one).  A case is a
dict of plain values; every tensor of a state is made on the GPU from the seed.  Steps rewind the committed lengths before
they run, so that a pass can be repeated on the same state.
"""
import numpy as np
import torch

from paper_2506_14158_b200 import drafter, s4c, target
from paper_2506_14158_b200 import workloads as W
from paper_2506_14158_b200.verify import VerifyStep

MODELS = {  # V, hidden width, query heads, KV heads, head width, MLP width, storage type
    "tiny": dict(V=1000, H=256, Hq=4, Hkv=4, d=64, inter=512, dtype=torch.float32),
    "7b": dict(V=32000, H=4096, Hq=32, Hkv=32, d=128, inter=11008, dtype=torch.bfloat16),
    "13b": dict(V=32000, H=5120, Hq=40, Hkv=40, d=128, inter=13824, dtype=torch.bfloat16),
    "8b": dict(V=128256, H=4096, Hq=32, Hkv=8, d=128, inter=14336, dtype=torch.bfloat16),
}
MAX_DEPTH = 8
TREES = {16: (3, 2, 2, 1), 21: (2, 3, 1, 1), 26: (4, 3, 2, 2, 1), 40: (4, 3, 2, 2, 2), 64: (4, 4, 3, 2, 1)}


def verify(name, model, layers, B, L, T, tau, top_k=0, top_p=1.0, page=0, ragged=False, build=False):
    """tau 0: greedy; top_k > 0: filtered sampling; page > 0: paged caches; ragged: lengths and tree sizes differ over the
    batch; build: the step builds its trees on the device from the draft distributions."""
    return dict(name=name, kind="verify", model=model, layers=layers, B=B, L=L, T=T, tau=tau, top_k=top_k, top_p=top_p, page=page,
                ragged=ragged, build=build)


def listed():
    return [
        # the smallest step: a toy model's single layer in float32, called eagerly -- launches and host time
        verify("verify tiny f32", "tiny", 1, 1, 128, 15, 1.0),
        # interactive decoding of one 7B chat at a short context, sampling at temperature 1: the benchmark's step
        verify("verify 7b L1024", "7b", 32, 1, 1024, 26, 1.0),
        # one 13B chat, larger tree, sampling as samplers usually run it (top-50, nucleus 0.9, temperature 0.7)
        verify("verify 13b filtered", "13b", 40, 1, 2048, 60, 0.7, top_k=50, top_p=0.9),
        # a small batch on an 8B model with grouped queries and a large vocabulary, sampling
        verify("verify 8b b4 L4096", "8b", 32, 4, 4096, 64, 1.0),
        # a serving batch of 16 on paged caches: lengths differ, greedy, trees built on the device
        verify("verify 8b b16 paged", "8b", 32, 16, 2000, 26, 0.0, page=128, ragged=True, build=True),
        # one long document: the attention streams 17 GB of cache
        verify("verify 7b L32768", "7b", 32, 1, 32768, 64, 1.0),
        # a single layer's call from a program's own decoder: odd length, small odd tree
        dict(name="attention 7b call", kind="attention", model="7b", B=1, L=777, T=19, f32=False, rows=False, ragged=False),
        # the LM head, greedy choice and walk behind a program's own decoder: two sequences, odd row count
        dict(name="head 8b greedy", kind="head", model="8b", B=2, T=27),
        # the target's whole pass for one 7B chat, greedy (Section 4.1)
        dict(name="target 7b greedy", kind="target", model="7b", layers=32, B=1, L=1024, T=26, tau=0.0, ragged=False),
        # the same for a batch of four on the 8B shapes, sampling, lengths and trees of different size
        dict(name="target 8b b4 sampling", kind="target", model="8b", layers=32, B=4, L=1024, T=64, tau=1.0, ragged=True),
        # the drafting round of one chat: a few rows per head, latency and weight streaming
        dict(name="draft 7b", kind="draft", model="7b", B=1, L=1024, T=21),
        # and of a batch of eight on the 8B shapes
        dict(name="draft 8b b8", kind="draft", model="8b", B=8, L=700, T=21),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(lo * (hi / lo) ** rng.random()))))


def _draw_once(rng):
    kind = rng.choice(["verify", "verify", "verify", "attention", "head", "target", "draft"])
    if kind == "verify":
        model = rng.choice(["tiny", "7b", "7b", "13b", "8b", "8b"])
        tau = rng.choice([0.0, 0.7, 1.0])
        filtered = tau > 0 and rng.random() < 0.4
        B = rng.choice([1, 1, 2, 3, 4, 8, 16])
        if model == "tiny":
            return verify("", model, 1, B, _log_int(rng, 64, 1024), rng.choice([15, 16, 26]), tau, 20 if filtered else 0, 0.9 if filtered else 1.0,
                          ragged=rng.random() < 0.5)
        build = rng.random() < 0.3
        T = rng.choice(sorted(TREES)) if build else _log_int(rng, 16, 128)
        return verify("", model, rng.choice([8, 16, 32]), B, _log_int(rng, 256, 32768), T, tau, rng.choice([20, 50]) if filtered else 0,
                      rng.choice([0.9, 1.0]) if filtered else 1.0, page=rng.choice([0, 0, 64, 128, 256]), ragged=rng.random() < 0.5, build=build)
    if kind == "attention":
        model = rng.choice(["tiny", "7b", "13b", "8b"])
        return dict(kind=kind, model=model, B=rng.choice([1, 1, 2, 4]), L=_log_int(rng, 128, 1024 if model == "tiny" else 16384),
                    T=_log_int(rng, 8, 128), f32=model == "tiny", rows=model != "tiny" and rng.random() < 0.3, ragged=rng.random() < 0.5)
    model = rng.choice(["7b", "8b"])
    if kind == "head":
        return dict(kind=kind, model=rng.choice(["7b", "13b", "8b"]), B=rng.choice([1, 2, 4, 8]), T=_log_int(rng, 8, 64))
    if kind == "target":
        return dict(kind=kind, model=model, layers=rng.choice([4, 8, 16]), B=rng.choice([1, 1, 2, 4, 8]), L=_log_int(rng, 256, 4096),
                    T=_log_int(rng, 16, 64), tau=rng.choice([0.0, 0.0, 1.0]), ragged=rng.random() < 0.5)
    return dict(kind=kind, model=model, B=rng.choice([1, 1, 2, 4, 8]), L=_log_int(rng, 256, 2048), T=rng.choice([16, 21, 26]))


def _cost(case):
    w = work(case)
    return max(w["bytes"] / 6.5e12, w["flops"] / 1.4e15)


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        c = _draw_once(rng)
        c.pop("name", None)
        if _cost(c) <= most and _state_bytes(c) < 24e9:
            return c


# ------------------------------------------------------------------------------------------------ inputs
class _Make:
    """Seeded tensors on the GPU."""

    def __init__(self, seed):
        self.dev = torch.device("cuda")
        self.g = torch.Generator(device=self.dev)
        self.g.manual_seed(seed)
        self.rng = np.random.default_rng(seed)

    def normal(self, *shape, dtype=torch.bfloat16, std=1.0):
        return torch.empty(*shape, dtype=dtype, device=self.dev).normal_(0.0, std, generator=self.g)

    def uniform(self, *shape):
        return torch.rand(*shape, generator=self.g, device=self.dev).clamp_(max=1.0 - 2.0 ** -24)

    def perm(self, n):
        return torch.randperm(n, generator=self.g, device=self.dev)

    def ints(self, x):
        return torch.as_tensor(np.ascontiguousarray(x, dtype=np.int32)).to(self.dev)

    def lengths(self, B, L, ragged):
        return [int(L - self.rng.integers(0, max(1, L // 2))) for _ in range(B)] if ragged else [L] * B

    def trees(self, B, T, ragged):
        """parent [B,T] and the real node counts: trees grown breadth first, padded to T nodes where they are smaller."""
        counts = [int(self.rng.integers(max(1, T // 2), T + 1)) for _ in range(B)] if ragged else [T] * B
        parent = np.full((B, T), -1, np.int32)
        for b, n in enumerate(counts):
            parent[b, :n] = W.random_tree(n, MAX_DEPTH, self.rng)
        return parent, counts


def _child_ranks(parent):
    """rank [B,T]: the how-manieth child of its parent a node is."""
    rank = np.zeros_like(parent)
    for b in range(parent.shape[0]):
        seen = {}
        for i in range(1, parent.shape[1]):
            p = int(parent[b, i])
            if p >= 0:
                rank[b, i] = seen.get(p, 0)
                seen[p] = rank[b, i] + 1
    return rank


def _capacity(L, T):
    return (L + T + 127) // 128 * 128


def _acceptance_inputs(m, B, T, V, tau, parent):
    """Logits of a language model (one preferred token a row, its lead varying), the drafter's distribution close to them, and
    each node's token: the drafter's next best under its parent."""
    logits = m.normal(B, T, V, dtype=torch.float32, std=3.0)
    best = torch.randint(0, V, (B, T, 1), generator=m.g, device=m.dev)
    logits.scatter_(2, best, 12.0 + 6.0 * torch.rand(B, T, 1, generator=m.g, device=m.dev))
    draft = m.normal(B, T, V, dtype=torch.float32).add_(logits).div_(tau if tau > 0 else 1.0).softmax(dim=2)
    rank = _child_ranks(parent)
    par = torch.as_tensor(np.maximum(parent, 0), dtype=torch.int64, device=m.dev)
    ranked = draft.topk(int(rank.max()) + 1, dim=2).indices
    rows = ranked.gather(1, par.unsqueeze(2).expand(-1, -1, ranked.shape[2]))
    tokens = rows.gather(2, torch.as_tensor(rank, dtype=torch.int64, device=m.dev).unsqueeze(2)).squeeze(2)
    tokens[:, 0] = torch.randint(0, V, (B,), generator=m.g, device=m.dev)
    return logits, draft, tokens.to(torch.int32).contiguous(), m.uniform(B, T)


def _captured(fn):
    """fn as a CUDA graph, after one run outside the capture."""
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        fn()
    torch.cuda.current_stream().wait_stream(s)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = fn()
    return g, out


def _prepare_verify(c, m, S):
    B, L, T, n, V, d, Hkv = c["B"], c["L"], c["T"], c["layers"], S["V"], S["d"], S["Hkv"]
    dt = S["dtype"]
    lens = m.lengths(B, L, c["ragged"])
    if c["build"]:
        parent = np.tile(W.tree_from_branching(TREES[T], T), (B, 1))
        counts = [parent.shape[1]] * B
    else:
        parent, counts = m.trees(B, T, c["ragged"])
    logits, draft, tokens, uniforms = _acceptance_inputs(m, B, T, V, c["tau"], parent)
    C = _capacity(L, T)
    table = None
    if c["page"]:
        blocks = (L + T + c["page"] - 1) // c["page"]
        shape = (n, B * blocks, Hkv, c["page"], d)
        table = m.ints(m.rng.permutation(B * blocks).reshape(B, blocks))
    else:
        shape = (n, B, Hkv, C, d)
    q, k, v = m.normal(n, B, S["Hq"], T, d, dtype=dt), m.normal(*shape, dtype=dt), m.normal(*shape, dtype=dt)
    tau = c["tau"]
    step = VerifyStep(list(q), list(k), list(v), m.ints(lens), m.ints(parent), tokens, logits, draft if tau > 0 or c["build"] else None,
                      uniforms if tau > 0 else None, tau, MAX_DEPTH, n_nodes=m.ints(counts) if c["ragged"] and not c["build"] else None,
                      feat_in=m.normal(B, T, S["H"], dtype=dt), max_cache_len=L, block_table=table,
                      branching=TREES[T] if c["build"] else None, root_token=tokens[:, 0].contiguous() if c["build"] else None)
    if c["top_k"]:
        step.set_filter(c["top_k"], c["top_p"])
    if n > 1:
        step.capture()
    # what compaction writes: the tree slots (lengths that differ, or pages: the caches as they are)
    written = (k, v) if c["ragged"] or c["page"] else (k[:, :, :, L:L + T], v[:, :, :, L:L + T])
    return dict(run=step.graph.replay if n > 1 else step.run,
                out=dict(attention=step.attn_out, accept_len=step.accept_len, path=step.path, next_token=step.next_token,
                         near_tie=step.near_tie if tau > 0 else None, cache_len=step.cache_len, features=step.feat_out, k=written[0], v=written[1],
                         tree=[step.tokens, step.parent, step.position, step.n_nodes] if c["build"] else None,
                         status=[step.status_attn, step.status_accept, step.status_compact]), keep=step)


def _vocabulary(m, V, H, weights):
    """Embedding and LM head of a model that has learnt successors: token t's hidden state ranks successor[r](t) r-th, with the
    clear leads that a trained model's choices have (random heads would leave near ties that any rounding decides)."""
    table = m.normal(V, H)
    successor = [m.perm(V) for _ in weights]
    head = torch.zeros(V, H, dtype=torch.bfloat16, device=m.dev)
    for w, s in zip(weights, successor):
        head[s] += table * w
    head *= 2.0 * H ** -0.5
    return table, head, successor


def _layer(m, S):
    H, Hq, Hkv, d, inter = S["H"], S["Hq"], S["Hkv"], S["d"], S["inter"]
    norm = lambda: (1.0 + m.normal(H, dtype=torch.float32, std=0.05)).to(torch.bfloat16)
    return dict(norm1=norm(), qkv=m.normal((Hq + 2 * Hkv) * d, H, std=H ** -0.5), o=m.normal(H, Hq * d, std=(Hq * d) ** -0.5), norm2=norm(),
                gate_up=m.normal(2 * inter, H, std=H ** -0.5), down=m.normal(H, inter, std=inter ** -0.5))


def _drafted_tokens(m, parent, successor, root):
    """Tokens of a tree whose first children mostly are the target's choice (three in four), the others misses."""
    B, T = parent.shape
    V = successor.numel()
    succ = successor.cpu().numpy()
    rank = _child_ranks(parent)
    tokens = m.rng.integers(0, V, (B, T))
    tokens[:, 0] = root
    for b in range(B):
        for i in range(1, T):
            if parent[b, i] >= 0 and rank[b, i] == 0 and m.rng.random() < 0.75:
                tokens[b, i] = succ[tokens[b, parent[b, i]]]
    return tokens


def _prepare_target(c, m, S):
    B, L, T, n, V, H, Hkv, d = c["B"], c["L"], c["T"], c["layers"], S["V"], S["H"], S["Hkv"], S["d"]
    table, head, successor = _vocabulary(m, V, H, (1.0,))
    w = target.TargetWeights(embedding=table, layers=[target.LayerWeights(**_layer(m, S)) for _ in range(n)],
                             final_norm=torch.ones(H, dtype=torch.bfloat16, device=m.dev), lm_head=head)
    lens = m.lengths(B, L, c["ragged"])
    parent, counts = m.trees(B, T, c["ragged"])
    tokens = m.ints(_drafted_tokens(m, parent, successor[0], m.rng.integers(0, V, B)))
    C = _capacity(L, T)
    k, v = m.normal(n, B, Hkv, C, d), m.normal(n, B, Hkv, C, d)
    tau = c["tau"]
    draft = uniforms = None
    if tau > 0:  # the drafter's rows: 0.9 of the mass on the children it proposed, the rest spread over the vocabulary
        draft = m.normal(B, T, V, dtype=torch.float32, std=3.0).softmax(dim=2).mul_(0.1)
        rank = _child_ranks(parent)
        b, i = np.nonzero(parent >= 0)
        at = [torch.as_tensor(x, device=m.dev, dtype=torch.int64) for x in (b, parent[b, i])] + [tokens[b, i].long()]
        draft.index_put_(tuple(at), torch.as_tensor(np.array([0.5, 0.25, 0.1, 0.05])[np.minimum(rank[b, i], 3)], dtype=torch.float32, device=m.dev), accumulate=True)
        draft /= draft.sum(dim=2, keepdim=True)
        uniforms = m.uniform(B, T)
    tv = target.TargetVerify(w, B, T, S["Hq"], Hkv, d, C, list(k), list(v), MAX_DEPTH, stochastic=tau > 0)
    tv.feat_out.zero_()
    lengths, live, par = m.ints(lens), m.ints(lens), m.ints(parent)
    nodes = m.ints(counts) if c["ragged"] else None

    def once():
        live.copy_(lengths)
        return tv.forward(tokens, live, par, nodes, max_cache_len=L, temperature=tau, draft_probs=draft, uniforms=uniforms)

    graph, _ = _captured(once)
    written = (k, v) if c["ragged"] else (k[:, :, :, L:L + T], v[:, :, :, L:L + T])
    return dict(run=graph.replay, keep=(tv, once, graph),
                out=dict(accept_len=tv.accept_len, path=tv.path, next_token=tv.next_token, features=tv.feat_out, cache_len=live, k=written[0], v=written[1],
                         choice=tv.logits if tau > 0 else tv.target_token,
                         status=[tv.status_qkv, tv.status_attn, tv.status_head, tv.status_accept, tv.status_compact]))


def _prepare_draft(c, m, S):
    B, L, T, V, H, Hkv, d = c["B"], c["L"], c["T"], S["V"], S["H"], S["Hkv"], S["d"]
    k_best = max(TREES[T])
    table, head, successor = _vocabulary(m, V, H, (1.0, 0.8, 0.6, 0.4))
    heads = []
    for _ in range(3):
        fc = m.normal(H, 2 * H, std=0.5 * (2 * H) ** -0.5)
        fc[:, :H].diagonal().add_(1.0)
        heads.append(drafter.DrafterWeights(embedding=table, fc=fc, fc_bias=m.normal(H, std=0.02), lm_head=head, **_layer(m, S)))
    C = _capacity(L, 1)
    mh = drafter.MultiHeadDrafter(heads, B, T, TREES[T], S["Hq"], Hkv, d, C, k_best)
    root = m.rng.integers(0, V, B)
    candidates = torch.stack([s[torch.as_tensor(root, device=m.dev)] for s in successor[:k_best]], dim=1).to(torch.int32).contiguous()
    lens = m.lengths(B, L, B > 1)
    caches = []
    for s, e in mh.levels[: mh.n_passes]:
        rows = B * (e - s)
        caches.append((m.normal(rows, Hkv, C, d), m.normal(rows, Hkv, C, d), m.ints(np.repeat(lens, e - s))))
    root_token, f0, position = m.ints(root), m.normal(B, H), m.ints(lens)
    graph, out = _captured(lambda: mh.draft(root_token, f0, candidates, position, caches))
    return dict(run=graph.replay, out=dict(tree=out, choices=mh.topk_all), keep=(mh, caches, root_token, f0, candidates, position, graph))


def _prepare_attention(c, m, S):
    B, L, T, d, dt = c["B"], c["L"], c["T"], S["d"], torch.float32 if c["f32"] else torch.bfloat16
    C = _capacity(L, T)
    parent, counts = m.trees(B, T, c["ragged"])
    a = dict(q=m.normal(B, S["Hq"], T, d, dtype=dt), k_cache=m.normal(B, S["Hkv"], C, d, dtype=dt), v_cache=m.normal(B, S["Hkv"], C, d, dtype=dt),
             cache_len=m.ints(m.lengths(B, L, c["ragged"])), parent=m.ints(parent), n_nodes=m.ints(counts) if c["ragged"] else None,
             status=torch.zeros(B, dtype=torch.int32, device=m.dev), max_cache_len=L, rows=c["rows"])
    return dict(run=lambda: s4c.tree_attention(**a), out=None, keep=a)


def _prepare_head(c, m, S):
    B, T, V, H = c["B"], c["T"], S["V"], S["H"]
    table, head, successor = _vocabulary(m, V, H, (1.0,))
    parent, _ = m.trees(B, T, False)
    tokens = m.ints(_drafted_tokens(m, parent, successor[0], m.rng.integers(0, V, B)))
    hidden = table[tokens.long().reshape(-1)] * 0.6 + m.normal(B * T, H, std=0.8)  # final states: the token's direction among others
    par = m.ints(parent)

    def once():
        best = s4c.lm_head_greedy(hidden, head)
        walk = s4c.tree_accept_tokens(best["token"].view(B, T), tokens, par, V, max_depth=MAX_DEPTH)
        return dict(best, walk=walk)

    return dict(run=once, out=None, keep=(hidden, head, tokens, par))


_PREPARE = dict(verify=_prepare_verify, target=_prepare_target, draft=_prepare_draft, attention=_prepare_attention, head=_prepare_head)


def prepare(case, seed):
    return _PREPARE[case["kind"]](case, _Make(seed), MODELS[case["model"]])


def run(state):
    got = state["run"]()
    return got if state["out"] is None else state["out"]


# ------------------------------------------------------------------------------------------------ what a pass cannot do without
def _mean_len(c):
    """Committed tokens of a sequence: lengths that differ are spread evenly over the upper half of L."""
    return c["L"] * (0.75 if c.get("ragged") or (c["kind"] == "draft" and c["B"] > 1) else 1.0)


def _attention_work(S, rows, L, T, size):
    """One layer over `rows` sequences: K and V of the committed slots and the tree once, Q in, the output out."""
    return (2 * rows * (S["Hkv"] * (L + T) + S["Hq"] * T) * S["d"] * size, 4 * rows * S["Hq"] * T * (L + T) * S["d"])


def _layer_weights(S):
    return (S["Hq"] + 2 * S["Hkv"]) * S["d"] * S["H"] + S["Hq"] * S["d"] * S["H"] + 3 * S["inter"] * S["H"]


def _levels(T):
    parent = W.tree_from_branching(TREES[T], T)
    depth = W.tree_depths(parent)
    return [int((depth == j).sum()) for j in range(1, 4)]


def work(case):
    c, S = case, MODELS[case["model"]]
    B, T, V, H = c["B"], c["T"], S["V"], S["H"]
    size = 4 if S["dtype"] == torch.float32 else 2
    if c["kind"] == "attention":
        b, f = _attention_work(S, B, _mean_len(c), T, size)
        return dict(bytes=b, flops=f)
    if c["kind"] == "head":
        return dict(bytes=2 * V * H + 2 * B * T * H + 8 * B * T, flops=2 * B * T * V * H)
    if c["kind"] == "verify":
        b, f = _attention_work(S, B, _mean_len(c), T, size)
        # acceptance reads every logits row, sampling the draft rows too; a built tree reads the rows of its inner nodes
        rows = 4 * B * T * V * (2 if c["tau"] > 0 else 1)
        if c["build"] and c["tau"] == 0:
            rows += 4 * B * V * len(set(W.tree_from_branching(TREES[T], T)[1:].tolist()))
        return dict(bytes=c["layers"] * b + rows, flops=c["layers"] * f)
    if c["kind"] == "target":
        b, f = _attention_work(S, B, _mean_len(c), T, 2)
        weights = c["layers"] * _layer_weights(S) + V * H
        # sampling writes the logits and reads the draft rows
        return dict(bytes=2 * weights + c["layers"] * b + (12 * B * T * V if c["tau"] > 0 else 0), flops=2 * B * T * weights + c["layers"] * f)
    bytes_, flops = 0, 0
    for n in _levels(T):
        b, f = _attention_work(S, B * n, _mean_len(c), 1, 2)
        weights = 2 * H * H + _layer_weights(S) + V * H
        bytes_, flops = bytes_ + 2 * weights + b, flops + 2 * B * n * weights + f
    return dict(bytes=bytes_, flops=flops)


def _state_bytes(c):
    """Device memory of a state, roughly (three of them have to fit)."""
    S = MODELS[c["model"]]
    cache = lambda rows, layers: 4.0 * layers * rows * S["Hkv"] * _capacity(c["L"], c["T"]) * S["d"]
    if c["kind"] == "verify":
        return cache(c["B"], c["layers"]) + 16.0 * c["B"] * c["T"] * S["V"]
    if c["kind"] == "target":
        return 2.0 * c["layers"] * _layer_weights(S) + 4.0 * S["V"] * S["H"] + cache(c["B"], c["layers"]) + 12.0 * c["B"] * c["T"] * S["V"]
    if c["kind"] == "draft":
        return 6.0 * _layer_weights(S) + 12.0 * S["H"] ** 2 + 4.0 * S["V"] * S["H"] + cache(c["B"] * sum(_levels(c["T"])), 1)
    return 4.0 * S["V"] * S["H"] if c["kind"] == "head" else cache(c["B"], 1)


def tolerance(case):
    """Decisions, tokens and lengths are the same; float results as the data types give them: 32-bit sums, bf16 results of one
    attention, bf16 through a chain of layers (whose roundings feed the next layer)."""
    if case["model"] == "tiny":
        return {"rel": 1e-5}
    return {"rel": 2e-2} if case["kind"] in ("target", "draft") else {"rel": 1e-2}
