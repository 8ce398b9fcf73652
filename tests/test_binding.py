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


def test_of_several_wrong_arguments_the_first_is_named(s4c_lib):
    # the order of the call decides, not the compiler's order of evaluation, and no CUDA call is made for arguments that are refused
    from paper_2506_14158_b200 import s4c

    q, kv = torch.zeros(1, 4, 8, 64), torch.zeros(1, 2, 128, 64)
    i, par = torch.zeros(1, dtype=torch.int32), torch.zeros(1, 8, dtype=torch.int32)
    with pytest.raises(ValueError, match="^q must be a CUDA tensor"):
        s4c.tree_attention(q, kv, kv, i, par, max_cache_len=128.0)
    with pytest.raises(ValueError, match="^hidden must be a CUDA tensor"):
        s4c.lm_head_greedy(torch.zeros(3, 64), torch.zeros(5, 64))
    with pytest.raises(ValueError, match="^target_token must be a CUDA tensor"):
        s4c.tree_accept_tokens(par, par, par, 100)
    with pytest.raises(ValueError, match="^target_logits must be a CUDA tensor"):
        s4c.tree_accept(torch.zeros(1, 8, 10), None, par, par, 0.0)
    with pytest.raises(RuntimeError, match="ambiguous"):  # what `rows` itself raises, not a SystemError
        s4c.tree_attention(q, kv, kv, i, par, rows=torch.ones(2))
    with pytest.raises(IndexError):
        s4c.kv_compact(None, None, 0, (1, 2, 128, 64), torch.float32, i, i, i, 8, status=i)


def test_a_binary_of_another_torch_is_neither_kept_nor_loaded(s4c_lib, monkeypatch, tmp_path):
    import os
    import subprocess
    import sys

    from paper_2506_14158_b200 import _build

    ran = []

    def compiler(cmd, check):
        ran.append(cmd)
        open(cmd[cmd.index("-o") + 1], "w").close()

    monkeypatch.setattr(_build, "_HERE", str(tmp_path))
    monkeypatch.setattr(_build.subprocess, "run", compiler)
    build = lambda: (ran.clear(), _build._build_bind(), len(ran))[-1]
    assert build() == 1 and build() == 0
    monkeypatch.setattr(torch, "__version__", "0.0.0")  # the sources are older than the binary all the same
    assert build() == 1 and build() == 0
    monkeypatch.undo()
    assert os.path.exists(_build.bind_path())
    code = "import torch; torch.__version__ = '0.0.0'; import paper_2506_14158_b200.s4c"
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, cwd=os.path.dirname(_build._HERE))
    assert r.returncode != 0 and "ImportError" in r.stderr and "0_0_0" in r.stderr
