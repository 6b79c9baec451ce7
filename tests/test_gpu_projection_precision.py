"""Accumulation error of the projections against fp64.  The tensor core truncates when it adds to its accumulator, so a sum is
biased toward zero in proportion to the products added in a row; kernels spread long sums over several accumulators."""
from types import SimpleNamespace

import numpy as np
import pytest
import torch

import synth
from gpu_util import anc_dev, i32

pytestmark = pytest.mark.gpu

# 128 products of 16 in a row measure 2.1e-6 (2-norm, normal inputs; 1.8e-6 of it bias); adding the pieces to nearest is below 0.3e-6
IN_A_ROW = 2.5e-6


@pytest.mark.parametrize("m", [129, 256, 257, 600])
@pytest.mark.parametrize("n,k", [(4096, 4096), (22016, 4096), (4096, 11008), (1028, 1000)])
def test_gemm_of_many_rows(trj, m, n, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(m + n + k)
    x = torch.randn(m, k, generator=g, device="cuda", dtype=torch.bfloat16)
    w = torch.randn(n, k, generator=g, device="cuda", dtype=torch.bfloat16)
    ws = torch.zeros(trj.lib().trj_gemm_workspace(m, n, k), dtype=torch.uint8, device="cuda")
    y = trj.gemm(x, w, workspace=ws)[:, -1024:].double()
    ref = x.double() @ w[-1024:].double().T
    assert float((y - ref).norm() / ref.norm()) <= IN_A_ROW


@pytest.mark.parametrize("rows", [1, 9, 33, 40, 64, 65, 96, 128, 129, 160, 300, 512])
def test_projections_of_a_step(trj, rows):
    """A decoder whose attention adds nothing (wo = 0) and whose one layer's SwiGLU output is large beside the embedding: the logits go
    through gate/up (as a bf16 pair, alone or with SwiGLU in its epilogue), down and LM head, nothing is rounded to bf16 on the way."""
    d, f, vocab, n_seq = 4096, 11008, 4096, -(-rows // 128)
    c = SimpleNamespace(n_layers=1, d_model=d, n_heads=32, head_dim=128, d_ff=f, vocab=vocab, dtype="bf16", n_kv_heads=32, rope_theta=10000.0, rms_eps=1e-5)
    g = torch.Generator(device="cuda")
    g.manual_seed(rows)
    mat = lambda r, k, std: torch.randn(r, k, generator=g, device="cuda", dtype=torch.bfloat16).mul_(std)
    one = torch.ones(d, device="cuda")
    layer = {"attn_norm": one, "wqkv": mat(3 * d, d, 0.02), "wo": torch.zeros(d, d, device="cuda", dtype=torch.bfloat16), "mlp_norm": one,
             "w_gate_up": mat(2 * f, d, 0.02), "w_down": mat(d, f, 0.2)}
    embed, head = mat(vocab, d, 1.0), mat(vocab, d, 0.02)
    model = trj.Model(c, [layer], {"embed": embed, "lm_head": head, "final_norm": one}, max_batch=n_seq, max_seq=160, max_rows=128)
    off = [rows * i // n_seq for i in range(n_seq + 1)]
    parents = [synth.random_tree(i, m, min(5, m - 1), 8) if m > 1 else np.array([-1], np.int32) for i, m in enumerate(np.diff(off))]
    trees = [trj.tree_from_parents(p) for p in parents]
    tokens = i32(synth.prompt(rows, rows, vocab))
    out = model.verify_step(tokens, i32(np.concatenate(parents)), i32(np.concatenate([t[0] for t in trees])), anc_dev(np.concatenate([t[1] for t in trees])),
                            i32(off), max_rows=int(max(np.diff(off))), max_len=130, want_logits=True)
    model.device_status()
    rms = lambda h: h * torch.rsqrt((h * h).mean(-1, keepdim=True) + c.rms_eps)
    h = embed[tokens.long()].double()
    gu = rms(h) @ layer["w_gate_up"].double().T
    ref = rms(h + (torch.nn.functional.silu(gu[:, :f]) * gu[:, f:]) @ layer["w_down"].double().T) @ head.double().T
    # Inputs rounded to 16 bits (uniform within 2^-18 relative to the top of their binade: 1.4e-6 rms) for gate/up, where gate and up
    # share the error, down and LM head, independent: 1.4e-6 * sqrt(4 + 1 + 1) = 3.5e-6.  Accumulation: the LM head's in full; of gate's and up's,
    # which add up in SwiGLU, and down's the last RMSNorm divides out the common bias and leaves the spread, (2 + 1) / 3 of it at most.
    err = float((out["logits"].double() - ref).norm() / ref.norm())
    print("rows", rows, "error", err)
    assert err <= 3.5e-6 + 2 * IN_A_ROW
