"""Op-level calls inside a stream capture, as a program with its own decoder makes them: behind kernels of other libraries, behind
a join of two streams, behind copies.  They are launched programmatically: a replay must read what the replayed predecessors wrote."""
import numpy as np
import pytest
import torch

import synth
from gpu_util import AttnCase, i32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prefixes,rows", [([700], [40]), ([900, 300, 1500], [20, 33, 64])])
def test_captured_ops_equal_eager_ones(trj, prefixes, rows):
    vocab, heads, n = 1000, 8, len(rows)
    total = sum(rows)
    parents = [synth.random_tree(5 + i, m, 6, 3) for i, m in enumerate(rows)]
    case = AttnCase(trj, 31, heads, 128, prefixes, rows, parents, "bf16")
    depth = i32(np.concatenate([synth.node_depths(p) for p in parents]))
    par, tokens = i32(np.concatenate(parents)), i32(np.arange(total) % vocab)
    ws = torch.zeros(trj.tree_attention_workspace(total, n, heads, 128, case.max_len), dtype=torch.uint8, device="cuda")
    aws = torch.zeros(trj.argmax_accept_workspace(total, n), dtype=torch.uint8, device="cuda")
    q0, w = torch.zeros_like(case.q), torch.randn(heads * 128, vocab, device="cuda", dtype=torch.bfloat16)
    k, v, length = case.k.clone()[None], case.v.clone()[None], case.seq_len.clone()

    def program(side):
        here = torch.cuda.current_stream()
        side.wait_stream(here)
        with torch.cuda.stream(side):
            q = q0 * 0.5 + 1.0                               # on the other stream
        k.copy_(case.k[None])                                # copies ahead of the join, on this one
        v.copy_(case.v[None])
        length.copy_(case.seq_len)
        here.wait_stream(side)
        out = trj.tree_attention(q, k[0], v[0], length, case.row_off, case.anc, max_rows=case.max_rows, max_len=case.max_len, workspace=ws)
        logits = out.view(total, -1) @ w
        got = trj.argmax_accept(logits, tokens, par, depth, case.row_off, workspace=aws)
        trj.compact_rows(k, v, length, got["k_acc"], got["path"])
        return out, got["node_argmax"], got["k_acc"], got["path"], k, v, length

    main, side = torch.cuda.Stream(), torch.cuda.Stream()
    main.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(main):
        q0.copy_(case.q)
        program(side)                                        # warm-up outside the capture
        main.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=main):
            held = program(side)
        for seed in range(4):
            g = torch.Generator(device="cuda")
            g.manual_seed(seed)
            q0.normal_(generator=g)
            graph.replay()
            replayed = [t.clone() for t in held]
            eager = [t.clone() for t in program(side)]
            main.synchronize()
            for a, b in zip(replayed, eager):
                assert torch.equal(torch.nan_to_num(a), torch.nan_to_num(b))
