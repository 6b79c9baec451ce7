"""The CTA-pair projection kernel (trees and prompts of more than 64 rows) at the edges of its tiles."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import anc_dev, i32, to_dev

pytestmark = pytest.mark.gpu


# one more row than the one-CTA kernel takes; N whose last 256-row tile has no row for the second CTA, or a few;
# K of one ragged block; the last row block short; several blocks and K ranges
@pytest.mark.parametrize("m,n,k", [(129, 132, 72), (160, 388, 64), (161, 256, 4096), (256, 128, 1376), (257, 1028, 200), (545, 4096, 11008)])
def test_gemm_of_many_rows(trj, m, n, k):
    g = synth.stream(m * n, "gemm")
    x = synth.round_bf16(g.standard_normal((m, k), dtype=np.float32))
    w = synth.round_bf16(g.standard_normal((n, k), dtype=np.float32) * 0.02)
    ws = torch.zeros(trj.lib().trj_gemm_workspace(m, n, k), dtype=torch.uint8, device="cuda")
    dx, dw = to_dev(x, "bf16"), to_dev(w, "bf16")
    y = trj.gemm(dx, dw, workspace=ws).cpu().numpy()
    assert int(ws[:4].view(torch.int32)[0]) == 0
    ref = x.astype(np.float64) @ w.astype(np.float64).T
    # fp32 accumulation of k products of magnitude |x||w|: error <= k * 2^-24 * (|x| . |w|), far below this for these k
    assert np.abs(y - ref).max() <= 1e-4 * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("rows,vocab", [(65, 1024), (96, 900), (97, 1156), (128, 1024)])
def test_step_of_many_rows_hi_lo_pairs_and_argmax(trj, rows, vocab):
    """Activations as bf16 pairs (two products per accumulator) and the arg-max candidates of the LM head's epilogue,
    with tied LM-head rows in one warp, in two warps, in the two CTAs of a pair and in two tiles."""
    from dataclasses import replace
    from paper_2406_17404_b200.decode import upload_weights
    cfg = replace(synth.TINY, dtype="bf16", vocab=vocab)
    layers = [synth.layer_weights(cfg, 5, l) for l in range(cfg.n_layers)]
    glob = dict(synth.global_weights(cfg, 5))
    lm = np.array(glob["lm_head"], np.float32)
    lm[5] *= 16.0                                            # wins for about half of the inputs (x16 is exact in bf16)
    for dup in (6, 40, 133, 300, vocab - 1):
        lm[dup] = lm[5]
    glob["lm_head"] = lm
    dl, dg = upload_weights(cfg, layers, glob)
    model = trj.Model(cfg, dl, dg, max_batch=1, max_seq=256, max_rows=128)
    f64 = lambda d: {k: np.asarray(v, np.float64) for k, v in d.items()}
    dec = oracle.Decoder(cfg, [f64(l) for l in layers], f64(glob))
    prompt = synth.prompt(9, 90, cfg.vocab)
    model.prefill(i32(prompt))
    cache = dec.new_cache(256)
    dec.forward_rows(cache, prompt, synth.chain_parents(len(prompt)))
    cache.seq_len = len(prompt)
    parent = synth.random_tree(rows, rows, 6, 4)
    tokens = synth.prompt(rows, rows, cfg.vocab)
    want = dec.forward_rows(cache, tokens, parent)
    depth, anc = trj.tree_from_parents(parent)
    out = model.verify_step(i32(tokens), i32(parent), i32(depth), anc_dev(anc), i32([0, rows]), max_rows=rows,
                            max_len=len(prompt) + rows, want_logits=True, want_margin=True)
    model.device_status()
    logits, pred = out["logits"].cpu().numpy(), out["node_argmax"].cpu().numpy()
    # q and K/V are stored as bf16 on both sides: two layers measure up to 5.8e-3 where logits are O(1); row 5 and its
    # copies are 16 times larger
    assert np.abs(logits - want).max() <= 2e-2 * max(1.0, np.abs(want).max())
    np.testing.assert_array_equal(pred, oracle.node_argmax(logits.astype(np.float64)))
    np.testing.assert_array_equal(out["margin"].cpu().numpy(), oracle.top2_margin(logits.astype(np.float64)).astype(np.float32))
    tied = np.isin(pred, [5, 6, 40, 133, 300, vocab - 1])
    assert tied.sum() >= 4 and (pred[tied] == 5).all()
