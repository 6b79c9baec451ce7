"""fp32 products of few tiles (the latency-bound kernel) at the edges of its tiles, and the first shapes past its range."""
import numpy as np
import pytest
import torch

import synth
from gpu_util import to_dev

pytestmark = pytest.mark.gpu


# one element, a tile more and a tile less than full, K of one vector and K at and past the bound, the last and the
# first tile count on either side of the rule (96 tiles of 64 x 64)
@pytest.mark.parametrize("m,n,k", [(1, 1, 4), (15, 7, 12), (16, 8, 1024), (17, 9, 688), (33, 1376, 256), (11, 770, 1028),
                                   (512, 768, 64), (512, 832, 64), (3, 5, 10)])
def test_small_f32_gemm(trj, m, n, k):
    g = synth.stream(m * n + k, "gemm")
    x, w = g.standard_normal((m, k), dtype=np.float32), g.standard_normal((n, k), dtype=np.float32)
    ws = torch.zeros(max(256, trj.lib().trj_gemm_workspace(m, n, k)), dtype=torch.uint8, device="cuda")
    out = torch.full((m + 1, n), 7.0, device="cuda")         # a row more than asked: it must stay as it is
    trj.gemm(to_dev(x, "f32"), to_dev(w, "f32"), out=out[:m], workspace=ws)
    ref = x.astype(np.float64) @ w.astype(np.float64).T
    bound = k * 2.0 ** -24 * (np.abs(x).astype(np.float64) @ np.abs(w).astype(np.float64).T) + 1e-30
    assert (np.abs(out[:m].cpu().numpy() - ref) <= bound).all()     # k roundings of fp32 sums, the worst case
    assert (out[m] == 7.0).all()


# K of the norms and of SwiGLU at and past the bound of 1024 (past it: the separate kernels), one row, a tile of 16 rows and
# one more, several row tiles
@pytest.mark.parametrize("d_model,d_ff,rows", [(256, 688, 1), (256, 688, 16), (256, 688, 17), (256, 688, 128), (256, 1024, 11),
                                               (256, 1100, 11), (1024, 260, 11), (1032, 260, 11)])
def test_norm_and_swiglu_inside_the_small_projections(trj, d_model, d_ff, rows):
    from dataclasses import replace
    import oracle
    from gpu_util import anc_dev, i32
    from paper_2406_17404_b200.decode import upload_weights
    cfg = replace(synth.TINY, d_model=d_model, d_ff=d_ff, n_kv_heads=2)
    layers = [synth.layer_weights(cfg, 6, l) for l in range(cfg.n_layers)]
    glob = synth.global_weights(cfg, 6)
    model = trj.Model(cfg, *upload_weights(cfg, layers, glob), max_batch=1, max_seq=256, max_rows=128)
    f64 = lambda d: {k: np.asarray(v, np.float64) for k, v in d.items()}
    dec = oracle.Decoder(cfg, [f64(l) for l in layers], f64(glob))
    prompt, tokens = synth.prompt(8, 9, cfg.vocab), synth.prompt(rows, rows, cfg.vocab)
    parent = synth.random_tree(rows, rows, min(5, rows - 1), 4) if rows > 1 else np.array([-1], np.int32)
    cache = dec.new_cache(256)
    lg = np.asarray(dec.forward_rows(cache, prompt, synth.chain_parents(9)))
    cache.seq_len = 9
    first = int(model.prefill(i32(prompt)).item())           # one row reaches the LM head
    assert first == int(oracle.node_argmax(lg[-1:])[0]) or oracle.top2_margin(lg[-1:])[0] < 1e-3
    depth, anc = trj.tree_from_parents(parent)
    out = model.verify_step(i32(tokens), i32(parent), i32(depth), anc_dev(anc), i32([0, rows]), max_rows=rows, max_len=9 + rows, want_logits=True)
    want = np.asarray(dec.forward_rows(cache, tokens, parent))
    # the fp32 bounds of the model tests
    assert np.abs(out["logits"].cpu().numpy() - want).max() < 1e-3
    for got, ref in ((model.k_cache, cache.k), (model.v_cache, cache.v)):
        assert np.abs(got[:, 0, :, :9 + rows].cpu().numpy() - np.asarray(ref)[:, :, :9 + rows]).max() < 1e-4
