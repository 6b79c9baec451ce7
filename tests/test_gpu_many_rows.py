"""Element-wise kernels on either side of the row counts where their form changes (one row per SM), through a decoder."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import anc_dev, i32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,heads", [("f32", 4), ("bf16", 2)])
@pytest.mark.parametrize("rows", [148, 149, 300])
def test_prompt_cache_rows_and_first_token(trj, dtype, heads, rows):
    """A prompt of `rows` tokens is one forward of that many rows: every layer's K/V rows (rotary table, RMSNorm and SwiGLU of
    many rows) and the greedy token against the oracle."""
    from dataclasses import replace
    from paper_2406_17404_b200.decode import upload_weights
    cfg = replace(synth.TINY, dtype=dtype, n_kv_heads=heads)
    layers = [synth.layer_weights(cfg, 3, l) for l in range(cfg.n_layers)]
    glob = synth.global_weights(cfg, 3)
    model = trj.Model(cfg, *upload_weights(cfg, layers, glob), max_batch=1, max_seq=512, max_rows=128)
    f64 = lambda d: {k: np.asarray(v, np.float64) for k, v in d.items()}
    dec = oracle.Decoder(cfg, [f64(l) for l in layers], f64(glob))
    prompt = synth.prompt(rows, rows, cfg.vocab)
    first = int(model.prefill(i32(prompt)).item())
    cache = dec.new_cache(512)
    want = dec.forward_rows(cache, prompt, synth.chain_parents(rows))
    k, v = (c[:, 0, :, :rows].float().cpu().numpy() for c in (model.k_cache, model.v_cache))
    # bf16: q and K/V roundings that fall the other way (2^-8 relative each) reach the next layer as input errors of that size
    # times its O(0.3) values, then each value is rounded itself: one bf16 step (2^-7) of the value, or of 0.25 below that;
    # fp32: sums of 256 and 688 products
    for got, ref in ((k, cache.k), (v, cache.v)):
        ref = np.asarray(ref)[:, :, :rows]
        tol = np.maximum(np.abs(ref), 0.25) * 2.0 ** -7 if dtype == "bf16" else 2e-5
        assert (np.abs(got - ref) <= tol).all()
    margin = oracle.top2_margin(np.asarray(want)[-1:])[0]
    assert margin < 1e-2 or first == int(oracle.node_argmax(np.asarray(want)[-1:])[0])


@pytest.mark.parametrize("rows", [148, 149, 592, 593])
def test_argmax_of_many_rows(trj, rows):
    """Either side of the row counts where a row gets fewer threads; ties inside a row, best and runner-up in its last elements."""
    b, vocab = 8, 1003
    logits = torch.from_numpy(synth.logits(rows, rows, vocab)).cuda().to(torch.bfloat16)
    logits[::3, 7] = logits[::3, 900] = 9.0                  # equal maxima: the smaller id
    logits[1::3, vocab - 1] = 8.0
    logits[1::3, vocab - 2] = 7.5
    off = [rows * i // b for i in range(b + 1)]
    parents = [synth.random_tree(i, off[i + 1] - off[i], 5, 4) for i in range(b)]
    host = logits.float().cpu().numpy().astype(np.float64)
    pred = oracle.node_argmax(host)
    tokens = np.concatenate([synth.planted_tokens(i, p, pred[off[i]:off[i + 1]], vocab) for i, p in enumerate(parents)])
    got = trj.argmax_accept(logits, i32(tokens), i32(np.concatenate(parents)), i32(np.concatenate([synth.node_depths(p) for p in parents])), i32(off))
    np.testing.assert_array_equal(got["node_argmax"].cpu().numpy(), pred)
    np.testing.assert_array_equal(got["margin"].cpu().numpy(), oracle.top2_margin(host).astype(np.float32))
    for i, p in enumerate(parents):
        k, path, bonus = oracle.accept_path(tokens[off[i]:off[i + 1]], p, pred[off[i]:off[i + 1]])
        assert (int(got["k_acc"][i]), got["path"][i, :k + 1].tolist(), int(got["bonus"][i])) == (k, list(path), bonus)


@pytest.mark.parametrize("rows", [256, 257, 300, 512])
def test_rotary_and_swiglu_in_the_projections_epilogue(trj, rows):
    """Either side of one row block of 256: a ragged batch of trees through a decoder whose heads are 128 wide (grouped keys) and
    whose d_ff ends inside a tile.  K/V rows of every layer (the second layer's rest on the first one's SwiGLU) and logits."""
    from dataclasses import replace
    from paper_2406_17404_b200.decode import upload_weights
    cfg = replace(synth.TINY, dtype="bf16", n_heads=4, n_kv_heads=2, head_dim=128, d_ff=328)
    layers = [synth.layer_weights(cfg, 4, l) for l in range(cfg.n_layers)]
    glob = synth.global_weights(cfg, 4)
    n_seq, prefix = 5, 9
    model = trj.Model(cfg, *upload_weights(cfg, layers, glob), max_batch=n_seq, max_seq=160, max_rows=128)
    f64 = lambda d: {k: np.asarray(v, np.float64) for k, v in d.items()}
    dec = oracle.Decoder(cfg, [f64(l) for l in layers], f64(glob))
    off = [rows * i // n_seq + (3 if 0 < i < n_seq else 0) for i in range(n_seq + 1)]
    parents = [synth.random_tree(i, off[i + 1] - off[i], 5, 4) for i in range(n_seq)]
    tokens = synth.prompt(rows, rows, cfg.vocab)
    trees = [trj.tree_from_parents(p) for p in parents]
    words = max(t[1].shape[1] for t in trees)
    anc = np.concatenate([np.pad(t[1], ((0, 0), (0, words - t[1].shape[1]))) for t in trees])
    caches = []
    for b in range(n_seq):
        prompt = synth.prompt(50 + b, prefix + b, cfg.vocab)
        model.prefill(i32(prompt), b=b)
        caches.append(dec.new_cache(160))
        dec.forward_rows(caches[b], prompt, synth.chain_parents(prefix + b))
        caches[b].seq_len = prefix + b
    out = model.verify_step(i32(tokens), i32(np.concatenate(parents)), i32(np.concatenate([t[0] for t in trees])), anc_dev(anc), i32(off),
                            max_rows=max(np.diff(off)), max_len=prefix + n_seq + max(np.diff(off)), want_logits=True)
    model.device_status()
    logits = out["logits"].float().cpu().numpy()
    for b in range(n_seq):
        n, m = prefix + b, off[b + 1] - off[b]
        want = dec.forward_rows(caches[b], tokens[off[b]:off[b + 1]], parents[b])
        # roundings that fall the other way, as for the prompt above
        for got, ref in ((model.k_cache, caches[b].k), (model.v_cache, caches[b].v)):
            got, ref = got[:, b, :, n:n + m].float().cpu().numpy(), np.asarray(ref)[:, :, n:n + m]
            assert (np.abs(got - ref) <= np.maximum(np.abs(ref), 0.25) * 2.0 ** -7).all()
            assert float(model.k_cache[:, b, :, n + m:].abs().max()) == 0.0
        assert np.abs(logits[off[b]:off[b + 1]] - np.asarray(want)).max() <= 2e-2


@pytest.mark.parametrize("rows", [1, 33, 64])
@pytest.mark.parametrize("d_ff", [7104, 7112, 9176, 9464, 9472, 9480, 18944, 18952])
def test_swiglu_of_few_rows_in_the_projections_epilogue(trj, d_ff, rows):
    """Either side of the range of d_ff whose items fit the grid (24 x 296 < d_ff <= 64 x 296: items of 32 to 64 gate rows, in
    eights; of 32 rows up to 32 x 296), ragged last items, both ends of the row range: logits of a two-layer decoder."""
    from dataclasses import replace
    from paper_2406_17404_b200.decode import upload_weights
    cfg = replace(synth.TINY, dtype="bf16", n_heads=2, n_kv_heads=2, head_dim=64, d_model=128, d_ff=d_ff)
    layers = [synth.layer_weights(cfg, 5, l) for l in range(cfg.n_layers)]
    glob = synth.global_weights(cfg, 5)
    model = trj.Model(cfg, *upload_weights(cfg, layers, glob), max_batch=1, max_seq=160, max_rows=128)
    f64 = lambda d: {k: np.asarray(v, np.float64) for k, v in d.items()}
    dec = oracle.Decoder(cfg, [f64(l) for l in layers], f64(glob))
    prompt, parent = synth.prompt(7, 9, cfg.vocab), synth.random_tree(rows, rows, min(5, rows - 1), 4) if rows > 1 else np.array([-1], np.int32)
    tokens = synth.prompt(rows, rows, cfg.vocab)
    model.prefill(i32(prompt))
    cache = dec.new_cache(160)
    dec.forward_rows(cache, prompt, synth.chain_parents(9))
    cache.seq_len = 9
    depth, anc = trj.tree_from_parents(parent)
    out = model.verify_step(i32(tokens), i32(parent), i32(depth), anc_dev(anc), i32([0, rows]), max_rows=rows, max_len=9 + rows, want_logits=True)
    model.device_status()
    want = np.asarray(dec.forward_rows(cache, tokens, parent))
    # the bf16 bound of the model tests: roundings of q and K/V that fall the other way
    assert np.abs(out["logits"].float().cpu().numpy() - want).max() <= 2e-2
    got = model.k_cache[:, 0, :, 9:9 + rows].float().cpu().numpy()
    ref = np.asarray(cache.k)[:, :, 9:9 + rows]
    assert (np.abs(got - ref) <= np.maximum(np.abs(ref), 0.25) * 2.0 ** -7).all()


@pytest.mark.parametrize("d_ff,rows,fused", [(7104, 1, False), (7112, 1, True), (7112, 40, True), (7112, 41, False), (9472, 40, True), (9472, 41, False),
                                             (9480, 41, True), (9480, 64, True), (18944, 64, True), (18952, 33, False)])
def test_which_projections_take_swiglu_into_their_epilogue(trj, d_ff, rows, fused):
    """By the launches of a step: one less per layer than a decoder whose d_ff is below the range."""
    from dataclasses import replace
    from paper_2406_17404_b200.decode import upload_weights

    def launches(f):
        cfg = replace(synth.TINY, dtype="bf16", n_heads=2, n_kv_heads=2, head_dim=64, d_model=128, d_ff=f)
        model = trj.Model(cfg, *upload_weights(cfg, [synth.layer_weights(cfg, 5, l) for l in range(cfg.n_layers)], synth.global_weights(cfg, 5)),
                          max_batch=1, max_seq=160, max_rows=128)
        parent = synth.chain_parents(rows)
        depth, anc = trj.tree_from_parents(parent)
        before = trj.launch_count()
        model.verify_step(i32(np.arange(rows)), i32(parent), i32(depth), anc_dev(anc), i32([0, rows]), max_rows=rows, max_len=rows)
        model.device_status()
        return trj.launch_count() - before, cfg.n_layers

    apart, n_layers = launches(2048)
    assert launches(d_ff)[0] == apart - (n_layers if fused else 0)
