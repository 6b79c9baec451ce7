"""Arg-max of logits that are infinite or NaN, by every route that a step's rows can take: candidates of the LM head's epilogue
(one-CTA and pair kernel), logits of an fp32 decoder, op level.  NaN is passed over; a prediction is always an id of the
vocabulary, since the next step reads its embedding."""
from dataclasses import replace

import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import anc_dev, i32

pytestmark = pytest.mark.gpu
ROUTES = [("bf16", 9), ("bf16", 64), ("bf16", 65), ("bf16", 96), ("bf16", 128), ("f32", 11), ("f32", 128)]


def verify(trj, dtype, rows, lm_head, final_norm):
    from paper_2406_17404_b200.decode import upload_weights
    cfg = replace(synth.TINY, dtype=dtype, vocab=lm_head.shape[0])
    glob = dict(synth.global_weights(cfg, 5), lm_head=lm_head, final_norm=final_norm)
    model = trj.Model(cfg, *upload_weights(cfg, [synth.layer_weights(cfg, 5, l) for l in range(cfg.n_layers)], glob), max_batch=1, max_seq=256, max_rows=128)
    model.prefill(i32(synth.prompt(9, 20, cfg.vocab)))
    parent = synth.random_tree(rows, rows, 6, 4)
    depth, anc = trj.tree_from_parents(parent)
    out = model.verify_step(i32(synth.prompt(rows, rows, cfg.vocab)), i32(parent), i32(depth), anc_dev(anc), i32([0, rows]), max_rows=rows,
                            max_len=20 + rows, want_logits=True, want_margin=True)
    model.device_status()
    return out["logits"].cpu().numpy(), out["node_argmax"].cpu().numpy(), out["margin"].cpu().numpy()


@pytest.mark.parametrize("dtype,rows", ROUTES)
def test_nan_logits_are_passed_over(trj, dtype, rows):
    lm = np.array(synth.global_weights(replace(synth.TINY, dtype=dtype), 5)["lm_head"], np.float32)
    for at in (0, 3, 500, lm.shape[0] - 1):                  # the first and the last id, inside a warp's 32
        lm[at] = np.nan
    lm[64:96] = np.nan                                       # all of a warp's
    logits, pred, margin = verify(trj, dtype, rows, lm, np.ones(synth.TINY.d_model, np.float32))
    assert np.isnan(logits[:, 3]).all() and not np.isnan(logits[:, 1]).any()
    host = np.where(np.isnan(logits), -np.inf, logits).astype(np.float64)
    np.testing.assert_array_equal(pred, oracle.node_argmax(host))
    np.testing.assert_array_equal(margin, oracle.top2_margin(host).astype(np.float32))


@pytest.mark.parametrize("sign", [-1, 1])
@pytest.mark.parametrize("dtype,rows", ROUTES)
def test_rows_of_infinite_logits(trj, dtype, rows, sign):
    """Every id has the same weights and they overflow: rows of +inf or -inf (with the other sign the other way round), all
    tied, so id 0 wins."""
    lm = np.zeros((1024, synth.TINY.d_model), np.float32)
    lm[:, 0] = synth.round_bf16(np.float32(sign * 3e38).reshape(1))[0]
    gain = np.ones(synth.TINY.d_model, np.float32)
    gain[0] = 8.0                                            # the high half overflows, the low half of a bf16 pair does not
    logits, pred, _ = verify(trj, dtype, rows, lm, gain)
    assert np.isinf(logits).all(1).any() and (logits == logits[:, :1]).all()
    assert (pred == 0).all()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("vocab", [1003, 1024])
def test_op_level(trj, dtype, vocab):
    rows = 12
    logits = torch.from_numpy(synth.logits(3, rows, vocab)).cuda().to(dtype)
    logits[0] = -torch.inf
    logits[1] = torch.nan
    logits[2, ::2] = torch.nan
    logits[3, 5] = logits[3, 9] = torch.inf
    logits[4] = -torch.inf
    logits[4, 700] = -1.0
    parent = synth.random_tree(rows, rows, 4, 3)
    host = logits.double().cpu().numpy()
    pred = oracle.node_argmax(np.where(np.isnan(host), -np.inf, host))
    got = trj.argmax_accept(logits, i32(synth.planted_tokens(1, parent, pred, vocab)), i32(parent), i32(synth.node_depths(parent)), i32([0, rows]))
    np.testing.assert_array_equal(got["node_argmax"].cpu().numpy(), pred)
