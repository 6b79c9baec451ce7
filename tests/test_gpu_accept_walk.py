"""The acceptance walk on trees whose depths are not those of the library's own builder."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import i32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 2, 33, 128])
@pytest.mark.parametrize("root_depth", [0, 3, 200, -1])
def test_the_root_is_accepted_at_depth_zero_whatever_it_carries(trj, rows, root_depth):
    """Only rows below the root compete for the deepest one: a depth at the root (absolute positions, say) must not be walked."""
    vocab = 500
    parent = synth.random_tree(rows, rows, min(6, rows - 1), 3) if rows > 1 else np.array([-1], np.int32)
    logits = torch.from_numpy(synth.logits(rows, rows, vocab)).cuda()
    pred = oracle.node_argmax(logits.cpu().numpy().astype(np.float64))
    tokens = synth.planted_tokens(2, parent, pred, vocab)
    depth = np.array(synth.node_depths(parent), np.int32)
    depth[0] = root_depth
    got = trj.argmax_accept(logits, i32(tokens), i32(parent), i32(depth), i32([0, rows]))
    k, path, bonus = oracle.accept_path(tokens, parent, pred)
    assert (int(got["k_acc"][0]), got["path"][0, :k + 1].tolist(), int(got["bonus"][0])) == (k, list(path), bonus)
    assert (got["path"][0, k + 1:] == -1).all()
