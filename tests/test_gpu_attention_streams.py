"""Tree attention on two streams per CTA: batches as whole heads and as equal shares, trees on either side of the 64-row line,
streams without work, segments that change inside a stream, programmatic launches back to back."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import AttnCase
from test_gpu_ops import TOL, check_attention

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h,hk,prefixes,rows", [
    (32, 32, [130] * 8, [40] * 8),                        # 256 heads of two tiles on 296 streams: whole heads, paired from both ends
    (32, 8, [100, 300, 500, 700, 900], [64, 1, 33, 32, 9]),      # whole heads of one to eight tiles
    (16, 16, [3000, 40, 1], [16, 64, 2]),                 # one long sequence: shares that cut heads, pieces merged afterwards
    (4, 4, list(range(0, 64)), [1 + i % 5 for i in range(64)]),  # as many sequences as a call takes
    (2, 2, [5, 0, 700], [65, 128, 3]),                    # wide streams in a batch; a tree without a prefix
    (40, 40, [260] * 9, [20] * 9),                        # 360 heads: more than streams, several per stream
])
def test_batches(trj, h, hk, prefixes, rows):
    parents = [synth.random_tree(90 + i, m, min(6, m - 1), 3) if m > 1 else np.array([-1], np.int32) for i, m in enumerate(rows)]
    case = AttnCase(trj, 11, h, 128, prefixes, rows, parents, "bf16", pad=3, kv_heads=hk)
    seqs = None if len(rows) <= 9 else [0, 1, 17, 40, 63]
    check_attention(trj, case, heads=None if h <= 4 else [0, 1, h // 2, h - 1], seqs=seqs)


@pytest.mark.parametrize("s,m", [(0, 1), (0, 64), (0, 65), (0, 128), (70, 58), (127, 1), (128, 64), (63, 65), (900, 64), (900, 65), (2500, 128)])
def test_one_sequence(trj, s, m):
    """1 to 21 tiles on the eight streams of a head's cluster; 64 and 65 rows take different kernels."""
    parent = synth.random_tree(s + m, m, min(8, m - 1), 3) if m > 1 else np.array([-1], np.int32)
    check_attention(trj, AttnCase(trj, 12, 32, 128, [s], [m], [parent], "bf16", pad=2), heads=[0, 9, 31])


def test_calls_back_to_back_see_each_others_results(trj):
    """An op-level call is set up while the kernel before it ends: it must still read what that kernel wrote.  Each call's q
    is the call before's output."""
    m, s = 48, 700
    case = AttnCase(trj, 13, 8, 128, [s], [m], [synth.random_tree(5, m, 6, 3)], "bf16")
    kw = dict(max_rows=case.max_rows, max_len=case.max_len)
    q, ws = case.q, torch.zeros(trj.tree_attention_workspace(m, 1, 8, 128, case.max_len), dtype=torch.uint8, device="cuda")
    step = lambda x: trj.tree_attention(x, case.k, case.v, case.seq_len, case.row_off, case.anc, workspace=ws, **kw)
    chained = q
    for _ in range(20):
        chained = step(chained)
    apart = q
    for _ in range(20):
        apart = step(apart)
        torch.cuda.synchronize()
    assert torch.equal(chained, apart)


def test_one_workspace_for_batches_of_other_sizes(trj):
    """The record of who worked on which head, and the pieces, of one batch must not reach the next one: batches of other B and H,
    split heads in each, through one workspace that starts as garbage."""
    cases = [AttnCase(trj, 20 + i, h, 128, prefixes, rows, [synth.random_tree(30 + i + j, m, min(6, m - 1), 3) for j, m in enumerate(rows)], "bf16", pad=1)
             for i, (h, prefixes, rows) in enumerate([(16, [3000, 40, 1], [16, 64, 2]), (4, [900, 1300], [20, 30]), (32, [100, 2500, 7, 600], [33, 9, 70, 12])])]
    need = max(trj.tree_attention_workspace(sum(c.rows), len(c.rows), c.h, 128, c.max_len) for c in cases)
    ws = torch.full((need,), 0x7f, dtype=torch.uint8, device="cuda")
    ws[:256] = 0                                             # the status word
    apart = [c.run(trj) for c in cases]
    together = [c.run(trj, workspace=ws) for c in cases + cases]
    for got, want in zip(together, apart + apart):
        assert torch.equal(got, want)
    for c in cases:
        check_attention(trj, c, heads=[0, c.h - 1])
