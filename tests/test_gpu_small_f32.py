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
