"""The top-k FF layer's candidate lists at the edges of their tiles: slices of a single ragged tile, fewer
candidates than a slice's share of k, tokens that keep nothing yet when the histogram starts, and the
finalize's in-memory selection.  Against the CPU oracle under the parity rules of _parity.py."""
import numpy as np
import pytest
import torch

import oracle
from paper_2106_06899_gb300 import topk as T
from paper_2106_06899_gb300 import workloads as W

from ._parity import check_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,d_model,d_ff,topk", [(5, 64, 255, 255), (130, 64, 257, 200), (129, 64, 513, 3),
                                                 (300, 64, 5000, 1), (40, 128, 20000, 700), (1, 64, 70000, 1024)])
@pytest.mark.parametrize("dist", ["ffn", "integer"])
def test_lists(N, d_model, d_ff, topk, dist):
    x, w1, w2 = W.ffn_inputs(N, d_model, d_ff, seed=800 + topk, dist=dist)
    if dist == "integer":
        w2 = w2 / 16  # exact: keeps outputs of integer-sized scores near 1
    x[0] = 0  # every score of a zero token ties
    out, idx, score = T.ffn(x.cuda(), w1.cuda(), w2.cuda(), topk, return_indices=True)
    T.topk_check()
    rows = np.arange(N)
    check_rows(q=x[None, None], k=w1[None, None], v=w2[None, None], rows=rows, gpu_out=out.cpu().numpy(),
               gpu_idx=idx.cpu().numpy(), gpu_score=score.cpu().numpy(), topk=topk, dtype="bf16", act=oracle.RELU)
    assert torch.equal(idx[0].cpu(), torch.arange(topk, dtype=torch.int32))
