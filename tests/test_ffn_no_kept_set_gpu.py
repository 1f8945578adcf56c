"""Tokens that have no k scores (NaN): the call reports an error, those tokens' selections read as empty, and
every other token is as without them.  Run only on a build whose gather never reads a kept list that was not
written."""
import numpy as np
import pytest
import torch

import oracle
from paper_2106_06899_gb300 import topk as T
from paper_2106_06899_gb300 import workloads as W

from ._parity import check_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,dm,dff,topk", [(5, 64, 300, 64), (300, 256, 5000, 200), (40, 128, 20000, 1024)])
def test_nan_tokens(N, dm, dff, topk):
    x, w1, w2 = W.ffn_inputs(N, dm, dff, seed=1040 + topk)
    x[::3, 7] = float("nan")
    out, idx, score = T.ffn(x.cuda(), w1.cuda(), w2.cuda(), topk, return_indices=True)
    with pytest.raises(T.TopkError):
        T.topk_check()
    T.topk_check()  # reported once
    bad = np.arange(N) % 3 == 0
    assert (idx.cpu().numpy()[bad] == -1).all() and np.isneginf(score.cpu().numpy()[bad]).all()
    assert (out.cpu().numpy()[bad] == 0).all()
    rows = np.nonzero(~bad)[0]
    x2 = torch.nan_to_num(x)
    check_rows(q=x2[None, None], k=w1[None, None], v=w2[None, None], rows=rows, gpu_out=out.cpu().numpy()[rows],
               gpu_idx=idx.cpu().numpy()[rows], gpu_score=score.cpu().numpy()[rows], topk=topk, dtype="bf16",
               act=oracle.RELU)
    # the empty selections pass through the backward call
    dx, dw1, dw2 = T.ffn_bwd(x2.cuda(), w1.cuda(), w2.cuda(), torch.ones(N, dm, device="cuda"), idx, score)
    T.topk_check()
    assert torch.isfinite(dw1).all() and torch.isfinite(dw2).all() and (dx[torch.from_numpy(bad)] == 0).all()
