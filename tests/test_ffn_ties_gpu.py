"""Tokens whose scores tie (padding: all-zero tokens) keep about k candidates per slice, so that they take no
longer than others; kept sets with ties everywhere, with k below and above a key tile's 256 keys."""
import numpy as np
import pytest
import torch

import oracle
from paper_2106_06899_gb300 import topk as T
from paper_2106_06899_gb300 import workloads as W

from ._parity import check_rows

pytestmark = pytest.mark.gpu


def _ms(x, w1, w2, topk):
    times = []
    for _ in range(8):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        T.ffn(x, w1, w2, topk)
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b))
    T.topk_check()
    return float(np.median(times[3:]))


def test_all_zero_tokens_take_no_longer():
    topk = 64
    x, w1, w2 = (t.cuda() for t in W.ffn_inputs(2048, 512, 16384, seed=1020))
    assert _ms(torch.zeros_like(x), w1, w2, topk) <= 1.5 * _ms(x, w1, w2, topk)


@pytest.mark.parametrize("topk", [3, 255, 256, 257, 700])
def test_few_distinct_scores(topk):
    # scores of four values: ties everywhere, and bounds that sit on a tied value
    N, dm, dff = 150, 64, 9000
    g = torch.Generator().manual_seed(1030 + topk)
    x, w1 = torch.zeros(N, dm), torch.zeros(dff, dm)
    x[:, 0] = torch.randint(0, 3, (N,), generator=g).float()
    w1[:, 0] = torch.randint(-1, 3, (dff,), generator=g).float()
    w2 = torch.randn(dff, dm, generator=g) / 64
    x, w1, w2 = x.bfloat16(), w1.bfloat16(), w2.bfloat16()
    out, idx, score = T.ffn(x.cuda(), w1.cuda(), w2.cuda(), topk, return_indices=True)
    T.topk_check()
    ref = oracle.ffn(x, w1, w2, topk)
    assert np.array_equal(idx.cpu().numpy(), ref["idx"])
    assert np.array_equal(score.cpu().double().numpy(), ref["score"])
    check_rows(q=x[None, None], k=w1[None, None], v=w2[None, None], rows=np.arange(N), gpu_out=out.cpu().numpy(),
               gpu_idx=idx.cpu().numpy(), gpu_score=score.cpu().numpy(), topk=topk, dtype="bf16", act=oracle.RELU,
               ref=ref)
