"""Scores of +inf: they rank first, ties among them go to the lower index, and the kept set below them is as
without them.  (The softmax over an infinite score is not a number, so only selections are compared.)"""
import numpy as np
import pytest
import torch

from paper_2106_06899_gb300 import topk as T

pytestmark = pytest.mark.gpu


def _check(idx, score, finite_scores, inf_keys, topk):
    # finite_scores [rows, keys] in fp64, -inf at the keys that score +inf
    n = min(len(inf_keys), topk)
    idx, score = idx.cpu().numpy(), score.cpu().numpy()
    assert np.isposinf(score[:, :n]).all() and np.isfinite(score[:, n:]).all()
    assert (idx[:, :n] == np.asarray(sorted(inf_keys))[:n]).all()
    want = np.sort(finite_scores.numpy(), axis=1)[:, ::-1][:, : topk - n]
    assert np.abs(score[:, n:] - want).max(initial=0.0) <= 1e-4 * np.abs(want).max(initial=1.0)


@pytest.mark.parametrize("dtype,d,Lq,Lk,topk", [("bf16", 64, 140, 900, 16), ("bf16", 128, 140, 5000, 16),
                                                ("bf16", 64, 140, 2000, 200), ("bf16", 64, 3, 20000, 16),
                                                ("f32", 64, 140, 900, 16)])
@pytest.mark.parametrize("n_inf", [1, 15, 16, 40])
def test_attention(dtype, d, Lq, Lk, topk, n_inf):
    g = torch.Generator().manual_seed(1080 + n_inf)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    q = (torch.rand(1, 2, Lq, d, generator=g) + 0.5).to(dt)
    k = torch.randn(1, 2, Lk, d, generator=g).to(dt)
    keys = torch.randperm(Lk, generator=g)[:n_inf].tolist()
    k[:, :, keys] = float("inf")
    v = torch.randn(1, 2, Lk, d, generator=g).to(dt)
    _, idx, score = T.attention(q.cuda(), k.cuda(), v.cuda(), topk, return_indices=True)
    T.topk_check()
    s = q.double() @ torch.nan_to_num(k, posinf=0.0).double().transpose(2, 3)
    s[..., keys] = -float("inf")
    _check(idx.reshape(-1, topk), score.reshape(-1, topk), s.reshape(-1, Lk), keys, topk)


@pytest.mark.parametrize("n_inf", [1, 15, 16, 40])
@pytest.mark.parametrize("N,dff", [(5, 700), (300, 9000)])
def test_ffn(N, dff, n_inf):
    topk, dm = 16, 128
    g = torch.Generator().manual_seed(1090 + n_inf)
    x = (torch.rand(N, dm, generator=g) + 0.5).bfloat16()
    w1 = torch.randn(dff, dm, generator=g).bfloat16()
    keys = torch.randperm(dff, generator=g)[:n_inf].tolist()
    w1[keys] = float("inf")
    w2 = torch.randn(dff, dm, generator=g).bfloat16()
    _, idx, score = T.ffn(x.cuda(), w1.cuda(), w2.cuda(), topk, return_indices=True)
    T.topk_check()
    s = x.double() @ torch.nan_to_num(w1, posinf=0.0).double().T
    s[:, keys] = -float("inf")
    _check(idx, score, s, keys, topk)
