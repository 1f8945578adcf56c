"""The bound pass of the tensor-core attention kernels at the sizes where a tile's slots and the class count
nearly miss each other (the class count is a fraction of the warp's memory, or the bound covers only a few
tiles): several units per CTA, early units of causal calls, key counts, and a row whose k-th score is
supported by one key.  Against the CPU oracle, as in test_attn_lists_gpu.py."""
import numpy as np
import pytest
import torch

import oracle
from paper_2106_06899_gb300 import topk as T
from paper_2106_06899_gb300 import workloads as W

from .test_attn_lists_gpu import _outputs_match, _selection_matches

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("topk,Lk,causal", [(292, 2500, False), (300, 3000, False), (320, 4700, False),
                                            (340, 4096, True), (24, 300, False), (5, 200, False)])
def test_units_of_fewer_rows(topk, Lk, causal):
    # more units than SMs, so that a CTA's epilogue is at work while its filters bound the next unit
    B, H, Lq = 1, 8, min(Lk, 2500)
    q, k, v = W.attention_inputs(B, H, Lq, Lk, 64, seed=810 + topk)
    _selection_matches(q, k, v, topk, W.sample_rows(B * H * Lq, 400, seed=topk).numpy(), causal)


@pytest.mark.parametrize("topk", [65, 66, 68])
def test_two_query_tiles_causal(topk):
    # rows 768 .. 1791 of each head lie in units of 5 to 8 bound tiles
    B, H, L = 1, 4, 17536
    q, k, v = W.attention_inputs(B, H, L, L, 64, seed=820 + topk, dist="lowrank")
    early = np.concatenate([h * L + np.arange(700, 1900, 12) for h in range(H)])
    rows = np.concatenate([early, W.sample_rows(B * H * L, 60, seed=topk).numpy()])
    _outputs_match(q, k, v, topk, np.unique(rows), causal=True)


def test_two_query_tiles_key_counts():
    B, H, Lq, Lk, d, topk = 4, 9, 2000, 8500, 64, 66
    q, k, v = W.attention_inputs(B, H, Lq, Lk, d, seed=830)
    kv_len = np.array([700, 1100, 8500, 30], dtype=np.int32)
    out = T.attention(q.cuda(), k.cuda(), v.cuda(), topk, kv_len=torch.from_numpy(kv_len).cuda())
    T.topk_check()
    rows = W.sample_rows(B * H * Lq, 600, seed=831).numpy()
    ref = oracle.topk_attention(q, k, v, topk, rows=rows, kv_len=kv_len)
    with np.errstate(invalid="ignore"):  # a batch of 30 keys has no k-th score
        tie = np.abs(ref["score"][:, -1] - ref["next_score"]) <= 1e-5 * np.abs(ref["score"][:, -1])
    err = np.abs(out.float().cpu().reshape(-1, d).numpy()[rows] - ref["out"])
    assert err[~tie].max() <= 2e-2


@pytest.mark.parametrize("topk", [292, 300])
def test_one_key_short_of_a_gap(topk):
    # rows 32 .. 63 of every 64 have k - 1 high keys, the rest tied far below; rows 0 .. 31 have high keys
    # everywhere.  Exact in every precision, so the kept lists must be identical.
    B, H, Lq, Lk, d = 1, 2, 2560, 3000, 64
    g = torch.Generator().manual_seed(840 + topk)
    q = torch.zeros(B, H, Lq, d)
    q[:, :, torch.arange(Lq) % 64 >= 32, 0] = 1.0
    q[:, :, torch.arange(Lq) % 64 < 32, 1] = 1.0
    k = torch.zeros(B, H, Lk, d)
    k[..., 0] = 0.25
    high = torch.arange(topk - 1) * 10 + 3
    k[:, :, high, 0] = 2.0 + (torch.arange(topk - 1) % 64).float() / 64
    k[..., 1] = 4.0 + (torch.arange(Lk) % 128).float() / 128
    v = torch.randn(B, H, Lk, d, generator=g)
    q, k, v = q.bfloat16(), k.bfloat16(), v.bfloat16()
    out, idx, _ = T.attention(q.cuda(), k.cuda(), v.cuda(), topk, return_indices=True)
    T.topk_check()
    rows = W.sample_rows(B * H * Lq, 800, seed=841).numpy()
    ref = oracle.topk_attention(q, k, v, topk, rows=rows)
    assert np.array_equal(idx.cpu().reshape(-1, topk).numpy()[rows], ref["idx"])
    assert np.abs(out.float().cpu().reshape(-1, d).numpy()[rows] - ref["out"]).max() <= 2e-2
