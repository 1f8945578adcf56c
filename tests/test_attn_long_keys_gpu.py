"""More than 65,536 keys, where an entry's position in its list gives the high bits of its index: kept sets at
the limits of the list memory, one and two query tiles per unit, key parts that begin and end inside a
stretch of 65,536 keys, masks, and key orders that cut the lists all the time.  Against the CPU oracle, under
the parity rules of _parity.py."""
import numpy as np
import pytest
import torch

import oracle
from paper_2106_06899_gb300 import topk as T
from paper_2106_06899_gb300 import workloads as W

from .test_attn_lists_gpu import _outputs_match, _selection_matches
from .test_mask_gpu import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("topk", [1, 64, 128, 300, 462, 463, 512])
@pytest.mark.parametrize("d", [64, 128])
def test_kept_sets(d, topk):
    H, Lq = 2, 1300 if topk > 300 else 5000  # too many query tiles to split the keys into parts
    q, k, v = W.attention_inputs(1, H, Lq, 70001, d, seed=850 + topk)
    _selection_matches(q, k, v, topk, W.sample_rows(H * Lq, 60, seed=topk).numpy())


@pytest.mark.parametrize("topk,Lk,causal", [(8, 65537, False), (64, 131072, True), (68, 140001, False)])
def test_two_query_tiles(topk, Lk, causal):
    H, Lq = 16, 2500
    q, k, v = W.attention_inputs(1, H, Lq, Lk, 64, seed=870 + topk, dist="lowrank")
    _outputs_match(q, k, v, topk, W.sample_rows(H * Lq, 40, seed=topk).numpy(), causal)


@pytest.mark.parametrize("d,topk", [(64, 16), (128, 200)])
@pytest.mark.parametrize("Lq,Lk", [(1, 65537), (5, 200001), (130, 131073)])
def test_key_parts(Lq, Lk, d, topk):
    q, k, v = W.attention_inputs(1, 2, Lq, Lk, d, seed=880 + topk)
    _selection_matches(q, k, v, topk, np.arange(2 * Lq)[:: max(1, Lq // 20)], causal=True)


def test_key_counts():
    B, H, Lq, Lk, d, topk = 5, 2, 1100, 140000, 64, 40
    q, k, v = W.attention_inputs(B, H, Lq, Lk, d, seed=890)
    _check(q, k, v, topk, kv_len=np.array([65536, 65537, 131073, 20, 0], dtype=np.int32),
           rows=W.sample_rows(B * H * Lq, 60, seed=891))


@pytest.mark.parametrize("topk", [5, 64, 300])
@pytest.mark.parametrize("order", ["rising", "falling", "constant"])
@pytest.mark.parametrize("Lq", [70, 10000])
def test_key_orders(Lq, order, topk):
    # one feature carries the score: exact in every precision, so the kept lists must be identical
    Lk, d = 140000, 64
    ramp = torch.arange(Lk) * 256 // Lk
    q, k = torch.zeros(1, 1, Lq, d), torch.zeros(1, 1, Lk, d)
    q[..., 0] = 1.0
    k[..., 0] = (ramp if order == "rising" else 255 - ramp if order == "falling" else ramp * 0).float() / 16
    v = torch.randn(1, 1, Lk, d, generator=torch.Generator().manual_seed(900 + topk))
    q, k, v = q.bfloat16(), k.bfloat16(), v.bfloat16()
    out, idx, _ = T.attention(q.cuda(), k.cuda(), v.cuda(), topk, return_indices=True)
    T.topk_check()
    rows = np.array([0, 33, Lq - 1])
    ref = oracle.topk_attention(q, k, v, topk, rows=rows)
    assert np.array_equal(idx.cpu().reshape(-1, topk).numpy()[rows], ref["idx"])
    assert (idx == idx[:, :, :1]).all()  # all query rows are the same
    assert np.abs(out.float().cpu().reshape(-1, d).numpy()[rows] - ref["out"]).max() <= 2e-2


@pytest.mark.parametrize("d,topk", [(64, 64), (64, 100), (128, 33)])
def test_a_million_keys(d, topk):
    # 18 breaks per row, kept where the parked lists leave room for them
    q, k, v = W.attention_inputs(1, 1, 10000, 1_200_000, d, seed=910 + topk)
    rows = W.sample_rows(10000, 12, seed=topk).numpy()
    _outputs_match(q, k, v, topk, rows)
    _selection_matches(q, k, v, topk, rows)
