"""The list-based selection of the tensor-core attention kernels at the sizes where it can go wrong:
two query tiles per unit, 32-bit key indices, every list size class, and key orders that keep every
list full (scores rising along the keys), constant (ties) or empty.  Against the CPU oracle, under the
parity rules of _parity.py; where no selection is asked for, outputs within 2e-2 as there."""
import numpy as np
import pytest
import torch

import oracle
from paper_2106_06899_gb300 import topk as T
from paper_2106_06899_gb300 import workloads as W

from ._parity import check_rows

pytestmark = pytest.mark.gpu


def _outputs_match(q, k, v, topk, rows, causal=False):
    """The call without selection outputs, on sampled rows, against the oracle."""
    d = q.shape[-1]
    out = T.attention(q.cuda(), k.cuda(), v.cuda(), topk, causal=causal)
    T.topk_check()
    ref = oracle.topk_attention(q, k, v, topk, causal=causal, rows=rows)
    tie = np.abs(ref["score"][:, -1] - ref["next_score"]) <= 1e-5 * np.abs(ref["score"][:, -1])
    err = np.abs(out.float().cpu().reshape(-1, d).numpy()[rows] - ref["out"])
    assert err[~tie].max() <= 2e-2


def _selection_matches(q, k, v, topk, rows, causal=False):
    d = q.shape[-1]
    out, idx, score = T.attention(q.cuda(), k.cuda(), v.cuda(), topk, causal=causal, return_indices=True)
    T.topk_check()
    check_rows(q=q, k=k, v=v, rows=rows, gpu_out=out.float().cpu().reshape(-1, d).numpy()[rows],
               gpu_idx=idx.cpu().reshape(-1, topk).numpy()[rows], gpu_score=score.cpu().reshape(-1, topk).numpy()[rows],
               topk=topk, dtype="bf16", causal=causal)


@pytest.mark.parametrize("topk,Lk,causal", [(1, 1001, False), (8, 1100, False), (8, 2100, True), (64, 8200, False)])
def test_two_query_tiles_per_unit(topk, Lk, causal):
    # 160 units of 256 query rows, the last one of each head ragged; rows of at least 128 k keys
    B, H, Lq = 2, 10, 2000
    q, k, v = W.attention_inputs(B, H, Lq, Lk, 64, seed=700 + topk, dist="lowrank")
    _outputs_match(q, k, v, topk, W.sample_rows(B * H * Lq, 400, seed=topk).numpy(), causal)


@pytest.mark.parametrize("d,topk", [(64, 33), (64, 100), (128, 64), (128, 300)])
def test_more_than_65536_keys(d, topk):
    B, H, Lq, Lk = 1, 1, 130, 70001
    q, k, v = W.attention_inputs(B, H, Lq, Lk, d, seed=720 + topk)
    rows = np.arange(B * H * Lq)
    _selection_matches(q, k, v, topk, rows)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("topk", [31, 32, 33, 68, 69, 129, 170, 257, 384, 512])
def test_list_size_classes(d, topk):
    B, H, Lq, Lk = 1, 2, 140, 1500
    q, k, v = W.attention_inputs(B, H, Lq, Lk, d, seed=740 + topk + d)
    _selection_matches(q, k, v, topk, np.arange(B * H * Lq))


@pytest.mark.parametrize("topk", [4, 64, 100, 300])
@pytest.mark.parametrize("order", ["rising", "falling", "constant", "zero_query"])
def test_key_orders(topk, order):
    # one feature carries the score: exact in every precision, so the kept lists must be identical
    B, H, Lq, Lk, d = 1, 2, 200, 2048, 64
    g = torch.Generator().manual_seed(760 + topk)
    q = torch.zeros(B, H, Lq, d)
    k = torch.zeros(B, H, Lk, d)
    q[..., 0] = 1.0
    ramp = torch.arange(Lk) // 8
    k[..., 0] = (ramp if order == "rising" else 255 - ramp if order == "falling" else torch.full((Lk,), 3)).float() / 16
    if order == "zero_query":
        q.zero_()
    v = torch.randn(B, H, Lk, d, generator=g)
    q, k, v = q.bfloat16(), k.bfloat16(), v.bfloat16()
    out, idx, _ = T.attention(q.cuda(), k.cuda(), v.cuda(), topk, return_indices=True)
    T.topk_check()
    ref = oracle.topk_attention(q, k, v, topk)
    assert np.array_equal(idx.cpu().reshape(-1, topk).numpy(), ref["idx"])
    assert np.abs(out.float().cpu().reshape(-1, d).numpy() - ref["out"]).max() <= 2e-2


def test_scores_of_infinity_and_nan_keys():
    # a key of +inf scores +inf, one of -inf or NaN is never kept, and value rows no key selects may hold anything
    B, H, Lq, Lk, d, topk = 1, 1, 140, 900, 64, 16
    g = torch.Generator().manual_seed(780)
    q = torch.rand(B, H, Lq, d, generator=g) + 0.5
    k = torch.randn(B, H, Lk, d, generator=g)
    v = torch.randn(B, H, Lk, d, generator=g)
    k[0, 0, 5] = -float("inf")
    k[0, 0, 700] = float("nan")
    v[0, 0, [0, 5, 700]] = float("nan")
    k[0, 0, 0] = -50.0  # the lowest finite scores: never among the best 16
    q, k, v = q.bfloat16(), k.bfloat16(), v.bfloat16()
    out, idx, score = T.attention(q.cuda(), k.cuda(), v.cuda(), topk, return_indices=True)
    T.topk_check()
    assert torch.isfinite(out).all() and torch.isfinite(score).all()
    assert not torch.isin(idx.cpu(), torch.tensor([0, 5, 700], dtype=torch.int32)).any()


@pytest.mark.parametrize("dtype,d", [("f32", 16), ("f32", 64), ("f32", 128), ("bf16", 128)])
@pytest.mark.parametrize("topk,Lk", [(1, 63), (64, 65), (128, 193), (129, 257), (128, 1000), (512, 700)])
@pytest.mark.parametrize("rows", ["few", "many"])
def test_cuda_core_lists(dtype, d, topk, Lk, rows):
    # lists that are cut never, once or often; one or four rows per warp; bf16 runs here under a bit mask
    B, H, Lq = (1, 1, 37) if rows == "few" else (7, 10, 140)
    q, k, v = W.attention_inputs(B, H, Lq, Lk, d, dtype=dtype, seed=790 + topk + d)
    mask = None
    if dtype == "bf16":
        mask = np.random.default_rng(topk).random((1, 1, Lq, Lk)) < 0.8
    out, idx, score = T.attention(q.cuda(), k.cuda(), v.cuda(), topk, return_indices=True,
                                  mask=None if mask is None else torch.from_numpy(mask).cuda())
    T.topk_check()
    sel = W.sample_rows(B * H * Lq, 300, seed=topk).numpy()
    check_rows(q=q, k=k, v=v, rows=sel, gpu_out=out.float().cpu().reshape(-1, d).numpy()[sel],
               gpu_idx=idx.cpu().reshape(-1, topk).numpy()[sel], gpu_score=score.cpu().reshape(-1, topk).numpy()[sel],
               topk=topk, dtype=dtype, mask=mask)
