"""Units of two query tiles: with and without the selection as output, causal, ragged last tiles, fewer units
than SMs, and both sides of the rule that picks them.  Against the CPU oracle as in test_attn_lists_gpu.py;
a workspace query, which is told neither, covers every call."""
import numpy as np
import pytest
import torch

from paper_2106_06899_gb300 import topk as T
from paper_2106_06899_gb300 import workloads as W

from .test_attn_lists_gpu import _outputs_match, _selection_matches

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("topk,H,Lq,Lk,causal", [
    (1, 9, 4200, 8300, False), (8, 9, 4200, 8191, False), (8, 9, 4200, 8192, False), (16, 3, 8192, 8192, False),
    (16, 3, 16400, 16400, True), (32, 9, 4161, 8192, False), (33, 9, 4161, 8200, False), (64, 9, 4200, 16500, False)])
def test_selection_and_outputs(topk, H, Lq, Lk, causal):
    q, k, v = W.attention_inputs(1, H, Lq, Lk, 64, seed=990 + topk, dist="lowrank")
    rows = W.sample_rows(H * Lq, 250, seed=topk).numpy()
    _outputs_match(q, k, v, topk, rows, causal)
    _selection_matches(q, k, v, topk, rows, causal)


@pytest.mark.parametrize("Lq,topk", [(1, 16), (3, 64), (128, 8)])
def test_second_tile_empty(Lq, topk):
    q, k, v = W.attention_inputs(10, 16, Lq, 8200, 64, seed=1005 + topk)
    _outputs_match(q, k, v, topk, W.sample_rows(160 * Lq, 150, seed=topk).numpy(), causal=True)


@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("Lk", [16384, 70000])
def test_scratch_within_the_query(Lk, causal):
    # 128 units of two query tiles, 256 of one; nothing else of the pool is in use
    q, k, v = (torch.randn(1, 4, n, 64, device="cuda").bfloat16() for n in (8192, Lk, Lk))
    need = T.topk_attn_workspace_bytes(1, 4, 8192, Lk, 64, 64, 1024, T.TOPK_BF16)
    for idx in (False, True):
        torch.cuda.synchronize()
        T.topk_pool_usage(reset_high=True)
        T.attention(q, k, v, 64, causal=causal, return_indices=idx)
        T.topk_check()
        used, _ = T.topk_pool_usage()
        assert used <= need + 4096


@pytest.mark.parametrize("Lk", [32767, 32768])
@pytest.mark.parametrize("d,topk", [(64, 1), (64, 64), (64, 130), (128, 90), (128, 128)])
def test_cut_in_the_filters_or_the_epilogue(Lk, d, topk):
    # on both sides of the key count that says which; ties at the cut included
    q, k, v = W.attention_inputs(1, 20, 1100, Lk, d, seed=1010 + topk)
    k[:, :, 1::2] = k[:, :, ::2][:, :, : Lk // 2]
    _selection_matches(q, k, v, topk, W.sample_rows(20 * 1100, 100, seed=topk).numpy())
