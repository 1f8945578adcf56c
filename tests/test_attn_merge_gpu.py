"""Key parts and their merge with large kept sets: few query rows, eight parts, up to k = 512.  Against the
CPU oracle, under the parity rules of _parity.py."""
import numpy as np
import pytest

from paper_2106_06899_gb300 import workloads as W

from .test_attn_lists_gpu import _selection_matches

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("topk", [454, 455, 512])
@pytest.mark.parametrize("H,Lq,Lk,causal", [(1, 128, 4096, False), (3, 9, 9000, True), (1, 1, 70001, False)])
def test_eight_parts(H, Lq, Lk, causal, d, topk):
    q, k, v = W.attention_inputs(1, H, Lq, Lk, d, seed=860 + topk)
    _selection_matches(q, k, v, topk, np.arange(H * Lq), causal)
