"""The tensor-core attention kernel on both sides of two lines: eight and four records per row at d = 128 (k = 90),
and units of 128 or 64 rows where the lists are nearly full (k = 137).  Against the CPU oracle as in
test_attn_lists_gpu.py."""
import numpy as np
import pytest

from paper_2106_06899_gb300 import workloads as W

from .test_attn_lists_gpu import _selection_matches

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("topk", [1, 16, 64, 89, 90, 91, 96])
@pytest.mark.parametrize("Lq,Lk,causal", [(300, 333, False), (1500, 1500, True), (3, 20000, True)])
def test_records(Lq, Lk, causal, topk):
    q, k, v = W.attention_inputs(1, 3, Lq, Lk, 128, seed=940 + topk)
    _selection_matches(q, k, v, topk, W.sample_rows(3 * Lq, 300, seed=topk).numpy(), causal)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("topk,Lk,causal", [(136, 500, False), (137, 500, False), (140, 2239, False), (140, 2240, False),
                                            (140, 4470, True)])
def test_lists_that_are_nearly_full(d, topk, Lk, causal):
    # on both sides of the line between units of 128 and 64 rows
    H, Lq = 12, min(Lk, 1700)
    q, k, v = W.attention_inputs(1, H, Lq, Lk, d, seed=1060 + topk)
    _selection_matches(q, k, v, topk, W.sample_rows(H * Lq, 200, seed=topk).numpy(), causal)
