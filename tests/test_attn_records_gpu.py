"""The d = 128 attention kernel on both sides of the line between eight and four records per row (k = 90),
against the CPU oracle as in test_attn_lists_gpu.py."""
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
