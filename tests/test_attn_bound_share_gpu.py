"""The bound pass over all, a part and very little of the keys: sizes on both sides of each of the divisor's
steps, against the CPU oracle as in test_attn_lists_gpu.py."""
import numpy as np
import pytest

from paper_2106_06899_gb300 import workloads as W

from .test_attn_lists_gpu import _selection_matches

pytestmark = pytest.mark.gpu


# keys per k: one step of the divisor lies at 4 per, 16 per, ... (per = 512, 64 and 128; 40 and 16 where the
# keys, more than 512 MB of them, are read from device memory)
@pytest.mark.parametrize("H,Lq,Lk,d,topk,causal", [
    (2, 200, 2047, 64, 1, False), (2, 200, 2048, 64, 1, False), (2, 200, 32768, 64, 4, False),
    (1, 150, 65536, 64, 1, True), (2, 3000, 40000, 64, 3, True),
    (2, 200, 4095, 128, 16, False), (2, 200, 4096, 128, 16, False), (2, 3000, 16384, 128, 1, True),
    (2, 200, 51200, 128, 100, False), (1, 150, 16384, 128, 256, False), (1, 150, 20000, 64, 300, False)])
def test_shares(H, Lq, Lk, d, topk, causal):
    q, k, v = W.attention_inputs(1, H, Lq, Lk, d, seed=960 + topk, dist="lowrank")
    _selection_matches(q, k, v, topk, W.sample_rows(H * Lq, 150, seed=topk).numpy(), causal)


@pytest.mark.parametrize("B,Lq,Lk,d,topk", [(4, 1, 65536, 64, 16), (4, 1, 65536, 64, 128), (4, 64, 33000, 128, 16)])
def test_keys_from_memory(B, Lq, Lk, d, topk):
    H = 16
    q, k, v = W.attention_inputs(B, H, Lq, Lk, d, seed=980 + topk)
    rows = np.unique(np.linspace(0, B * H * Lq - 1, 40).astype(np.int64))
    _selection_matches(q, k, v, topk, rows, causal=True)
