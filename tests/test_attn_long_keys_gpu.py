"""More than 65,536 keys with kept sets at the limits of the list memory.  Against the CPU oracle, under the
parity rules of _parity.py."""
import pytest

from paper_2106_06899_gb300 import workloads as W

from .test_attn_lists_gpu import _selection_matches

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("topk", [462, 463, 512])
@pytest.mark.parametrize("d", [64, 128])
def test_largest_kept_sets(d, topk):
    H, Lq = 2, 1300  # too many query tiles to split the keys into parts
    q, k, v = W.attention_inputs(1, H, Lq, 70001, d, seed=850 + topk)
    _selection_matches(q, k, v, topk, W.sample_rows(H * Lq, 60, seed=topk).numpy())
