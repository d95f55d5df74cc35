"""A launch that the runtime refuses (nothing runs) is this call's status and nobody else's error."""
import pytest
import torch

from paper_2510_20787_b200 import lte

pytestmark = pytest.mark.gpu


def test_refused_launch_leaves_no_error_behind():
    # more heads than the grid of a chunk's kernels takes
    empty, s = (lte.shape(1, 66000, T, 32, 1, 0, lte.F32) for T in (0, 1))
    c = lte.conv(torch.zeros((s.H, 1, 64), device="cuda"))
    cache = torch.empty(lte.lte_cache_bytes(s), dtype=torch.uint8, device="cuda")
    lte.lte_cache_init(empty, c, cache=cache)
    x = torch.zeros((1, s.H, 1, 32), device="cuda")
    with pytest.raises(lte.LteError) as e:
        lte.lte_attn_prefill_chunk(s, c, cache, 0, x, x, x)
    assert e.value.status == -4
    assert float(torch.ones(3, device="cuda").sum()) == 3.0    # torch looks at the runtime's last error after its own launches
    lte.lte_cache_init(empty, c, cache=cache)
    assert not bool(cache[:256].any())
