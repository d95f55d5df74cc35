"""What the native Python binding refuses of the tensors that it is given."""
import pytest
import torch

from paper_2510_20787_b200 import lte

pytestmark = pytest.mark.gpu


def test_workspaces_count_in_bytes():
    d, H, T = 64, 2, 100
    s = lte.shape(1, H, T, d, 20, 8, lte.BF16)
    ch = [2 * d, d, d // 2, d // 4]
    c = lte.conv_stack([torch.zeros((H, ch[i + 1], 3, ch[i]), device="cuda") for i in range(3)], torch.zeros((H, ch[3]), device="cuda"))
    x = torch.zeros((1, H, T, d), dtype=torch.bfloat16, device="cuda")
    need = lte.lte_workspace_bytes(lte.OP_SCORES, s, c)
    with pytest.raises(AssertionError):                        # lte_scores: bytes only
        lte.lte_scores(s, c, x, x, ws=torch.empty(need, dtype=torch.float32, device="cuda"))
    lte.lte_scores(s, c, x, x, ws=torch.empty(need, dtype=torch.uint8, device="cuda"))
    cache = torch.zeros(lte.lte_cache_bytes(s), dtype=torch.uint8, device="cuda")
    need = lte.lte_workspace_bytes(lte.OP_DECODE, s, c)
    with pytest.raises(lte.LteError) as e:                     # elsewhere an element counts as one byte
        lte.lte_cache_score(s, c, cache, ws=torch.empty((need + 3) // 4, dtype=torch.float32, device="cuda"))
    assert e.value.status == -3
    lte.lte_cache_score(s, c, cache, ws=torch.empty(need, dtype=torch.float32, device="cuda"))
