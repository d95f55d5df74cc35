"""lte_cache_init, lte_cache_score and lte_cache_score_unrope beyond their usual arguments: more heads than a grid's second dimension,
tensors that start between 16-byte boundaries."""
import pytest
import torch

from paper_2510_20787_b200 import lte

pytestmark = pytest.mark.gpu


def test_empty_cache_of_many_heads():
    B, H, W, R = 4096, 17, 20, 4                               # 69,632 heads
    s = lte.shape(B, H, 0, 32, W, R, lte.BF16)
    c = lte.conv(torch.zeros((H, 7, 64), device="cuda"))
    cache = torch.full((lte.lte_cache_bytes(s),), 255, dtype=torch.uint8, device="cuda")
    lte.lte_cache_init(s, c, cache=cache)
    blocks = cache[256:].view(B * H, -1)
    n = 2 * (W + R) * 32 * 2                                   # keys and values, then logits, then the rest
    logits = blocks[:, n:n + 4 * (W + R)].view(torch.float32)
    assert bool((logits == -float("inf")).all())
    assert not bool(cache[:256].any()) and not bool(blocks[:, :n].any()) and not bool(blocks[:, n + 4 * (W + R):].any())


def test_ring_of_many_heads_is_scored():
    B, H, d, W, R, T = 4096, 17, 32, 20, 4, 20
    g = torch.Generator(device="cuda").manual_seed(1)
    ch = [2 * d, d, d // 2, d // 4]
    c = lte.conv_stack([torch.randn((H, ch[i + 1], 3, ch[i]), generator=g, device="cuda") * 0.1 for i in range(3)],
                       torch.randn((H, ch[3]), generator=g, device="cuda"))
    s = lte.shape(B, H, T, d, W, R, lte.BF16)
    k, v = (torch.randn((B, H, T, d), generator=g, device="cuda").to(torch.bfloat16) for _ in "kv")
    z = lte.lte_scores(s, c, k, v)
    unscored = torch.full_like(z, -float("inf"))
    idx, cnt = (torch.zeros(n, dtype=torch.int32, device="cuda") for n in ((B, H, R), (B, H)))
    cache = lte.lte_cache_init(s, c, k, v, unscored, idx, cnt)
    lte.lte_cache_score(s, c, cache)
    n = 2 * (W + R) * d * 2
    got = cache[256:].view(B * H, -1)[:, n:n + 4 * W].view(torch.float32).view(B, H, W)
    assert torch.equal(got[:, :, :T - 6], z[:, :, :T - 6])     # the last six tokens' right context is not there yet
    assert bool((got[:, :, T - 6:] == -float("inf")).all())
    assert lte.lte_device_status() == 0


def _at(t, offset):
    """A contiguous copy of t that starts `offset` elements behind a 16-byte boundary."""
    buf = torch.empty(t.numel() + 8, dtype=t.dtype, device=t.device)
    out = buf[offset:offset + t.numel()].view(t.shape)
    return out.copy_(t)


@pytest.mark.parametrize("dtype,d,W,R,ok,ov", [
    (lte.BF16, 64, 20, 12, 1, 0), (lte.BF16, 64, 130, 140, 0, 2), (lte.BF16, 32, 20, 12, 4, 7), (lte.BF16, 128, 20, 12, 3, 3),
    (lte.F32, 32, 20, 12, 1, 0), (lte.F32, 64, 20, 0, 0, 3), (lte.F32, 128, 70, 12, 2, 1),
])
def test_cache_from_unaligned_tensors(dtype, d, W, R, ok, ov):
    B, H, T = 2, 3, 300
    g = torch.Generator(device="cuda").manual_seed(2)
    k, v = (torch.randn((B, H, T, d), generator=g, device="cuda").to(torch.bfloat16 if dtype == lte.BF16 else torch.float32) for _ in "kv")
    s = lte.shape(B, H, T, d, W, R, dtype)
    c = lte.conv(torch.randn((H, 5, 2 * d), generator=g, device="cuda") * 0.1)
    z = lte.lte_scores(s, c, k, v)
    idx, cnt = lte.lte_select(s, z)
    want = lte.lte_cache_init(s, c, k, v, z, idx, cnt)
    assert torch.equal(lte.lte_cache_init(s, c, _at(k, ok), _at(v, ov), z, idx, cnt), want)


@pytest.mark.parametrize("dtype,d,W,oc,os", [(lte.BF16, 64, 70, 1, 0), (lte.BF16, 64, 300, 0, 2), (lte.BF16, 32, 20, 3, 1), (lte.F32, 64, 65, 2, 3), (lte.F32, 32, 20, 1, 1)])
def test_unaligned_rotary_tables(dtype, d, W, oc, os):
    B, H, R, T = 2, 2, 8, 2 * W + 5
    g = torch.Generator(device="cuda").manual_seed(3)
    ch = [2 * d, d, d // 2, d // 4]
    c = lte.conv_stack([torch.randn((H, ch[i + 1], 3, ch[i]), generator=g, device="cuda") * 0.1 for i in range(3)],
                       torch.randn((H, ch[3]), generator=g, device="cuda"))
    s = lte.shape(B, H, T, d, W, R, dtype)
    k, v = (torch.randn((B, H, T, d), generator=g, device="cuda").to(torch.bfloat16 if dtype == lte.BF16 else torch.float32) for _ in "kv")
    z = torch.full((B, H, T), -float("inf"), device="cuda")    # nothing is scored yet
    idx, cnt = lte.lte_select(s, z)
    angle = torch.rand((T, d // 2), generator=g, device="cuda") * 6.0
    cos, sin = angle.cos(), angle.sin()
    caches = [lte.lte_cache_init(s, c, k, v, z, idx, cnt) for _ in range(3)]
    lte.lte_cache_score_unrope(s, c, caches[0], cos, sin)
    lte.lte_cache_score_unrope(s, c, caches[1], _at(cos, oc), _at(sin, os))
    assert torch.equal(caches[0], caches[1]) and not torch.equal(caches[0], caches[2])
    assert lte.lte_device_status() == 0
