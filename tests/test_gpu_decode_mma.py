"""GPU parity of the bf16 decode step whose rows go straight into mma operands (decode_mma.cu), where its splits change:
one to eight warps a head, clusters of two to eight blocks, rows that do not fill the last span of 16, more query heads
than a pass takes, the swizzled cache layout, more scorer taps than warps."""
import numpy as np
import pytest
import torch

from oracle import lte_oracle as orc
from paper_2510_20787_b200 import lte, synth
from tests.gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,W,R,G,K,sink,T0,steps", [
    (32, 13, 6, 1, 13, 0, 0, 40),          # one warp, 13 taps
    (32, 20, 12, 3, 7, 2, 25, 30),         # two warps
    (64, 257, 0, 1, 7, 0, 255, 5),         # no pool, the ring fills up
    (64, 100, 99, 8, 5, 1, 120, 20),       # swizzled rows, a full pass of query heads
    (128, 33, 15, 1, 7, 0, 40, 20),        # three warps
    (128, 250, 70, 9, 7, 3, 400, 6),       # a cluster, two passes of query heads
    (64, 768, 512, 4, 7, 4, 1500, 6),      # a cluster of eight, pool full
    (128, 1, 16, 2, 1, 0, 10, 25),         # the smallest window
    (32, 3000, 1096, 1, 3, 0, 3100, 3),    # the most rows a cache may hold
])
def test_decode_mma(d, W, R, G, K, sink, T0, steps):
    T = T0 + steps
    cfg = synth.Config("mma", "bf16", 1, 2, d, T, W, R, K, 0.1, sink=sink)
    x, q = synth.make(cfg, 3), synth.make(cfg.with_(H=cfg.H * G), 103)["q"]
    s = lte.shape(cfg.B, cfg.H, T0, d, W, R, lte.BF16, sink=sink, group=G)
    c = lte.conv(torch.from_numpy(x["w"]).cuda())
    qd, k, v = dev(q, "bf16"), dev(x["k"], "bf16"), dev(x["v"], "bf16")
    if T0 > 0:
        kp, vp = k[:, :, :T0].contiguous(), v[:, :, :T0].contiguous()
        z = lte.lte_scores(s, c, kp, vp)
        cache = lte.lte_cache_init(s, c, kp, vp, z, *lte.lte_select(s, z))
    else:
        cache = lte.lte_cache_init(s, c)
    got = [lte.lte_attn_decode(s, c, cache, qd[:, :, n].contiguous(), k[:, :, n].contiguous(), v[:, :, n].contiguous()) for n in range(T0, T)]
    o = np.stack([a.float().cpu().numpy() for a, _ in got], axis=2)
    lse = np.stack([b.cpu().numpy() for _, b in got], axis=2)
    rep = lambda a: np.repeat(a, G, axis=1)
    z64 = orc.scores(x["k"], x["v"], x["w"])
    o64, l64, _, _ = orc.stream(q, rep(x["k"]), rep(x["v"]), rep(z64), W, R, sink, n_from=T0)
    assert np.max(np.abs(o - o64)) <= 2e-2 and np.max(np.abs(lse - l64)) <= 2e-3
    assert lte.lte_device_status() == 0


@pytest.mark.parametrize("d,W,R,G", [(32, 20, 12, 1), (64, 300, 80, 1), (64, 100, 99, 4), (128, 250, 70, 9), (128, 768, 256, 1)])
@pytest.mark.parametrize("size", [30.0, 1e9, 1e18])
def test_decode_mma_large_logits(d, W, R, G, size):
    """Logits of about `size`: o and lse stay finite and as close to 64 bits as sums in fp32 of exact products are."""
    H, T0 = 2, W + 50
    g = torch.Generator(device="cuda").manual_seed(int(size) % 97 + d)
    n = lambda *shape: torch.randn(shape, generator=g, device="cuda")
    s, c = lte.shape(1, H, T0, d, W, R, lte.BF16, group=G), lte.conv(n(H, 7, 2 * d) * 1e-3)
    k, v, q1, k1, v1 = (t.to(torch.bfloat16) for t in (n(1, H, T0, d), n(1, H, T0, d), n(1, H * G, d) * size, n(1, H, d), n(1, H, d)))
    z = lte.lte_scores(s, c, k, v)
    idx, cnt = lte.lte_select(s, z)
    cache = lte.lte_cache_init(s, c, k, v, z, idx, cnt)
    o, lse = lte.lte_attn_decode(s, c, cache, q1, k1, v1)
    for h in range(H):
        # after the step: the window's rows, and what the pool holds (its positions stand behind the logits)
        e, alloc = 2, 256 if d == 64 and W + R <= 256 else W + R
        tail = cache[256:].view(H, -1)[h, 2 * alloc * d * e + 4 * (W + R):]
        pool = tail[:4 * R].view(torch.int32)[:int(tail[4 * R + 4:4 * R + 8].view(torch.int32)[0])].long()
        kr = torch.cat([k[0, h, pool], k[0, h, T0 - W + 1:], k1[:, h]]).double()
        vr = torch.cat([v[0, h, pool], v[0, h, T0 - W + 1:], v1[:, h]]).double()
        qh = q1[0, h * G:(h + 1) * G].double()
        x = qh @ kr.T / d ** 0.5
        l64 = torch.logsumexp(x, -1)
        # fp32 sums of d exact products, the scale, the sum of weights, the logarithm, their sum
        bound = 2.0 ** -24 * ((d + 2) * (qh.abs() @ kr.abs().T).amax(-1) / d ** 0.5 + 8)
        assert bool(((lse[0, h * G:(h + 1) * G].double() - l64).abs() <= bound).all())
        if size > 1e6:                                         # one weight is 1, the others 0
            assert torch.equal(o[0, h * G:(h + 1) * G].double(), vr[x.argmax(-1)])
    assert lte.lte_device_status() == 0


@pytest.mark.parametrize("d", [64, 128])
def test_decode_mma_lse_is_as_accurate_as_fp32(d):
    """lse's error against 64 bits stays near that of the same logits in plain fp32 (sums rounded to the nearest): at most 1.5 times as
    large in the mean square over 4,096 query heads, whose sampling error is a few per cent; a running sum rounded towards zero makes it twice."""
    B, H, G, W, R = 8, 128, 4, 64, 0
    g = torch.Generator(device="cuda").manual_seed(d)
    n = lambda *shape: torch.randn(shape, generator=g, device="cuda").to(torch.bfloat16)
    s, c = lte.shape(B, H, W - 1, d, W, R, lte.BF16, group=G), lte.conv(torch.zeros((H, 7, 2 * d), device="cuda"))
    k, v, q1, k1, v1 = n(B, H, W - 1, d), n(B, H, W - 1, d), n(B, H * G, d) * 6, n(B, H, d), n(B, H, d)
    idx, cnt = torch.zeros((B, H, 0), dtype=torch.int32, device="cuda"), torch.zeros((B, H), dtype=torch.int32, device="cuda")
    cache = lte.lte_cache_init(s, c, k, v, torch.zeros((B, H, W - 1), device="cuda"), idx, cnt)
    _, lse = lte.lte_attn_decode(s, c, cache, q1, k1, v1)
    rows, q = torch.cat([k, k1[:, :, None]], dim=2), q1.view(B, H, G, d)
    l64 = torch.logsumexp(q.double() @ rows.double().transpose(2, 3) / d ** 0.5, -1)
    l32 = torch.logsumexp(((q.float() * d ** -0.5)[:, :, :, None] * rows.float()[:, :, None]).sum(-1), -1)
    rms = lambda x: float((x.double() - l64).square().mean().sqrt())
    assert rms(lse.view(B, H, G)) <= 1.5 * rms(l32), (rms(lse.view(B, H, G)), rms(l32))
