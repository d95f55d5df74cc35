"""GPU parity of the d = 128 prefill kernel that works on pairs of query tiles (taken where there are two pairs for every SM), at the
edges of its 128-query and 64-key tiles: a second query tile without rows, with one, full; window and list lengths around a tile and
around a thread's half of one; query groups; logits that grow far beyond the exponentials' first reference; a chunk on a cache."""
import numpy as np
import pytest
import torch

from oracle import lte_oracle as orc
from paper_2510_20787_b200 import lte, synth
from tests.gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,G,T,W,R", [
    (19, 16, 1, 1, 7, 3), (19, 16, 1, 128, 8, 1), (19, 16, 1, 129, 64, 65), (19, 16, 1, 256, 63, 128), (10, 16, 1, 257, 65, 64),
    (5, 8, 4, 300, 33, 129), (10, 16, 1, 384, 300, 200), (7, 16, 1, 640, 31, 257), (7, 16, 1, 515, 128, 96),
])
@pytest.mark.parametrize("growing", [False, True])
def test_pairs(B, H, G, T, W, R, growing):
    cfg = synth.Config("pairs", "bf16", B, H, 128, T, W, R, 7, 0.1)
    x, q = synth.make(cfg, 17), synth.make(cfg.with_(H=H * G), 18)["q"]
    if growing:                                   # by hundreds from one tile of keys to the next
        x["k"] = synth.round_bf16(x["k"] * np.linspace(0.1, 1500.0, T, dtype=np.float32)[None, None, :, None])
    s = lte.shape(B, H, T, 128, W, R, lte.BF16, group=G)
    c = lte.conv(torch.from_numpy(x["w"]).cuda())
    qd, k, v = dev(q, "bf16"), dev(x["k"], "bf16"), dev(x["v"], "bf16")
    idx, cnt = lte.lte_select(s, lte.lte_scores(s, c, k, v))
    o, lse = lte.lte_attn_prefill(s, qd, k, v, idx, cnt)
    assert lte.lte_device_status() == 0
    rep = lambda a: np.repeat(a, G, axis=1)
    o64, l64 = orc.attn_prefill(q, rep(x["k"]), rep(x["v"]), rep(idx.cpu().numpy()), rep(cnt.cpu().numpy()), W)
    assert np.max(np.abs(o.float().cpu().numpy() - o64) - 4e-3 * np.abs(o64)) <= 2e-2   # (o is rounded to bf16)
    assert np.max(np.abs(lse.cpu().numpy() - l64)) <= 2e-3 * max(1.0, float(np.max(np.abs(l64))))


def test_chunk_of_many_heads_agrees_with_few():
    B, H, T0, Tc, W, R = 19, 16, 150, 140, 40, 30
    cfg = synth.Config("chunk", "bf16", B, H, 128, T0 + Tc, W, R, 7, 0.1)
    x = synth.make(cfg, 3)
    c = lte.conv(torch.from_numpy(x["w"]).cuda())

    def run(b):
        q, k, v = (dev(np.ascontiguousarray(x[n][:b]), "bf16") for n in "qkv")
        s0, s1 = (lte.shape(b, H, n, 128, W, R, lte.BF16) for n in (T0, Tc))
        kp, vp = k[:, :, :T0].contiguous(), v[:, :, :T0].contiguous()
        z = lte.lte_scores(s0, c, kp, vp)
        cache = lte.lte_cache_init(s0, c, kp, vp, z, *lte.lte_select(s0, z))
        return lte.lte_attn_prefill_chunk(s1, c, cache, T0, *(t[:, :, T0:].contiguous() for t in (q, k, v)))
    (o, lse), (o1, lse1) = run(B), run(1)
    assert lte.lte_device_status() == 0
    assert float((o[:1].float() - o1.float()).abs().max()) <= 2e-2 and float((lse[:1] - lse1).abs().max()) <= 2e-3


def test_pair_large_values_and_growing_logits():
    """Weights are taken relative to a reference that follows the row's maximum within 2^8, so that values of 1e30 do not overflow on the
    way to outputs of 1e30."""
    B, H, T, d, W, R = 2, 16, 2500, 128, 300, 64                # 320 pairs of query tiles: two for every SM
    s = lte.shape(B, H, T, d, W, R, lte.BF16)
    g = torch.Generator(device="cuda").manual_seed(5)
    n = lambda *shape: torch.randn(shape, generator=g, device="cuda")
    up = torch.ones(d, device="cuda") * torch.arange(T, device="cuda")[:, None] * 0.02   # q.k / sqrt(d) grows by 0.23 per key
    q, k, v = torch.ones((B, H, T, d), device="cuda").to(torch.bfloat16), (n(B, H, T, d) * 0.1 + up).to(torch.bfloat16), (n(B, H, T, d) * 1e30).to(torch.bfloat16)
    idx, cnt = lte.lte_select(s, n(B, H, T))
    o, lse = lte.lte_attn_prefill(s, q, k, v, idx, cnt)
    j, i = torch.arange(T, device="cuda")[None], torch.arange(T, device="cuda")[:, None]
    for b, h in ((0, 0), (1, 15)):
        sees = (j <= i) & (j > i - W)
        sees[:, idx[b, h, :int(cnt[b, h])].long()] |= (j <= i - W)[:, idx[b, h, :int(cnt[b, h])].long()]
        x = (q[b, h].double() @ k[b, h].double().T / d ** 0.5).masked_fill(~sees, -float("inf"))
        o64 = torch.softmax(x, -1) @ v[b, h].double()
        # weights rounded to bf16, and o: 2^-9 each
        assert bool(((o[b, h].double() - o64).abs() <= 2.0 ** -8 * v[b, h].double().abs().max()).all())
        assert bool(((lse[b, h].double() - torch.logsumexp(x, -1)).abs() <= 2e-3 * x[sees].abs().max()).all())
    assert lte.lte_device_status() == 0
