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
