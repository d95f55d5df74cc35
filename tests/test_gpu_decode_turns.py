"""GPU parity of decode steps over caches larger than three quarters of L2, which go through a block's heads or a head's rows forwards and
backwards in turn, on sampled sequences: both kernels, one warp a head and several, clusters, more query heads than a pass takes, fewer spans of
rows than warps, remainders of a span, rows swizzled and not, pools empty, growing and full."""
import numpy as np
import pytest
import torch

from oracle import lte_oracle as orc
from paper_2510_20787_b200 import lte

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,W,R,G,K,sink,B,H,T0,steps", [
    (64, 64, 64, 1, 7, 0, 256, 16, 201, 5),        # the tensor-core step, 128 rows
    (64, 101, 120, 1, 7, 2, 150, 16, 300, 4),      # its variant of 256 rows
    (64, 128, 128, 1, 1, 0, 200, 8, 130, 4),       # blocks of three heads and of four
    (64, 128, 101, 2, 7, 0, 128, 16, 300, 4),      # mma, swizzled rows
    (32, 300, 100, 1, 5, 0, 128, 16, 421, 4),      # a warp a head, all heads at once: alternating
    (32, 300, 100, 1, 5, 0, 160, 16, 421, 4),      # more heads than that: forwards only
    (64, 768, 512, 4, 7, 4, 32, 16, 1500, 4),      # several warps a head
    (128, 401, 111, 1, 7, 0, 32, 16, 540, 4),
    (64, 3000, 96, 1, 7, 0, 8, 16, 21, 4),         # a cluster of two, two spans of rows
    (128, 2950, 1146, 9, 7, 3, 6, 8, 5300, 3),     # a cluster, two passes of query heads
])
def test_decode_turns(d, W, R, G, K, sink, B, H, T0, steps):
    l2 = torch.cuda.get_device_properties(0).L2_cache_size
    assert B * H * (W + R) * d * 4 > l2 * 3 // 4
    g = torch.Generator(device="cuda").manual_seed(d + W + R)
    n = lambda *shape: torch.randn(shape, generator=g, device="cuda")
    T = T0 + steps
    q, k = (n(B, H * G, steps, d) * d ** -0.25).to(torch.bfloat16), (n(B, H, T, d) * d ** -0.25).to(torch.bfloat16)
    v, w = n(B, H, T, d).to(torch.bfloat16), n(H, K, 2 * d) * 0.1
    s, c = lte.shape(B, H, T0, d, W, R, lte.BF16, sink=sink, group=G), lte.conv(w)
    kp, vp = k[:, :, :T0].contiguous(), v[:, :, :T0].contiguous()
    z = lte.lte_scores(s, c, kp, vp)
    cache = lte.lte_cache_init(s, c, kp, vp, z, *lte.lte_select(s, z))
    got = [lte.lte_attn_decode(s, c, cache, q[:, :, t].contiguous(), k[:, :, T0 + t].contiguous(), v[:, :, T0 + t].contiguous()) for t in range(steps)]
    assert lte.lte_device_status() == 0
    for b in (0, B // 2, B - 1):
        host = lambda t: t[b:b + 1].float().cpu().numpy()
        o, lse = (np.stack([host(x[i]) for x in got], axis=2) for i in (0, 1))
        kb, vb = host(k), host(v)
        qb = np.zeros((1, H * G, T, d), np.float32)
        qb[:, :, T0:] = host(q)
        rep = lambda a: np.repeat(a, G, axis=1)
        z64 = orc.scores(kb, vb, w.cpu().numpy())
        o64, l64, _, _ = orc.stream(qb, rep(kb), rep(vb), rep(z64), W, R, sink, n_from=T0)
        assert np.max(np.abs(o - o64)) <= 2e-2 and np.max(np.abs(lse - l64)) <= 2e-3
