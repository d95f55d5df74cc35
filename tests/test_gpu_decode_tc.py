"""GPU parity of the tcgen05 decode step (bf16, d = 64, one query head, at most 256 rows) where its variants change: 128 and 129
rows, all 256, hardly any; thirteen scorer taps; a pool that is full; more heads than blocks fit on the chip (a block then walks several)."""
import numpy as np
import pytest
import torch

from oracle import lte_oracle as orc
from paper_2510_20787_b200 import lte, synth
from tests.gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,W,R,K,sink,T0,steps", [
    (1, 2, 8, 3, 5, 0, 0, 30), (1, 2, 80, 48, 7, 2, 300, 12), (1, 2, 80, 49, 13, 0, 300, 12), (1, 2, 128, 128, 7, 4, 500, 8),
    (1, 2, 13, 200, 13, 0, 0, 30), (1, 1, 128, 0, 7, 0, 126, 5), (53, 16, 24, 16, 7, 1, 90, 3), (53, 16, 70, 60, 7, 1, 200, 3),
])
def test_decode_tc(B, H, W, R, K, sink, T0, steps):
    d, T = 64, T0 + steps
    cfg = synth.Config("tc", "bf16", B, H, d, T, W, R, K, 0.1, sink=sink)
    x = synth.make(cfg, 5)
    s = lte.shape(B, H, T0, d, W, R, lte.BF16, sink=sink)
    c = lte.conv(torch.from_numpy(x["w"]).cuda())
    q, k, v = (dev(x[n], "bf16") for n in "qkv")
    if T0 > 0:
        kp, vp = k[:, :, :T0].contiguous(), v[:, :, :T0].contiguous()
        z = lte.lte_scores(s, c, kp, vp)
        cache = lte.lte_cache_init(s, c, kp, vp, z, *lte.lte_select(s, z))
    else:
        cache = lte.lte_cache_init(s, c)
    got = [lte.lte_attn_decode(s, c, cache, *(t[:, :, n].contiguous() for t in (q, k, v))) for n in range(T0, T)]
    o = np.stack([a.float().cpu().numpy() for a, _ in got], axis=2)
    lse = np.stack([b.cpu().numpy() for _, b in got], axis=2)
    o64, l64, _, _ = orc.stream(x["q"], x["k"], x["v"], orc.scores(x["k"], x["v"], x["w"]), W, R, sink, n_from=T0)
    assert np.max(np.abs(o - o64)) <= 2e-2 and np.max(np.abs(lse - l64)) <= 2e-3
    assert lte.lte_device_status() == 0


@pytest.mark.parametrize("B,H,W,R,K,sink,T0,steps", [
    (1, 2, 60, 192, 7, 0, 400, 6),         # the longest tail with which three blocks share an SM
    (1, 2, 64, 192, 7, 2, 400, 6),         # the first with which two do
    (2, 2, 1, 255, 1, 4, 300, 6),          # the longest there is
    (53, 16, 20, 236, 7, 1, 300, 3),       # ... nearly, with more heads than blocks
])
def test_decode_tc_long_pools(B, H, W, R, K, sink, T0, steps):
    test_decode_tc(B, H, W, R, K, sink, T0, steps)
