"""GPU parity of the d = 64 / 32 prefill kernel at the edges of its 96-key tiles: window spans and lists around one and two tiles, items of
a single tile, warps that see nothing of a tile, and logits whose maximum grows within an item's first tiles, within one tile and between
later ones (the sums, O and what has been written of P are rescaled)."""
import numpy as np
import pytest
import torch

from oracle import lte_oracle as orc
from paper_2510_20787_b200 import lte, synth
from tests.gpu_util import dev, shape_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,T,W,R,ws", [
    (64, 96, 96, 8, None), (64, 97, 97, 8, None), (64, 400, 65, 95, None), (64, 400, 66, 97, None), (64, 500, 161, 96, False),
    (64, 900, 162, 193, None), (64, 130, 1000, 0, None), (32, 400, 64, 97, None), (64, 1200, 31, 288, False),
])
@pytest.mark.parametrize("slope", [0.0, 0.1, 4.0])                # growth of q.k / sqrt(d) per key: over a tile none, 10, 400
def test_tiles_of_96(d, T, W, R, ws, slope):
    cfg = synth.Config("rows", "bf16", 2, 3, d, T, W, R, 7, 0.1)
    x = synth.make(cfg, 23)
    if slope:
        ramp = (np.arange(T, dtype=np.float32) * slope / d ** 0.5)[None, None, :, None]
        x["q"] = np.ones_like(x["q"])
        x["k"] = synth.round_bf16(x["k"] + ramp)
    s = shape_of(cfg)
    c = lte.conv(torch.from_numpy(x["w"]).cuda())
    q, k, v = (dev(x[t], "bf16") for t in "qkv")
    idx, cnt = lte.lte_select(s, lte.lte_scores(s, c, k, v))
    o, lse = lte.lte_attn_prefill(s, q, k, v, idx, cnt, ws=ws)
    assert lte.lte_device_status() == 0
    o64, l64 = orc.attn_prefill(x["q"], x["k"], x["v"], idx.cpu().numpy(), cnt.cpu().numpy(), W)
    # weights and o are rounded to bf16 (2^-9 each); a logit carries the rounding of its sum and of the exponent's difference (2^-23 each)
    big = max(1.0, float(np.max(np.abs(l64))))
    vmax = float(np.max(np.abs(x["v"])))
    assert np.max(np.abs(o.float().cpu().numpy() - o64)) <= vmax * (2.0 ** -8 + 2 * big * 2.0 ** -22)
    assert np.max(np.abs(lse.cpu().numpy() - l64)) <= 1e-5 + big * 2.0 ** -21
