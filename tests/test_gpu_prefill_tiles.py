"""GPU parity of the d = 64 / 32 prefill kernel around its items of 128 queries and at small shapes: sequence, window and list lengths around 128
and 64, one tile per item, more items than blocks fit on the chip (blocks then take over the work of blocks that have not started), a row
maximum that keeps growing (the accumulator is rescaled).  The edges of its 96-key tiles are in test_gpu_prefill_rows.py."""
import numpy as np
import pytest
import torch

from oracle import lte_oracle as orc
from paper_2510_20787_b200 import lte, synth
from tests.gpu_util import dev, shape_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,d,T,W,R,ws", [
    (1, 1, 64, 1, 7, 3, None), (1, 2, 64, 128, 64, 16, None), (1, 2, 64, 129, 7, 128, None), (2, 1, 64, 383, 127, 127, None),
    (1, 2, 64, 640, 129, 129, None), (1, 2, 64, 520, 65, 256, False), (1, 2, 32, 300, 33, 31, None), (2, 3, 64, 257, 300, 8, None),
    (4, 16, 64, 700, 40, 70, None), (4, 16, 64, 700, 40, 70, False),
])
@pytest.mark.parametrize("growing", [False, True])
def test_tiles(B, H, d, T, W, R, ws, growing):
    cfg = synth.Config("tiles", "bf16", B, H, d, T, W, R, 7, 0.1)
    x = synth.make(cfg, 17)
    if growing:                                   # logits that grow along the keys by far more than the rescale threshold
        x["k"] = synth.round_bf16(x["k"] * np.linspace(0.1, 30.0, T, dtype=np.float32)[None, None, :, None])
    s = shape_of(cfg)
    c = lte.conv(torch.from_numpy(x["w"]).cuda())
    q, k, v = (dev(x[t], "bf16") for t in "qkv")
    idx, cnt = lte.lte_select(s, lte.lte_scores(s, c, k, v))
    o, lse = lte.lte_attn_prefill(s, q, k, v, idx, cnt, ws=ws)
    o64, l64 = orc.attn_prefill(x["q"], x["k"], x["v"], idx.cpu().numpy(), cnt.cpu().numpy(), W)
    assert np.max(np.abs(o.float().cpu().numpy() - o64)) <= 2e-2
    assert np.max(np.abs(lse.cpu().numpy() - l64)) <= 2e-3 * max(1.0, float(np.max(np.abs(l64))))
    assert lte.lte_device_status() == 0


@pytest.mark.parametrize("d,T,W,R,ws", [(64, 700, 200, 100, None), (64, 700, 200, 100, False), (32, 500, 60, 200, None), (64, 100, 128, 0, None)])
def test_equal_values_come_out_as_they_are(d, T, W, R, ws):
    """Where every value row is the same, so is every output: the weights' rounding to bf16 cancels against their sum, whatever the reference
    of the exponentials is (the rest are sums in fp32, some 1e-6 of the value, which is itself a bf16 number)."""
    B, H = 2, 3
    cfg = synth.Config("equal", "bf16", B, H, d, T, W, R, 7, 0.1)
    s = shape_of(cfg)
    g = torch.Generator(device="cuda").manual_seed(T + d)
    n = lambda *shape: torch.randn(shape, generator=g, device="cuda")
    q, k = n(B, H, T, d).to(torch.bfloat16), (n(B, H, T, d) * torch.linspace(0.2, 3.0, T, device="cuda")[:, None]).to(torch.bfloat16)
    v = n(B, H, 1, d).to(torch.bfloat16).expand(B, H, T, d).contiguous()
    idx, cnt = lte.lte_select(s, n(B, H, T))
    o, _ = lte.lte_attn_prefill(s, q, k, v, idx, cnt, ws=ws)
    assert torch.equal(o, v)
    assert lte.lte_device_status() == 0
