"""A chunk on top of a cache that lacks logits of its ring (the single-layer scorer): the tokens are scored by the chunk, with no larger error against
64 bits than lte_scores has, and everything else is as on the cache that has them.  Gaps in single tokens, in whole heads among heads without, in all
of the ring; rings that are not full."""
import pytest
import torch

from paper_2510_20787_b200 import lte

pytestmark = pytest.mark.gpu


def _exact(k, v, w, bias):
    x, K = torch.cat([k, v], -1).double(), w.shape[1]
    x = torch.nn.functional.pad(x, (0, 0, K // 2, K // 2))
    T = k.shape[2]
    return sum(torch.einsum("bhtc,hc->bht", x[:, :, t:t + T], w[:, t].double()) for t in range(K)) + bias.double()[:, None]


@pytest.mark.parametrize("dtype,d,B,H,G,K,W,R,sink,T0,Tc", [
    ("bf16", 64, 4, 16, 1, 7, 500, 300, 4, 1200, 130),
    ("bf16", 64, 1, 3, 2, 13, 440, 64, 0, 700, 200),
    ("bf16", 128, 2, 5, 1, 5, 400, 20, 0, 900, 1),
    ("bf16", 32, 2, 4, 1, 7, 260, 70, 2, 700, 97),
    ("bf16", 64, 2, 2, 1, 1, 300, 64, 0, 400, 50),
    ("f32", 32, 2, 4, 1, 5, 300, 40, 1, 600, 60),
    ("f32", 64, 1, 2, 1, 7, 300, 40, 0, 280, 20),        # the ring is not full: rows are zero before position 0
    ("f32", 128, 1, 2, 1, 7, 300, 40, 0, 280, 20),
    ("bf16", 128, 1, 2, 1, 7, 900, 10, 0, 480, 400),
])
@pytest.mark.parametrize("gaps", ["few", "heads", "all"])
def test_gaps_are_scored(dtype, d, B, H, G, K, W, R, sink, T0, Tc, gaps):
    dt, code, e = (torch.bfloat16, lte.BF16, 2) if dtype == "bf16" else (torch.float32, lte.F32, 4)
    g = torch.Generator(device="cuda").manual_seed(d + K + T0)
    n = lambda *shape: torch.randn(shape, generator=g, device="cuda")
    half, T = K // 2, T0 + Tc
    w, bias = n(H, K, 2 * d) * 0.1, n(H) * 0.1
    c = lte.conv(w, bias)
    s0, s1 = (lte.shape(B, H, t, d, W, R, code, sink=sink, group=G) for t in (T0, Tc))
    k, v, q = n(B, H, T, d).to(dt), n(B, H, T, d).to(dt), n(B, H * G, Tc, d).to(dt)
    kp, vp, kc, vc = (x.contiguous() for x in (k[:, :, :T0], v[:, :, :T0], k[:, :, T0:], v[:, :, T0:]))
    z = lte.lte_scores(s0, c, kp, vp)
    idx, cnt = lte.lte_select(s0, z)
    first = T0 - W + half if T0 > W else 0                     # (tokens before it have lost their left neighbours)
    lost = torch.zeros((B, H, T0), dtype=torch.bool, device="cuda")
    if gaps == "few":
        lost[:, :, [first, first + 1, (first + T0) // 2, T0 - half - 1]] = True
    else:
        lost[:, :, first:] = True
        if gaps == "heads":
            lost &= (torch.arange(B * H, device="cuda").view(B, H, 1) % 3 == 1)
    out, parts = [], []
    for zz in (z, torch.where(lost, -float("inf"), z)):
        cache = torch.zeros(lte.lte_cache_bytes(s0), dtype=torch.uint8, device="cuda")
        lte.lte_cache_init(s0, c, kp, vp, zz, idx, cnt, cache=cache)
        out.append(lte.lte_attn_prefill_chunk(s1, c, cache, T0, q, kc, vc))
        rows = W + R
        blocks = cache[256:].view(B * H, -1)
        a = 2 * (256 if dtype == "bf16" and d == 64 and rows <= 256 else rows) * d * e
        parts.append((blocks[:, :a], blocks[:, a + 4 * rows:], blocks[:, a:a + 4 * rows].view(torch.float32)))
    assert lte.lte_device_status() == 0
    for a, b in list(zip(*out)) + list(zip(*parts))[:2]:
        assert torch.equal(a, b)
    # the ring's logits: slot p mod W holds position p
    pos = torch.arange(max(T - W, 0), T - half, device="cuda")
    z64 = _exact(k, v, w, bias)[:, :, pos]
    have, scored = (p[2].view(B, H, rows)[:, :, pos % W] for p in parts)
    assert torch.equal(have == -float("inf"), scored == -float("inf"))
    was = torch.zeros((B, H, T), dtype=torch.bool, device="cuda")
    was[:, :, :T0] = lost
    was = was[:, :, pos] & (scored > -float("inf"))
    assert torch.equal(have[~was], scored[~was]) and int(was.sum()) > 0
    # A chain of 2 K d additions in a row is several times further off than lte_scores.  (The rms of n errors has a sampling error of
    # 1 / (2 n)^(1/2), so the ratio of two of them one of n^(-1/2): three of those.)
    rms = lambda x: float((x[was].double() - z64[was]).square().mean().sqrt())
    assert rms(scored) <= (1.1 + 3 * int(was.sum()) ** -0.5) * rms(have), (rms(scored), rms(have))
