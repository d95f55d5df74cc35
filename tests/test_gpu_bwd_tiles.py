"""GPU parity of the tensor-core backward at the edges of its 128-row items and 128- or 64-wide tiles: sequence, window and list
lengths around a tile and around a thread's quarter of one, items of one tile and of many, lists of more than one item, parts of the
list that are empty, retained keys without a far query, query groups, more items than blocks fit on the chip (blocks then take over
the work of blocks that have not started)."""
import numpy as np
import pytest
import torch

from oracle import lte_oracle as orc
from paper_2510_20787_b200 import lte, synth
from tests.gpu_util import assert_grad_close, dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,G,d,T,W,R", [
    (1, 1, 1, 64, 2, 7, 3), (1, 2, 1, 64, 128, 32, 16), (1, 2, 1, 64, 129, 97, 127), (1, 1, 2, 64, 385, 128, 130), (2, 1, 1, 64, 300, 300, 0),
    (1, 2, 1, 64, 640, 31, 300), (1, 1, 3, 32, 257, 33, 40), (2, 1, 1, 32, 130, 129, 129), (3, 16, 1, 64, 700, 40, 70),
    (1, 1, 1, 128, 2, 7, 3), (1, 2, 1, 128, 127, 16, 64), (1, 2, 1, 128, 193, 63, 65), (1, 1, 2, 128, 450, 64, 257), (2, 1, 1, 128, 260, 300, 0),
    (3, 16, 1, 128, 700, 40, 70),
])
def test_tiles(B, H, G, d, T, W, R):
    cfg = synth.Config("tiles", "bf16", B, H, d, T, W, R, 7, 0.1)
    x = synth.make(cfg, 23)
    y = synth.make(cfg.with_(H=H * G), 24, with_dO=True)
    s = lte.shape(B, H, T, d, W, R, lte.BF16, group=G)
    c = lte.conv(torch.from_numpy(x["w"]).cuda())
    k, v, q, dO = (dev(a, "bf16") for a in (x["k"], x["v"], y["q"], y["dO"]))
    z = lte.lte_scores(s, c, k, v)
    idx, cnt = lte.lte_select(s, z)
    o, lse = lte.lte_attn_prefill(s, q, k, v, idx, cnt)
    dq, dk, dv, _, _ = lte.lte_attn_bwd(s, c, q, k, v, o, lse, dO, z, idx, cnt, flags=0)
    assert lte.lte_device_status() == 0
    rep = lambda a: np.repeat(a, G, axis=1)
    idx_n, cnt_n = idx.cpu().numpy(), cnt.cpu().numpy()
    ref = orc.attn_bwd(y["q"], rep(x["k"]), rep(x["v"]), y["dO"], rep(orc.scores(x["k"], x["v"], x["w"])), rep(idx_n), rep(cnt_n),
                       np.repeat(x["w"], G, axis=0), W, cnn_input_grad=False)
    assert_grad_close("dq", dq.float().cpu().numpy(), ref["dq"], 5e-2)
    for name, got in (("dk", dk), ("dv", dv)):
        assert_grad_close(name, got.float().cpu().numpy(), ref[name].reshape(B, H, G, T, d).sum(axis=2), 5e-2, idx_n, cnt_n)
