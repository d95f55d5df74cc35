"""GPU parity of the backward's last pass (K = 5, 7; scorer gradients, input gradient, far-query shares) where its ring of row stages
can go wrong: fewer rows than a stage, a stage and one row, several rounds of the ring with a remainder, two blocks per sequence."""
import numpy as np
import pytest
import torch

from oracle import lte_oracle as orc
from paper_2510_20787_b200 import lte, synth
from tests.gpu_util import assert_grad_close, dev, shape_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,K,T", [(64, 7, 9), (64, 5, 33), (64, 7, 227), (32, 7, 65), (32, 5, 300), (128, 7, 17), (128, 5, 131), (64, 7, 1100), (128, 7, 1029)])
@pytest.mark.parametrize("flags", [0, 1])
def test_row_stages(d, K, T, flags):
    cfg = synth.Config("tail", "bf16", 1, 2, d, T, 8, 6, K, 0.1)
    x = synth.make(cfg, 31, with_dO=True)
    s = shape_of(cfg)
    c = lte.conv(torch.from_numpy(x["w"]).cuda())
    q, k, v, dO = (dev(x[n], "bf16") for n in ("q", "k", "v", "dO"))
    z = lte.lte_scores(s, c, k, v)
    idx, cnt = lte.lte_select(s, z)
    o, lse = lte.lte_attn_prefill(s, q, k, v, idx, cnt)
    lam = torch.tensor([0.3, 0.0]).cuda()
    _, dk, dv, dw, db = lte.lte_attn_bwd(s, c, q, k, v, o, lse, dO, z, idx, cnt, lam=lam, flags=flags)
    assert lte.lte_device_status() == 0
    idx_n, cnt_n = idx.cpu().numpy(), cnt.cpu().numpy()
    g = orc.attn_bwd(x["q"], x["k"], x["v"], x["dO"], orc.scores(x["k"], x["v"], x["w"]), idx_n, cnt_n, x["w"], cfg.W,
                     lam=np.array([0.3, 0.0]), cnn_input_grad=bool(flags))
    assert_grad_close("dk", dk.float().cpu().numpy(), g["dk"], 5e-2, idx_n, cnt_n)
    assert_grad_close("dv", dv.float().cpu().numpy(), g["dv"], 5e-2, idx_n, cnt_n)
    assert_grad_close("dw", dw.cpu().numpy(), g["dw"], 5e-2)
    assert_grad_close("dbias", db.cpu().numpy(), g["dbias"], 5e-2)
