"""The tensor-core scorer stack where the resident weights change with almost every tile: more heads than thread blocks, so that a block
goes through several heads of one, two or three tiles each (120 logits per tile), and through batch entries of one head between."""
import numpy as np
import pytest
import torch

from oracle import lte_oracle as orc
from paper_2510_20787_b200 import lte, synth
from tests.gpu_util import dev, shape_of
from tests.test_gpu_scores_stack import _stack_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,T,d", [(1, 700, 40, 64), (1, 300, 127, 64), (2, 160, 130, 64), (3, 150, 13, 64), (1, 200, 247, 64), (1, 500, 60, 32)])
def test_many_heads(B, H, T, d):
    cfg = synth.Config("heads", "bf16", B, H, d, T, 7, 4, 7, 0.1)
    x = synth.make(cfg, 31)
    wl, wout, bl, bout = _stack_params(H, d, 31, True)
    z64 = orc.scores_stack(x["k"], x["v"], wl, bl, wout, bout)
    t = lambda a: torch.from_numpy(a).cuda()
    c = lte.conv_stack([t(w) for w in wl], t(wout), [t(b) for b in bl], t(bout))
    z = lte.lte_scores(shape_of(cfg, B=B), c, dev(x["k"], "bf16"), dev(x["v"], "bf16"))
    assert lte.lte_device_status() == 0
    zn = z.cpu().numpy().astype(np.float64)
    fin = np.isfinite(z64)
    assert np.array_equal(np.isfinite(zn), fin)
    # a few ulp of fp32 sums of up to 384 products, through three layers (the bound of the other tests of this kernel)
    assert np.max(np.abs(zn[fin] - z64[fin])) <= 2e-5 * max(1.0, np.max(np.abs(z64[fin])))
