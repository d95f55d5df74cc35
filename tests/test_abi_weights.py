"""The tensor-core scorers read their weights in 16-byte pieces, so calls that run them refuse weights that start elsewhere (a read there would fault
the GPU); fp32 calls and the decode step read them element by element and do not.  Needs no GPU: what passes the check ends at the next one."""
import ctypes

import pytest

from paper_2510_20787_b200 import lte

FAKE = 4096          # never dereferenced: validation fails first


@pytest.mark.parametrize("dtype,offset,refused", [(lte.BF16, 4, True), (lte.BF16, 8, True), (lte.BF16, 0, False), (lte.F32, 4, False)])
def test_weights_off_a_16_byte_boundary(dtype, offset, refused):
    L, a = lte.lib(), ctypes.addressof
    s, conv = lte.shape(1, 2, 128, 64, 16, 8, dtype), lte.LteConv(1, 5, 1, FAKE + offset, 0)
    if refused:                                               # (what is accepted would go on to the device)
        assert L.lte_scores(a(s), a(conv), FAKE, FAKE, FAKE, None, None, 0, None) == -1
    chunk = L.lte_attn_prefill_chunk(a(s), a(conv), FAKE, 0, FAKE, FAKE, FAKE, FAKE, FAKE, None, 0, None)
    assert chunk == (-1 if refused else -3)                   # -3: the workspace, which is asked for next
