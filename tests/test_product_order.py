"""Two tensor-core products are known to run in their order only if they have the same accumulator.  Where P takes the place of the S it came
from, the next S of that buffer is another accumulator's product over columns that P V reads, so it may be issued only when P V is known to be
complete.  This is read off the sources: between the issue of P V and of that S there is a wait for P V's barrier."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_20787_b200", "csrc")


@pytest.mark.parametrize("source", ["prefill_tc.cu", "prefill_tc_long.cu"])
def test_s_is_issued_over_p_only_behind_its_product(source):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, source)).read())
    loop = text[text.index("umma_ts("):]
    assert text.count("umma_ts(") == 1 and "umma_commit(" in loop
    behind = loop[:loop.index("mma_s()")]
    assert re.search(r"umma_commit\([^;]*bar_pv", behind)
    assert re.search(r"mbar_wait(_u)?\([^;]*bar_pv", behind[behind.index("bar_pv"):])
