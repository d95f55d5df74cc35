"""CPU-side checks of the native Python binding: wrong arguments raise, they do not reach the library."""
import os
import subprocess
import sys

import pytest
import torch

from paper_2510_20787_b200 import lte

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_missing_structs_raise():
    """None in the place of the shape or of the scorer is a TypeError (in a process of its own: it once ended the interpreter)."""
    code = """
import torch
from paper_2510_20787_b200 import lte
s, c, x = lte.shape(1, 2, 8, 32, 5, 2, lte.F32), lte.LteConv(1, 5, 1, 256, 0), torch.zeros(4)
calls = {
    "lte_scores": (s, c, x, x), "lte_select": (s, x), "lte_select_rule": (s, lte.RULE_ACCUM_ATTN, x), "lte_attn_colsum": (s, x, x, x, x, x),
    "lte_attn_prefill": (s, x, x, x, x, x), "lte_cache_init": (s, c, x, x, x, x, x, x), "lte_attn_decode": (s, c, x, x, x, x),
    "lte_attn_prefill_chunk": (s, c, x, 0, x, x, x), "lte_sparsity_stats": (s, x), "lte_cache_score": (s, c, x),
    "lte_cache_score_unrope": (s, c, x, x, x), "lte_attn_bwd": (s, c) + (x,) * 9, "lte_attn_bwd_static": (s, c) + (x,) * 9,
}
for name, args in calls.items():
    for i, a in enumerate(args):
        if a is s or a is c:
            try:
                getattr(lte, name)(*args[:i], None, *args[i + 1:])
            except TypeError:
                continue
            raise SystemExit("%s took None as argument %d" % (name, i))
print("done")
"""
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "done", (r.returncode, r.stdout, r.stderr)


def test_outputs_are_never_allocated_off_the_gpu():
    """lte_select_rule is told where to allocate: on the host the library's kernels could not write them."""
    s = lte.shape(1, 2, 64, 32, 8, 4, lte.F32)
    with pytest.raises(AssertionError):
        lte.lte_select_rule(s, lte.RULE_UNIFORM, device="cpu")


def test_an_exception_on_the_way_to_the_library_is_raised():
    """Without a GPU torch has no current stream and throws; with one the library refuses the missing cache.  Either way Python sees an
    exception (in a process of its own: thrown without the interpreter lock it ended the process)."""
    code = """
from paper_2510_20787_b200 import lte
try:
    lte._load().cache_init(lte.shape(1, 2, 0, 32, 5, 2, lte.F32), lte.LteConv(1, 5, 1, 256, 0), None, None, None, None, None, None)
except RuntimeError:
    print("done")
"""
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "done", (r.returncode, r.stdout, r.stderr[-500:])


def test_rotary_tables_are_required():
    """lte_cache_score_unrope without its tables would score rotated keys as they are: lte_cache_score is the call for that."""
    s, c, x = lte.shape(1, 2, 0, 32, 20, 2, lte.F32), lte.LteConv(3, 3, 2, 256, 0), torch.zeros(4)
    for tables in ((None, None), (x, None), (None, x)):
        with pytest.raises(TypeError):
            lte.lte_cache_score_unrope(s, c, x, *tables)
