"""When the native Python binding is built again."""
import subprocess
import types

import pytest
import torch

from paper_2510_20787_b200 import build, lte


def test_binding_is_built_again_for_another_torch(monkeypatch):
    """It is compiled against torch's C++ interface: a module built for another torch may not be kept."""
    assert torch.__version__ in lte._load().built_for
    tried = []
    monkeypatch.setattr(subprocess, "run", lambda cmd, **kw: tried.append(cmd) or types.SimpleNamespace(returncode=1, stdout="", stderr=""))
    monkeypatch.setattr(torch, "__version__", "0.0.0+other")
    with pytest.raises(RuntimeError):                          # (the compiler above always fails)
        build.build_binding()
    assert len(tried) == 1 and tried[0][0] == "g++"
