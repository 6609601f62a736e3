"""What the build needs and when it repeats itself: the C library takes the CUDA
toolkit alone, with or without a torch to build the Python binding against."""
import os
import subprocess
import sys

import pytest

from paper_2607_21475_gb300 import build as b

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_the_library_builds_without_torch(tmp_path):
    """A fresh build directory, one small source, and an interpreter in which torch
    cannot be imported."""
    code = f"""
import sys
sys.modules["torch"] = None  # import torch raises ImportError
from paper_2607_21475_gb300 import build as b
b.BUILD = {str(tmp_path)!r}
b.LIB, b.CALL = b.BUILD + "/libebd.so", b.BUILD + "/ebd_call.so"
b._sources = lambda: [b.CSRC + "/selftest.cu"]
import os
assert b.build() == b.LIB and os.path.exists(b.LIB) and not os.path.exists(b.CALL)
before = os.stat(b.LIB).st_mtime_ns
b.build()
assert os.stat(b.LIB).st_mtime_ns == before  # nothing changed: not built again
"""
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr


def test_the_binding_is_built_again_for_another_torch_or_python(monkeypatch):
    here = b._call_digest("2.9.1")
    assert here == b._call_digest("2.9.1") != b._call_digest("2.11.0")
    monkeypatch.setattr(sys, "version", "3.99.0")
    assert b._call_digest("2.9.1") != here


def test_the_binding_takes_the_python_way_where_it_was_not_built(monkeypatch, tmp_path):
    torch = pytest.importorskip("torch")
    b.build()
    from paper_2607_21475_gb300 import ebd as E
    monkeypatch.setattr(E, "CALL", str(tmp_path / "missing.so"))
    monkeypatch.setattr(E, "_CALL", None)
    c = E.alloc_compact(1, 1, 64, 64, torch.float32, "cpu")
    des = E.design_for(batch=1, n_kv_heads=1, group=1, head_dim=64, n_ctx=64, k_head=1,
                       budget_tokens=40)
    with pytest.raises(ValueError):  # the Python checks' answer to a CPU tensor
        E.ebd_select(des, torch.zeros(1, 1, 64), c)
