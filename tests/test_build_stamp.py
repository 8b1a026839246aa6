"""What a rebuild depends on: a change of anything that goes into libxkv.so or its Python module changes the stamp."""
import sysconfig

import torch
from torch.utils import cpp_extension

from paper_2503_18893_b200 import build


def test_the_stamp_follows_torch(monkeypatch):
    stamp = build._stamp()
    assert build._stamp() == stamp
    with monkeypatch.context() as m:
        m.setattr(torch, "__version__", torch.__version__ + ".other")
        assert build._stamp() != stamp
    with monkeypatch.context() as m:
        m.setattr(cpp_extension, "include_paths", lambda *a, **k: ["/somewhere/else/include"])
        assert build._stamp() != stamp
    with monkeypatch.context() as m:
        m.setattr(cpp_extension, "library_paths", lambda *a, **k: ["/somewhere/else/lib"])
        assert build._stamp() != stamp
    with monkeypatch.context() as m:
        m.setattr(sysconfig, "get_paths", lambda *a, **k: {"include": "/somewhere/else/python"})
        assert build._stamp() != stamp
    assert build._stamp() == stamp
