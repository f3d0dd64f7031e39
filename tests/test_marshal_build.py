"""Which build of the binding's marshalling module is used (host only)."""
import os

import torch

from paper_2312_00752_b200 import binding as K, build as B


def test_a_module_built_for_another_torch_is_not_taken_for_this_one(monkeypatch):
    here = B.build_marshal()
    assert os.path.exists(here) and not B.marshal_is_stale()
    assert K._native().__file__ == here
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    assert B.marshal_path() != here and B.marshal_is_stale()
    monkeypatch.undo()
    monkeypatch.setattr(torch.version, "git_version", "0123456789abcdef")
    assert B.marshal_path() != here and B.marshal_is_stale()
    monkeypatch.undo()
    monkeypatch.setattr(B.sysconfig, "get_config_var", lambda name: "cpython-399-other")
    assert B.marshal_path() != here and B.marshal_is_stale()
