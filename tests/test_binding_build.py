"""The CPython binding belongs to one torch: which object is built, which one is found, and what happens without it."""
import os
import sys
import warnings

import pytest
import torch

from paper_2502_05003_b200 import _lib, build


def test_the_name_carries_the_torch_version_and_the_module_loads(monkeypatch):
    build.build()
    name = build.binding_name()
    monkeypatch.setattr(torch, "__version__", "9.8.7+other")
    assert build.binding_name() != name and build.binding_name().isidentifier()
    monkeypatch.undo()
    monkeypatch.setattr(_lib, "_binding", None)
    assert _lib.binding().__name__.split(".")[-1] == name


def test_another_torch_is_built_for_although_an_object_is_there(monkeypatch, tmp_path):
    build.build()
    commands = []

    def compiled(cmd):
        commands.append(cmd)
        open(cmd[cmd.index("-o") + 1], "w").close()
    monkeypatch.setattr(build.subprocess, "check_call", compiled)
    assert os.path.exists(build.build_binding()) and not commands           # up to date for this torch
    here = build.build_binding()
    monkeypatch.setattr(torch, "__version__", "9.8.7+other")
    target = build.build_binding()
    try:
        assert len(commands) == 1 and target != here and os.path.exists(target)
        assert f"-DQUEST_BINDING={build.binding_name()}" in commands[0]
    finally:
        os.remove(target)
    monkeypatch.setattr(torch.version, "cuda", None)
    assert build.build_binding() is None and len(commands) == 1             # a torch without CUDA: nothing to compile against


def test_calls_go_through_ctypes_where_there_is_no_binding(monkeypatch):
    import paper_2502_05003_b200 as quest
    build.build()
    monkeypatch.setattr(_lib, "_binding", None)
    monkeypatch.setattr(torch, "__version__", "9.8.7+other")
    with pytest.warns(RuntimeWarning, match="go through ctypes"):
        assert _lib.binding().linear_fwd(1, 2, 3) is None
    with warnings.catch_warnings():
        warnings.simplefilter("error")                                      # said once
        with pytest.raises(ValueError):
            quest.quest_quantize(torch.zeros(4, 128), 4, 128)
    assert "_binding_torch_9_8_7_other" not in " ".join(sys.modules)


def test_an_object_that_does_not_load_is_passed_over(monkeypatch):
    build.build()
    monkeypatch.setattr(_lib, "_binding", None)
    monkeypatch.setattr(torch, "__version__", "9.8.7+broken")
    path = os.path.join(build.HERE, build.binding_name() + ".so")
    with open(path, "w") as f:
        f.write("not an object")
    try:
        with pytest.warns(RuntimeWarning, match="does not load"):
            assert _lib.binding().quantize() is None
    finally:
        os.remove(path)
