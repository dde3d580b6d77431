"""What the build script builds, in which order and when again; no compiler runs."""
import importlib.util
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture
def built(monkeypatch, tmp_path):
    """The build script with its targets in a folder of their own, and the targets of the compilers it called."""
    spec = importlib.util.spec_from_file_location("_build_under_test", os.path.join(ROOT, "paper_2505_00232_b200", "build.py"))
    b = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(b)
    b.LIB, b.NATIVE, calls = str(tmp_path / "lib.so"), str(tmp_path / "native.so"), []

    def compiler(cmd, **kw):
        target = cmd[cmd.index("-o") + 1]
        calls.append(os.path.basename(target))
        with open(target, "w") as f:
            f.write("".join(c[len('-DQL_BUILT_FOR="'):-1] + "\0" for c in cmd if c.startswith("-DQL_BUILT_FOR")))
    monkeypatch.setattr(b.subprocess, "check_call", compiler)
    return b, calls


def test_the_library_comes_first_and_needs_no_torch(built, monkeypatch):
    b, calls = built
    b.build()
    assert calls == ["lib.so", "native.so"]
    find_spec = importlib.util.find_spec
    monkeypatch.setattr(b.importlib.util, "find_spec", lambda name, *a: None if name == "torch" else find_spec(name, *a))
    assert b.build(force=True) == b.LIB and calls == ["lib.so", "native.so", "lib.so"]


def test_the_module_is_built_again_for_another_torch_or_python(built, monkeypatch):
    b, calls = built
    b.build()
    b.build()
    assert calls == ["lib.so", "native.so"]
    folder, name = b.installed_torch()
    for other in (name.replace("torch ", "torch 9."), name[:-1]):
        monkeypatch.setattr(b, "installed_torch", lambda: (folder, other))
        b.build()
        b.build()
        assert calls.pop() == "native.so" and calls == ["lib.so", "native.so"]


def test_a_module_for_another_torch_is_not_loaded(_built_library, monkeypatch):
    import paper_2505_00232_b200 as P
    native = P.binding._bind_torch()
    import torch
    assert torch.__version__ in native.built_for
    monkeypatch.setattr(P.binding, "_native", None)
    monkeypatch.setattr("paper_2505_00232_b200.build.installed_torch", lambda: ("", "torch 9"))
    with pytest.raises(ImportError):
        P.binding._bind_torch()
