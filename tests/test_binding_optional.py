"""The native call path is an addition: without it, or with one that was built
for another torch, every call still has its Python path, and a build replaces a
module that does not fit."""
import os

import pytest

torch = pytest.importorskip("torch")


@pytest.fixture()
def parts(monkeypatch):
    from paper_2510_15095_gb300 import build as B
    from paper_2510_15095_gb300 import hive as H

    L = H.load_library(B.build())
    monkeypatch.setattr(H, "_native", None)
    return B, H, L


def test_the_built_module_fits(parts):
    B, H, L = parts
    assert B.binding_fits()
    assert H._load_native(L).__name__ == "hive_binding"


@pytest.mark.parametrize("why", ["missing", "another torch", "broken"])
def test_python_takes_the_calls(parts, monkeypatch, tmp_path, why):
    B, H, L = parts
    so, stamp = tmp_path / "hive_binding.so", tmp_path / "built_for"
    if why != "missing":
        so.write_bytes(b"not a module")
    stamp.write_text(B.binding_key() if why == "broken" else "torch 0.1 cpython-39")
    monkeypatch.setattr(B, "BINDING", str(so))
    monkeypatch.setattr(B, "BINDING_STAMP", str(stamp))
    with pytest.warns(RuntimeWarning, match="ctypes"):
        n = H._load_native(L)
    for f in (n.insert, n.erase, n.find, n.execute, n.multi):
        assert f(1, 2, 3) is NotImplemented
    assert all(H._fn.values())


def test_build_replaces_a_module_for_another_torch(parts, monkeypatch):
    B, H, L = parts
    with open(B.BINDING_STAMP, "w") as f:
        f.write("torch 0.1 cpython-39")
    assert not B.binding_fits()
    before = os.path.getmtime(B.LIB)
    B.build()
    assert B.binding_fits() and os.path.getmtime(B.LIB) == before


def test_build_goes_on_without_the_module(parts, monkeypatch, capsys):
    B, H, L = parts
    monkeypatch.setattr(B, "BINDING_SRC", "no_such_file.cpp")
    monkeypatch.setattr(B, "_older", lambda path, sources: path == B.BINDING)
    assert B.build() == B.LIB
    assert "ctypes" in capsys.readouterr().err
