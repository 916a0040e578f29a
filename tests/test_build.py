"""What the build and the loader need, and what they do without it: the
library needs nvcc, the autograd node of render() torch's headers and a host
compiler, and neither is needed once its product is current."""
import os
import types
import warnings

import pytest

from paper_2508_06768_gb300 import binding as B
from paper_2508_06768_gb300 import build as _build
from paper_2508_06768_gb300 import render as R


@pytest.fixture
def tree(tmp_path, monkeypatch):
    """An empty output folder and compilers that only write their output; those
    named in `missing` fail."""
    monkeypatch.setattr(_build, "OUT_DIR", str(tmp_path))
    monkeypatch.setattr(_build, "LIB", str(tmp_path / "libdiffus.so"))
    monkeypatch.setattr(_build, "NODE", str(tmp_path / "diffus_torch.so"))
    monkeypatch.setattr(_build, "_nvcc", lambda: "nvcc")
    monkeypatch.setenv("CXX", "g++")
    t = types.SimpleNamespace(missing=set(), ran=[])

    def run(cmd, **kw):
        t.ran.append(cmd[0])
        if cmd[0] in t.missing:
            raise FileNotFoundError(cmd[0])
        open(cmd[cmd.index("-o") + 1], "w").close()
        return types.SimpleNamespace(returncode=0, stdout="", stderr="")

    monkeypatch.setattr(_build.subprocess, "run", run)
    return t


def _no_nvcc():
    raise RuntimeError("nvcc not found")


def test_current_build_needs_no_tools(tree, monkeypatch):
    assert _build.build() == _build.LIB and os.path.exists(_build.NODE)
    assert {"nvcc", "g++"} == set(tree.ran)
    tree.ran.clear()
    monkeypatch.setattr(_build, "_nvcc", _no_nvcc)
    tree.missing = {"nvcc", "g++"}
    assert _build.build() == _build.LIB and not tree.ran


@pytest.mark.parametrize("what", ["compiler", "torch"])
def test_library_builds_without_the_node(tree, monkeypatch, what):
    if what == "compiler":
        tree.missing = {"g++"}
    else:
        monkeypatch.setitem(__import__("sys").modules, "torch", None)
    with pytest.warns(RuntimeWarning, match="not built"):
        assert _build.build() == _build.LIB
    assert os.path.exists(_build.LIB) and not os.path.exists(_build.NODE)
    # the library is current all the same, and the node comes when it can
    tree.missing, n = {"nvcc"}, tree.ran.count("nvcc")
    if what == "compiler":
        _build.build()
        assert os.path.exists(_build.NODE) and tree.ran.count("nvcc") == n


def test_node_follows_the_installed_torch(tree, monkeypatch):
    import torch
    _build.build()
    assert _build.node_current()
    monkeypatch.setattr(torch, "__version__", "0.0.0")
    assert not _build.node_current()
    tree.ran.clear()
    _build.build_node()
    assert _build.node_current() and set(tree.ran) == {"g++"}
    # a missing library is an error as before
    tree.missing = {"nvcc"}
    os.remove(_build.LIB)
    with pytest.raises(OSError):
        _build.build()


def test_render_without_the_node(monkeypatch):
    def fail():
        raise RuntimeError("no headers")
    monkeypatch.setattr(B, "_node", None)
    monkeypatch.setattr(B, "load", lambda: None)
    monkeypatch.setattr(_build, "build_node", fail)
    with pytest.warns(RuntimeWarning, match="no headers"):
        assert B.load_node() is None
    monkeypatch.setattr(R, "_native_call", lambda *a: b"packed")
    monkeypatch.setattr(R, "_Render", types.SimpleNamespace(apply=lambda *a: a))
    with warnings.catch_warnings():
        warnings.simplefilter("error")
        assert R.render("v", "p", "fan", "prm") == ("v", "p", (1.0,) * 3, (0.0,) * 3, "fan", "prm", 0)
