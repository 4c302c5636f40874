"""The build's host logic, with compilers that only pretend: what it leaves behind and what it goes on without."""
import importlib
import os
import stat
import sys
import types

import pytest
import torch

from paper_2412_19829_b200 import binding as gf
from paper_2412_19829_b200 import build as gf_build

FAKE = """#!{python}
import sys
args = sys.argv[1:]
open(args[args.index("-o") + 1], "w").write("built")
sys.exit(1 if any(x in " ".join(args) for x in {fails!r}) else 0)
"""


@pytest.fixture
def tree(tmp_path, monkeypatch):
    """A package folder of its own; tree(fails) installs compilers that fail on commands with one of these words."""
    src = tmp_path / "csrc"
    src.mkdir()
    for f in ("a.cu", "b.cu", "fastcall.cpp"):
        (src / f).write_text("")
    (tmp_path / "include").mkdir()
    for name, value in (("HERE", tmp_path), ("CSRC", src), ("INCLUDE", tmp_path / "include"), ("LIB", tmp_path / "libgformer.so"),
                        ("FASTCALL", tmp_path / "_fastcall.so")):
        monkeypatch.setattr(gf_build, name, str(value))
    monkeypatch.setattr(gf_build, "SOURCES", ["a.cu", "b.cu"])

    def install(*fails):
        bin_dir = tmp_path / "bin"
        bin_dir.mkdir(exist_ok=True)
        for tool in ("nvcc", "g++"):
            f = bin_dir / tool
            f.write_text(FAKE.format(python=sys.executable, fails=fails))
            f.chmod(f.stat().st_mode | stat.S_IXUSR)
        monkeypatch.setenv("NVCC", str(bin_dir / "nvcc"))
        monkeypatch.setenv("PATH", f"{bin_dir}{os.pathsep}{os.environ['PATH']}")
        return tmp_path

    return install


def _left_behind(root):
    return [f for _, _, files in os.walk(root) for f in files if f.endswith(".tmp")]


@pytest.mark.parametrize("fails", ["a.cu", "-shared -o"])
def test_a_build_that_fails_leaves_nothing_behind(tree, fails):
    root = tree(fails)
    with pytest.raises(Exception):
        gf_build.build(force=True)
    assert _left_behind(root) == [] and not os.path.exists(gf_build.LIB)


def test_a_build_puts_both_files_in_place(tree):
    root = tree()
    assert gf_build._stale()
    assert gf_build.build(force=True) == gf_build.LIB
    assert os.path.exists(gf_build.LIB) and os.path.exists(gf_build.FASTCALL) and _left_behind(root) == []
    assert not gf_build._stale()


def test_the_library_is_built_where_the_module_of_the_binding_cannot_be(tree):
    tree()
    gf_build.build(force=True)
    root = tree("fastcall.cpp")
    assert gf_build.build(force=True) == gf_build.LIB
    assert os.path.exists(gf_build.LIB) and _left_behind(root) == []
    assert not os.path.exists(gf_build.FASTCALL)  # (no module of an earlier library beside this one)
    assert gf_build._stale()


def test_a_module_built_for_another_torch_is_stale(tree, monkeypatch):
    tree()
    gf_build.build(force=True)
    assert not gf_build._stale()
    monkeypatch.setattr(torch, "__version__", "9.9.9")
    assert gf_build._stale()


@pytest.mark.parametrize("case", ["missing", "other torch"])
def test_calls_go_through_ctypes_where_the_module_cannot_be_used(case, monkeypatch):
    real = importlib.import_module

    def fake(name, package=None):
        if name != "._fastcall":
            return real(name, package)
        if case == "missing":
            raise ImportError("no module")
        return types.SimpleNamespace(built_for="another")

    monkeypatch.setattr(gf, "_fast", None)
    monkeypatch.setattr(importlib, "import_module", fake)
    x = torch.zeros(1, 1, 4, 64)
    with pytest.warns(UserWarning, match="through ctypes"), pytest.raises(ValueError, match="CUDA tensors"):
        gf.window_attn(x, x, x, 4)
    with pytest.raises(ValueError, match="CUDA tensors"):
        gf.hybrid_attn(x, x, x, 4)
