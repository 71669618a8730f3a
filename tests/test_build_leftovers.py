"""A build that fails leaves nothing behind, no built file is in the history, and what was built for another torch is not used."""
import os
import shutil
import subprocess

import pytest

from paper_2607_03229_b200 import binding as B
from paper_2607_03229_b200 import build as build_mod

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_a_failed_build_leaves_no_library_behind(tmp_path, monkeypatch):
    pkg = tmp_path / "pkg"
    pkg.mkdir()
    src = pkg / "broken.cpp"
    src.write_text("int whole;\n")
    monkeypatch.setattr(build_mod, "HERE", str(pkg))
    monkeypatch.setattr(build_mod, "LIB", str(pkg / "libx.so"))
    monkeypatch.setattr(build_mod, "HOST_LIB", str(pkg / "_host.so"))
    monkeypatch.setattr(build_mod, "HOST_SRC", str(src))
    monkeypatch.setattr(build_mod, "sources", lambda: [str(pkg / "a.cu")])
    monkeypatch.setattr(build_mod, "host_command", lambda out: ["g++", "-shared", "-fPIC", str(src), "-o", out])
    monkeypatch.setenv("NVCC", shutil.which("false"))
    with pytest.raises(RuntimeError):
        build_mod.build()
    assert [f for _, _, files in os.walk(pkg) for f in files if ".so" in f] == []


def test_no_built_file_is_tracked():
    if shutil.which("git") is None or not os.path.isdir(os.path.join(ROOT, ".git")):
        pytest.skip("no history here")
    got = subprocess.run(["git", "-c", "safe.directory=*", "ls-files"], cwd=ROOT, capture_output=True, text=True)
    names = got.stdout.split()
    assert got.returncode == 0 and names
    assert [n for n in names if ".so" in os.path.basename(n) or n.endswith((".o", ".a", ".tmp", ".cubin"))] == []


def test_a_module_of_another_torch_is_rebuilt_and_not_loaded(monkeypatch):
    build_mod.build()
    assert build_mod.host_is_current() and not build_mod.is_stale()
    monkeypatch.setattr(build_mod, "built_for", lambda: "marshalling for torch 0.0.0, cpython-27")
    assert build_mod.is_stale()
    monkeypatch.setattr(B, "_lib", None)
    with pytest.raises(RuntimeError, match="another torch"):
        B.load()
