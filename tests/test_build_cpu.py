"""What the build notices and what a failed load says: an extension compiled for another Python or torch is rebuilt, the C
library is built where there is no torch, and an extension that cannot be loaded is not reported as missing."""
import os
import shutil
import subprocess
import sys

from paper_2601_19675_b200 import build

PACKAGE = os.path.dirname(os.path.abspath(build.__file__))


def test_an_extension_for_another_torch_is_stale(tmp_path, monkeypatch):
    build.build()
    stamp = tmp_path / "binding.txt"
    monkeypatch.setattr(build, "STAMP", str(stamp))
    stamp.write_text(build._binding_for())
    assert not build._stale()
    stamp.write_text("cpython-39 torch 1.0")
    assert build._stale()


def test_the_c_library_is_built_without_torch(tmp_path, monkeypatch):
    # the compiler is a stand-in that succeeds; what it was asked for shows what would have been built
    asked = tmp_path / "asked.txt"
    fake = tmp_path / "nvcc"
    fake.write_text(f'#!/bin/sh\necho "$@" >> {asked}\n')
    fake.chmod(0o755)
    monkeypatch.setattr(build, "_nvcc", lambda: str(fake))
    monkeypatch.setattr(build, "_torch_version", lambda: None)
    monkeypatch.setattr(build, "HERE", str(tmp_path))
    assert build.build(force=True) == build.LIB
    assert "api.cu" in asked.read_text() and "binding.cpp" not in asked.read_text()


def test_an_extension_that_cannot_be_loaded_is_named_so(tmp_path):
    build.build()
    there = tmp_path / "paper_2601_19675_b200"
    there.mkdir()
    for name in ("__init__.py", "lopro.py", "build.py"):
        shutil.copy(os.path.join(PACKAGE, name), there / name)
    os.symlink(build.LIB, there / "liblopro.so")
    (there / "_binding.so").write_bytes(b"not an extension")
    run = [sys.executable, "-c", "from paper_2601_19675_b200 import lopro; lopro.lib()"]
    out = subprocess.run(run, cwd=tmp_path, capture_output=True, text=True).stderr
    assert "_binding.so cannot be loaded here" in out
    (there / "_binding.so").unlink()
    out = subprocess.run(run, cwd=tmp_path, capture_output=True, text=True).stderr
    assert "_binding.so is missing" in out
