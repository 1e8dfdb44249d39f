"""The build leaves nothing behind that it does not replace and knows what its products are good for; no compiled code is
part of the source tree."""
import os
import subprocess

import pytest

from paper_2609_35465_b200 import build as tbuild

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture
def away(tmp_path, monkeypatch):
    """The build's products in a folder of their own, without the compilers."""
    monkeypatch.setattr(tbuild, "LIB", str(tmp_path / "lib.so"))
    monkeypatch.setattr(tbuild, "BINDING", str(tmp_path / "binding.so"))
    monkeypatch.setattr(tbuild, "SOURCES", ["tetra_tables.cpp"])
    monkeypatch.setattr(tbuild, "_binding_command", lambda out: ["touch", out])
    return tmp_path


def test_a_failed_compiler_leaves_no_files(away, monkeypatch):
    monkeypatch.setattr(tbuild, "NVCC", "false")
    with pytest.raises(RuntimeError):
        tbuild.build(force=True)
    assert os.listdir(away) == []


def test_an_interrupted_build_leaves_no_files(away, monkeypatch):
    def interrupted(*args, **kwargs):
        raise KeyboardInterrupt
    monkeypatch.setattr(tbuild, "NVCC", "true")
    monkeypatch.setattr(tbuild.subprocess, "run", interrupted)
    with pytest.raises(KeyboardInterrupt):
        tbuild.build(force=True)
    assert os.listdir(away) == []


def test_a_finished_build_is_not_stale(away, monkeypatch):
    """Its objects lie beside the sources and may be younger than the first of its two products."""
    csrc, old = away / "csrc", 1_000_000_000
    csrc.mkdir()
    monkeypatch.setattr(tbuild, "CSRC", str(csrc))
    monkeypatch.setattr(tbuild, "HERE", str(away / "include"))
    for name, at in (("a.cu", old), ("binding.cpp", old), ("a.o", old + 20)):
        (csrc / name).write_text("")
        os.utime(csrc / name, (at, at))
    (away / "include").mkdir()
    for h in ("tetra.h", "tetra_q4.h"):
        (away / "include" / h).write_text("")
        os.utime(away / "include" / h, (old, old))
    for path, at in ((tbuild.BINDING, old + 10), (tbuild.LIB, old + 30)):
        with open(path, "w") as f:
            f.write(tbuild.built_for())
        os.utime(path, (at, at))
    assert not tbuild._stale()
    os.utime(csrc / "a.cu", (old + 15, old + 15))
    assert tbuild._stale()


def test_a_binding_for_another_torch_is_stale_and_refused(monkeypatch):
    tbuild.build()
    assert not tbuild._stale()
    from paper_2609_35465_b200 import tetra
    monkeypatch.setattr(tetra, "_nat", None)
    tetra._native()
    monkeypatch.setattr(tetra, "_nat", None)
    monkeypatch.setattr(tbuild.sys, "version_info", (3, 99))
    assert tbuild._stale()
    with pytest.raises(tetra.TetraError, match="built for"):
        tetra._native()


def test_no_compiled_code_is_tracked():
    if not os.path.exists(os.path.join(ROOT, ".git")):
        pytest.skip("not a checkout")
    files = subprocess.run(["git", "ls-files", "-z"], cwd=ROOT, capture_output=True, check=True).stdout.decode().split("\0")
    for f in filter(None, files):
        path = os.path.join(ROOT, f)
        if os.path.isfile(path):
            with open(path, "rb") as fh:
                assert fh.read(4) != b"\x7fELF", f
