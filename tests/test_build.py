"""What build() makes anew: the CUDA library and the marshalling extension, each by its own sources."""
import os

import pytest

from paper_2509_16989_b200 import build


@pytest.fixture
def tree(tmp_path, monkeypatch):
    """Sources and artefacts of a tree of its own, the artefacts the newer ones; compilers only leave a trace."""
    csrc, include = tmp_path / "csrc", tmp_path / "include"
    csrc.mkdir()
    include.mkdir()
    for name in ("a.cu", "b.h", "marshal.cpp"):
        (csrc / name).touch()
    (include / "ptqtp.h").touch()
    for name, value in (("ROOT", tmp_path), ("CSRC", csrc), ("LIB", tmp_path / "libptqtp.so")):
        monkeypatch.setattr(build, name, str(value))
    monkeypatch.setattr(build, "marshal_path", lambda: str(tmp_path / "_marshal.so"))
    ran = []

    def run(cmd, **kw):
        ran.append(os.path.basename(cmd[0]))
        fails = ran[-1] == "false"
        if not fails:
            open(cmd[cmd.index("-o") + 1], "w").close()
        return type("Result", (), {"returncode": int(fails), "stdout": "no compiler"})()

    monkeypatch.setattr(build.subprocess, "run", run)
    monkeypatch.setenv("CXX", "g++")
    monkeypatch.setenv("NVCC", "nvcc")
    build.build()
    assert sorted(ran) == ["g++", "nvcc"] and not build.needs_build()
    ran.clear()
    return tmp_path, ran


def later(path):
    os.utime(str(path), (2e9, 2e9))


@pytest.mark.parametrize("changed,compiler", [("csrc/a.cu", "nvcc"), ("csrc/b.h", "nvcc"), ("csrc/marshal.cpp", "g++")])
def test_a_changed_source_makes_one_of_the_two_anew(tree, changed, compiler):
    root, ran = tree
    build.build()
    assert ran == []
    later(root / changed)
    assert build.needs_build()
    build.build()
    assert ran == [compiler]


def test_without_a_host_compiler_the_library_is_built_once(tree, monkeypatch, capsys):
    root, ran = tree
    monkeypatch.setenv("CXX", "false")
    later(root / "csrc/marshal.cpp")
    for _ in range(2):
        assert build.build() == build.LIB and os.path.exists(build.LIB)
        assert not os.path.exists(build.marshal_path())         # rather none than one of older sources
        assert "was not built" in capsys.readouterr().err
    assert ran == ["false", "false"]                     # and no nvcc
