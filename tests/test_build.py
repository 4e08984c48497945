"""What the build considers stale, with the compilers replaced by a function that only writes their output."""
import os

import pytest

from paper_2505_03254_b200 import build


@pytest.fixture
def tree(tmp_path, monkeypatch):
    for name in ("api.cu", "tc.cuh", "native.cpp", "prom.h"):
        (tmp_path / name).write_text("")
    monkeypatch.setattr(build, "CSRC", str(tmp_path))
    monkeypatch.setattr(build, "INCLUDE", str(tmp_path))
    monkeypatch.setattr(build, "LIB", str(tmp_path / "libprom.so"))
    monkeypatch.setattr(build, "NATIVE", str(tmp_path / "_native.so"))
    monkeypatch.setattr(build, "NATIVE_SOURCE", str(tmp_path / "native.cpp"))
    built = []

    def compiler(cmd):
        target = cmd[cmd.index("-o") + 1]
        built.append(os.path.basename(target).split(".")[0])
        with open(target, "w"):
            pass
    monkeypatch.setattr(build.subprocess, "check_call", compiler)
    build.build()
    assert built == ["libprom", "_native"] and not build.needs_build()
    del built[:]
    build.build()
    assert built == []
    return tmp_path, built


@pytest.mark.parametrize("changed,rebuilt", [("tc.cuh", ["libprom"]), ("native.cpp", ["_native"]), ("prom.h", ["libprom", "_native"])])
def test_a_newer_source_is_noticed(tree, changed, rebuilt):
    path, built = tree
    later = max(os.path.getmtime(p) for p in path.iterdir()) + 10
    os.utime(path / changed, (later, later))
    assert build.needs_build()
    build.build()
    assert built == rebuilt
