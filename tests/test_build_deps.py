"""The in-tree build recompiles every translation unit that a changed source file reaches through #include (no compiler is
run: a stand-in writes the objects)."""
import glob
import os
import re
import shutil
import types

import pytest

from paper_2307_12607_gb300 import build


@pytest.fixture
def tree(tmp_path, monkeypatch):
    csrc, include, out = tmp_path / "csrc", tmp_path / "include", tmp_path / "out"
    shutil.copytree(build.CSRC, csrc)
    shutil.copytree(build.INCLUDE, include)
    monkeypatch.setattr(build, "CSRC", str(csrc))
    monkeypatch.setattr(build, "INCLUDE", str(include))
    monkeypatch.setattr(build, "OUT", str(out))
    monkeypatch.setattr(build, "LIB", str(out / "libexw.so"))
    monkeypatch.setattr(build, "nvcc", lambda: "nvcc")
    compiled = []

    def run(cmd, **kwargs):
        if "-c" in cmd:
            compiled.append(os.path.basename(cmd[cmd.index("-c") + 1]))
        open(cmd[cmd.index("-o") + 1], "w").close()
        return types.SimpleNamespace(returncode=0, stdout="", stderr="")

    monkeypatch.setattr(build.subprocess, "run", run)
    return compiled


def included(path, seen=()):
    """The files of the tree that path includes, directly or not."""
    files = set()
    for name in re.findall(r'#include\s+[<"]([^">]+)[">]', open(path).read()):
        for folder in (os.path.dirname(path), build.CSRC, build.INCLUDE):
            f = os.path.join(folder, name)
            if os.path.exists(f) and f not in seen:
                files |= {f} | included(f, seen + (f,))
    return files


def test_a_changed_file_rebuilds_every_unit_that_includes_it(tree):
    build.build()
    units = {os.path.basename(u): {u} | included(u) for u in glob.glob(os.path.join(build.CSRC, "*.cu"))}
    assert sorted(tree) == sorted(units)
    later = max(os.path.getmtime(f) for f in glob.glob(os.path.join(build.OUT, "*"))) + 10
    for f in sorted(set().union(*units.values())):
        tree.clear()
        os.utime(f, (later, later))
        build.build()
        missing = {u for u, files in units.items() if f in files} - set(tree)
        assert not missing, f"{os.path.basename(f)} changed and {sorted(missing)} were not compiled again"
        for o in glob.glob(os.path.join(build.OUT, "*")):
            os.utime(o, (later + 1, later + 1))
        later += 10
