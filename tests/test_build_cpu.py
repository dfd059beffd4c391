"""What makes the native side of the binding stale."""
import importlib.metadata
import os

import pytest

from paper_2406_07368_b200 import build


class _Compiled(Exception):
    pass


def test_host_module_is_built_anew_for_another_torch(tmp_path, monkeypatch):
    monkeypatch.setattr(build, "HOST", str(tmp_path / "_host.so"))
    monkeypatch.setattr(build, "OBJ", str(tmp_path))

    def run(cmd, **kw):
        raise _Compiled

    monkeypatch.setattr(build.subprocess, "run", run)
    with pytest.raises(_Compiled):                               # nothing there yet
        build._build_host([])
    (tmp_path / "_host.so").write_bytes(b"")
    os.utime(tmp_path / "_host.so", (2 ** 31, 2 ** 31))          # newer than its source
    with pytest.raises(_Compiled):                               # built, but nobody knows for what
        build._build_host([])

    class _Done:
        returncode = 0

    monkeypatch.setattr(build.subprocess, "run", lambda cmd, **kw: _Done)
    build._build_host([])
    monkeypatch.setattr(build.subprocess, "run", run)
    build._build_host([])                                        # up to date
    monkeypatch.setattr(importlib.metadata, "version", lambda name: "0.0")
    with pytest.raises(_Compiled):
        build._build_host([])
