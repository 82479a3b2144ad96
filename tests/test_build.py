"""The incremental build looks at every file that a translation unit includes."""
import os
import re

from paper_1704_01127_gb300 import build


def test_every_included_file_is_a_dependency():
    known = {os.path.realpath(h) for h in build._headers()}
    files = [os.path.join(build.CSRC, f) for f in os.listdir(build.CSRC)]
    included = set()
    for f in files:
        for name in re.findall(r'^\s*#\s*include\s*"([^"]+)"', open(f).read(), flags=re.M):
            included.add(os.path.realpath(os.path.join(os.path.dirname(f), name)))
    assert included
    assert included <= known, sorted(included - known)


def test_a_changed_header_recompiles(monkeypatch, tmp_path):
    src = os.path.join(build.CSRC, "qs_pass.cu")
    obj = tmp_path / "qs_pass.cu.o"
    obj.write_bytes(b"")
    monkeypatch.setattr(build, "BUILD", str(tmp_path))
    compiled = []
    monkeypatch.setattr(build.subprocess, "check_call", compiled.append)
    newest = max(os.path.getmtime(f) for f in [src] + build._headers())
    os.utime(obj, (newest + 1, newest + 1))
    build._compile(src)
    assert not compiled
    newer = os.path.join(build.CSRC, "qs_launch.cuh")
    real = os.path.getmtime
    monkeypatch.setattr(build.os.path, "getmtime", lambda f: newest + 2 if f == newer else real(f))
    build._compile(src)
    assert len(compiled) == 1
