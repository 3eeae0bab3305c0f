"""An edit of any source that the library is compiled from makes it out of date."""
import glob
import os
import re

from paper_2108_08769_gb300 import build


def test_every_included_file_is_a_dependency():
    seen, todo = set(), [os.path.abspath(p) for p in build.sources()]
    while todo:
        path = todo.pop()
        if path in seen:
            continue
        seen.add(path)
        for name in re.findall(r'^#include "([^"]+)"', open(path).read(), re.M):
            for d in (os.path.dirname(path), build.CSRC, build.INCLUDE):
                p = os.path.abspath(os.path.join(d, name))
                if os.path.exists(p):
                    todo.append(p)
                    break
            else:
                raise AssertionError(f"{path} includes {name}, which is nowhere")
    deps = {os.path.abspath(p) for p in build._deps()}
    assert seen <= deps, sorted(os.path.basename(p) for p in seen - deps)
    assert {os.path.abspath(p) for p in glob.glob(os.path.join(build.CSRC, "*.*"))} <= deps


def test_a_newer_header_means_a_new_build(monkeypatch, tmp_path):
    lib = tmp_path / "lib.so"
    lib.write_bytes(b"")
    monkeypatch.setattr(build, "LIB", str(lib))
    newest = max(os.path.getmtime(p) for p in glob.glob(os.path.join(build.CSRC, "*")) + build._deps())
    os.utime(lib, (newest + 10, newest + 10))
    assert build.up_to_date()
    header = next(p for p in glob.glob(os.path.join(build.CSRC, "*.h")))
    real = os.path.getmtime

    monkeypatch.setattr(build.os.path, "getmtime", lambda p: newest + 20 if p == header else real(p))
    assert not build.up_to_date()
