"""The in-tree build: an edit of any file the library is compiled from makes it stale."""
import os
import re

import pytest

from paper_1712_10279_gb300 import build as B


def _included(path, seen):
    """Every header of this repository that `path` includes, directly or not."""
    for name in re.findall(r'^\s*#include\s+"([^"]+)"', open(path).read(), flags=re.M):
        for d in (B.CSRC, B.INCLUDE):
            p = os.path.join(d, name)
            if os.path.exists(p) and p not in seen:
                seen.add(p)
                _included(p, seen)
    return seen


def test_every_included_header_is_a_dependency():
    headers = set()
    for src in B._sources():
        _included(src, headers)
    assert any(h.endswith(".cuh") for h in headers) and any(h.endswith(".h") for h in headers)
    assert headers <= set(B._deps())


@pytest.mark.parametrize("name", ["march2d.cuh", "resident_kernel.cuh", "internal.h", "api.cu"])
def test_a_newer_file_makes_the_library_stale(name, tmp_path, monkeypatch):
    lib = tmp_path / "lib.so"
    lib.write_bytes(b"")
    newest = max(os.path.getmtime(d) for d in B._deps())
    os.utime(lib, (newest + 10, newest + 10))
    monkeypatch.setattr(B, "LIB", str(lib))
    assert B.up_to_date()
    real = os.path.getmtime
    monkeypatch.setattr(B.os.path, "getmtime",
                        lambda p: newest + 20 if os.path.basename(p) == name else real(p))
    assert not B.up_to_date()
