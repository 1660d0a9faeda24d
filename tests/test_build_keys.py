"""Objects and the library are rebuilt by content and flags, not by times: a
stand-in for the compiler writes what it was given."""
import os
import stat

import pytest

from paper_2303_16999_gb300 import build as B

FAKE = """#!/usr/bin/env python3
import sys
a = sys.argv[1:]
out = a[a.index("-o") + 1]
if "-c" in a:
    src = a[a.index("-c") + 1]
    text = open(src).read() + "|" + open(%r).read() + "|" + ",".join(x for x in a if x[:2] == "-D")
    open(%r, "a").write(src + "\\n")
else:
    text = ";".join(open(x).read() for x in a if x.endswith(".o"))
open(out, "w").write(text)
"""


@pytest.fixture
def tree(tmp_path, monkeypatch):
    csrc, inc, out = tmp_path / "csrc", tmp_path / "include", tmp_path / "_build"
    csrc.mkdir()
    inc.mkdir()
    (csrc / "a.cu").write_text("A1")
    (csrc / "b.cpp").write_text("B1")
    (csrc / "h.cuh").write_text("H1")
    nvcc = tmp_path / "nvcc"
    nvcc.write_text(FAKE % (str(csrc / "h.cuh"), str(tmp_path / "log")))
    nvcc.chmod(nvcc.stat().st_mode | stat.S_IXUSR)
    for name, v in (("ROOT", tmp_path), ("CSRC", csrc), ("OUT_DIR", out),
                    ("LIB", out / "lib.so"), ("NVCC", nvcc)):
        monkeypatch.setattr(B, name, str(v))

    class Tree:
        def compiled(self):
            log = tmp_path / "log"
            lines = log.read_text().split() if log.exists() else []
            log.write_text("")
            return sorted(os.path.basename(x) for x in lines)

        def lib(self):
            return (out / "lib.so").read_text()
    t = Tree()
    t.csrc = csrc
    return t


def test_nothing_is_compiled_twice(tree):
    B.build()
    assert tree.compiled() == ["a.cu", "b.cpp"] and tree.lib() == "A1|H1|;B1|H1|"
    B.build()
    assert tree.compiled() == []


def test_a_plain_build_after_one_with_flags(tree):
    B.build()
    B.build(extra=["-DX=1"])
    assert tree.lib() == "A1|H1|-DX=1;B1|H1|-DX=1"
    B.build()
    assert tree.lib() == "A1|H1|;B1|H1|"
    tree.compiled()
    B.build(extra=["-DX=1"])
    assert tree.compiled() == [] and tree.lib() == "A1|H1|-DX=1;B1|H1|-DX=1"


def test_a_header_of_an_older_time(tree):
    """A header changed back to an earlier file (with its time): every object
    follows it."""
    B.build()
    tree.compiled()
    (tree.csrc / "h.cuh").write_text("H0")
    os.utime(tree.csrc / "h.cuh", (1, 1))
    B.build()
    assert tree.compiled() == ["a.cu", "b.cpp"] and tree.lib() == "A1|H0|;B1|H0|"


def test_objects_without_their_keys_are_rebuilt(tree):
    B.build()
    tree.compiled()
    os.remove(os.path.join(B.OUT_DIR, "a.cu.o.key"))
    os.remove(os.path.join(B.OUT_DIR, "b.cpp.o"))
    B.build()
    assert tree.compiled() == ["a.cu", "b.cpp"] and tree.lib() == "A1|H1|;B1|H1|"
