"""A library older than any file it is made from is built again: the dependency list holds every source
and every header that the sources include, directly or through another header."""
import os
import re

from paper_2205_02380_gb300 import build as B


def test_dependencies_hold_every_included_file():
    deps = {os.path.realpath(p) for p in B.dependencies()}
    todo = [os.path.join(B.CSRC, s) for s in B.SOURCES]
    seen = set()
    while todo:
        path = os.path.realpath(todo.pop())
        if path in seen:
            continue
        seen.add(path)
        with open(path) as fh:
            for name in re.findall(r'^\s*#include "([^"]+)"', fh.read(), re.M):
                inc = os.path.join(os.path.dirname(path), name)
                todo.append(inc if os.path.exists(inc) else os.path.join(B.HERE, "..", "include", name))
    assert len(seen) > len(B.SOURCES)
    assert seen <= deps


def test_a_changed_header_makes_the_library_stale(tmp_path, monkeypatch):
    lib = tmp_path / "lib.so"
    lib.write_text("")
    monkeypatch.setattr(B, "LIB", str(lib))
    monkeypatch.setattr(B, "BUILD", str(tmp_path / "o"))
    newest = max(os.path.getmtime(p) for p in B.dependencies())
    built = []

    def compile_one(src, verbose):
        built.append(src)
        raise RuntimeError("compiler called")

    monkeypatch.setattr(B, "_compile", compile_one)
    os.utime(lib, (newest + 10, newest + 10))
    assert B.build() == str(lib) and not built
    header = os.path.join(B.CSRC, "fft_fx.cuh")
    monkeypatch.setattr(B.os.path, "getmtime", lambda p, get=os.path.getmtime: newest + 20
                        if os.path.realpath(p) == os.path.realpath(header) else get(p))
    try:
        B.build()
    except RuntimeError as e:
        assert "compiler called" in str(e)
    assert built
