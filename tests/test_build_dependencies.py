"""A change in any file that a source includes makes the library stale."""
import os
import re

from paper_2203_07820_gb300 import _build


def test_every_included_file_is_a_dependency():
    deps = {os.path.realpath(d) for d in _build.dependencies()}
    assert {os.path.realpath(os.path.join(_build.CSRC, s)) for s in _build.sources()} <= deps
    seen = 0
    for d in sorted(deps):
        for inc in re.findall(r'^\s*#include "([^"]+)"', open(d).read(), flags=re.M):
            assert os.path.realpath(os.path.join(os.path.dirname(d), inc)) in deps, (d, inc)
            seen += 1
    assert seen > 20


def test_a_newer_header_triggers_a_build(tmp_path, monkeypatch):
    lib = tmp_path / "lib.so"
    lib.write_text("built")
    newest = max(os.path.getmtime(d) for d in _build.dependencies())
    os.utime(lib, (newest, newest))
    monkeypatch.setattr(_build, "LIB", str(lib))
    monkeypatch.setattr(_build, "BUILD", str(tmp_path / "b"))
    compiled = []

    def compile_(src, verbose):
        compiled.append(src)
        raise RuntimeError("compiled")

    monkeypatch.setattr(_build, "_compile", compile_)
    assert _build.build() == str(lib) and not compiled
    real = os.path.getmtime
    monkeypatch.setattr(_build.os.path, "getmtime",
                        lambda f: newest + 1 if os.path.basename(f) == "nonlocal.cuh" else real(f))
    try:
        _build.build()
    except RuntimeError:
        pass
    assert compiled
