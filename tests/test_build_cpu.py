"""The in-tree build rebuilds every object when a header it includes changes."""
import os
import re

from paper_2203_05665_gb300 import _build


def test_every_included_header_is_a_dependency():
    deps = {os.path.realpath(os.path.join(_build.CSRC, h)) for h in _build.HEADERS}
    assert all(os.path.exists(d) for d in deps)
    for name in os.listdir(_build.CSRC):
        with open(os.path.join(_build.CSRC, name)) as f:
            for inc in re.findall(r'^\s*#include "([^"]+)"', f.read(), re.M):
                assert os.path.realpath(os.path.join(_build.CSRC, inc)) in deps, (name, inc)


def test_sources_are_all_compiled():
    assert sorted(_build.SOURCES) == sorted(f for f in os.listdir(_build.CSRC) if f.endswith((".cu", ".cpp")))


def test_newer_dependency_makes_an_object_stale(tmp_path):
    obj, hdr = tmp_path / "a.o", tmp_path / "a.hpp"
    hdr.write_text("")
    obj.write_text("")
    os.utime(hdr, (1, 1))
    assert not _build._stale(str(obj), [str(hdr)])
    os.utime(hdr, (2**31, 2**31))
    assert _build._stale(str(obj), [str(hdr)])
