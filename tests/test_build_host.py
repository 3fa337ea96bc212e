"""Objects are rebuilt when a header changes: every quoted include of the CUDA
sources and headers is among the files that the build watches."""
import glob
import os
import re

from paper_1102_3094_gb300 import _build


def test_every_include_is_watched():
    watched = {os.path.basename(f) for f in _build.headers()}
    for path in glob.glob(os.path.join(_build.CSRC, "*")) + glob.glob(os.path.join(_build.INCLUDE, "*")):
        for name in re.findall(r'^#include "([^"]+)"', open(path).read(), flags=re.M):
            assert name in watched, f"{os.path.basename(path)} includes {name}"


def test_a_newer_header_makes_objects_stale(monkeypatch):
    newest = _build._deps_mtime()
    times = {os.path.join(_build.CSRC, "lf_cvt.h"): newest + 100.0}
    real = os.path.getmtime
    monkeypatch.setattr(_build.os.path, "getmtime", lambda f: times.get(f, real(f)))
    assert _build._deps_mtime() == newest + 100.0
