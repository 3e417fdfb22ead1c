"""The library is rebuilt when any file that its sources include has changed."""
import os
import re


def test_every_included_file_is_a_dependency():
    from paper_1809_02390_gb300 import build

    deps = {os.path.basename(d) for d in build.dependencies()}
    assert all(os.path.exists(d) for d in build.dependencies())
    for path in build.dependencies():
        for name in re.findall(r'^#include "([^"]+)"', open(path).read(), flags=re.M):
            assert os.path.basename(name) in deps, (path, name)
    assert {"lbm_launch.cuh", "lbm.h", "lbm3d.h", "lbm_capi.cu"} <= deps


def test_a_newer_dependency_makes_the_library_stale(monkeypatch):
    from paper_1809_02390_gb300 import build

    build.build()
    assert not build._stale()
    t = os.path.getmtime(build.LIB)
    for path in build.dependencies():
        real = os.path.getmtime
        monkeypatch.setattr(os.path, "getmtime", lambda p, f=path: t + 1 if p == f else real(p))
        assert build._stale(), path
        monkeypatch.undo()
