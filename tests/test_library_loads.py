"""Host-side checks that need no GPU: the library builds for sm_100a, loads, and exports every
symbol the header declares; the binding refuses to run without a device."""
import os
import re
import shutil
import subprocess
import sys
import sysconfig

import pytest
import torch

import paper_2202_02365_b200 as mg
from paper_2202_02365_b200 import api, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared():
    text = open(os.path.join(ROOT, "include", "mgdense.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(mg_[a-z0-9_]+)\s*\(", text)))


def test_builds_and_exports_every_declared_symbol():
    import __graft_entry__ as ge
    ge.build()
    lib = mg.load_library()
    names = _declared()
    assert len(names) >= 20
    for name in names:
        assert hasattr(lib, name), name
    assert sorted(api.EXPORTS) == names


# the library needs nothing of the native views: a copy of it loads, and plans, where they were not built
def test_loads_without_the_native_views(tmp_path):
    package = tmp_path / "paper_2202_02365_b200"
    package.mkdir()
    for name in ("__init__.py", "api.py", "build.py", "inputs.py", "libmgdense.so"):
        shutil.copy(os.path.join(api.HERE, name), package / name)
    code = ("import paper_2202_02365_b200 as mg; from paper_2202_02365_b200 import api; assert api.HERE != %r; "
            "assert mg.load_library().mg_kernel_launches(None) == 0 and len(api.comet_plan(8, 4, 2, 1)['sets']) >= 1" % api.HERE)
    ran = subprocess.run([sys.executable, "-c", code], cwd=tmp_path, capture_output=True, text=True)
    assert ran.returncode == 0, ran.stderr[-2000:]


# native views that were built for another torch or another Python are not taken for those of this one: neither loaded nor left unbuilt
def test_native_views_belong_to_their_versions(monkeypatch):
    build.build()
    assert os.path.exists(build.views_path())
    for module, name, value in ((torch, "__version__", "0.0.0+other"), (sysconfig, "get_config_var", lambda name: "cpython-00-other")):
        with monkeypatch.context() as m:
            m.setattr(module, name, value)
            m.setattr(api, "_views", None)
            asked = []
            m.setattr(build.subprocess, "run", lambda command, **_: asked.append(command) or subprocess.CompletedProcess(command, 0, "", ""))
            build.build()
            assert [c[c.index("-o") + 1] for c in asked] == [build.views_path()]      # (the library itself is as it was)
            with pytest.warns(RuntimeWarning, match="missing"):
                assert api._load_views() is False


# the library is built where the views cannot be: without Python's headers, and where their compiler fails (which is said, behind the library)
def test_builds_the_library_whatever_becomes_of_the_views(monkeypatch, tmp_path, capsys):
    asked = []

    def run(command, **_):
        asked.append(command)
        return subprocess.CompletedProcess(command, int(command[0] == "g++"), "", "")
    monkeypatch.setattr(build.subprocess, "run", run)
    with monkeypatch.context() as m:
        m.setattr(sysconfig, "get_paths", lambda: {"include": str(tmp_path)})
        assert build.build(force=True) == build.LIB
    assert "Python.h" in capsys.readouterr().err and build.LIB in asked[-1] and all(c[0] != "g++" for c in asked)
    asked.clear()
    with pytest.raises(RuntimeError, match="compiler failed"):
        build.build(force=True)
    assert any(build.LIB in c for c in asked)


@pytest.mark.skipif(torch.cuda.is_available(), reason="checks the no-GPU behaviour")
def test_no_cpu_fallback():
    with pytest.raises(RuntimeError):
        mg.Context(0)
    import ctypes as C
    lib = mg.load_library()
    h = C.c_void_p(0)
    assert lib.mg_create(C.byref(h), 0, None) != 0      # fails cleanly, no crash
    assert not h.value
