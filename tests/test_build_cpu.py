"""How the libraries get into the tree: stand-ins for the compilers, in a folder of their own."""
import os
import shutil
import subprocess
import time
from concurrent.futures import ThreadPoolExecutor

import pytest
import torch

from paper_2506_18952_b200 import build as b


@pytest.fixture
def compiler(tmp_path, monkeypatch):
    """Both libraries are built in an empty folder by a script; returns a function that sets what it does with $out."""
    folder = tmp_path / "pkg"
    folder.mkdir()
    monkeypatch.setattr(b, "_PKG", str(folder))
    monkeypatch.setattr(b, "LIB", str(folder / "lib.so"))

    def does(body):
        script = tmp_path / "cc"
        script.write_text(f'#!/bin/sh\necho run >> {tmp_path}/runs\n'
                          'while [ "$1" != -o ]; do shift; done\nout=$2\n' + body + "\n")
        script.chmod(0o755)
        for name in ("NVCC", "CXX"):
            monkeypatch.setenv(name, str(script))
    does.runs = lambda: len((tmp_path / "runs").read_text().split()) if (tmp_path / "runs").exists() else 0
    return does


@pytest.mark.parametrize("build", ["build", "build_host"])
def test_an_interrupted_build_leaves_what_was_there(compiler, build):
    compiler("printf whole > $out")
    lib = getattr(b, build)()
    assert open(lib).read() == "whole" and compiler.runs() == 1
    getattr(b, build)()
    assert compiler.runs() == 1                            # (up to date)
    os.utime(lib, (0, 0))
    compiler("printf ha > $out; exit 1")
    with pytest.raises(subprocess.CalledProcessError):
        getattr(b, build)()
    assert open(lib).read() == "whole" and os.listdir(b._PKG) == [os.path.basename(lib)]
    compiler("printf ha > $out; kill -9 $$")
    with pytest.raises(subprocess.CalledProcessError):
        getattr(b, build)()
    assert open(lib).read() == "whole" and os.listdir(b._PKG) == [os.path.basename(lib)]


@pytest.mark.parametrize("build", ["build", "build_host"])
def test_builds_that_start_together_compile_once_and_see_a_whole_library(compiler, build):
    compiler("printf ha > $out; sleep 0.3; printf lf >> $out")

    def one(delay):
        time.sleep(delay)
        return open(getattr(b, build)()).read()
    with ThreadPoolExecutor(8) as pool:
        assert list(pool.map(one, [0.05 * i for i in range(8)])) == ["half"] * 8
    assert compiler.runs() == 1


@pytest.fixture
def helpers(tmp_path):
    """(a helper that loads, one that wants a symbol which nothing has)"""
    bad = tmp_path / "bad.so"
    src = tmp_path / "bad.c"
    src.write_text("extern int nobody_has_this(void);\nvoid* PyInit__host_call(void) { return nobody_has_this() ? 0 : 0; }\n")
    subprocess.run(["gcc", "-w", "-shared", "-fPIC", "-o", bad, src], check=True)
    return b.build_host(), bad


def test_a_helper_that_cannot_be_imported_is_built_once_more(helpers, compiler, monkeypatch):
    good, bad = helpers
    shutil.copy(bad, b.host_lib())                         # (younger than its source)
    compiler(f"cp {good} $out")
    assert callable(b.load_host().call) and compiler.runs() == 1
    assert callable(b.load_host().call) and compiler.runs() == 1
    monkeypatch.setattr(torch, "__version__", "98.0")      # (another file: this one stays loaded)
    shutil.copy(bad, b.host_lib())
    compiler(f"cp {bad} $out")
    with pytest.raises(ImportError, match="nobody_has_this"):
        b.load_host()
    assert compiler.runs() == 2


def test_processes_that_meet_the_same_unusable_helper_replace_it_once(helpers, compiler):
    good, bad = helpers
    shutil.copy(bad, b.host_lib())
    compiler(f"sleep 0.2; cp {good} $out")
    found = os.stat(b.host_lib())
    with ThreadPoolExecutor(4) as pool:
        list(pool.map(lambda _: b.build_host(unusable=found), range(4)))
    assert compiler.runs() == 1


def test_a_helper_of_another_torch_or_python_is_not_looked_at(helpers, compiler, monkeypatch):
    good, bad = helpers
    shutil.copy(bad, b.host_lib())
    compiler(f"cp {good} $out")
    with monkeypatch.context() as m:
        m.setattr(torch, "__version__", "99.0")
        assert callable(b.load_host().call) and compiler.runs() == 1
    with monkeypatch.context() as m:
        m.setattr(b.sysconfig, "get_config_var", lambda name: "cpython-399" if name == "SOABI" else None)
        assert callable(b.load_host().call) and compiler.runs() == 2
    assert len(os.listdir(b._PKG)) == 3


def test_the_build_succeeds_without_the_helper(monkeypatch):
    """As on a box without Python headers: calls are then filled from Python."""
    import __graft_entry__
    from paper_2506_18952_b200 import binding

    def no_headers(*args, **kw):
        raise subprocess.CalledProcessError(1, "g++")
    monkeypatch.setattr(b, "build_host", no_headers)
    for name, empty in (("_lib", None), ("_host", None), ("_entry", {})):
        monkeypatch.setattr(binding, name, empty)
    with pytest.warns(UserWarning, match="host-side helper not available"):
        __graft_entry__.build()
    assert binding._lib is not None and binding._host is None
