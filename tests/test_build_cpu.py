"""How the libraries get into the tree: stand-ins for the compilers, in a folder of their own."""
import os
import subprocess
import time
from concurrent.futures import ThreadPoolExecutor

import pytest

from paper_2506_18952_b200 import build as b


@pytest.fixture
def compiler(tmp_path, monkeypatch):
    """Both libraries are built in an empty folder by a script; returns a function that sets what it does with $out."""
    folder = tmp_path / "pkg"
    folder.mkdir()
    monkeypatch.setattr(b, "_PKG", str(folder))
    monkeypatch.setattr(b, "LIB", str(folder / "lib.so"))
    monkeypatch.setattr(b, "HOST_LIB", str(folder / "host.so"))

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
