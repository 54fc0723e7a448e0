"""Builds libhola_verify.so (nvcc, sm_100a; cross-compiles without a GPU) and the host-side helper (g++, against the running
Python and torch, which its file name says) in-tree."""
from __future__ import annotations

import contextlib
import fcntl
import importlib.util
import os
import subprocess
import sys
import sysconfig

_PKG = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(_PKG, "csrc", "hola_verify.cu")
HEADER = os.path.join(os.path.dirname(_PKG), "include", "hola_verify.h")
LIB = os.path.join(_PKG, "libhola_verify.so")
HOST_SRC = os.path.join(_PKG, "csrc", "host_call.cpp")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
              "-shared", "-Xcompiler", "-fPIC"]


def _older(out: str, *sources: str) -> bool:
    if not os.path.exists(out):
        return True
    t = os.path.getmtime(out)
    return any(os.path.getmtime(f) > t for f in sources)


@contextlib.contextmanager
def _build_lock():
    """One build at a time in this tree: a lock on the package's folder.  (Where the file system has none, processes that
    start together build more often than needed, nothing else.)"""
    fd = os.open(_PKG, os.O_RDONLY)
    try:
        with contextlib.suppress(OSError):
            fcntl.flock(fd, fcntl.LOCK_EX)
        yield
    finally:
        os.close(fd)


def _link(cmd: list, out: str, wanted) -> None:
    """Runs the compiler on a file of its own beside `out` and moves it there whole, so that nobody meets the half of a
    library, now or after an interrupted build.  `wanted` is asked again once the lock is held: another process may have
    built meanwhile."""
    with _build_lock():
        if not wanted():
            return
        tmp = f"{out.removesuffix('.so')}.{os.getpid()}.tmp.so"
        try:
            subprocess.run([*cmd, "-o", tmp], check=True)
            os.replace(tmp, out)
        finally:
            with contextlib.suppress(FileNotFoundError):
                os.unlink(tmp)


def needs_build() -> bool:
    return _older(LIB, SRC, HEADER)


def build(force: bool = False, verbose: bool = False) -> str:
    def wanted():
        return force or needs_build()
    if wanted():
        nvcc = os.environ.get("NVCC", "nvcc")
        _link([nvcc, *NVCC_FLAGS, *(["-Xptxas", "-v"] if verbose else []), SRC], LIB, wanted)
    return LIB


def host_lib() -> str:
    import torch
    return os.path.join(_PKG, f"_host_call.{sysconfig.get_config_var('SOABI')}-torch-{torch.__version__}.so")


def build_host(force: bool = False, unusable=None) -> str:
    """`unusable`: os.stat of a helper that is to be replaced whatever its age."""
    lib = host_lib()

    def wanted():
        return force or _older(lib, HOST_SRC, HEADER) or (
            unusable is not None and os.path.samestat(os.stat(lib), unusable) and os.stat(lib).st_mtime_ns == unusable.st_mtime_ns)
    if wanted():
        import torch
        root = os.path.dirname(os.path.abspath(torch.__file__))
        _link([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC",
               f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
               f"-I{os.path.join(root, 'include')}", f"-I{sysconfig.get_paths()['include']}", HOST_SRC,
               f"-L{os.path.join(root, 'lib')}", "-ltorch_python", "-ltorch_cpu", "-lc10"], lib, wanted)
    return lib


def load_host():
    """The helper as a module, built first where it is missing or older than its source, and once more where the one in place
    cannot be imported (symbols of another build of the same torch version).  Raises if it cannot be had."""
    def load(path):
        spec = importlib.util.spec_from_file_location(__package__ + "._host_call", path)
        module = importlib.util.module_from_spec(spec)
        spec.loader.exec_module(module)
        return module
    path = build_host()
    found = os.stat(path)
    try:
        return load(path)
    except ImportError:
        return load(build_host(unusable=found))


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
    print(build_host(force="--force" in sys.argv))
