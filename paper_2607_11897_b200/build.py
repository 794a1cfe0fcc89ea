"""Build ``libsfda.so`` (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and the small extension beside it.

A build is current when the hash of its sources, kept in a small file beside the library, equals the hash of the
sources in the tree: file times say nothing once a source file has been put back to an earlier state.  The extension's
hash also covers the torch and the interpreter that it was built against; the library depends on neither."""
import glob
import hashlib
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libsfda.so")
HOST = os.path.join(HERE, "_host.so")          # native marshalling of the decode calls (CPython extension)
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "--fmad=true", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
    "--expt-relaxed-constexpr",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return sorted(sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h"))
                  + glob.glob(os.path.join(HERE, "..", "include", "*.h")))


def source_hash(extra_flags=()) -> str:
    """SHA-256 over the compiler flags and the names and contents of every source and header of the library."""
    h = hashlib.sha256(" ".join(FLAGS + list(extra_flags)).encode())
    for path in _deps():
        h.update(os.path.basename(path).encode() + b"\0")
        with open(path, "rb") as f:
            h.update(f.read())
    return h.hexdigest()


def _recorded(target: str):
    """The hash kept beside a build, or None where there is no such build."""
    try:
        with open(target + ".srchash") as f:
            return f.read().strip() if os.path.exists(target) else None
    except OSError:
        return None


def _record(target: str, value: str) -> None:
    with open(target + ".srchash", "w") as f:
        f.write(value + "\n")


def _current(lib: str, extra_flags=()) -> bool:
    return _recorded(lib) == source_hash(extra_flags)


def is_stale() -> bool:
    """True when the library is missing or was not built from the sources now in the tree."""
    return not _current(LIB)


def _host_command(out: str):
    """g++ command of the extension; its torch and CUDA symbols come from the libraries torch has loaded."""
    import sysconfig

    import torch
    root = os.path.dirname(os.path.abspath(torch.__file__))
    return ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
            "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
            "-isystem", os.path.join(root, "include"), "-isystem", os.path.join(root, "include", "torch", "csrc", "api", "include"),
            "-isystem", os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include"), "-isystem", sysconfig.get_paths()["include"],
            os.path.join(CSRC, "sfda_host.cpp"), "-o", out, "-L" + os.path.join(root, "lib"),
            "-ltorch_python", "-ltorch_cpu", "-lc10_cuda", "-lc10"]


def host_hash() -> str:
    """SHA-256 over the extension's source, its build command and the torch and interpreter whose ABI it is built for."""
    import sysconfig

    import torch
    h = hashlib.sha256(" ".join(_host_command("") + [torch.__version__, sys.version, str(sysconfig.get_config_var("SOABI"))]).encode())
    with open(os.path.join(CSRC, "sfda_host.cpp"), "rb") as f:
        h.update(f.read())
    return h.hexdigest()


def host_is_stale() -> bool:
    """True when the extension is missing or was built from another source or for another torch or interpreter."""
    return _recorded(HOST) != host_hash()


def _start(cmd):
    return cmd, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)


def _finish(procs, verbose=False):
    for cmd, p in procs:
        out, _ = p.communicate()
        if verbose and out:
            print(out)
        if p.returncode != 0:
            raise RuntimeError("build failed: %s\n%s" % (" ".join(cmd), out))


def build_host() -> str:
    """Compile the extension."""
    tmp = HOST + ".tmp.%d" % os.getpid()
    _finish([_start(_host_command(tmp))])
    os.replace(tmp, HOST)
    _record(HOST, host_hash())
    return HOST


def build_library(verbose: bool = False) -> str:
    """Compile every ``csrc/*.cu`` into ``libsfda.so``."""
    objdir = os.path.join(HERE, "build")
    os.makedirs(objdir, exist_ok=True)
    _link(objdir, LIB, [], verbose)
    return LIB


def _link(objdir, lib, extra_flags, verbose=False):
    procs, objs = [], []
    for src in sources():
        obj = os.path.join(objdir, os.path.basename(src)[:-3] + ".o")
        procs.append(_start([NVCC] + FLAGS + list(extra_flags) + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", obj]))
        objs.append(obj)
    _finish(procs, verbose)
    tmp = lib + ".tmp.%d" % os.getpid()
    subprocess.run([NVCC, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", tmp] + objs, check=True)
    os.replace(tmp, lib)
    _record(lib, source_hash(extra_flags))


def build(force: bool = False, verbose: bool = False) -> str:
    """Build the library and the extension where they are missing or stale; returns the library's path."""
    if force or is_stale():
        build_library(verbose)
    if force or host_is_stale():
        build_host()
    return LIB


def build_variant(name: str, extra_flags):
    """Compile every source with `extra_flags` added into ``build/<name>/`` and link ``build/libsfda_<name>.so``
    (used by the tests for the development build whose roles pause at random, ``-DSFDA_WS_CHAOS``)."""
    objdir = os.path.join(HERE, "build", name)
    lib = os.path.join(HERE, "build", "libsfda_%s.so" % name)
    if _current(lib, extra_flags):
        return lib
    os.makedirs(objdir, exist_ok=True)
    _link(objdir, lib, extra_flags)
    return lib


if __name__ == "__main__":
    import sys
    print(build(force=True, verbose="-v" in sys.argv))
