"""Builds libdiffus.so (sm_103a) in-tree with nvcc.

Each translation unit is compiled in parallel, then linked into one shared
library under ``paper_2508_06768_gb300/_build``.  The native autograd node of
``render()`` (the one piece of host code that needs torch's headers and a host
compiler) is a module of its own beside it, which links the library.  Neither
build depends on the other's tools: the library builds without torch, and each
is left alone, whatever is installed, while its stamp says that it is current.
"""
from __future__ import annotations

import concurrent.futures as cf
import hashlib
import os
import shutil
import subprocess
import sys
import sysconfig
import warnings

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
OUT_DIR = os.path.join(HERE, "_build")
LIB = os.path.join(OUT_DIR, "libdiffus.so")
NODE_NAME = "diffus_torch"
NODE = os.path.join(OUT_DIR, NODE_NAME + ".so")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
              "--expt-relaxed-constexpr", "-I", INCLUDE, "-I", CSRC]


def _nvcc():
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libdiffus")


def sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _fingerprint():
    h = hashlib.sha256()
    for d in (CSRC, INCLUDE):
        for f in sorted(os.listdir(d)):
            p = os.path.join(d, f)
            if os.path.isfile(p):
                h.update(f.encode())
                h.update(open(p, "rb").read())
    h.update(" ".join(ARCH + NVCC_FLAGS).encode())
    return h.hexdigest()


def _node_fingerprint():
    """What a built node depends on: its source, the C header, the installed
    torch and the interpreter."""
    import torch

    h = hashlib.sha256()
    for p in (os.path.join(CSRC, "torch_node.cpp"), os.path.join(INCLUDE, "diffus.h")):
        h.update(open(p, "rb").read())
    return "%s torch %s %s" % (h.hexdigest(), torch.__version__, sysconfig.get_config_var("SOABI"))


def _node_object():
    # of this process: load_node() may find the node out of date in several
    return os.path.join(OUT_DIR, "torch_node.%d.o" % os.getpid())


def _node_commands(obj, out):
    """Compile and link commands of the autograd node (g++, torch's headers
    and libraries as installed)."""
    import torch

    base = os.path.dirname(torch.__file__)
    inc = [os.path.join(base, "include"), os.path.join(base, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include"), INCLUDE]
    flags = ["-O1", "-std=c++17", "-fPIC", "-w", "-DTORCH_EXTENSION_NAME=" + NODE_NAME,
             "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI)]
    cxx = os.environ.get("CXX", "g++")
    compile_ = [cxx, *flags, *[a for i in inc for a in ("-isystem", i)], "-c", os.path.join(CSRC, "torch_node.cpp"),
                "-o", obj]
    lib = os.path.join(base, "lib")
    link = [cxx, "-shared", obj, "-L" + lib, "-ltorch_python", "-ltorch", "-ltorch_cpu", "-ltorch_cuda", "-lc10",
            "-lc10_cuda", "-L" + OUT_DIR, "-l:libdiffus.so", "-Wl,-rpath,$ORIGIN", "-Wl,-rpath," + lib, "-o", out]
    return compile_, link


def _run(cmd, verbose=False):
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("compilation failed:\n" + " ".join(cmd) + "\n" + r.stdout + r.stderr)
    if verbose and (r.stdout or r.stderr):
        sys.stderr.write(r.stdout + r.stderr)


def _stamped(stamp, product, fp):
    return os.path.exists(product) and os.path.exists(stamp) and open(stamp).read() == fp


def _finish(tmp, product, stamp, fp):
    os.replace(tmp, product)
    with open(stamp, "w") as f:
        f.write(fp)


def node_current() -> bool:
    """Whether the built node fits its source, the installed torch and this
    interpreter."""
    return _stamped(os.path.join(OUT_DIR, "node_stamp"), NODE, _node_fingerprint())


def build_node(force: bool = False, verbose: bool = False, compiled=None) -> str:
    """Compile and link the autograd node of render() against the built
    libdiffus.so; returns its path.  Raises if it cannot be built here."""
    if not force and node_current():
        return NODE
    fp = _node_fingerprint()
    tmp = NODE + ".tmp%d" % os.getpid()
    compile_, link = _node_commands(_node_object(), tmp)
    if compiled is None:
        _run(compile_, verbose)
    else:
        compiled.result()      # the same command, started by build()
    _run(link, verbose)
    os.remove(_node_object())
    _finish(tmp, NODE, os.path.join(OUT_DIR, "node_stamp"), fp)
    return NODE


def build(force: bool = False, verbose: bool = False, extra_flags=None) -> str:
    """Compile and link libdiffus.so; returns its path.  Rebuilds only when a
    source, header or flag changed.  The autograd node is brought up to date
    beside it; where that is not possible (no torch, no host compiler) the
    library stands alone, with a warning, and render() takes its Python
    function."""
    os.makedirs(OUT_DIR, exist_ok=True)
    stamp = os.path.join(OUT_DIR, "stamp")
    fp = _fingerprint() + (" ".join(extra_flags) if extra_flags else "")
    with cf.ThreadPoolExecutor(max_workers=12) as ex:
        compiled = None
        try:
            if force or not node_current():
                compiled = ex.submit(_run, _node_commands(_node_object(), NODE)[0], verbose)
        except (ImportError, OSError, RuntimeError):
            pass               # reported below
        if force or not _stamped(stamp, LIB, fp):
            nvcc = _nvcc()
            flags = ARCH + NVCC_FLAGS + list(extra_flags or [])
            objs = [os.path.join(OUT_DIR, os.path.basename(src)[:-3] + ".o") for src in sources()]
            list(ex.map(lambda so: _run([nvcc, *flags, "-c", so[0], "-o", so[1]], verbose), zip(sources(), objs)))
            tmp = LIB + ".tmp%d" % os.getpid()
            _run([nvcc, *ARCH, "-shared", "-o", tmp, *objs, "-lcudart"], verbose)
            _finish(tmp, LIB, stamp, fp)
        try:
            build_node(force=force, verbose=verbose, compiled=compiled)
        except (ImportError, OSError, RuntimeError) as e:
            warnings.warn("the autograd node of render() was not built: %s" % e, RuntimeWarning, stacklevel=2)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
