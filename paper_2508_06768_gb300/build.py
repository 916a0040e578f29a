"""Builds libdiffus.so (sm_103a) in-tree with nvcc.

Each translation unit is compiled in parallel, then linked into one shared
library under ``paper_2508_06768_gb300/_build``; the native autograd node of
``render()`` (the one piece of host code that needs torch's headers) is
compiled beside them into its own module, which links the library.
"""
from __future__ import annotations

import concurrent.futures as cf
import hashlib
import os
import shutil
import subprocess
import sys

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


def _node_commands(obj):
    """Compile and link commands of the autograd node (g++, torch's headers
    and libraries as installed)."""
    import sysconfig

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
            "-lc10_cuda", "-L" + OUT_DIR, "-l:libdiffus.so", "-Wl,-rpath,$ORIGIN", "-Wl,-rpath," + lib]
    return compile_, link, torch.__version__


def build(force: bool = False, verbose: bool = False, extra_flags=None) -> str:
    """Compile and link libdiffus.so; returns its path.  Rebuilds only when a
    source, header or flag changed."""
    os.makedirs(OUT_DIR, exist_ok=True)
    stamp = os.path.join(OUT_DIR, "stamp")
    node_obj = os.path.join(OUT_DIR, "torch_node.o")
    node_compile, node_link, torch_version = _node_commands(node_obj)
    fp = _fingerprint() + (" ".join(extra_flags) if extra_flags else "") + " torch " + torch_version
    if (not force and os.path.exists(LIB) and os.path.exists(NODE) and os.path.exists(stamp)
            and open(stamp).read() == fp):
        return LIB
    nvcc = _nvcc()
    flags = ARCH + NVCC_FLAGS + list(extra_flags or [])
    objs = []
    cmds = [node_compile]
    for src in sources():
        obj = os.path.join(OUT_DIR, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        cmds.append([nvcc, *flags, "-c", src, "-o", obj])

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("compilation failed:\n" + " ".join(cmd) + "\n" + r.stdout + r.stderr)
        if verbose and (r.stdout or r.stderr):
            sys.stderr.write(r.stdout + r.stderr)

    with cf.ThreadPoolExecutor(max_workers=min(12, len(cmds))) as ex:
        list(ex.map(run, cmds))
    tmp = LIB + ".tmp%d" % os.getpid()
    run([nvcc, *ARCH, "-shared", "-o", tmp, *objs, "-lcudart"])
    os.replace(tmp, LIB)
    tmp = NODE + ".tmp%d" % os.getpid()
    run([*node_link, "-o", tmp])
    os.replace(tmp, NODE)
    with open(stamp, "w") as f:
        f.write(fp)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
