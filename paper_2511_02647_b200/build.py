"""Builds the FedAttn CUDA library for sm_100a with nvcc, in-tree."""
from __future__ import annotations

import glob
import os
import subprocess
import sys

_PKG = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_PKG)
CSRC = os.path.join(_PKG, "csrc")
LIB_DIR = os.path.join(_PKG, "lib")
LIB_PATH = os.path.join(LIB_DIR, "libfedattn.so")
MARSHAL_SRC = os.path.join(CSRC, "marshal.cpp")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC"]


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    t = os.path.getmtime(LIB_PATH)
    deps = _sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(_ROOT, "include", "*.h"))
    return any(os.path.getmtime(p) > t for p in deps)


def marshal_path() -> str:
    """Where the marshalling module for the running interpreter and torch is.  It is compiled against the layouts in torch's
    headers, which no symbol version guards: one built for another torch must not be found, let alone loaded."""
    import sysconfig
    import torch
    tag = "%s-%s" % (torch.__version__, (torch.version.git_version or "")[:8])
    return os.path.join(LIB_DIR, "_fedattn_marshal-torch%s%s" % (tag, sysconfig.get_config_var("EXT_SUFFIX")))


def missing() -> list:
    """The files that build() makes and that are not there."""
    return [p for p in (LIB_PATH, marshal_path()) if not os.path.exists(p)]


def build_marshal(force: bool = False) -> str:
    """Compile the binding's native marshalling module (a CPython extension against torch's headers)."""
    path = marshal_path()
    if not force and os.path.exists(path) and os.path.getmtime(path) >= os.path.getmtime(MARSHAL_SRC):
        return path
    import sysconfig
    import torch
    inc = os.path.join(os.path.dirname(torch.__file__), "include")
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    tmp = path + ".tmp%d" % os.getpid()
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC",
                           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
                           "-I", sysconfig.get_paths()["include"], "-I", inc,
                           "-I", os.path.join(inc, "torch", "csrc", "api", "include"), MARSHAL_SRC, "-o", tmp,
                           "-L", lib, "-ltorch_python", "-ltorch_cpu", "-lc10"])
    os.replace(tmp, path)
    return path


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into lib/libfedattn.so, and the marshalling module (no-op when up to date)."""
    os.makedirs(LIB_DIR, exist_ok=True)
    try:
        build_marshal(force)
    except (OSError, subprocess.CalledProcessError) as e:      # no g++, no Python headers: the binding works without it
        sys.stderr.write("marshalling module not built: %s\n" % e)
    if not force and not _stale():
        return LIB_PATH
    objs = []
    procs = []
    for src in _sources():
        obj = os.path.join(LIB_DIR, os.path.basename(src)[:-3] + ".o")
        cmd = ["nvcc", *NVCC_FLAGS, "-I", os.path.join(_ROOT, "include"), "-I", CSRC, "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode != 0:
            sys.stderr.write(out)
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    tmp = LIB_PATH + ".tmp%d" % os.getpid()
    subprocess.check_call(["nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", tmp, *objs,
                           "-cudart", "static"])
    os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose="-v" in sys.argv)
    print(LIB_PATH)
