"""Build ``libllattn.so`` in-tree with nvcc for sm_100a (no torch in the link), and the binding's marshalling module with the host compiler."""
from __future__ import annotations

import os
import shlex
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libllattn.so")
MARSHAL = os.path.join(HERE, "_marshal" + sysconfig.get_config_var("EXT_SUFFIX"))
MARSHAL_SOURCE = os.path.join(CSRC, "marshal.c")
SOURCES = ["ll_host.cu", "rope_append.cu", "attn_sm100.cu", "attn_simt.cu", "rope_static.cu", "qkv_gemm.cu", "attn_bwd.cu"]
HEADERS = ["ll_internal.h", "ptx.cuh", "bounded_wait.cuh", "exp2_poly.cuh", "rope_math.cuh", os.path.join(ROOT, "include", "llattn.h"),
           os.path.join(ROOT, "include", "llattn_debug.h")]

NVCC_FLAGS = [
    "-std=c++17", "-O3", "-lineinfo",
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-Xcompiler", "-fPIC",
    "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


def _nvcc() -> str:
    cand = os.environ.get("NVCC") or "/usr/local/cuda/bin/nvcc"
    return cand if os.path.exists(cand) else "nvcc"


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, s) for s in SOURCES] + \
           [h if os.path.isabs(h) else os.path.join(CSRC, h) for h in HEADERS] + [os.path.abspath(__file__)]
    return any(os.path.getmtime(d) > t for d in deps)


def build_marshal(force: bool = False) -> None:
    """The marshalling module.  Without Python's headers or a compiler that builds it there is none (nor an older one), and the
    binding's ctypes functions serve every call."""
    include = sysconfig.get_paths()["include"]
    header = os.path.join(ROOT, "include", "llattn.h")
    if not force and os.path.exists(MARSHAL) and os.path.getmtime(MARSHAL) > max(map(os.path.getmtime, (MARSHAL_SOURCE, header, __file__))):
        return
    tmp = MARSHAL + ".tmp%d" % os.getpid()
    try:
        if not os.path.exists(os.path.join(include, "Python.h")):
            raise OSError("no Python.h in %s" % include)
        subprocess.check_call(shlex.split(os.environ.get("CC") or "gcc") + ["-O2", "-Wall", "-shared", "-fPIC", "-I", include, "-I",
                                                                            os.path.join(ROOT, "include"), MARSHAL_SOURCE, "-o", tmp])
        os.replace(tmp, MARSHAL)
    except (OSError, ValueError, subprocess.CalledProcessError) as e:
        sys.stderr.write("the marshalling module has not been built, calls go through ctypes: %s\n" % e)
        if os.path.exists(MARSHAL):
            os.remove(MARSHAL)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every translation unit and link the shared library; returns its path."""
    build_marshal(force)
    if not force and not _stale():
        return LIB
    objs = []
    procs = []
    bdir = os.path.join(HERE, "_build")
    os.makedirs(bdir, exist_ok=True)
    for s in SOURCES:
        obj = os.path.join(bdir, s.replace(".cu", ".o"))
        cmd = [_nvcc()] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + \
              ["-c", os.path.join(CSRC, s), "-o", obj]
        procs.append((s, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    failed = False
    for s, pr in procs:
        out, _ = pr.communicate()
        if verbose or pr.returncode != 0:
            sys.stderr.write(out)
        failed |= pr.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    tmp = LIB + ".tmp%d" % os.getpid()
    subprocess.check_call([_nvcc(), "-shared", "-o", tmp] + objs +
                          ["-gencode", "arch=compute_100a,code=sm_100a", "-Xcompiler", "-fPIC", "-ldl"])
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
