"""Build libpatconv.so in-tree with nvcc for sm_100a (cross-compiles without a GPU)."""
from __future__ import annotations

import hashlib
import os
import subprocess
import sys
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
_CSRC = os.path.join(_HERE, "csrc")
_INC = os.path.join(os.path.dirname(_HERE), "include")
LIB_PATH = os.path.join(_HERE, "libpatconv.so")
CALLS_PATH = os.path.join(_HERE, "_calls.abi3.so")     # the enqueueing calls for Python
_SOURCES = ["patconv.cu", "tapgemm.cu", "tapgemm_f32.cu", "tapgemm_f16.cu", "tapgemm_f16_cut.cu", "tapgemm_i8.cu", "fewconv.cu", "blockgemm.cu", "dwconv.cu", "probe.cu", "pack.cpp"]
_DEPS = _SOURCES + ["patconv_internal.h", "ptx.cuh", "tapgemm.h", "tapgemm_kernel.cuh", "fewconv.h", "gen_core.py", "gen_blockgemm.py", os.path.join(_INC, "patconv.h"),
                    os.path.join(_INC, "blockgemm.h"), os.path.join(_INC, "dwconv.h")]


_OBJ_DIR = os.path.join(_HERE, "_build")
# what each source includes besides itself
_INCLUDES = {
    "patconv.cu": ["patconv_internal.h", "ptx.cuh", "tapgemm.h", "fewconv.h", "gen_core.py", os.path.join(_INC, "patconv.h")],
    **{"tapgemm%s.cu" % part: ["patconv_internal.h", "ptx.cuh", "tapgemm.h", "tapgemm_kernel.cuh", os.path.join(_INC, "patconv.h")]
       for part in ("", "_f32", "_f16", "_f16_cut", "_i8")},
    "fewconv.cu": ["patconv_internal.h", "fewconv.h", os.path.join(_INC, "patconv.h")],
    "blockgemm.cu": ["patconv_internal.h", "tapgemm.h", "gen_blockgemm.py", os.path.join(_INC, "patconv.h"),
                     os.path.join(_INC, "blockgemm.h")],
    "dwconv.cu": ["patconv_internal.h", os.path.join(_INC, "patconv.h"), os.path.join(_INC, "dwconv.h")],
    "probe.cu": [os.path.join(_INC, "patconv.h")],
    "pack.cpp": ["patconv_internal.h", os.path.join(_INC, "patconv.h")],
}


def _mtime(name: str) -> float:
    return os.path.getmtime(os.path.join(_CSRC, name))


def build_calls(force: bool = False) -> str:
    """Compile the CPython extension that marshals the enqueueing calls (host code only), unless the one
    that is there was made from these sources."""
    src = os.path.join(_CSRC, "calls.cpp")
    digest = hashlib.sha256()
    for f in [src] + [os.path.join(_INC, h) for h in ("patconv.h", "blockgemm.h", "dwconv.h")]:
        with open(f, "rb") as fh:
            digest.update(fh.read())
    tag = "sources " + digest.hexdigest()          # stands in the file: a copy of the tree need not keep its times
    if not force and os.path.exists(CALLS_PATH):
        with open(CALLS_PATH, "rb") as fh:
            force = tag.encode() not in fh.read()
    if force or not os.path.exists(CALLS_PATH):
        tmp = CALLS_PATH + ".tmp%d" % os.getpid()
        subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-I", _INC,
                               "-I", sysconfig.get_paths()["include"], '-DXGEN_CALLS_TAG="%s"' % tag, src, "-o", tmp])
        os.replace(tmp, CALLS_PATH)
    return CALLS_PATH


def _stale() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    t = os.path.getmtime(LIB_PATH)
    return any(_mtime(d) > t for d in _DEPS)


def build(force: bool = False, verbose: bool = False) -> str:
    """Generate the per-pattern code, compile every source that changed to an object of its
    own, and link the shared library."""
    build_calls(force)
    if not force and not _stale():
        return LIB_PATH
    gen = os.path.join(_CSRC, "core_gen.inc")
    subprocess.check_call([sys.executable, os.path.join(_CSRC, "gen_core.py"), gen])
    subprocess.check_call([sys.executable, os.path.join(_CSRC, "gen_blockgemm.py"),
                           os.path.join(_CSRC, "blockgemm_core.inc")])
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    os.makedirs(_OBJ_DIR, exist_ok=True)
    flags = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
             "-Xcompiler", "-fPIC", "-I", _INC, "-I", _CSRC]
    if verbose:
        flags += ["-Xptxas", "-v"]
    objs, jobs = [], []
    for src in _SOURCES:
        obj = os.path.join(_OBJ_DIR, os.path.splitext(src)[0] + ".o")
        objs.append(obj)
        newest = max([_mtime(src)] + [_mtime(d) for d in _INCLUDES[src]])
        if force or verbose or not os.path.exists(obj) or os.path.getmtime(obj) < newest:
            jobs.append((obj, subprocess.Popen([nvcc] + flags + ["-c", os.path.join(_CSRC, src), "-o", obj + ".tmp"])))
    for obj, job in jobs:                       # the compilations run side by side
        if job.wait() != 0:
            raise subprocess.CalledProcessError(job.returncode, "nvcc -c (%s)" % obj)
        os.replace(obj + ".tmp", obj)
    tmp = LIB_PATH + ".tmp%d" % os.getpid()
    subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", tmp] + objs)
    os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
