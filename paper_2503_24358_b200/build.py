"""Builds libsquat.so in-tree with nvcc for sm_100a (cross-compiles without a GPU).

`build(checked=True)` (or `python -m paper_2503_24358_b200.build --checked`) builds libsquat_checked.so from the same
sources with -DSQUAT_CHECKED: the key and value kernels then test every address they form against the extent of the
buffer or on-chip region it belongs to and report through SQUAT_FLAG_BOUNDS instead of accessing.  Select it with the
environment variable SQUAT_LIBRARY=<path> before the package is first used."""
import os
import shutil
import subprocess
import sysconfig
from importlib.machinery import EXTENSION_SUFFIXES
from concurrent.futures import ThreadPoolExecutor

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(_HERE), "include")
OBJ_DIR = os.path.join(_HERE, "build")
LIB = os.path.join(_HERE, "libsquat.so")
OBJ_DIR_CHECKED = os.path.join(_HERE, "build_checked")
LIB_CHECKED = os.path.join(_HERE, "libsquat_checked.so")
PYCALL = os.path.join(_HERE, "_squatcall" + EXTENSION_SUFFIXES[0])
SOURCES = ["api.cu", "values.cu", "keys.cu", "keys_lane.cu", "subspace.cu", "gram_i8.cu", "eig.cu", "power.cu", "attention.cu", "attention_mma.cu", "attention_rope.cu", "peak.cu", "keys_lowrank.cu", "keys_block.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I", INCLUDE]


def _nvcc():
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def _deps_mtime():
    paths = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(INCLUDE, "squat.h")]
    return max(os.path.getmtime(p) for p in paths)


def _compile(src, verbose, obj_dir=OBJ_DIR, extra=()):
    obj = os.path.join(obj_dir, src.replace(".cu", ".o"))
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cuh")] + [os.path.join(INCLUDE, "squat.h")]
    hdr_time = max(os.path.getmtime(p) for p in headers)
    src_path = os.path.join(CSRC, src)
    if os.path.exists(obj) and os.path.getmtime(obj) >= max(os.path.getmtime(src_path), hdr_time):
        return obj
    cmd = [_nvcc()] + NVCC_FLAGS + list(extra) + (["-Xptxas", "-v"] if verbose else []) + ["-c", src_path, "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or r.returncode != 0:
        print(r.stdout + r.stderr)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed on {src}")
    return obj


def build_pycall(force: bool = False):
    """The extension module through which the binding makes its per-token and per-window calls (gcc, the CPython C API).  Its
    file name carries the interpreter's ABI tag.  Without a C compiler or the CPython headers there is none (None is returned)
    and the binding calls through ctypes."""
    src, out = os.path.join(CSRC, "pycall.c"), PYCALL
    include, cc = sysconfig.get_paths()["include"], shutil.which(os.environ.get("CC") or "gcc")
    if cc is None or not os.path.exists(os.path.join(include, "Python.h")):
        return None
    if force or not os.path.exists(out) or os.path.getmtime(out) < max(os.path.getmtime(src), os.path.getmtime(os.path.join(INCLUDE, "squat.h"))):
        subprocess.run([cc, "-O2", "-Wall", "-shared", "-fPIC", "-I", include, src, "-o", out], check=True)
    return out


def build(force: bool = False, verbose: bool = False, checked: bool = False) -> str:
    obj_dir, lib = (OBJ_DIR_CHECKED, LIB_CHECKED) if checked else (OBJ_DIR, LIB)
    extra = ("-DSQUAT_CHECKED",) if checked else ()
    os.makedirs(obj_dir, exist_ok=True)
    build_pycall(force)
    if not force and os.path.exists(lib) and os.path.getmtime(lib) >= _deps_mtime():
        return lib
    if force:
        for f in os.listdir(obj_dir):
            if f.endswith(".o"):
                os.remove(os.path.join(obj_dir, f))
    with ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(lambda s: _compile(s, verbose, obj_dir, extra), SOURCES))
    cmd = [_nvcc(), "-shared", "-cudart", "static", "-gencode", "arch=compute_100a,code=sm_100a", "-o", lib] + objs
    subprocess.run(cmd, check=True)
    return lib


if __name__ == "__main__":
    import sys
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, checked="--checked" in sys.argv))
