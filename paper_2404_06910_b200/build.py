"""Builds the CUDA library in-tree: every csrc/*.cu -> libsp_b200.so (sm_100a only), and the same
sources with -DSP_DEBUG_BOUNDS (extra device-side layout checks) -> libsp_b200_debug.so; and the Python argument
marshalling, csrc/marshal.c -> _marshal (with the interpreter's suffix)."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libsp_b200.so")
OBJ_DEBUG = os.path.join(HERE, "_build_debug")
LIB_DEBUG = os.path.join(HERE, "libsp_b200_debug.so")
MARSHAL = os.path.join(HERE, "_marshal" + sysconfig.get_config_var("EXT_SUFFIX"))     # an interpreter's own
MARSHAL_FLAGS = ["-O2", "-Wall", "-Werror=int-conversion", "-Werror=incompatible-pointer-types", "-shared", "-fPIC",
                 "-I", sysconfig.get_paths()["include"]]

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xptxas", "-v",
]


def _sources():
    return sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))


def _deps_mtime():
    hdrs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    hdrs.append(os.path.join(HERE, "..", "include", "sp.h"))
    return max(os.path.getmtime(h) for h in hdrs)


def _compile(src: str, verbose: bool, obj_dir: str = OBJ, extra=()) -> str:
    obj = os.path.join(obj_dir, src[:-3] + ".o")
    path = os.path.join(CSRC, src)
    if os.path.exists(obj) and os.path.getmtime(obj) >= max(os.path.getmtime(path), _deps_mtime()):
        return obj
    cmd = ["nvcc", *NVCC_FLAGS, *extra, "-c", path, "-o", obj]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode:
        sys.stderr.write(f"$ {' '.join(cmd)}\n{res.stdout}{res.stderr}")
    if res.returncode:
        raise RuntimeError(f"nvcc failed on {src}")
    return obj


def _build_one(lib: str, obj_dir: str, extra, force: bool, verbose: bool) -> str:
    os.makedirs(obj_dir, exist_ok=True)
    if force:
        for f in os.listdir(obj_dir):
            os.remove(os.path.join(obj_dir, f))
    with ThreadPoolExecutor(max_workers=8) as ex:
        objs = list(ex.map(lambda s: _compile(s, verbose, obj_dir, extra), _sources()))
    if force or not os.path.exists(lib) or os.path.getmtime(lib) < max(os.path.getmtime(o) for o in objs):
        tmp = lib + f".tmp{os.getpid()}"
        subprocess.check_call(["nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", tmp, *objs,
                               "-Xcompiler", "-fPIC"])
        os.replace(tmp, lib)
    return lib


def _build_marshal(force: bool) -> None:
    src = os.path.join(CSRC, "marshal.c")
    newest = max(os.path.getmtime(f) for f in (src, os.path.join(HERE, "..", "include", "sp.h"), os.path.abspath(__file__)))
    if force or not os.path.exists(MARSHAL) or os.path.getmtime(MARSHAL) < newest:
        tmp = MARSHAL + f".tmp{os.getpid()}"
        subprocess.check_call(["gcc", *MARSHAL_FLAGS, src, "-o", tmp])
        os.replace(tmp, MARSHAL)


def build(force: bool = False, verbose: bool = False, debug: bool = True) -> str:
    """Builds the library and (debug=True) its bounds-checking twin; returns the library's path."""
    _build_marshal(force)
    lib = _build_one(LIB, OBJ, (), force, verbose)
    if debug:
        _build_one(LIB_DEBUG, OBJ_DEBUG, ("-DSP_DEBUG_BOUNDS",), force, verbose)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
