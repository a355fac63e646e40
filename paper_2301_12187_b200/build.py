"""Builds libdepthc.so (sm_100a, nvcc) and the Python module _dccall (gcc) next to this file.  `python -m paper_2301_12187_b200.build`."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig
import warnings

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libdepthc.so")
CALL_SRC = os.path.join(CSRC, "dccall.c")
CALL_LIB = os.path.join(HERE, "_dccall" + sysconfig.get_config_var("EXT_SUFFIX"))     # marshals the forward calls of dc.py; one per Python ABI

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
    "-Xcompiler", "-fPIC", "-shared", "-cudart", "static",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def needs_build() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + [os.path.join(ROOT, "include", "dc.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def build_call(force: bool = False) -> None:
    if not force and os.path.exists(CALL_LIB) and os.path.getmtime(CALL_LIB) >= os.path.getmtime(CALL_SRC):
        return
    tmp = CALL_LIB + ".tmp.%d" % os.getpid()
    subprocess.check_call([os.environ.get("CC", "gcc"), "-O2", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"], "-o", tmp,
                           CALL_SRC])
    os.replace(tmp, CALL_LIB)


def build(force: bool = False, verbose: bool = False) -> str:
    try:
        build_call(force)
    except (OSError, subprocess.CalledProcessError) as e:          # no compiler or no headers of Python: ctypes makes those calls
        warnings.warn("_dccall could not be built, calls are marshalled by ctypes: %r" % (e,))
    if not force and not needs_build():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + ".tmp.%d" % os.getpid()
    cmd = [nvcc] + NVCC_FLAGS + ["-I", os.path.join(ROOT, "include"), "-I", CSRC]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += ["-o", tmp] + sources()
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
