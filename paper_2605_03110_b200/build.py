"""Build libada.so in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the binding's native
marshalling (_pycall, plain C, one file per interpreter ABI) beside it."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libada.so")
# the suffix names the interpreter's ABI: another interpreter does not import it, and builds its own
PYCALL = os.path.join(HERE, "_pycall" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
PYCALL_SRC = os.path.join(CSRC, "pycall.c")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-shared",
    "-Xptxas", "-v", "-cudart", "static",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def is_stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(PYCALL):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(PYCALL))
    deps = sources() + [PYCALL_SRC] + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + \
        [os.path.join(os.path.dirname(HERE), "include", "ada.h")]
    return any(os.path.getmtime(p) > t for p in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not is_stale():
        return LIB
    cmd = [NVCC] + FLAGS + ["-o", LIB] + sources()
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed building libada.so")
    # Python's include directory is only looked up, the interpreter provides the symbols
    cc = ["gcc", "-O2", "-Wall", "-fPIC", "-shared", "-I", sysconfig.get_paths()["include"], "-o", PYCALL, PYCALL_SRC,
          "-L", HERE, "-l:libada.so", "-Wl,-rpath,$ORIGIN"]
    res_c = subprocess.run(cc, capture_output=True, text=True)
    if verbose or res_c.returncode != 0:
        sys.stderr.write(res_c.stdout + res_c.stderr)
    if res_c.returncode != 0:
        raise RuntimeError("gcc failed building " + os.path.basename(PYCALL))
    with open(os.path.join(HERE, "build.log"), "w") as f:
        f.write(" ".join(cmd) + "\n" + res.stdout + res.stderr)
    return LIB


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose=True)
    print(LIB)
