"""Build step, in-tree: the CUDA library (one nvcc invocation for sm_100a) and the CPython module that marshals its calls."""
from __future__ import annotations

import hashlib
import os
import subprocess
import sysconfig

_PKG = os.path.dirname(os.path.abspath(__file__))
_CSRC = os.path.join(_PKG, "csrc")
LIB_PATH = os.path.join(_PKG, "libcomet_b200.so")
MARSHAL_PATH = os.path.join(_PKG, "_marshal.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-shared", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
]


def _sources():
    return sorted(os.path.join(_CSRC, f) for f in os.listdir(_CSRC) if f.endswith(".cu"))


STAMP_PATH = LIB_PATH + ".stamp"


def source_digest() -> str:
    """Hash of everything the library is built from (sources, the public header, the flags) and, for the marshalling
    module, the torch it is compiled against."""
    import torch

    h = hashlib.sha256(" ".join([*NVCC_FLAGS, torch.__version__]).encode())
    paths = sorted(os.path.join(_CSRC, f) for f in os.listdir(_CSRC))
    paths.append(os.path.join(os.path.dirname(_PKG), "include", "comet.h"))
    for path in paths:
        with open(path, "rb") as fh:
            h.update(os.path.basename(path).encode())
            h.update(fh.read())
    return h.hexdigest()


def is_current() -> bool:
    """True when both shared objects exist and were built from the sources as they are now."""
    if not all(os.path.exists(p) for p in (LIB_PATH, MARSHAL_PATH, STAMP_PATH)):
        return False
    with open(STAMP_PATH) as fh:
        return fh.read().strip() == source_digest()


def _marshal_command():
    """The compiler line of csrc/marshal.cpp: torch's headers, linked to the library beside it.  torch's own libraries are in
    the process already when the module is imported."""
    import torch

    root = os.path.dirname(torch.__file__)
    include = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
               sysconfig.get_paths()["include"]]
    return [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
            f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", *(x for p in include for x in ("-isystem", p)),
            "-o", MARSHAL_PATH, os.path.join(_CSRC, "marshal.cpp"), "-L" + _PKG, "-l:libcomet_b200.so",
            "-Wl,-rpath,$ORIGIN", "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10"]


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile csrc/*.cu into libcomet_b200.so and csrc/marshal.cpp into _marshal.so next to this file (skipped when the
    stamp written by the last build matches the current sources)."""
    if not force and is_current():
        return LIB_PATH
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, *NVCC_FLAGS, *(["-Xptxas", "-v"] if verbose else []), "-o", LIB_PATH, *_sources()]
    subprocess.check_call(cmd)
    subprocess.check_call(_marshal_command())
    with open(STAMP_PATH, "w") as fh:
        fh.write(source_digest() + "\n")
    return LIB_PATH


if __name__ == "__main__":
    import sys

    print(build_library(force=True, verbose="-v" in sys.argv))
