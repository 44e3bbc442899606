"""In-tree build of the CUDA library (sm_100a only) and of its Python call extension.  `python -m paper_2306_08162_b200.build` or build_library()."""
from __future__ import annotations

import os
import shutil
import subprocess
import sysconfig

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG_DIR)
CSRC = os.path.join(PKG_DIR, "csrc")
INCLUDE = os.path.join(ROOT, "include")
LIB_PATH = os.path.join(PKG_DIR, "libqlora_b200.so")
CALL_PATH = os.path.join(PKG_DIR, "_pycall" + sysconfig.get_config_var("EXT_SUFFIX"))   # (tagged: another interpreter builds its own)

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-shared"]


def sources() -> list[str]:
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _stale() -> bool:
    if not os.path.exists(LIB_PATH) or not os.path.exists(CALL_PATH):
        return True
    built = min(os.path.getmtime(LIB_PATH), os.path.getmtime(CALL_PATH))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE)]
    return any(os.path.getmtime(p) > built for p in deps)


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into one shared library next to this file.  Returns its path."""
    if not force and not _stale():
        return LIB_PATH
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        raise RuntimeError("nvcc not found: the CUDA library cannot be built")
    tmp = LIB_PATH + ".tmp"
    cmd = [nvcc, *NVCC_FLAGS, "-I", INCLUDE, "-I", CSRC, *sources(), "-o", tmp]
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + res.stdout + res.stderr)
    if verbose:
        print(res.stderr)
    os.replace(tmp, LIB_PATH)
    _build_calls()
    return LIB_PATH


def _build_calls() -> None:
    """csrc/pycall.cpp -> the CPython extension beside the library, which it finds through its own directory."""
    tmp = CALL_PATH + ".tmp"
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-I", INCLUDE, "-I", sysconfig.get_paths()["include"],
           os.path.join(CSRC, "pycall.cpp"), "-L", PKG_DIR, "-lqlora_b200", "-Wl,-rpath,$ORIGIN", "-o", tmp]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("the call extension failed to build:\n" + res.stdout + res.stderr)
    os.replace(tmp, CALL_PATH)


if __name__ == "__main__":
    print(build_library(force=True, verbose=True))
