"""Build step: compile the CUDA sources in ``csrc/`` into ``libkeydiff.so`` (sm_100a only) and the binding's C entry into
``_pycall.<ABI>.so``."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from pathlib import Path

PKG = Path(__file__).resolve().parent
CSRC = PKG / "csrc"
LIB = PKG / "libkeydiff.so"
SOURCES = [CSRC / "keydiff_api.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-shared", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden"]


def _stale(lib: Path) -> bool:
    if not lib.exists():
        return True
    t = lib.stat().st_mtime
    deps = list(CSRC.glob("*.cu")) + list(CSRC.glob("*.cuh")) + list(CSRC.glob("*.h")) + list((PKG.parent / "include").glob("*.h"))
    return any(p.stat().st_mtime > t for p in deps)


# CPython entry of KeyDiff.evict (argument marshalling in C); its name carries the interpreter's ABI, so that another one does not load it
PYCALL = PKG / ("_pycall" + sysconfig.get_config_var("EXT_SUFFIX"))


def build_pycall(force: bool = False) -> Path | None:
    """Compile the C entry in-tree if missing or older than its source.  None without Python's headers: the binding then makes the same call
    through ctypes."""
    src, include = CSRC / "pycall.c", Path(sysconfig.get_paths()["include"])
    (PKG / "_pycall.so").unlink(missing_ok=True)   # (named without the ABI before: any interpreter would load it)
    if not (include / "Python.h").exists():
        print(f"{include}/Python.h not found: KeyDiff.evict goes through ctypes", file=sys.stderr)
        return None
    if force or not PYCALL.exists() or src.stat().st_mtime > PYCALL.stat().st_mtime:
        tmp = PYCALL.with_suffix(f".{os.getpid()}.tmp")
        subprocess.run([os.environ.get("CC", "gcc"), "-O2", "-Wall", "-shared", "-fPIC", f"-I{include}", str(src), "-o", str(tmp)], check=True)
        os.replace(tmp, PYCALL)
    return PYCALL


STAMPS_LIB = PKG / "libkeydiff_stamps.so"   # diagnostic build: fused kernel with per-phase timers (phase_times.py)
DEBUG_LIB = PKG / "libkeydiff_debug.so"     # debug build: computed row indices are range-checked into the status word


def build_library(force: bool = False, verbose: bool = False, phase_stamps: bool = False, debug_checks: bool = False) -> Path:
    """Compile libkeydiff.so in-tree if missing or older than its sources.  phase_stamps=True builds the
    diagnostic variant libkeydiff_stamps.so instead (-DKEYDIFF_PHASE_STAMPS: the fused kernel times its phases),
    debug_checks=True the variant libkeydiff_debug.so (-DKEYDIFF_DEBUG_CHECKS: row indices are range-checked)."""
    build_pycall(force)
    out = STAMPS_LIB if phase_stamps else DEBUG_LIB if debug_checks else LIB
    if not force and not _stale(out):
        return out
    nvcc = os.environ.get("NVCC", "nvcc")
    tmp = out.with_suffix(f".{os.getpid()}.tmp")
    cmd = [nvcc, *NVCC_FLAGS, *(["-DKEYDIFF_PHASE_STAMPS"] if phase_stamps else []),
           *(["-DKEYDIFF_DEBUG_CHECKS"] if debug_checks else []), *(["-Xptxas", "-v"] if verbose else []),
           *map(str, SOURCES), "-o", str(tmp)]
    subprocess.run(cmd, check=True)
    os.replace(tmp, out)
    return out


if __name__ == "__main__":
    print(build_library(force=True, verbose="-v" in sys.argv, phase_stamps="--phase-stamps" in sys.argv,
                        debug_checks="--debug-checks" in sys.argv))
