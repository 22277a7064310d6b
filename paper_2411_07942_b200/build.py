"""Build libtpq.so in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the extension module _calls."""
from __future__ import annotations

import os
import shlex
import subprocess
import sys
import sysconfig
import warnings
from pathlib import Path

PKG = Path(__file__).resolve().parent
CSRC = PKG / "csrc"
INCLUDE = PKG.parent / "include"
LIB = PKG / "libtpq.so"
# csrc/calls.c: the step's calls for Python (binding.py).  Its name says which interpreter it is built for, so that no other one
# takes it for its own.
CALLS = PKG / f"_calls{sysconfig.get_config_var('EXT_SUFFIX')}"

OBJ = PKG / "build"   # object files (git-ignored)

NVCC_FLAGS = [
    "-std=c++17", "-O3", "-lineinfo",
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-Xcompiler", "-fPIC",
    # IEEE arithmetic everywhere: no fast-math; the kernels use explicit _rn intrinsics
    # wherever the rounding sequence is part of the result.
]
LINK_FLAGS = ["-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-Xcompiler", "-fPIC"]


def sources():
    return sorted(CSRC.glob("*.cu"))


def _stale(target: Path, deps) -> bool:
    return (not target.exists()) or target.stat().st_mtime < max(d.stat().st_mtime for d in deps)


def needs_build() -> bool:
    return _stale(LIB, [f for f in CSRC.glob("*") if f.suffix != ".c"] + [INCLUDE / "tpq.h", Path(__file__)])


def build_calls(force: bool = False) -> Path:
    """Compile the extension module.  Raises RuntimeError if that fails, and then leaves none behind: an older one might call the
    library by another table."""
    src = CSRC / "calls.c"
    (CALLS.parent / "_calls.so").unlink(missing_ok=True)   # (without a tag: any interpreter would load it)
    if not force and not _stale(CALLS, [src, INCLUDE / "tpq.h", Path(__file__)]):
        return CALLS
    tmp = CALLS.with_suffix(f".{os.getpid()}.tmp")
    cmd = [*shlex.split(os.environ.get("CC", "gcc")), "-std=c11", "-O2", "-Wall", "-fPIC", "-shared",
           f"-I{sysconfig.get_paths()['include']}", f"-I{INCLUDE}", "-o", str(tmp), str(src)]
    try:
        res = subprocess.run(cmd, capture_output=True, text=True)
        failed = f"status {res.returncode}\n{res.stdout}{res.stderr}" if res.returncode != 0 else None
    except OSError as e:   # no such compiler
        failed = str(e)
    if failed is not None:
        CALLS.unlink(missing_ok=True)
        raise RuntimeError("calls.c: " + failed)
    os.replace(tmp, CALLS)
    return CALLS


def build(force: bool = False, verbose: bool = False) -> Path:
    """Build the library, then the extension module.  The library needs no C compiler and no Python headers, and every call
    can go through ctypes: where the module cannot be compiled, that is a warning."""
    build_lib(force, verbose)
    try:
        build_calls(force)
    except RuntimeError as e:
        warnings.warn(f"the extension module is not built (the calls of a step will go through ctypes): {e}", RuntimeWarning)
    return LIB


def build_lib(force: bool = False, verbose: bool = False) -> Path:
    """Compile every translation unit to an object file (only the stale ones unless ``force``), side by side,
    and link them into libtpq.so."""
    if not force and not needs_build():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    OBJ.mkdir(exist_ok=True)
    headers = list(CSRC.glob("*.h")) + [INCLUDE / "tpq.h", Path(__file__)]
    jobs = []
    for src in sources():
        obj = OBJ / (src.stem + ".o")
        if force or _stale(obj, [src] + headers):
            cmd = [nvcc, *NVCC_FLAGS, "-c", f"-I{INCLUDE}", f"-I{CSRC}", "-o", str(obj), str(src)]
            if verbose:
                cmd[1:1] = ["-Xptxas", "-v"]
            jobs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.PIPE, text=True)))
    failed = []
    for src, proc in jobs:
        out, err = proc.communicate()
        if verbose:
            sys.stderr.write(err)
        if proc.returncode != 0:
            failed.append(f"{src.name}:\n{out}{err}")
    if failed:
        raise RuntimeError("nvcc failed:\n" + "\n".join(failed))
    tmp = LIB.with_suffix(f".{os.getpid()}.tmp")
    objs = [str(OBJ / (src.stem + ".o")) for src in sources()]
    res = subprocess.run([nvcc, *LINK_FLAGS, "-o", str(tmp), *objs], capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("link failed:\n" + res.stdout + res.stderr)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
