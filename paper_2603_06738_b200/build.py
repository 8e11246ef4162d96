"""Builds the CUDA library in-tree: csrc/*.cu -> paper_2603_06738_b200/librib_window_attn.so, and the native form of the
binding's argument marshalling, csrc/rib_marshal.cpp -> paper_2603_06738_b200/_rib_marshal.<ABI tag of this Python>.so.

nvcc cross-compiles for sm_100a without a GPU.  Run as ``python -m paper_2603_06738_b200.build``.
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
import warnings
from pathlib import Path

PKG = Path(__file__).resolve().parent
CSRC = PKG / "csrc"
LIB = PKG / "librib_window_attn.so"
HEADER = PKG.parent / "include" / "rib_window_attn.h"
MARSHAL_SOURCE, MARSHAL = CSRC / "rib_marshal.cpp", PKG / f"_rib_marshal{sysconfig.get_config_var('EXT_SUFFIX')}"

NVCC_FLAGS = [
    "-std=c++17", "-O3", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
    "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr", "-Xptxas", "-v",
]


def sources() -> list[Path]:
    return sorted(CSRC.glob("*.cu"))


def stale() -> bool:
    if not LIB.exists():
        return True
    newest = max(f.stat().st_mtime for f in list(CSRC.glob("*.cu*")) + [HEADER])
    return LIB.stat().st_mtime < newest


def marshal_identity() -> str:
    """What a marshaller is compiled for.  It reads the fields of torch's tensors at places that are fixed when it is compiled, so it is
    of use to this torch and this Python only."""
    import torch
    return f"torch {torch.__version__} ({torch.version.git_version}), {sysconfig.get_config_var('SOABI')}"


def marshal_stale() -> bool:
    """No marshaller, one older than its sources (this file holds its compiler flags), or one for another torch or Python."""
    note = PKG / "_build" / "rib_marshal.built_for"
    if not MARSHAL.exists() or not note.exists() or note.read_text() != marshal_identity():
        return True
    return MARSHAL.stat().st_mtime < max(f.stat().st_mtime for f in (MARSHAL_SOURCE, HEADER, Path(__file__)))


def build_marshal(force: bool = False) -> Path:
    """Compile the marshaller against the installed torch (host code only).  Raises on failure."""
    if not force and not marshal_stale():
        return MARSHAL
    import torch
    root = Path(torch.__file__).resolve().parent
    cuda = Path(os.environ.get("CUDA_HOME", "/usr/local/cuda"))
    includes = [root / "include", root / "include" / "torch" / "csrc" / "api" / "include", sysconfig.get_path("include"), cuda / "include"]
    tmp = MARSHAL.with_suffix(f".{os.getpid()}.tmp")
    run = subprocess.run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared",
                          f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DRIB_BUILT_FOR="{marshal_identity()}"', *[f"-I{p}" for p in includes], str(MARSHAL_SOURCE),
                          f"-L{root / 'lib'}", "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python", "-o", str(tmp)], capture_output=True, text=True)
    if run.returncode:
        sys.stderr.write(run.stdout + run.stderr)
        raise RuntimeError("g++ failed on rib_marshal.cpp")
    note = PKG / "_build" / "rib_marshal.built_for"
    note.parent.mkdir(exist_ok=True)
    note.unlink(missing_ok=True)            # (never beside a marshaller that it does not describe)
    os.replace(tmp, MARSHAL)
    note.write_text(marshal_identity())
    return MARSHAL


def build(force: bool = False, verbose: bool = False) -> Path:
    """Compile every .cu for sm_100a and link the shared library; raises on failure.  Then the marshaller, which the library does
    not need: where it cannot be compiled (no g++, no headers of Python or torch), a warning says so, none of an earlier build is
    left behind, and the binding marshals in Python."""
    lib = build_library(force, verbose)
    try:
        build_marshal(force)
    except Exception as e:      # noqa: BLE001 - whatever is missing, the library is there
        MARSHAL.unlink(missing_ok=True)
        warnings.warn(f"{MARSHAL.name} was not built, calls are marshalled in Python (a few us more each): {e}", RuntimeWarning, stacklevel=2)
    return lib


def build_library(force: bool = False, verbose: bool = False) -> Path:
    """Compile every .cu for sm_100a and link the shared library (nvcc alone is needed).  Raises on failure."""
    if not force and not stale():
        return LIB
    nvcc = os.environ.get("NVCC", "nvcc")
    obj_dir = PKG / "_build"
    obj_dir.mkdir(exist_ok=True)
    objs = []
    log = []
    for src in sources():
        obj = obj_dir / (src.stem + ".o")
        run = subprocess.run([nvcc, *NVCC_FLAGS, "-c", str(src), "-o", str(obj)], capture_output=True, text=True)
        log.append(run.stderr)
        if run.returncode:
            sys.stderr.write(run.stdout + run.stderr)
            raise RuntimeError(f"nvcc failed on {src.name}")
        objs.append(str(obj))
    tmp = LIB.with_suffix(f".{os.getpid()}.tmp")
    run = subprocess.run([nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", *objs, "-o", str(tmp)],
                         capture_output=True, text=True)
    if run.returncode:
        sys.stderr.write(run.stdout + run.stderr)
        raise RuntimeError("link failed")
    os.replace(tmp, LIB)
    (obj_dir / "ptxas.log").write_text("\n".join(log))
    if verbose:
        print("\n".join(log))
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
