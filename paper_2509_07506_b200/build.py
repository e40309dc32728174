"""Build ``libastra.so`` (the CUDA kernels and their C ABI) for sm_100a with nvcc, the ablation
library beside it, and with the host compilers two small CPython extensions that issue calls without
ctypes: ``_astra_fastcall`` (prepared calls) and ``_astra_torchcall`` (direct calls on the tensors of the
installed torch).

Usage: ``python -m paper_2509_07506_b200.build [--force]``.  The shared objects are written next
to this file; nothing is installed outside the source tree.
"""
from __future__ import annotations

import hashlib
import os
import re
import shutil
import subprocess
import sys
import sysconfig

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG_DIR)
CSRC = os.path.join(PKG_DIR, "csrc")
INCLUDE = os.path.join(ROOT, "include")
LIB_PATH = os.path.join(PKG_DIR, "libastra.so")
ABLATION_LIB_PATH = os.path.join(PKG_DIR, "libastra_ablation.so")
FASTCALL_PATH = os.path.join(PKG_DIR, "_astra_fastcall.so")
TORCHCALL_PATH = os.path.join(PKG_DIR, "_astra_torchcall.so")

SOURCES = ["astra.cu", "astra_allreduce.cu", "astra_runs.cu"]
ABLATION_SOURCES = ["ablation.cu"]
FASTCALL_SOURCE = "fastcall.c"
TORCHCALL_SOURCE = "torchcall.cpp"
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-std=c++17", "-lineinfo",
    "-Xcompiler", "-fPIC", "-shared",
    "-cudart", "static",
    "--threads", "0",
]


def _nvcc() -> str:
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found: libastra.so cannot be built")
    return exe


def _inputs():
    files = [os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE) if f.endswith(".h")]
    files += [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh", ".h", ".c", ".cpp"))]
    return files


_ID_MARKER = b"astra-build-id:"


def source_hash(extra_flags=()) -> str:
    """SHA-256 over the names and contents of every header and CUDA source (and the extra compiler
    flags of a variant build).  It is compiled into each library, so a library can be matched to the
    sources beside it by content; file times, which a copy or a checkout rewrites, play no part."""
    h = hashlib.sha256()
    for path in sorted(_inputs()):
        h.update(os.path.basename(path).encode() + b"\0")
        with open(path, "rb") as fh:
            h.update(fh.read())
        h.update(b"\0")
    for flag in extra_flags:
        h.update(flag.encode() + b"\0")
    return h.hexdigest()


def embedded_hash(lib_path: str):
    """The source hash compiled into a built library (read from the file, without loading it), or None."""
    try:
        with open(lib_path, "rb") as fh:
            blob = fh.read()
    except OSError:
        return None
    m = re.search(re.escape(_ID_MARKER) + rb"([0-9a-f]{64})", blob)
    return m.group(1).decode() if m else None


def is_stale(lib_path: str = LIB_PATH, extra_flags=()) -> bool:
    """True when the library is missing or was not built from the sources now on disk."""
    return embedded_hash(lib_path) != source_hash(extra_flags)


def _compile(lib_path: str, sources, force: bool, verbose: bool, extra_flags=()) -> str:
    if not force and not is_stale(lib_path, extra_flags):
        return lib_path
    tmp = lib_path + f".tmp{os.getpid()}"
    cmd = [_nvcc(), *NVCC_FLAGS, *extra_flags, f'-DASTRA_BUILD_ID="{source_hash(extra_flags)}"',
           "-I", INCLUDE, "-I", CSRC, "-o", tmp]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [os.path.join(CSRC, s) for s in sources]
    subprocess.check_call(cmd)
    os.replace(tmp, lib_path)
    return lib_path


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile libastra.so (and the extensions the binding loads with it) if missing or built from other
    sources; returns the library's path."""
    build_fastcall(force)
    try:
        build_torchcall(force)
    except (RuntimeError, OSError, subprocess.CalledProcessError) as exc:  # no torch headers, say: direct calls do without
        print(f"_astra_torchcall not built, direct calls take the slower route: {exc}", file=sys.stderr)
    return _compile(LIB_PATH, SOURCES, force, verbose)


def build_fastcall(force: bool = False) -> str:
    """Compile the _astra_fastcall extension (plain C against the CPython headers) if it is missing or was
    built from other sources; returns its path."""
    if not force and not is_stale(FASTCALL_PATH):
        return FASTCALL_PATH
    cc = shutil.which("gcc") or shutil.which("cc")
    if cc is None:
        raise RuntimeError("no C compiler found: _astra_fastcall cannot be built")
    tmp = FASTCALL_PATH + f".tmp{os.getpid()}"
    subprocess.check_call([cc, "-O2", "-std=c11", "-shared", "-fPIC", "-fvisibility=hidden", f'-DASTRA_BUILD_ID="{source_hash()}"',
                           "-I", sysconfig.get_paths()["include"], "-I", INCLUDE, "-I", CSRC, "-o", tmp,
                           os.path.join(CSRC, FASTCALL_SOURCE)])
    os.replace(tmp, FASTCALL_PATH)
    return FASTCALL_PATH


def torchcall_torch(path: str = TORCHCALL_PATH):
    """The torch release a built _astra_torchcall belongs to (read from the file, without loading it), or None."""
    try:
        with open(path, "rb") as fh:
            m = re.search(rb"astra-torch:([^;]+);", fh.read())
    except OSError:
        return None
    return m.group(1).decode() if m else None


def build_torchcall(force: bool = False) -> str:
    """Compile the _astra_torchcall extension (against the CPython and torch headers) if it is missing or
    was built from other sources or for another torch; returns its path."""
    import torch
    if not force and not is_stale(TORCHCALL_PATH) and torchcall_torch() == str(torch.__version__):
        return TORCHCALL_PATH
    from torch.utils import cpp_extension
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        raise RuntimeError("no C++ compiler found")
    tmp = TORCHCALL_PATH + f".tmp{os.getpid()}"
    subprocess.check_call([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
                           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DASTRA_BUILD_ID="{source_hash()}"',
                           f'-DASTRA_TORCH_VERSION="{torch.__version__}"', "-I", sysconfig.get_paths()["include"], "-I", INCLUDE,
                           "-I", CSRC, *(flag for d in cpp_extension.include_paths("cuda") for flag in ("-isystem", d)),
                           "-o", tmp, os.path.join(CSRC, TORCHCALL_SOURCE), "-L", os.path.join(os.path.dirname(torch.__file__), "lib"),
                           "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"])
    os.replace(tmp, TORCHCALL_PATH)
    return TORCHCALL_PATH


def ensure_built(ablation: bool = False) -> str:
    """Build if the library is missing or does not match the sources on disk.  A library that cannot
    be rebuilt (no compiler on this machine) and does not match is an error: results must never come
    from a library other than the one the sources describe."""
    return build_ablation() if ablation else build()


def build_variant(lib_path: str, defines: dict) -> str:
    """Compile libastra's sources to `lib_path` with extra preprocessor definitions (used by the
    tests to lower the per-launch limits so that the multi-launch splitting runs on small inputs)."""
    flags = [f"-D{k}={v}" for k, v in sorted(defines.items())]
    return _compile(lib_path, SOURCES, False, False, flags)


def build_ablation(force: bool = False, verbose: bool = False) -> str:
    """Compile libastra_ablation.so (the paper's design pairs, for the ablation measurements)."""
    return _compile(ABLATION_LIB_PATH, ABLATION_SOURCES, force, verbose)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
    print(FASTCALL_PATH)
    print(TORCHCALL_PATH)
    print(build_ablation(force="--force" in sys.argv, verbose="-v" in sys.argv))
