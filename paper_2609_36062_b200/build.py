"""Builds libsmat.so in-tree with nvcc for sm_100a, then the Python extension over it (both without a GPU).  The library
needs neither torch nor a C++ compiler of its own; where one of them is missing it is built alone, for C callers."""
from __future__ import annotations

import glob
import importlib.metadata
import os
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
LIB = os.path.join(HERE, "libsmat.so")
EXT = os.path.join(HERE, "_smat_torch.so")       # argument checks and launches of binding.SmatPlan
EXT_SRC = os.path.join(HERE, "csrc", "smat_torch.cpp")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
CXX = os.environ.get("CXX", "g++")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC"]
OBJ_DIR = os.path.join(HERE, "csrc", ".obj")     # per-source objects (git-ignored), compiled in parallel
EXT_VERSIONS = os.path.join(OBJ_DIR, "smat_torch.versions")   # Python and torch that the extension was compiled for


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(HERE, "csrc", "*.cu")))


def _older(target: str, deps: list[str]) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(f) > os.path.getmtime(target) for f in deps)


def _headers() -> list[str]:
    return glob.glob(os.path.join(HERE, "..", "include", "*.h"))


def _library_is_old() -> bool:
    return _older(LIB, sources() + _headers() + [f for x in ("h", "cuh", "inc") for f in glob.glob(os.path.join(HERE, "csrc", f"*.{x}"))])


def _host_versions() -> str | None:
    """What the extension is compiled against; None where it cannot be (no torch, no C++ compiler)."""
    try:
        torch_version = importlib.metadata.version("torch")
    except importlib.metadata.PackageNotFoundError:
        return None
    return f"python {sys.version} torch {torch_version}" if shutil.which(CXX) else None


def _extension_is_old() -> bool:
    versions = _host_versions()
    if versions is None:
        return False
    if _older(EXT, [EXT_SRC] + _headers()) or not os.path.exists(EXT_VERSIONS):
        return True
    with open(EXT_VERSIONS) as f:
        return f.read() != versions


def needs_build() -> bool:
    return _library_is_old() or _extension_is_old()


def _run(commands: list[list[str]], what: str, verbose: bool) -> None:
    """All commands at once; when one fails the others are ended."""
    jobs = [subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True) for cmd in commands]
    try:
        for proc in jobs:
            out, _ = proc.communicate()
            if verbose or proc.returncode != 0:
                sys.stderr.write(out)
            if proc.returncode != 0:
                raise RuntimeError(f"{what} failed")
    finally:
        for proc in jobs:
            if proc.poll() is None:
                proc.terminate()
                proc.wait()


def _build_library(verbose: bool) -> None:
    extra = os.environ.get("SMAT_NVCC_FLAGS", "").split()   # e.g. -D switches of a kernel variant under test
    objects, commands = [], []
    for src in sources():                                    # one nvcc per translation unit, all at once
        objects.append(os.path.join(OBJ_DIR, os.path.basename(src)[:-3] + ".o"))
        commands.append([NVCC] + FLAGS + extra + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", objects[-1]])
    _run(commands, "compiling libsmat.so", verbose)
    _run([[NVCC] + FLAGS + ["-shared", "-o", LIB] + objects], "linking libsmat.so", verbose)


def _build_extension(versions: str, verbose: bool) -> None:
    """Torch's headers and libraries; no CUDA code in it."""
    import torch
    root = os.path.dirname(torch.__file__)
    obj = os.path.join(OBJ_DIR, "smat_torch.o")
    cuda = os.path.dirname(os.path.dirname(NVCC))
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           os.path.join(cuda, "include"), sysconfig.get_paths()["include"]]
    compile_ = [CXX, "-O2", "-std=c++17", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    compile_ += [f"-I{d}" for d in inc] + ["-c", EXT_SRC, "-o", obj]
    link = [CXX, "-shared", "-o", EXT, obj, f"-L{os.path.join(root, 'lib')}", "-ltorch_python", "-ltorch", "-ltorch_cpu",
            "-lc10", "-lc10_cuda", f"-L{HERE}", "-l:libsmat.so", "-Wl,-rpath,$ORIGIN"]
    _run([compile_], "compiling _smat_torch.so", verbose)
    _run([link], "linking _smat_torch.so", verbose)
    with open(EXT_VERSIONS, "w") as f:
        f.write(versions)


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(OBJ_DIR, exist_ok=True)
    if force or _library_is_old():
        _build_library(verbose)
    versions = _host_versions()
    if versions is None:
        sys.stderr.write("no torch or no C++ compiler here: libsmat.so alone, without the Python call layer\n")
    elif force or _extension_is_old():
        _build_extension(versions, verbose)
    return LIB


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose="-v" in sys.argv)
    print(LIB)
