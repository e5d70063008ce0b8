"""Builds libsmat.so in-tree with nvcc for sm_100a, and the Python extension over it (both without a GPU)."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
LIB = os.path.join(HERE, "libsmat.so")
EXT = os.path.join(HERE, "_smat_torch.so")       # argument checks and launches of binding.SmatPlan
EXT_SRC = os.path.join(HERE, "csrc", "smat_torch.cpp")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC"]
OBJ_DIR = os.path.join(HERE, "csrc", ".obj")     # per-source objects (git-ignored), compiled in parallel


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(HERE, "csrc", "*.cu")))


def needs_build() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(EXT):
        return True
    stamp = min(os.path.getmtime(LIB), os.path.getmtime(EXT))
    deps = (sources() + glob.glob(os.path.join(HERE, "csrc", "*.h")) + glob.glob(os.path.join(HERE, "csrc", "*.cuh")) +
            glob.glob(os.path.join(HERE, "csrc", "*.inc")) + glob.glob(os.path.join(HERE, "..", "include", "*.h")) + [EXT_SRC])
    return any(os.path.getmtime(f) > stamp for f in deps)


def _extension_commands() -> tuple[list[str], list[str]]:
    """Compile and link commands of the Python extension (torch's headers and libraries; no CUDA code in it)."""
    import torch
    root = os.path.dirname(torch.__file__)
    obj = os.path.join(OBJ_DIR, "smat_torch.o")
    cuda = os.path.dirname(os.path.dirname(NVCC))
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           os.path.join(cuda, "include"), sysconfig.get_paths()["include"]]
    cxx = os.environ.get("CXX", "g++")
    compile_ = [cxx, "-O2", "-std=c++17", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    compile_ += [f"-I{d}" for d in inc] + ["-c", EXT_SRC, "-o", obj]
    link = [cxx, "-shared", "-o", EXT, obj, f"-L{os.path.join(root, 'lib')}", "-ltorch_python", "-ltorch", "-ltorch_cpu",
            "-lc10", "-lc10_cuda", f"-L{HERE}", "-l:libsmat.so", "-Wl,-rpath,$ORIGIN"]
    return compile_, link


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
    extra = os.environ.get("SMAT_NVCC_FLAGS", "").split()   # e.g. -D switches of a kernel variant under test
    os.makedirs(OBJ_DIR, exist_ok=True)
    jobs = []
    for src in sources():                                    # one nvcc per translation unit, all at once
        obj = os.path.join(OBJ_DIR, os.path.basename(src)[:-3] + ".o")
        cmd = [NVCC] + FLAGS + extra + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", obj]
        jobs.append((obj, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    ext_compile, ext_link = _extension_commands()
    ext = subprocess.Popen(ext_compile, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    failed = False
    for obj, proc in jobs + [(None, ext)]:
        out, _ = proc.communicate()
        if verbose or proc.returncode != 0:
            sys.stderr.write(out)
        failed = failed or proc.returncode != 0
    if failed:
        raise RuntimeError("compiling libsmat.so failed")
    link = [NVCC] + FLAGS + ["-shared", "-o", LIB] + [obj for obj, _ in jobs]
    for cmd, what in ((link, "libsmat.so"), (ext_link, "_smat_torch.so")):
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode != 0:
            sys.stderr.write(res.stdout + res.stderr)
            raise RuntimeError(f"linking {what} failed")
    return LIB


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose="-v" in sys.argv)
    print(LIB)
