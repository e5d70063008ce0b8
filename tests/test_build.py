"""The build on stand-ins for the compilers: the C library does not depend on torch, a failed compilation leaves no process
behind, and the extension follows the Python and torch that it is used with."""
import os
import stat
import sys
import time

import pytest

from paper_2609_36062_b200 import build


@pytest.fixture
def tree(tmp_path, monkeypatch):
    """A build that writes under tmp_path, with compilers that create the file behind -o."""
    def tool(name, body):
        path = tmp_path / name
        path.write_text(f"#!{sys.executable}\nimport os, sys, time\nout = sys.argv[sys.argv.index('-o') + 1]\n{body}\n")
        path.chmod(path.stat().st_mode | stat.S_IXUSR)
        return str(path)

    monkeypatch.setattr(build, "LIB", str(tmp_path / "libsmat.so"))
    monkeypatch.setattr(build, "EXT", str(tmp_path / "_smat_torch.so"))
    monkeypatch.setattr(build, "OBJ_DIR", str(tmp_path / "obj"))
    monkeypatch.setattr(build, "EXT_VERSIONS", str(tmp_path / "obj" / "versions"))
    monkeypatch.setattr(build, "NVCC", tool("nvcc", "open(out, 'w').close()"))
    monkeypatch.setattr(build, "CXX", tool("cxx", "open(out, 'w').close()"))
    return tool


def test_the_library_is_built_where_torch_is_missing(tree, monkeypatch):
    monkeypatch.setattr(build, "_host_versions", lambda: None)
    monkeypatch.setitem(sys.modules, "torch", None)       # an import of it would raise
    assert build.needs_build()
    build.build()
    assert os.path.exists(build.LIB) and not os.path.exists(build.EXT)
    assert not build.needs_build()


def test_a_failed_compilation_ends_the_others(tree, monkeypatch, tmp_path):
    first = os.path.basename(build.sources()[0])[:-3] + ".o"
    monkeypatch.setattr(build, "NVCC", tree("slow_nvcc", f"""
open(out + '.pid', 'w').write(str(os.getpid()))
if out.endswith('{first}'):
    n = 0
    while len([f for f in os.listdir(os.path.dirname(out)) if f.endswith('.pid')]) < {len(build.sources())} and n < 300:
        time.sleep(0.1); n += 1
    sys.exit(1)
time.sleep(600)"""))
    began = time.monotonic()
    with pytest.raises(RuntimeError, match="libsmat"):
        build.build()
    assert time.monotonic() - began < 300
    pids = [int((tmp_path / "obj" / f).read_text()) for f in os.listdir(tmp_path / "obj") if f.endswith(".pid")]
    assert len(pids) == len(build.sources())
    for pid in pids:
        with pytest.raises(ProcessLookupError):
            os.kill(pid, 0)


def test_the_extension_follows_torch_and_python(tree, monkeypatch):
    build.build()
    assert not build.needs_build()
    lib = os.path.getmtime(build.LIB)
    monkeypatch.setattr(build, "_host_versions", lambda: "another torch")
    assert build.needs_build()
    build.build()
    assert not build.needs_build() and os.path.getmtime(build.LIB) == lib
