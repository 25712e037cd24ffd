"""Small C++ files that call the library's own internal functions, compiled by
a test against the sources and linked with libann.so."""
import ctypes
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2201_13007_gb300", "csrc")


def compile_and_load(source, tmp_path):
    """Compiles `source` (host C++ that may include the library's .cuh headers of host functions) and loads it."""
    from paper_2201_13007_gb300 import _build
    lib = _build.build()
    src, so = os.path.join(tmp_path, "shim.cpp"), os.path.join(tmp_path, "shim.so")
    with open(src, "w") as f:
        f.write(source)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(_build._nvcc())))
    includes = [os.path.join(ROOT, "include"), CSRC, os.path.join(cuda, "include")]
    includes += [p for p in (os.path.join(cuda, "targets", t, "include") for t in ("x86_64-linux", "sbsa-linux"))
                 if os.path.isdir(p)]
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC"] + [f"-I{p}" for p in includes] +
                       [src, lib, f"-Wl,-rpath,{os.path.dirname(lib)}", "-o", so], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(so)
