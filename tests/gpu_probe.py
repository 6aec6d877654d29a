"""Compiles a few lines of CUDA against the library's own headers, so that a test can call a device
function by itself."""
import ctypes as C
import os
import subprocess


def compile_probe(source, path):
    from paper_2503_18682_gb300 import build
    src, lib = os.path.join(path, "probe.cu"), os.path.join(path, "probe.so")
    with open(src, "w") as f:
        f.write(source)
    r = subprocess.run([build.NVCC] + build._flags() + ["-shared", "-cudart", "static", "-o", lib, src],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return C.CDLL(lib)
