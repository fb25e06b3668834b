"""Compiles a CUDA source of tests/kernels/ into a shared library, for tests of device code that no entry
point of the library reaches by itself."""
import ctypes
import os
import subprocess
import tempfile

from conftest import ROOT

_loaded = {}


def load(name: str) -> ctypes.CDLL:
    if name not in _loaded:
        from paper_2312_16335_gb300 import build_lib
        out = os.path.join(tempfile.mkdtemp(prefix="kernel_unit_"), name + ".so")
        src = os.path.join(ROOT, "tests", "kernels", name + ".cu")
        r = subprocess.run([build_lib._nvcc(), *build_lib.ARCH, *build_lib.NVCC_FLAGS, "-shared", "-cudart", "static", src,
                            "-o", out], capture_output=True, text=True)
        assert r.returncode == 0, r.stdout + r.stderr
        _loaded[name] = ctypes.CDLL(out)
    return _loaded[name]
