"""Host code of the CUDA sources, compiled with the host compiler for the tests."""
import ctypes
import os
import subprocess
import tempfile

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(os.path.dirname(HERE))
_libs = {}


def load(name):
    """The shared library of <name>.cpp, which includes headers of csrc/."""
    if name not in _libs:
        cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
        with tempfile.TemporaryDirectory() as tmp:
            so = os.path.join(tmp, name + ".so")
            subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-fPIC", "-shared",
                            "-I", os.path.join(ROOT, "paper_2606_14173_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                            "-isystem", os.path.join(cuda, "include"), os.path.join(HERE, name + ".cpp"), "-o", so],
                           check=True, capture_output=True, text=True)
            _libs[name] = ctypes.CDLL(so)
    return _libs[name]
