"""The library's objects linked with tests/fake_cuda_runtime.cpp in place of the
CUDA runtime, so that host code runs without a GPU and failures of the runtime
can be had on request."""
import ctypes as C
import importlib
import os
import subprocess

import paper_2507_17094_gb300 as A

B = importlib.import_module("paper_2507_17094_gb300.build")   # the package's `build` is the function

HERE = os.path.dirname(os.path.abspath(__file__))


def load(folder):
    """A ctypes library of its own (fresh state) with the binding's argument types."""
    A.build()
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B._nvcc()))), "include")
    out = os.path.join(str(folder), "libann_fake.so")
    objs = [os.path.join(B.BUILD, os.path.basename(s)[:-3] + ".o") for s in B.sources()]
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-w", "-I" + include, "-I" + B.INCLUDE, "-I" + B.CSRC,
                    os.path.join(HERE, "fake_cuda_runtime.cpp"), *objs, "-Wl,-Bsymbolic", "-ldl", "-lpthread",
                    "-o", out], check=True)
    L = C.CDLL(out)
    real = A.lib()
    for f in A.EXPORTS:
        getattr(L, f).argtypes = getattr(real, f).argtypes
        getattr(L, f).restype = getattr(real, f).restype
    return L
