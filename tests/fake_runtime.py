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
    """A ctypes library of its own (fresh state) with the binding's argument
    types. Only the entry points are exported: what C++ makes unique in a process
    (the static variables of inline functions, the tensor-map encoder among them)
    would otherwise be shared with the real library, whichever is used first."""
    A.build()
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B._nvcc()))), "include")
    out, exports = os.path.join(str(folder), "libann_fake.so"), os.path.join(str(folder), "exports")
    with open(exports, "w") as f:
        f.write("{ global: ann_*; fake_*; local: *; };\n")
    objs = [os.path.join(B.BUILD, os.path.basename(s)[:-3] + ".o") for s in B.sources()]
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-w", "-I" + include, "-I" + B.INCLUDE, "-I" + B.CSRC,
                    os.path.join(HERE, "fake_cuda_runtime.cpp"), *objs, "-Wl,--version-script=" + exports, "-Wl,-Bsymbolic",
                    "-ldl", "-lpthread", "-o", out], check=True)
    symbols = subprocess.run(["nm", "-D", "--defined-only", out], check=True, capture_output=True, text=True).stdout
    for line in symbols.splitlines():
        kind, name = line.split()[-2:]
        assert kind != "u" and name.split("@")[0].startswith(("ann_", "fake_")), line
    L = C.CDLL(out)
    real = A.lib()
    for f in A.EXPORTS:
        getattr(L, f).argtypes = getattr(real, f).argtypes
        getattr(L, f).restype = getattr(real, f).restype
    return L
