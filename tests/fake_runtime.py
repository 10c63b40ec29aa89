"""The library's host code without a GPU: its objects linked against the stand-in runtime of fake_cudart.cpp, behind a
copy of the binding.  ``load()`` returns that binding; ``launches()`` what the last calls launched."""
import ctypes as C
import importlib.util
import os
import re
import subprocess
import typing

from paper_1702_03818_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))


def load(tmp):
    """The binding over the stand-in runtime (built in the folder ``tmp``)."""
    objs = [os.path.join(B.OUTDIR, "obj", os.path.basename(s) + ".o") for s in B.sources()]
    if not all(os.path.exists(o) and os.path.getmtime(o) >= os.path.getmtime(s) for o, s in zip(objs, B.sources())):
        B.build()
    nvcc = B._nvcc()
    fake, lib = os.path.join(tmp, "fake_cudart.o"), os.path.join(tmp, "libfrkc2_fake.so")
    subprocess.run([nvcc, "-std=c++17", "-O1", "-Xcompiler", "-fPIC", "-c", os.path.join(HERE, "fake_cudart.cpp"), "-o", fake], check=True)
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-Wl,-z,defs", "-o", lib, *objs, fake, "-ldl", "-lpthread"], check=True)
    spec = importlib.util.spec_from_file_location("frkc2_fake", os.path.join(B.PKG, "frkc2.py"))
    F = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(F)
    F._lib = C.CDLL(lib)
    for name, (res, args) in F._sig.items():
        f = getattr(F._lib, name)
        f.restype, f.argtypes = res, args
    F._lib.fake_launch.restype = C.c_char_p
    return F


class Buffer:
    """Stands for a device buffer: an address and a size, no memory."""

    def __init__(self, nbytes, at=1 << 40):
        self.nbytes, self.at = int(nbytes), at

    def data_ptr(self):
        return self.at

    def numel(self):
        return self.nbytes

    def element_size(self):
        return 1


class Launch(typing.NamedTuple):
    kernel: str  # its name, without namespaces and template arguments
    mangled: str
    grid: tuple
    threads: int
    smem: int  # dynamic
    cooperative: bool
    device: int


def launches(F):
    """What was launched since the last reset."""
    out = []
    for i in range(F._lib.fake_count()):
        f = F._lib.fake_launch(i).decode().split()
        out.append(Launch(re.search(r"\d(k_[a-z0-9_]+)", f[0])[1], f[0], tuple(map(int, f[1:4])), int(f[4]), int(f[5]), f[6] == "1", int(f[7])))
    return out
