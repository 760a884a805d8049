"""The library's host code on a CUDA runtime without a GPU (runtime.cpp): its objects linked with the fake
instead of CUDA's runtime. `load()` gives the C ABI, `use(monkeypatch)` lets the qs module call it."""
import ctypes
import os
import subprocess

from paper_2603_14641_gb300 import build, qs

HERE = os.path.dirname(os.path.abspath(__file__))
_lib = None


def load():
    global _lib
    if _lib is None:
        build.build()
        objs = [os.path.join(build.LIBDIR, "obj", os.path.basename(s) + ".o") for s in build._sources()]
        if not all(os.path.exists(o) for o in objs):
            build.build(force=True)
        out = os.path.join(build.LIBDIR, f"libqs_fake.{os.getpid()}.so")
        cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
        subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I", cuda,
                        os.path.join(HERE, "runtime.cpp"), *objs, "-o", out, "-ldl", "-lpthread"], check=True)
        L = ctypes.CDLL(out)
        os.remove(out)
        for name, (res, args) in qs.SIGNATURES.items():
            getattr(L, name).restype, getattr(L, name).argtypes = res, args
        L.fake_count.restype, L.fake_count.argtypes = ctypes.c_long, [ctypes.c_char_p]
        L.fake_reset.restype, L.fake_reset.argtypes = None, [ctypes.c_long, ctypes.c_int]
        _lib = L
    return _lib


def use(monkeypatch):
    L = load()
    monkeypatch.setattr(qs, "_lib", L)
    L.fake_reset(-1, 0)
    return L


def count(name):
    return _lib.fake_count(name.encode())
