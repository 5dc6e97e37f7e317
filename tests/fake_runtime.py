"""The library's host code on a stand-in for the CUDA runtime (fake_cudart.cpp), for tests of what
it asks the runtime for: no GPU, the kernels do nothing.  load() links the objects of the built
library with it and returns a second copy of the binding on the result."""
import ctypes as C
import glob
import importlib.util
import os
import subprocess
import tempfile

from paper_2401_07965_gb300 import build

FIELDS = ("grid", "block", "cluster", "smem", "device", "priority", "captured", "chained")
_binding = None


class Stream:
    """A stream of the current device, as torch's have it."""

    def __init__(self, lib, priority=0):
        self.cuda_stream = lib.fake_stream(priority)


def load():
    global _binding
    if _binding is None:
        build.build()
        objs = sorted(glob.glob(os.path.join(build.LIBDIR, "obj", "*.o")))
        if len(objs) < len(build.SOURCES):
            build.build(force=True)
        objs = [os.path.join(build.LIBDIR, "obj", s.replace(".cu", ".o")) for s in build.SOURCES]
        tmp = tempfile.mkdtemp()
        so = os.path.join(tmp, "libpa_fake.so")
        inc = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
        subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I", inc,
                        os.path.join(os.path.dirname(__file__), "fake_cudart.cpp"), *objs, "-o", so,
                        "-Wl,-Bsymbolic", "-Wl,--no-undefined"], check=True, capture_output=True)
        spec = importlib.util.spec_from_file_location(
            "paper_2401_07965_gb300.pa_on_fake", os.path.join(build.PKG, "pa.py"))
        mod = importlib.util.module_from_spec(spec)
        real = build.LIB
        build.LIB = so
        try:
            spec.loader.exec_module(mod)
        finally:
            build.LIB = real
        lib = mod._lib
        lib.fake_stream.restype = C.c_void_p
        lib.fake_launch.restype = C.c_longlong
        lib.fake_capture.argtypes = [C.c_void_p, C.c_int]
        lib.fake_static_smem.argtypes = [C.c_char_p, C.c_int]
        _binding = mod
    _binding._lib.fake_reset(1)
    return _binding


def launches(lib, first=0):
    """The launches from number `first` on: dicts of FIELDS and the kernel's name."""
    out = []
    for k in range(first, lib.fake_launches()):
        name = C.create_string_buffer(200)
        d = {f: lib.fake_launch(k, i, name, 200) for i, f in enumerate(FIELDS)}
        d["name"] = name.value.decode()
        out.append(d)
    return out
