"""The binding loaded over a build of the library whose CUDA runtime is a host stand-in (fake_cudart.cpp)."""
import ctypes
import importlib.util
import os
import subprocess

from paper_2603_21835_gb300 import build as gbuild

HERE = os.path.dirname(os.path.abspath(__file__))


def load(tmpdir):
    """(module like paper_2603_21835_gb300.gint, its library): CPU tensors stand for device tensors."""
    objs = [os.path.join(gbuild.BUILD, s.replace(".cu", ".o")) for s in gbuild.SOURCES]
    gbuild.build(force=not all(os.path.exists(o) for o in objs))
    path = os.path.join(str(tmpdir), "libgint_fake.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(gbuild.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", inc, "-o", path,
                    os.path.join(HERE, "fake_cudart.cpp")] + objs, check=True)
    real = ctypes.CDLL
    spec = importlib.util.spec_from_file_location("gint_over_fake_cudart",
                                                  os.path.join(gbuild.HERE, "gint.py"))
    G = importlib.util.module_from_spec(spec)
    ctypes.CDLL = lambda name, *a, **k: real(path, *a, **k)
    try:
        import sys

        sys.modules[spec.name] = G  # (dataclasses look their module up)
        spec.loader.exec_module(G)
    finally:
        ctypes.CDLL = real
    G._dptr = lambda t, dtype=None, numel=None: None if t is None else ctypes.c_void_p(t.data_ptr())
    G._stream = lambda stream: None
    lib = G._lib
    lib.fake_log.restype = ctypes.c_char_p
    lib.fake_live.restype = ctypes.c_size_t
    lib.fake_limit.argtypes = [ctypes.c_size_t]
    lib.fake_list_entries.argtypes = [ctypes.c_longlong]
    lib.fake_tiles.argtypes = [ctypes.c_longlong]
    return G, lib
