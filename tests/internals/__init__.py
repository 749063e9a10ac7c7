"""Builds internals.cu against the library's objects and loads it (tests only).  The functions
take the handle of a package Lattice: both libraries are built from the same headers."""
import ctypes
import importlib.util
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(os.path.dirname(HERE))


def load():
    spec = importlib.util.spec_from_file_location("_qs_build", os.path.join(ROOT, "paper_2108_11989_gb300", "build.py"))
    b = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(b)
    b.build()
    out = os.path.join(HERE, "_build")
    os.makedirs(out, exist_ok=True)
    src, obj, so = os.path.join(HERE, "internals.cu"), os.path.join(out, "internals.o"), os.path.join(out, "libqsinternals.so")
    objs = [os.path.join(b.BUILD, os.path.basename(s)[:-3] + ".o") for s in b.sources() if not s.endswith("solver.cu")]
    newest = max(os.path.getmtime(f) for f in [src, b.LIB] + objs)
    if not os.path.exists(so) or os.path.getmtime(so) < newest:
        subprocess.run([b.NVCC, *b.ARCH, *b.FLAGS, "-c", src, "-o", obj], check=True)
        subprocess.run([b.NVCC, *b.ARCH, "-shared", "-o", so, obj, *objs], check=True)
    lib = ctypes.CDLL(so)
    P, I, D, L = ctypes.c_void_p, ctypes.c_int, ctypes.c_double, ctypes.c_int64
    for name, args in {"t_ntile": [P], "t_nvariants": [], "t_fixed_variant": [P, I],
                      "t_d32": [P, I, I, I, I, D, P, P, P, P, D, D, D, P, P, P],
                       "t_norm2": [P, I, P, I, L, P, P], "t_resid2": [P, P, P, P, I, L, P, P],
                       "t_cg": [P, I, D, D, I, P, P, P],
                       "t_rr32": [P, I, D, P, P, P]}.items():
        getattr(lib, name).argtypes = args
    lib.t_ntile.restype = L
    return lib
