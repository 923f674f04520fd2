"""Builds tests/native/probe.cu against libpf.so and loads it."""
import ctypes as C
import os
import subprocess

from paper_2007_12908_gb300 import _binding as B
from paper_2007_12908_gb300 import build

SRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "native", "probe.cu")
OUT = os.path.join(build.BUILD, "probe.so")


def load() -> C.CDLL:
    lib = build.build()
    B.lib()
    newest = max(os.path.getmtime(p) for p in (SRC, lib))
    if not os.path.exists(OUT) or os.path.getmtime(OUT) < newest:
        cmd = [build._nvcc(), *build.FLAGS, *build.ARCH, "-I", build.CSRC, "-shared", SRC, "-o", OUT + ".tmp",
               lib, "-Xlinker", "-rpath," + os.path.dirname(lib)]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(r.stdout + r.stderr)
        os.replace(OUT + ".tmp", OUT)
    return C.CDLL(OUT)


def ptr(t):
    return C.c_void_p(t.data_ptr() if t is not None else None)
