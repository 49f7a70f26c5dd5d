"""Runs the package in a process of its own on a CUDA runtime without a GPU (tests/cuda/fake_runtime.cpp): the
objects of the library's build, linked with that runtime."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "tests", "cuda", "fake_runtime.cpp")
OUT = os.path.join(ROOT, "tests", "cuda", "librewl_fake.so")

PRELUDE = """
import ctypes, sys
sys.modules["torch"] = None
import numpy as np
import paper_1411_4212_gb300 as rw
lib = rw.load_library({out!r})
lib.fake_pool_reserved.restype = lib.fake_pool_used.restype = lib.fake_plain_bytes.restype = lib.fake_stream.restype = ctypes.c_size_t
lib.fake_refuse_from.argtypes = [ctypes.c_size_t]
lib.fake_work.argtypes = [ctypes.c_size_t]
"""


def library():
    from paper_1411_4212_gb300 import _build
    _build.build()
    objs = [os.path.join(_build.BUILD, os.path.splitext(s)[0] + ".o") for s in _build.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        _build.build(force=True)
    include = os.path.join(os.path.dirname(os.path.dirname(_build.nvcc())), "include")
    if not os.path.exists(OUT) or os.path.getmtime(OUT) < max(map(os.path.getmtime, objs + [SRC])):
        subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", include, "-o", OUT, SRC,
                        *objs], check=True)
    return OUT


def run(script):
    """Run `script` after the prelude; it fails by an exception, an assertion or a crash."""
    r = subprocess.run([sys.executable, "-c", PRELUDE.format(out=library()) + script], cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, f"exit {r.returncode}\n{r.stdout}\n{r.stderr}"
    return r.stdout
