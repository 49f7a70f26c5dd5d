"""Compile the test-only probes: cuRAND's Philox (tests/cuda/libcurand_probe.so) and the library's own elementary
functions (tests/cuda/libmath_probe.so)."""
import os
import shutil
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(os.path.dirname(HERE)), "paper_1411_4212_gb300", "csrc")
SRC = os.path.join(HERE, "curand_philox_probe.cu")
OUT = os.path.join(HERE, "libcurand_probe.so")
MATH_SRC = os.path.join(HERE, "math_probe.cu")
MATH_OUT = os.path.join(HERE, "libmath_probe.so")


def _compile(out, deps, force):
    if not force and os.path.exists(out) and all(os.path.getmtime(out) >= os.path.getmtime(d) for d in deps):
        return out
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "-I", CSRC, "-shared",
                    "-Xcompiler", "-fPIC", "-cudart", "shared", "-o", out, deps[0]], check=True)
    return out


def build(force=False):
    _compile(MATH_OUT, [MATH_SRC, os.path.join(CSRC, "device_math.cuh")], force)
    return _compile(OUT, [SRC], force)


if __name__ == "__main__":
    print(build(force=True))
