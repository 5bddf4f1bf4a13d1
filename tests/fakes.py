"""The library linked with cuda_fakes.cpp in front of the CUDA runtime, and a
process that runs a script on it."""
import os
import subprocess
import sys

from paper_1208_4247_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
WRAPPED = ["cudaFuncSetAttribute", "cudaLaunchKernelExC", "cudaOccupancyMaxActiveClusters",
           "cudaMemcpyAsync", "sinl", "cosl", "sincosl"]


def link(path):
    """libgmg.so's objects and the fakes -> path"""
    build.build()
    objs = [os.path.join(build.OUT_DIR, "obj", os.path.basename(s)[:-3] + ".o")
            for s in build.sources()]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    r = subprocess.run([build.nvcc(), "-shared", *build.ARCH, "-Xcompiler", "-fPIC", "-o", path,
                        os.path.join(HERE, "cuda_fakes.cpp"), *objs, "-lcudart", "-lm",
                        *[x for w in WRAPPED for x in ("-Xlinker", f"--wrap={w}")]],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return path


PREAMBLE = """
import ctypes, sys
import numpy as np
import torch
from paper_1208_4247_gb300 import gmg, inputs
gmg.LIB_PATH = sys.argv[1]
fake = ctypes.CDLL(sys.argv[1])
"""


def run(path, script):
    """The script's output lines, in a process of its own (PREAMBLE first)."""
    r = subprocess.run([sys.executable, "-c", PREAMBLE + script, path], capture_output=True,
                       text=True, timeout=300, cwd=os.path.dirname(HERE))
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout.strip().splitlines()
