"""narrow_sixth (a double's sixth as a float, on the FP32 pipe) over the whole
range of the float format, on the host."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1208_4247_gb300", "csrc")


def test_narrow_sixth(tmp_path):
    gxx, cuda_inc = shutil.which("g++"), "/usr/local/cuda/include"
    if not gxx or not os.path.exists(os.path.join(cuda_inc, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path / "narrow_sixth")
    subprocess.run([gxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, "-I", cuda_inc, "-o",
                    exe, os.path.join(HERE, "narrow_sixth_check.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
