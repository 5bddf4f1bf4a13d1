"""cvt::narrow (double to float on the integer pipe) against the C cast, bit for
bit, on the host."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1208_4247_gb300", "csrc")


def test_narrow_equals_cast(tmp_path):
    gxx, cuda_inc = shutil.which("g++"), "/usr/local/cuda/include"
    if not gxx or not os.path.exists(os.path.join(cuda_inc, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path / "narrow")
    subprocess.run([gxx, "-std=c++17", "-O2", "-I", CSRC, "-I", cuda_inc, "-o", exe,
                    os.path.join(HERE, "narrow_host_check.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
