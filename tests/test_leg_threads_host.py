"""The batched legs' launch shapes against their launch bounds, on the host."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1208_4247_gb300", "csrc")


def test_threads_within_the_launch_bounds(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("needs g++")
    exe = str(tmp_path / "threads")
    subprocess.run([gxx, "-std=c++17", "-O2", "-I", CSRC, "-o", exe,
                    os.path.join(HERE, "leg_threads_check.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
