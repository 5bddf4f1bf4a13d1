"""The batched legs' tiles, on the host: every output in exactly one tile, every
operand of it inside the tile."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1208_4247_gb300", "csrc")


def test_tiles_cover_each_level_once(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("needs g++")
    exe = str(tmp_path / "tiles")
    subprocess.run([gxx, "-std=c++17", "-O2", "-I", CSRC, "-o", exe,
                    os.path.join(HERE, "batch_tiles_check.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
