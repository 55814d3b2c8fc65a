"""How a host encryption is cut into pieces, checked without a GPU."""
import os
import shutil
import subprocess

import pytest

from paper_2111_11924_gb300 import _native_build as NB

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_pieces_over_random_messages(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "host_pieces_check")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-Wall", "-Wextra", "-Werror", "-o", exe,
                           os.path.join(ROOT, "tests", "c", "host_pieces_check.cpp"), "-I", NB.CSRC])
    res = subprocess.run([exe], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout
