"""The NTT passes' index arithmetic on the host, for every size (n = 1..24, one
and two digits, 1 to 64 slices, every tile, whole and part-filled, and the
commitment's row encodings): each column, factor and shared-memory index is in
range and what its definition says, and every output element is stored once."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_every_index(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "check")
    subprocess.run([cxx, "-std=c++17", "-O2", os.path.join(HERE, "ntt_index_check.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.startswith("ok "), r.stdout
