"""Memory that a product with several right-hand sides takes (host logic): what a lockstep solve counts is what is
allocated.  Compiles tests/batch_bytes_check.cpp with the system C++ compiler."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_bytes_of_a_batch(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "batch_bytes_check")
    subprocess.run([cxx, "-std=c++17", "-O1", "-o", exe, os.path.join(HERE, "batch_bytes_check.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout
