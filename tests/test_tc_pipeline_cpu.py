"""Control flow of the copy and MMA lanes of the tensor-core M2L when a bounded wait runs out (host logic): nothing
is issued afterwards, and exactly the stages in flight are waited for.  Compiles tests/tc_pipeline_check.cpp with
the system C++ compiler."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_lanes_stop_and_drain(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "tc_pipeline_check")
    subprocess.run([cxx, "-std=c++17", "-O1", "-o", exe, os.path.join(HERE, "tc_pipeline_check.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout
