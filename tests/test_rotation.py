"""The rotating accumulators of the residue product (csrc/rotation.h) in a model of
the warps that use and drain them: no wait is answered by an older phase."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2006_08498_gb300", "csrc")


def test_no_buffer_is_used_before_it_is_drained(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "rotation_model")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, os.path.join(HERE, "rotation_model.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe, "5000"], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
