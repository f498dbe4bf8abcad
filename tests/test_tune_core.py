"""The tuner's candidate settings (no GPU), built with g++."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_candidates_begin_with_the_present_settings(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "tune_core_check")
    subprocess.check_call([gxx, "-std=c++17", "-O1", "-Wall",
                           "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(ROOT, "paper_1501_05387_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "tune_core_check.cpp"), "-o", exe])
    res = subprocess.run([exe], capture_output=True, text=True)
    assert res.returncode == 0 and res.stdout.strip() == "ok", res.stdout + res.stderr
