"""The rule by which smaller batches earn the transposed copy, on the host."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_sequence_loses_more_than_one_copy(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("needs a C++ compiler")
    exe = str(tmp_path / "copyrule_check")
    subprocess.run([cxx, "-O1", "-std=c++17", os.path.join(ROOT, "tests", "copyrule_check.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
