"""Settled slot moves (host half of a large batch of cuckoo writes) against the
ordered moves they stand for, on arbitrary lists and on those of inserts with
evictions, collection and failed walks."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_settled_moves_leave_every_slot_as_the_ordered_ones(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("needs the CUDA toolkit's headers")
    exe = str(tmp_path / "settle_check")
    src = [os.path.join(ROOT, "tests", "settle_check.cpp"),
           os.path.join(ROOT, "paper_2001_08250_gb300", "csrc", "cuckoo.cpp")]
    subprocess.run([nvcc, "-O1", "-std=c++17", "-I", os.path.join(ROOT, "include"), *src, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
