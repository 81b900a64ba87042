"""Shared-memory layout of the one-cluster Rayleigh-Ritz kernel, checked on the CPU with the
kernel's own index functions (tests/ritz_layout_dump.cu): for every subspace size, what a sweep
reads of a copy of the matrix lies inside that copy and the copies inside the memory that the launch
asks for, every matrix entry has a place of its own, and the threads that take part cover all
blocks."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_sweep_reads_stay_inside_the_copy(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "ritz_layout_dump")
    subprocess.run([nvcc, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1602_01421_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "ritz_layout_dump.cu"), "-o", exe], check=True, capture_output=True)
    lines = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()
    assert len(lines) == 160
    for line in lines:
        m, threads, active, items, top, copy, end, asked, once = map(int, line.split())
        pairs = (m + 1) // 2
        assert top < copy, f"m = {m}: reads float {top} of a copy of {copy}"
        assert end <= asked and once == 1, m
        assert active % 32 == 0 and pairs <= active <= threads and items * active >= pairs * (pairs - 1) // 2, m
