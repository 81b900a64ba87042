"""Shared-memory layout of the one-cluster Rayleigh-Ritz kernel, checked on the CPU with the
kernel's own index functions (tests/ritz_layout_dump.cu): for every subspace size, on clusters of 8 and
of 16 CTAs, what a sweep reads of a copy of the matrix lies inside that copy and the copies inside the memory that the launch
asks for, every matrix entry has a place of its own, and the threads that take part cover all
blocks."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = str(tmp_path_factory.mktemp("ritz") / "ritz_layout_dump")
    subprocess.run([nvcc, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1602_01421_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "ritz_layout_dump.cu"), "-o", exe], check=True, capture_output=True)
    return subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()


def test_sweep_reads_stay_inside_the_copy(lines):
    rows = [line for line in lines if not line.startswith("sweeps")]
    assert len(rows) == 2 * 160
    for line in rows:
        m, threads, active, items, top, copy, end, asked, once = map(int, line.split())
        pairs = (m + 1) // 2
        assert top < copy, f"m = {m}: reads float {top} of a copy of {copy}"
        assert end <= asked and once == 1, m
        assert active % 32 == 0 and pairs <= active <= threads and items * active >= pairs * (pairs - 1) // 2, m


def test_sweeps_allowed(lines):
    """max_sweeps bounds the sweeps after the first iteration's FP32 ones, all iterations together, and
    leaves those of the first one alone."""
    rows = [line.split()[1:] for line in lines if line.startswith("sweeps")]
    assert rows
    for row in rows:
        max_sweeps, first, later = map(int, row)
        assert first == 15 and later == max_sweeps
