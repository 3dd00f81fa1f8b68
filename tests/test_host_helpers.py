"""Host-side logic of the library checked on the CPU (no GPU, no kernel launch).

aligned_prefetch_range: logq_linear_grouped accepts an L2 prefetch hint at any
alignment, and the bulk prefetch it issues wants a 16-byte aligned start and a
whole number of 16-byte units.  The helper is compiled with the host compiler
from the library's own header and checked over every start offset and length
in a window, against the largest aligned range inside the caller's range.

reads_codes_early: which launches may read packed codes before the kernel ahead of
them on the stream has completed, checked the same way.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"


def run_host_check(name, tmp_path):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.isdir(CUDA_INC):
        pytest.skip("host compiler or CUDA headers missing")
    exe = tmp_path / name
    subprocess.run([cxx, "-std=c++17", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2607_01127_gb300", "csrc"), "-I", CUDA_INC,
                    os.path.join(ROOT, "tests", "host", name + ".cpp"), "-o", str(exe)],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr


def test_aligned_prefetch_range(tmp_path):
    run_host_check("prefetch_range_check", tmp_path)


def test_larger_batches_read_codes_in_stream_order(tmp_path):
    run_host_check("reads_codes_check", tmp_path)
