"""Candidate generation of light rows (straight lines, B-splines of few dimensions or
of rows that are not whole 16-byte pieces) fits five blocks of 256 threads on an SM: at
most 48 registers a thread, without spills.  With the 56 that heavy rows need, and four
blocks, they took up to 1.45 times as long."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_light_rows_leave_room_for_five_blocks(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    csrc = os.path.join(ROOT, "paper_2505_01059_gb300", "csrc")
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-Xptxas", "-v", "-I",
                        os.path.join(ROOT, "include"), "-I", csrc, "-c", os.path.join(csrc, "candidates.cu"), "-o",
                        str(tmp_path / "candidates.o")], check=True, capture_output=True, text=True)
    use = re.findall(r"entry function '\w*?k_candidates(I\w*?E)?E\w*'.*?(\d+) bytes spill stores.*?Used (\d+) registers",
                     r.stderr, re.S)
    assert use
    blocks = sorted(65536 // (256 * (-(-int(regs) // 8) * 8)) for _, _, regs in use)
    assert blocks[-1] >= 5 and all(spilled == "0" for _, spilled, _ in use)
