"""Which lone chain rollouts stage their controls: by link count, whether the rows
are whole cache lines apart (H n a multiple of 32), and how many candidates there
are, at sizes where the other form took 5 to 60 % longer."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "rollout_kernels.cuh"
namespace mtp {
int device_sms() { return 152; }
}
int main() {
  int links, H, rows;
  while (std::scanf("%d %d %d", &links, &H, &rows) == 3) std::putchar(mtp::stages_alone(links, H, rows) ? 's' : 'd');
}
"""

# links, steps, candidates (on 152 SMs), form: s staged, d direct
CASES = [(8, 36, 64, "s"), (8, 128, 2048, "s"), (6, 64, 2048, "s"), (3, 48, 8192, "s"), (2, 256, 64, "s"),
         (7, 128, 4096, "d"), (4, 64, 8192, "d"), (5, 48, 1000, "d"), (9, 36, 2048, "d"), (11, 36, 2048, "d"),
         (7, 48, 16384, "d"), (9, 36, 16384, "d"), (5, 36, 16384, "d"), (12, 36, 40000, "d"), (1, 48, 1000, "d"),
         (7, 128, 16384, "s"), (4, 48, 16384, "s"), (9, 64, 40000, "s"), (1, 64, 40000, "s"), (11, 64, 64, "s")]


def test_rule(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "rule.cu", tmp_path / "rule"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17",
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2505_01059_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], input="\n".join("%d %d %d" % c[:3] for c in CASES), capture_output=True, text=True,
                       timeout=120)
    assert r.stdout == "".join(c[3] for c in CASES)
