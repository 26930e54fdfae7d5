"""Which lone chain rollouts of shared models stage their controls, where the other
form took 3 to 11 % longer, and which rollouts take their angles' whole turns on the
SFU: many candidates, whose issue slots are full."""
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
  while (std::scanf("%d %d %d", &links, &H, &rows) == 3) {
    std::putchar(mtp::stages_alone(links, H, rows, true) ? 's' : 'd');
    std::putchar(mtp::turns_by_sfu(rows) ? 'S' : 'f');
  }
}
"""

# links, steps, candidates (on 152 SMs): s staged, d direct; S turns on the SFU, f off it
CASES = [(10, 50, 1000, "df"), (12, 97, 32, "df"), (12, 50, 4096, "df"), (6, 100, 2000, "df"), (2, 50, 1000, "df"),
         (3, 100, 256, "sf"), (8, 50, 4096, "sf"), (12, 48, 1000, "sf"), (10, 128, 4096, "sf"), (6, 128, 4096, "sf"),
         (12, 36, 16384, "sf"), (10, 36, 16384, "sf"), (6, 36, 16384, "df"), (2, 36, 16384, "df"),
         (7, 128, 4096, "df"), (11, 36, 2048, "df"), (12, 36, 40000, "dS"), (9, 36, 40000, "dS"), (9, 36, 16384, "df")]


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
