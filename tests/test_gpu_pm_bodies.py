"""A lone point-mass rollout takes one of three bodies by its size (a warp per tile
of candidates, a lane per candidate with staged rows, a thread per candidate with
direct loads): the choice at sizes on both sides of its lines, and the same bits
from each of them, whichever candidates a call holds."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2505_01059_gb300 import workloads as W

torch = pytest.importorskip("torch")
DEV = "cuda:0"
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# axes, candidates, steps, rows of whole 16-byte pieces, body: t tile, l lanes, d direct.
# on 152 SMs
CHOICES = [
    (2, 512, 64, 1, "t"), (12, 8192, 256, 1, "t"), (7, 4096, 33, 0, "t"), (16, 1, 200, 1, "t"), (4, 1000, 16, 1, "t"),
    (7, 30000, 33, 0, "d"), (9, 16384, 45, 0, "d"), (3, 65536, 101, 0, "d"), (5, 1 << 24, 31, 0, "d"),
    (12, 32768, 64, 1, "l"), (2, 200000, 64, 1, "l"), (16, 200000, 20, 1, "l"),
    (2, 8192, 9, 0, "d"), (12, 8192, 11, 1, "d"), (4, 300, 15, 1, "d"), (1, 24000, 20, 1, "d"), (1, 24000, 31, 0, "d"),
]

PROGRAM = r"""
#include <cstdio>
#include "rollout_pm.cuh"
namespace mtp {
int device_sms() { return 152; }
}
using namespace mtp;
template <int K>
PmBody choose(int k, long long rows, int H, bool pieces) {
  if constexpr (K < kMaxPmAxes)
    if (k != K) return choose<K + 1>(k, rows, H, pieces);
  return pm_body<K>(rows, H, pieces);
}
int main() {
  long long rows;
  int k, H, pieces;
  while (std::scanf("%d %lld %d %d", &k, &rows, &H, &pieces) == 4) {
    const PmBody b = choose<1>(k, rows, H, pieces != 0);
    std::putchar(b == PmBody::kTile ? 't' : b == PmBody::kLanes ? 'l' : 'd');
  }
}
"""


def test_choice(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "pm_body.cu", tmp_path / "pm_body"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17",
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2505_01059_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    text = "\n".join("%d %d %d %d" % c[:4] for c in CHOICES)
    r = subprocess.run([str(exe)], input=text, capture_output=True, text=True, timeout=120)
    assert r.stdout == "".join(c[4] for c in CHOICES)


@pytest.fixture(scope="module")
def mtp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_01059_gb300 import _build, mtp as m
    _build.build_library()
    m.load_library()
    torch.cuda.set_device(0)
    return m


# all candidates at once: direct, lanes, direct, lanes, lanes, direct; 257 of them: a tile each
@pytest.mark.gpu
@pytest.mark.parametrize("k,B,H,extra", [
    (7, 30000, 33, dict(dr_mode="per_sample", dr_lo=0.8, dr_hi=1.2)),
    (3, 40001, 20, {}),
    (9, 20000, 45, dict(flags=0x1)),
    (16, 33000, 65, dict(dr_mode="per_sample", dr_lo=0.8, dr_hi=1.2)),
    (4, 60000, 36, dict(dr_mode="shared", R=3, dr_lo=0.9, dr_hi=1.1)),
    (1, 70003, 26, dict(n_obstacles=8)),
])
def test_every_body_gives_the_same_bits(mtp, k, B, H, extra):
    spec = W.pointmass(**dict(dict(seed=k, k=k, B=B, H=H, E=1, M=4, N=8, degree=2, w_ctrl=0.01), **extra))
    h = mtp.mtp_create(spec)
    g = torch.Generator(device=DEV).manual_seed(H)
    U = torch.rand(B, H, k, generator=g, device=DEV) * 2 - 1
    U[5] = float("inf")
    U[B - 2] = float("nan")
    x0 = torch.tensor(np.random.default_rng(B).uniform(-0.2, 0.8, size=2 * k).astype(np.float32), device=DEV)
    cost = torch.full((B,), -1.0, device=DEV)
    mtp.mtp_rollout_cost(h, 3, x0, U, cost)
    for row0 in (0, B // 3, B - 257):
        part = torch.empty(257, device=DEV)
        mtp.mtp_rollout_cost(h, 3, x0, U[row0:row0 + 257].contiguous(), part, row0=row0)
        assert torch.equal(part, cost[row0:row0 + 257]), row0
    assert torch.isinf(cost[[5, B - 2]]).all() and torch.isfinite(cost).sum() == B - 2
    mtp.mtp_destroy(h)
