"""The shared-memory layout of a lone point-mass rollout's tile depends on the
axis count alone, so choosing a tile at a launch is a few comparisons: a program
around the library's own headers checks every row against the search that defines
it (the shortest 16-byte row with the fewest bank conflicts), that a block's
tiles fit its shared memory, and that a choice takes well under a microsecond of
the host (searching the rows at each launch took 20 to 60)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <chrono>
#include <cstdio>
#include "rollout_pm.cuh"
namespace mtp {
int device_sms() { return 152; }
}
using namespace mtp;

static int conflicts(int K, int row) {
  int most = 0;
  for (int b = 0; b < 32; ++b) {
    int hits = 0;
    for (int q = 0; q < 32; ++q) hits += (q / K * row + q % K) % 32 == b;
    if (hits > most) most = hits;
  }
  return most;
}
static int shortest(int K, int T) {
  const int least = (T * (K % 8 ? K : K + 4) + 3) / 4 * 4;
  int best = least;
  for (int y = least; y < least + 32; y += 4)
    if (conflicts(K, y) < conflicts(K, best)) best = y;
  return best;
}

static int bad = 0;
template <int K>
void check() {
  for (long long rows : {1LL, 7LL, 512LL, 911LL, 912LL, 1823LL, 1824LL, 7296LL, 8192LL, 30000LL, 1LL << 24}) {
    const PmTile t = pm_tile<K>(rows);
    const bool ok = t.T >= 4 && t.T % 4 == 0 && t.C >= 1 && t.C <= 32 && t.row == shortest(K, t.T) &&
                    t.floats >= t.C * (2 * t.row + 3 * K + t.T + 1) && t.floats % 4 == 0 &&
                    t.block / 32 * t.floats * 4 <= kPmSmemMax;
    if (!ok) {
      ++bad;
      std::printf("K %d rows %lld: C %d T %d row %d (%d) floats %d\n", K, rows, t.C, t.T, t.row, shortest(K, t.T), t.floats);
    }
  }
  double best = 1e9;
  long long sum = 0;
  for (int rep = 0; rep < 5; ++rep) {
    const auto t0 = std::chrono::steady_clock::now();
    for (int i = 0; i < 1000; ++i) sum += pm_tile<K>(1000 + i).floats;
    best = std::min(best, std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count() * 1e3);
  }
  if (best > 1.0) ++bad;
  std::printf("K %d: %.3f us a choice (%lld)\n", K, best, sum % 10);
  if constexpr (K < kMaxPmAxes) check<K + 1>();
}

int main() {
  check<1>();
  return bad != 0;
}
"""


def test_tiles_are_chosen_without_a_search(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "pm_tile.cu", tmp_path / "pm_tile"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17",
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2505_01059_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
