// rollout_pm.cu -- launcher of the standalone k-D point-mass rollout
// (rollout_pm.cuh).
#include "rollout_pm.cuh"

namespace mtp {
namespace {

// Candidates C and steps T of a warp's tile, and threads per block, for `rows`
// candidates.  About six warps per SM or more before a warp takes a second
// candidate; up to eight candidates per warp, two beyond 8 axes, whose rows fill
// the shared memory first.  T up to 64 steps, as far as a tile takes 16 KB.
// Measured (us a call, replayed from a graph; C and T swept over 1 .. 32 and
// 8 .. 128): 2 axes, B 512, H 64: C 1 / 2 / 8 at T 64: 5.4 / 5.6 / 7.9 (21 as one
// candidate per lane); 2 axes, B 8192, H 128: C 1 / 2 / 4 / 8: 29 / 19 / 14 / 14;
// 12 axes, B 8192, H 256: C 1 / 2 / 4 / 8: 63 / 49 / 56 / 55 (227 as one candidate
// per lane); 16 axes, B 8192, H 128: C 2, T 32 / 64: 34 / 47.
struct PmTile {
  int C, T, block;
};
template <int K>
PmTile pm_tile(long long rows) {
  PmTile t{K > 8 ? 2 : 8, 64, 128};
  const long long want = (long long)device_sms() * 6;
  while (t.C > 1 && rows / t.C < want) t.C >>= 1;
  while (t.T > 4 && PmTileShape<K>::floats(t.C, t.T) > 4096) t.T >>= 1;
  while (t.block > 32 && rows / t.C * 32 < (long long)t.block * device_sms()) t.block >>= 1;
  return t;
}

template <int K>
cudaError_t pm_dispatch(const RolloutArgs& a, const PointMassModel& m, cudaStream_t s) {
  if constexpr (K <= kMaxPmAxes) {
    if (a.n == K) {
      const PmTile t = pm_tile<K>(a.rows);
      const int tiles = (a.rows + t.C - 1) / t.C, warps = t.block / 32, grid = (tiles + warps - 1) / warps;
      const int row = PmTileShape<K>::row(t.T), floats = PmTileShape<K>::floats(t.C, t.T);
      const size_t smem = warps * floats * sizeof(float);
      if (a.X) k_rollout_pm<K, true><<<grid, t.block, smem, s>>>(a, m, t.C, t.T, row, floats);
      else k_rollout_pm<K, false><<<grid, t.block, smem, s>>>(a, m, t.C, t.T, row, floats);
      return cudaGetLastError();
    }
    return pm_dispatch<K + 1>(a, m, s);
  } else {
    return cudaErrorInvalidValue;
  }
}

template <int K>
cudaError_t pm_attributes() {
  if constexpr (K <= kMaxPmAxes) {
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(k_rollout_pm<K, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPmSmemMax)) ||
        (e = cudaFuncSetAttribute(k_rollout_pm<K, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPmSmemMax)))
      return e;
    return pm_attributes<K + 1>();
  } else {
    return cudaSuccess;
  }
}

}  // namespace

cudaError_t init_rollout_pm_attributes() { return pm_attributes<1>(); }

cudaError_t launch_rollout_pointmass(const RolloutArgs& a, const PointMassModel& m, cudaStream_t s) {
  if (a.rows <= 0) return cudaSuccess;
  return pm_dispatch<1>(a, m, s);
}

}  // namespace mtp
