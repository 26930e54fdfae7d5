// rollout_pm.cu -- launcher of the standalone k-D point-mass rollout
// (rollout_pm.cuh).
#include "rollout_pm.cuh"

namespace mtp {
namespace {

template <int K>
cudaError_t pm_dispatch(const RolloutArgs& a, const PointMassModel& m, cudaStream_t s) {
  if constexpr (K <= kMaxPmAxes) {
    if (a.n == K) {
      const PmBody body = a.X ? PmBody::kTile : pm_body<K>(a.rows, a.H, can_stage(a, K));
      if (body != PmBody::kTile) {
        const int block = body == PmBody::kLanes ? 64 : rollout_block(a.rows), grid = (a.rows + block - 1) / block;
        if (body == PmBody::kLanes)
          k_rollout_pm_lanes<K><<<grid, block, block / 32 * PmLane<K>::floats * sizeof(float), s>>>(a, m);
        else k_rollout_pm_direct<K><<<grid, block, 0, s>>>(a, m);
        return cudaGetLastError();
      }
      const PmTile t = pm_tile<K>(a.rows);
      const int tiles = (a.rows + t.C - 1) / t.C, warps = t.block / 32, grid = (tiles + warps - 1) / warps;
      const size_t smem = warps * t.floats * sizeof(float);
      if (a.X) k_rollout_pm<K, true><<<grid, t.block, smem, s>>>(a, m, t.C, t.T, t.row, t.floats);
      else k_rollout_pm<K, false><<<grid, t.block, smem, s>>>(a, m, t.C, t.T, t.row, t.floats);
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
        (e = cudaFuncSetAttribute(k_rollout_pm<K, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPmSmemMax)) ||
        (e = cudaFuncSetAttribute(k_rollout_pm_lanes<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPmSmemMax)))
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
