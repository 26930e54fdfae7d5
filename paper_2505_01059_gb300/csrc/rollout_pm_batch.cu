// rollout_pm_batch.cu -- launcher of the batched k-D point-mass rollout (one
// launch over many instances of one dimension; rollout_pm.cuh).
#include "rollout_pm.cuh"

namespace mtp {
namespace {

template <int K>
cudaError_t pm_batch_dispatch(const RolloutArgs* ra, const PointMassModel* pm, const int* row_start, int count,
                              int total_rows, int k, int block, bool staged, cudaStream_t s) {
  if constexpr (K <= kMaxPmAxes) {
    if (k == K) {
      const int grid = (total_rows + block - 1) / block;
      if (staged)
        k_rollout_pm_batch<K, true><<<grid, block, block / 32 * PmLane<K>::floats * sizeof(float), s>>>(ra, pm, row_start, count);
      else k_rollout_pm_batch<K, false><<<grid, block, 0, s>>>(ra, pm, row_start, count);
      return cudaGetLastError();
    }
    return pm_batch_dispatch<K + 1>(ra, pm, row_start, count, total_rows, k, block, staged, s);
  } else {
    return cudaErrorInvalidValue;
  }
}

template <int K>
cudaError_t pm_batch_attributes() {
  if constexpr (K <= kMaxPmAxes) {
    const cudaError_t e =
        cudaFuncSetAttribute(k_rollout_pm_batch<K, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPmSmemMax);
    if (e != cudaSuccess) return e;
    return pm_batch_attributes<K + 1>();
  } else {
    return cudaSuccess;
  }
}

}  // namespace

cudaError_t init_rollout_pm_batch_attributes() { return pm_batch_attributes<1>(); }

cudaError_t launch_rollout_pointmass_batch(const RolloutArgs* d_ra, const PointMassModel* d_pm, const int* d_row_start,
                                           int count, int total_rows, int k, int block, bool staged, cudaStream_t s) {
  if (total_rows <= 0) return cudaSuccess;
  return pm_batch_dispatch<1>(d_ra, d_pm, d_row_start, count, total_rows, k, block, staged, s);
}

}  // namespace mtp
