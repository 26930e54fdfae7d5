// rollout_chain.cu -- launcher of the standalone planar-chain rollout, with
// direct or staged control loads (rollout_kernels.cuh).
#include "rollout_kernels.cuh"

namespace mtp {
namespace {

constexpr int kMaxChainLinks = 12;

template <int NL, int T, bool SFU = kSfuTurns<NL, kPrefetchAlone>>
cudaError_t chain_launch(const RolloutArgs& a, const ChainModel& m, cudaStream_t s) {
  const int bd = rollout_block(a.rows);
  k_rollout_chain<NL, T, SFU><<<(a.rows + bd - 1) / bd, bd, staged_smem<NL, T>(bd), s>>>(a, m);
  return cudaGetLastError();
}

template <int NL>
cudaError_t chain_dispatch(const RolloutArgs& a, const ChainModel& m, int links, bool staged,
                           cudaStream_t s) {
  if constexpr (NL <= kMaxChainLinks) {
    if (links == NL) {
      if (staged) return chain_launch<NL, chain_chunk(NL)>(a, m, s);
      return turns_by_sfu(a.rows) ? chain_launch<NL, 0, true>(a, m, s) : chain_launch<NL, 0>(a, m, s);
    }
    return chain_dispatch<NL + 1>(a, m, links, staged, s);
  } else {
    return cudaErrorInvalidValue;
  }
}

template <int NL>
cudaError_t chain_attributes() {
  if constexpr (NL <= kMaxChainLinks) {
    cudaError_t e = cudaFuncSetAttribute(k_rollout_chain<NL, chain_chunk(NL), kSfuTurns<NL, kPrefetchAlone>>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)staged_smem<NL, chain_chunk(NL)>(kThreads));
    if (e != cudaSuccess) return e;
    return chain_attributes<NL + 1>();
  } else {
    return cudaSuccess;
  }
}

}  // namespace

cudaError_t init_rollout_chain_attributes() { return chain_attributes<1>(); }

cudaError_t launch_rollout_chain(const RolloutArgs& a, const ChainModel& m, int links, cudaStream_t s) {
  if (a.rows <= 0) return cudaSuccess;
  const bool shared = a.dr_mode == MTP_DR_SHARED && a.R > 1;
  return chain_dispatch<1>(a, m, links, can_stage(a, links) && stages_alone(links, a.H, a.rows, shared), s);
}

int rollout_blocks(int rows) {
  if (rows <= 0) return 0;
  const int bd = rollout_block(rows);
  return (rows + bd - 1) / bd;
}

}  // namespace mtp
