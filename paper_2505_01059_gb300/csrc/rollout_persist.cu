// rollout_persist.cu -- the rollouts of a whole batch in one persistent
// launch, or two (Alg. 2 rollout fused with the Eq. 2 cost, the bodies of
// rollout_kernels.cuh and rollout_pm.cuh).
//
// Work items are warp tiles: 32 consecutive candidates of one instance.  The
// instances are listed group by group, the longest group first and within a
// group the longest expected rollout first (H times the time per step of the
// group's dynamics and dimension), and numbered by a prefix of their warp
// tiles, so item w belongs to the instance whose range holds w.  Each warp of
// the launch repeatedly takes the next item from a device counter (one
// atomic add per item), looks its instance up by binary search, and runs
// that tile's rollout: a point mass of K axes, or a planar chain of L links with
// direct or staged control loads.  A warp therefore
// moves between instances of different sizes and dynamics, while the warps
// running at one time mostly run the same body.  The bodies are the
// per-candidate rollouts of the other kernels (the same templates), so every
// cost is the same bits as in a per-group or standalone launch.  The
// two-launch mode of the batch runs the same kernel over two ranges of the
// entries (w_base numbers the second range's tiles).
//
// The warps never wait on one another: an item, once taken, depends only on
// the candidates generated before the launch.
//
// The bodies are inlined into the kernel: as separate functions their
// arguments went through a 240-byte stack frame and the launch was 7-8 %
// slower on the batch of 256.  The launch is bounded at three 128-thread
// CTAs per SM, i.e. at most 170 registers per thread (168 used, no spills).
//
// Measured on GB300 on the 256-instance batch (the bench's timed region):
// 1.90 ms per iteration with two launches: 2.68 before the point masses
// evaluated several steps' costs at once (2.43 then), 2.09 before the chains'
// controls were staged by asynchronous copies and not by bulk copies with
// their barriers, the rest in generation.  The order of the
// tiles matters: sorted by length alone across all groups, the warps of an
// SM ran different bodies at once, half of their stall samples were
// instruction fetches, and the iteration took 3.5 ms; tiles are therefore
// taken group by group (longest group first, longest tiles first within it).
#include <algorithm>
#include <map>
#include <mutex>

#include "rollout_kernels.cuh"
#include "rollout_pm.cuh"

namespace mtp {
namespace {

constexpr int kPersistThreads = 128;

template <int K, bool DIRECT>
__device__ __forceinline__ void pm_item(int k, bool pieces, const RolloutArgs& a, const PointMassModel& m, int r0,
                                        float* buf) {
  if constexpr (K <= kPersistMaxAxes) {
    using L = PmLane<K>;
    if (k == K) {
      if constexpr (DIRECT)
        if (!pieces) return rollout_pm_lanes_direct<K, L::P>(a, m, r0);
      rollout_pm_lanes<K, L::P, L::T>(a, m, r0, buf);
    } else {
      pm_item<K + 1, DIRECT>(k, pieces, a, m, r0, buf);
    }
  }
}

template <int NL>
__device__ __forceinline__ void chain_item(int links, bool staged, const RolloutArgs& a, const ChainModel& m, int r0,
                                           float* buf) {
  if constexpr (NL <= kPersistMaxLinks) {
    if (links != NL) return chain_item<NL + 1>(links, staged, a, m, r0, buf);
    const int r = r0 + (threadIdx.x & 31);
    if (staged) {
      constexpr int T = chain_chunk(NL);
      const StagedRows<NL, T> st{a.U + (size_t)r0 * a.H * NL, min(32, a.rows - r0), buf};
      rollout_chain_body<NL, kPrefetchBatch, T>(a, m, r, r < a.rows, &st);
    } else if (r < a.rows) {
      rollout_chain_body<NL, kPrefetchBatch, 0>(a, m, r, true, nullptr);
    }
  }
}

// DIRECT: some point mass's rows are not whole 16-byte pieces and are loaded
// directly.  A kernel of its own: with both forms of every point mass in it, the
// batch of 256, which has no such rows, took 1.913 ms instead of 1.899.
template <bool DIRECT>
__global__ void __launch_bounds__(kPersistThreads, 3) k_rollout_persistent(const PersistArgs p) {
  __shared__ PointMassModel models[kPersistThreads / 32];
  extern __shared__ __align__(16) unsigned char persist_smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* const buf = reinterpret_cast<float*>(persist_smem + (size_t)warp * p.warp_bytes);
  for (;;) {
    int w = 0;
    if (lane == 0) w = (int)atomicAdd(p.head, 1u);
    w = __shfl_sync(0xffffffffu, w, 0);
    if (w >= p.total_warps) break;
    w += p.w_base;
    // the instance whose warp range holds w: the last k with wstart[k] <= w
    int lo = 0, hi = p.count;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (__ldg(p.wstart + mid) <= w) lo = mid;
      else hi = mid;
    }
    const int code = __ldg(p.code + lo);
    const int model = __ldg(p.model + lo);
    const RolloutArgs a = p.ra[__ldg(p.order + lo)];
    const int r0 = (w - __ldg(p.wstart + lo)) * 32;
    const int dim = (code >> 8) & 0xff;
    if ((code & 0xff) == MTP_DYN_POINTMASS) {
      load_pm_model(models[warp], p.pm[model]);
      pm_item<1, DIRECT>(dim, (code >> 16) != 0, a, models[warp], r0, buf);
    } else {
      const ChainModel cm = p.cm[model];
      // staged only where the instance's rows allow it and the launch asks for it
      chain_item<1>(dim, p.staged && (code >> 16) != 0, a, cm, r0, buf);
    }
    __syncwarp();  // the model slot and the staging buffers are reused by the next item
  }
}

}  // namespace

template <int K>
static size_t pm_floats_of(int k) {
  if constexpr (K <= kPersistMaxAxes) return k == K ? PmLane<K>::floats : pm_floats_of<K + 1>(k);
  else return 0;
}
size_t persist_pm_floats(int axes) { return pm_floats_of<1>(axes); }

template <int NL>
static size_t chain_bytes_of(int links) {
  if constexpr (NL <= kPersistMaxLinks)
    return std::max(NL <= links ? StageShape<NL, chain_chunk(NL)>::kWarpBytes : size_t(0), chain_bytes_of<NL + 1>(links));
  else return 0;
}
size_t persist_warp_bytes(size_t pm_floats, int max_links_staged) {
  return std::max({pm_floats * sizeof(float), chain_bytes_of<1>(max_links_staged), size_t(16)});
}

template <bool DIRECT>
static int blocks_per_sm_of(size_t warp_bytes) {
  // per device and shared-memory size, computed once: a batch refilled every
  // serving cycle asks again each time
  static std::mutex mu;
  static std::map<std::pair<int, size_t>, int> cache;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  std::lock_guard<std::mutex> lock(mu);
  auto it = cache.find({dev, warp_bytes});
  if (it != cache.end()) return it->second;
  // the attribute is the ceiling of every launch's shared memory: the
  // largest tile any batch can have
  const int warps = kPersistThreads / 32;
  const size_t ceiling = persist_warp_bytes(kPmLaneFloats, kPersistMaxLinks) * warps;
  if (cudaFuncSetAttribute(k_rollout_persistent<DIRECT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ceiling) !=
      cudaSuccess)
    return 0;
  int blocks = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k_rollout_persistent<DIRECT>, kPersistThreads,
                                                    warp_bytes * warps) != cudaSuccess)
    return 0;
  cache[{dev, warp_bytes}] = blocks;
  return blocks;
}
int persist_blocks_per_sm(size_t warp_bytes, bool pm_direct) {
  return pm_direct ? blocks_per_sm_of<true>(warp_bytes) : blocks_per_sm_of<false>(warp_bytes);
}

cudaError_t launch_rollout_persistent(const PersistArgs& p, int blocks_per_sm, cudaStream_t s) {
  if (p.total_warps <= 0) return cudaSuccess;
  const int warps_per_block = kPersistThreads / 32;
  const int grid = std::max(1, std::min(blocks_per_sm * device_sms(),
                                        (p.total_warps + warps_per_block - 1) / warps_per_block));
  cudaError_t e = cudaMemsetAsync(p.head, 0, sizeof(unsigned), s);
  if (e != cudaSuccess) return e;
  const size_t smem = p.warp_bytes * warps_per_block;
  if (p.pm_direct) k_rollout_persistent<true><<<grid, kPersistThreads, smem, s>>>(p);
  else k_rollout_persistent<false><<<grid, kPersistThreads, smem, s>>>(p);
  return cudaGetLastError();
}

}  // namespace mtp
