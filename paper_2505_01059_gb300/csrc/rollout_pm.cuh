// rollout_pm.cuh -- Alg. 2 batch rollout fused with the cost reduction (Eq. 2)
// for the k-D point mass: device bodies and kernels, instantiated by
// rollout_pm.cu, rollout_pm_batch.cu and rollout_persist.cu.
//
// The double integrator's recursion is two fused multiply-adds per axis and
// step; nearly all of a step's work is its cost (the distances to the goal and
// to every obstacle), which nothing of a later step waits for.  The bodies use
// the same operations in the same order for every value, so a cost does not
// depend on which one ran (pm_body says which one a lone instance takes, and why).
//
// Many candidates (rollout_pm_lanes: batches, large lone instances): a lane walks
// its candidate's horizon, P steps' costs in flight.  Bound by the issue slots of
// the distances; one step at a time left fixed latencies in the open (the batch of
// 256: 2.68 -> 2.43 ms per iteration).
//
// Short horizons, and rows that cannot be staged (rollout_pm_direct): the same a
// step at a time, with nothing through shared memory and the model as constant
// operands.
//
// Few candidates (rollout_pm_tile: lone instances): a warp takes C candidates
// T steps at a time, and its lanes share each of three passes over the chunk:
//   1. the C K axes' recursions, one per lane: the control of (candidate, step,
//      axis) in shared memory is replaced by the position before that step;
//   2. the C T stage costs, one (candidate, step) per lane, P in flight;
//   3. the C compensated sums over the chunk's costs in step order, one per lane.
// Its passes go through shared memory and leave lanes idle in the third, so it
// issues about twice the instructions of the first body, but on many more warps.
// Bound, for small problems, by the latency of passes 1 and 3 (about 8 and 20
// cycles a step): the 2-axis problem of 512 candidates and 64 steps went from 21
// to about 5 us, 12 axes, 8192 candidates and 256 steps from 227 to 49 us.
#pragma once

#include <algorithm>

#include "rollout_common.cuh"

namespace mtp {
namespace {

constexpr int kPmThreads = 128;  // at most four warps per block
constexpr int kMaxPmAxes = 16;
constexpr int kPmSmemMax = 68 * 1024;  // dynamic shared memory of a block, at most

// Copies an instance's model to this warp's slot in shared memory.
__device__ __forceinline__ void load_pm_model(PointMassModel& m, const PointMassModel& src) {
  const int* s = reinterpret_cast<const int*>(&src);
  int* d = reinterpret_cast<int*>(&m);
  for (int w = threadIdx.x & 31; w < (int)(sizeof(PointMassModel) / sizeof(int)); w += 32) d[w] = s[w];
  __syncwarp();
}

// K consecutive floats at a 16-byte aligned address.
template <int K>
__device__ __forceinline__ void load_axes(const float* p, float (&v)[K]) {
#pragma unroll
  for (int k = 0; k + 3 < K; k += 4) {
    const float4 x = *reinterpret_cast<const float4*>(p + k);
    v[k] = x.x;
    v[k + 1] = x.y;
    v[k + 2] = x.z;
    v[k + 3] = x.w;
  }
#pragma unroll
  for (int k = K / 4 * 4; k < K; ++k) v[k] = p[k];
}

// State costs (Eq. 2 without the control term) of P positions, interleaved so
// that their latencies overlap.  An obstacle's distance is d2 * rsqrt(d2)
// (relative error ~1e-7), the argument kept normal: at d2 = 0 that is 0.
template <int K, int P>
__device__ __forceinline__ void pm_state_costs(const PointMassModel& pm, const float (&p)[P][K], float (&out)[P]) {
  float dist2[P], pen[P], c[K];
#pragma unroll
  for (int j = 0; j < P; ++j) dist2[j] = pen[j] = 0.f;
  load_axes<K>(pm.target, c);
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int j = 0; j < P; ++j) {
      const float e = p[j][k] - c[k];
      dist2[j] = fmaf(e, e, dist2[j]);
    }
  // obstacles in flight (slots past n_obs have radius 0 and add exactly +0)
  constexpr int kSlots = P == 1 ? (K <= 4 ? 4 : 2) : 1;
  const int n_obs = pm.n_obs;
#pragma unroll 1
  for (int o = 0; o < n_obs; o += kSlots) {
    float d2[kSlots][P];
#pragma unroll
    for (int z = 0; z < kSlots; ++z) {
      load_axes<K>(pm.obs_c[o + z], c);
#pragma unroll
      for (int j = 0; j < P; ++j) d2[z][j] = 0.f;
#pragma unroll
      for (int k = 0; k < K; ++k)
#pragma unroll
        for (int j = 0; j < P; ++j) {
          const float e = p[j][k] - c[k];
          d2[z][j] = fmaf(e, e, d2[z][j]);
        }
    }
#pragma unroll
    for (int z = 0; z < kSlots; ++z) {
      const float r = pm.obs_r[o + z];
#pragma unroll
      for (int j = 0; j < P; ++j) {
        const float dist = __fmul_rn(d2[z][j], rsqrt_normal(fmaxf(d2[z][j], kMinNormal)));
        pen[j] += fmaxf(r - dist, 0.f);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < P; ++j) out[j] = fmaf(pm.w_target, dist2[j], pm.w_obs * pen[j]);
}

// Controls (or positions) of one step, or of several, from shared memory at
// an address aligned to 16 bytes where N is a multiple of 4, to 8 where it is even.
template <int N>
__device__ __forceinline__ void load_steps(const float* p, float (&u)[N]) {
  if constexpr (N % 4 == 0) {
    load_axes<N>(p, u);
  } else if constexpr (N % 2 == 0) {
#pragma unroll
    for (int k = 0; k < N; k += 2) {
      const float2 x = *reinterpret_cast<const float2*>(p + k);
      u[k] = x.x;
      u[k + 1] = x.y;
    }
  } else {
#pragma unroll
    for (int k = 0; k < N; ++k) u[k] = p[k];
  }
}

// copy_controls into rows whose steps are KS floats apart (a 16-byte piece lies
// inside one step where KS is not K).
template <int K, int KS>
__device__ __forceinline__ void copy_steps(const float* src, int H, int n, int steps, bool vec, float* dst, int row) {
  if constexpr (KS == K) {
    copy_controls<K>(src, H, n, steps, vec, dst, row);
  } else {
    const int lane = threadIdx.x & 31;
    const int len = vec ? steps * K / 4 : steps * K;  // pieces per candidate
    int i = lane / len, o = lane - i * len;
    const int di = 32 / len, dlen = 32 - di * len;
    while (i < n) {
      const int f = vec ? 4 * o : o;
      const int at = f / K * KS + f % K;
      if (vec) copy_async_16(dst + i * row + at, src + (size_t)i * H * K + f);
      else copy_async_f32(dst + i * row + at, src + (size_t)i * H * K + f);
      i += di;
      o += dlen;
      if (o >= len) {
        o -= len;
        ++i;
      }
    }
    copy_async_commit();
  }
}

// Whether an instance's control rows can be copied in 16-byte pieces.
__device__ __forceinline__ bool vector_rows(const RolloutArgs& a, int K) {
  return (((uintptr_t)a.U & 15) == 0) && (((long long)a.H * K) & 3) == 0;
}

// ---------------------------------------------------------------------------
// A lane per candidate.
// ---------------------------------------------------------------------------

// Floats of a candidate's row of two chunks of T steps: 16-byte pieces, an odd
// number, so that the lanes' rows start on different banks.
__host__ __device__ constexpr int pm_lane_row(int K, int T) {
  const int quads = (2 * T * K + 3) / 4;
  return 4 * (quads % 2 ? quads : quads + 1);
}

// Candidates r0 .. r0 + 31 (those below a.rows) of one instance by one warp;
// every lane calls it.  pm: in shared memory; sm: 32 rows of pm_lane_row(K, T)
// floats, 16-byte aligned; T: a multiple of P and of 4 (a chunk of a 16-byte
// aligned row of H K floats, a multiple of 4, is then whole 16-byte pieces).
template <int K, int P, int T>
__device__ __forceinline__ void rollout_pm_lanes(const RolloutArgs& a, const PointMassModel& pm, int r0, float* sm) {
  static_assert(T % P == 0 && T % 4 == 0, "whole turns and pieces");
  constexpr int row = pm_lane_row(K, T);
  const int lane = threadIdx.x & 31;
  const int n = min(32, a.rows - r0);  // the other lanes compute on what shared memory holds, and store nothing
  const int r = r0 + lane;
  const int H = a.H;
  const uint32_t iter = a.d_iter ? *a.d_iter : a.iter;
  const float* const U = a.U + (size_t)r0 * H * K;
  const bool vec = vector_rows(a, K);
  const int models = (a.dr_mode == MTP_DR_SHARED) ? a.R : 1;
  const float dt = a.dt;
  const float w_ctrl = pm.w_ctrl;
  auto request = [&](int t0) {
    if (t0 < H) copy_controls<K>(U + (size_t)t0 * K, H, n, min(T, H - t0), vec, sm + (t0 / T & 1) * T * K, row);
  };
  float total = 0.f;
  for (int mdl = 0; mdl < models; ++mdl) {
    request(0);
    float gain[K], v[K], x[K];
    dr_scales<K>(a, iter, (a.dr_mode == MTP_DR_SHARED) ? (uint32_t)mdl : (uint32_t)(a.row0 + r), gain);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      gain[k] *= dt;
      x[k] = a.x0[k];
      v[k] = a.x0[K + k];
    }
    KahanSum J;
    // step H stands for the terminal cost
    for (int t0 = 0; t0 <= H; t0 += T) {
      copy_async_wait_all();
      __syncwarp();  // this chunk is there, and the other one has been used
      request(t0 + T);
      const float* u_row = sm + lane * row + (t0 / T & 1) * T * K;
      for (int t = t0; t < t0 + T && t <= H; t += P, u_row += P * K) {
        float p[P][K], uu[P], u[P * K];
        load_steps<P * K>(u_row, u);
#pragma unroll
        for (int q = 0; q < P; ++q) {
          uu[q] = 0.f;
#pragma unroll
          for (int k = 0; k < K; ++k) {
            p[q][k] = x[k];
            uu[q] = fmaf(u[q * K + k], u[q * K + k], uu[q]);
            v[k] = fmaf(gain[k], u[q * K + k], v[k]);
            x[k] = fmaf(dt, v[k], x[k]);
          }
        }
        float state[P];
        pm_state_costs<K, P>(pm, p, state);
        if (t + P <= H) {
          if (a.kahan) {
#pragma unroll
            for (int q = 0; q < P; ++q) J.add(fmaf(w_ctrl, uu[q], state[q]), true);
          } else {
#pragma unroll
            for (int q = 0; q < P; ++q) J.add(fmaf(w_ctrl, uu[q], state[q]), false);
          }
        } else {
#pragma unroll
          for (int q = 0; q < P; ++q)
            if (t + q <= H)
              J.add(t + q < H ? fmaf(w_ctrl, uu[q], state[q]) : __fmul_rn(pm.w_term, state[q]), a.kahan);
        }
      }
    }
    total += J.s;
    __syncwarp();  // the next model's controls overwrite the rows
  }
  if (lane < n) {
    float cost = total / (float)models;
    if (!isfinite(cost)) cost = __int_as_float(0x7f800000);
    a.cost[r] = cost;
  }
}

// The same for rows that cannot be staged in 16-byte pieces: each lane loads its
// own row, the next P steps while the current ones' costs are evaluated.  (Copied
// into shared memory by single floats, such rows took 1.2 to 1.7 times as long as
// with the direct loads one step ahead that came before: a persistent launch of 600
// candidates of 7 axes and 101 steps 57 us, 38 so.)
template <int K, int P>
__device__ __forceinline__ void rollout_pm_lanes_direct(const RolloutArgs& a, const PointMassModel& pm, int r0) {
  const int r = r0 + (int)(threadIdx.x & 31);
  const int H = a.H;
  const uint32_t iter = a.d_iter ? *a.d_iter : a.iter;
  const float* const row = a.U + (size_t)min(r, a.rows - 1) * H * K;
  const int models = (a.dr_mode == MTP_DR_SHARED) ? a.R : 1;
  const float dt = a.dt;
  const float w_ctrl = pm.w_ctrl;
  float total = 0.f;
  for (int mdl = 0; mdl < models; ++mdl) {
    float gain[K], v[K], x[K], u[P * K];
    dr_scales<K>(a, iter, (a.dr_mode == MTP_DR_SHARED) ? (uint32_t)mdl : (uint32_t)(a.row0 + r), gain);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      gain[k] *= dt;
      x[k] = a.x0[k];
      v[k] = a.x0[K + k];
    }
    auto load = [&](int t) {
#pragma unroll
      for (int q = 0; q < P; ++q) {
        const float* const s = row + min(t + q, H - 1) * K;
#pragma unroll
        for (int k = 0; k < K; ++k) u[q * K + k] = __ldg(s + k);
      }
    };
    load(0);
    KahanSum J;
    // step H stands for the terminal cost
    for (int t = 0; t <= H; t += P) {
      float p[P][K], uu[P], state[P];
#pragma unroll
      for (int q = 0; q < P; ++q) {
        uu[q] = 0.f;
#pragma unroll
        for (int k = 0; k < K; ++k) {
          p[q][k] = x[k];
          uu[q] = fmaf(u[q * K + k], u[q * K + k], uu[q]);
          v[k] = fmaf(gain[k], u[q * K + k], v[k]);
          x[k] = fmaf(dt, v[k], x[k]);
        }
      }
      if (t + P < H) load(t + P);
      pm_state_costs<K, P>(pm, p, state);
      if (t + P <= H) {
#pragma unroll
        for (int q = 0; q < P; ++q) J.add(fmaf(w_ctrl, uu[q], state[q]), a.kahan);
      } else {
#pragma unroll
        for (int q = 0; q < P; ++q)
          if (t + q <= H)
            J.add(t + q < H ? fmaf(w_ctrl, uu[q], state[q]) : __fmul_rn(pm.w_term, state[q]), a.kahan);
      }
    }
    total += J.s;
  }
  if (r < a.rows) {
    float cost = total / (float)models;
    if (!isfinite(cost)) cost = __int_as_float(0x7f800000);
    a.cost[r] = cost;
  }
}

// The lane body's steps in flight and chunk length: more steps where a position
// takes few registers, and as long a chunk as kPmLaneFloats hold.
constexpr int kPmLaneFloats = 4352;
template <int K>
struct PmLane {
  static constexpr int P = K <= 4 ? 4 : 2;
  static constexpr int T = 32 * pm_lane_row(K, 16) <= kPmLaneFloats ? 16 : 32 * pm_lane_row(K, 8) <= kPmLaneFloats ? 8 : 4;
  static constexpr int floats = 32 * pm_lane_row(K, T);
  static_assert(floats <= kPmLaneFloats, "a warp's rows fit");
};

// Many instances: their rows are padded to multiples of 32 (row_start), so a
// warp's candidates belong to one instance.  STAGED: all of them have vector_rows.
template <int K, bool STAGED>
__global__ void __launch_bounds__(kPmThreads) k_rollout_pm_batch(const RolloutArgs* __restrict__ ra,
                                                                 const PointMassModel* __restrict__ pm,
                                                                 const int* __restrict__ row_start, int count) {
  extern __shared__ __align__(16) float pm_smem[];
  __shared__ PointMassModel models[kPmThreads / 32];
  const int warp = threadIdx.x >> 5;
  const int g = (blockIdx.x * blockDim.x + threadIdx.x) & ~31;
  if (g >= __ldg(row_start + count)) return;
  const int i = batch_instance(row_start, count, g);
  load_pm_model(models[warp], pm[i]);
  const RolloutArgs a = ra[i];
  using L = PmLane<K>;
  const int r0 = g - __ldg(row_start + i);
  if constexpr (STAGED) rollout_pm_lanes<K, L::P, L::T>(a, models[warp], r0, pm_smem + warp * L::floats);
  else rollout_pm_lanes_direct<K, L::P>(a, models[warp], r0);
}

// ---------------------------------------------------------------------------
// A warp per tile of candidates.
// ---------------------------------------------------------------------------

// Floats between a tile's steps: the axes, padded where their count would put
// the steps of pass 2's lanes on the same banks.
constexpr int pm_tile_step(int K) { return K % 8 == 0 ? K + 4 : K; }

// Floats between a tile's candidates: the shortest 16-byte row of T steps on which
// the fewest lanes of pass 1, q on candidate q / K and axis q % K, share a bank.
constexpr int pm_tile_conflicts(int K, int row) {
  int hits[32] = {}, most = 0;
  for (int q = 0; q < 32; ++q) most = std::max(most, ++hits[(q / K * row + q % K) % 32]);
  return most;
}
constexpr int pm_tile_row(int K, int T) {
  const int least = (T * pm_tile_step(K) + 3) / 4 * 4;
  int best = least, fewest = pm_tile_conflicts(K, least);
  for (int y = least + 4; y < least + 32; y += 4) {
    const int conflicts = pm_tile_conflicts(K, y);
    if (conflicts < fewest) {
      best = y;
      fewest = conflicts;
    }
  }
  return best;
}

// Shared-memory layout of a tile of T = 4 << i steps, i = 0 .. 4.  The rows are
// found by the compiler: searched at every launch they took 20 to 60 us of the
// host, more than the launch and a small rollout themselves (4 axes, 1384
// candidates of 44 steps, called one after another: 20.3 us, now 9.7).
template <int K>
struct PmTileShape {
  static constexpr int kStep = pm_tile_step(K);
  static constexpr int kLengths = 5;
  static constexpr int kRow[kLengths] = {pm_tile_row(K, 4), pm_tile_row(K, 8), pm_tile_row(K, 16), pm_tile_row(K, 32),
                                         pm_tile_row(K, 64)};
  // two buffers of controls, velocity, position and gain of every axis, costs
  static constexpr int floats(int C, int i) { return (C * (2 * kRow[i] + 3 * K + (4 << i) + 1) + 3) / 4 * 4; }
};

// A warp's tile: C candidates, T steps, its row and floats of shared memory; and
// the threads per block.  About six warps per SM or more before a warp takes a
// second candidate; up to eight candidates per warp, two beyond 8 axes, whose rows
// fill the shared memory first.  T up to 64 steps, as far as a tile takes 16 KB.
// Measured (us a call, replayed from a graph; C and T swept over 1 .. 32 and
// 8 .. 128): 2 axes, B 512, H 64: C 1 / 2 / 8 at T 64: 5.4 / 5.6 / 7.9 (21 as one
// candidate per lane); 2 axes, B 8192, H 128: C 1 / 2 / 4 / 8: 29 / 19 / 14 / 14;
// 12 axes, B 8192, H 256: C 1 / 2 / 4 / 8: 63 / 49 / 56 / 55 (227 as one candidate
// per lane); 16 axes, B 8192, H 128: C 2, T 32 / 64: 34 / 47.
constexpr int pm_tile_most(int K) { return K > 8 ? 2 : 8; }
constexpr int kPmTileFloats = 4096;
struct PmTile {
  int C, T, row, floats, block;
};
template <int K>
PmTile pm_tile(long long rows) {
  using Shape = PmTileShape<K>;
  int C = pm_tile_most(K), i = Shape::kLengths - 1, block = 128;
  const long long want = (long long)device_sms() * 6;
  while (C > 1 && rows / C < want) C >>= 1;
  while (i > 0 && Shape::floats(C, i) > kPmTileFloats) --i;
  while (block > 32 && rows / C * 32 < (long long)block * device_sms()) block >>= 1;
  return {C, 4 << i, Shape::kRow[i], Shape::floats(C, i), block};
}

// Candidates r0 .. r0 + C - 1 (those below a.rows) of one instance by one warp;
// every lane calls it.  pm: in shared memory; sm: this warp's
// PmTileShape<K>::floats of C and T, 16-byte aligned; row: its kRow; C <= 32, T a
// multiple of 4.
// STATES: also writes the states of the one candidate asked for to a.X.
template <int K, bool STATES>
__device__ __forceinline__ void rollout_pm_tile(const RolloutArgs& a, const PointMassModel& pm, int r0, int C, int T,
                                                int row, float* sm) {
  constexpr int KS = PmTileShape<K>::kStep;
  constexpr int P = K <= 4 ? 4 : 2;  // costs in flight per lane
  const int lane = threadIdx.x & 31;
  const int n = min(C, a.rows - r0);  // this tile's candidates
  const int H = a.H;
  const uint32_t iter = a.d_iter ? *a.d_iter : a.iter;
  const float* const U = a.U + (size_t)r0 * H * K;
  const bool vec = vector_rows(a, K);
  const int models = (a.dr_mode == MTP_DR_SHARED) ? a.R : 1;
  const float dt = a.dt;
  const float w_ctrl = pm.w_ctrl;
  float* const V = sm + 2 * C * row;
  float* const X = V + C * K;
  float* const G = X + C * K;
  float* const cst = G + C * K;
  const int ld = T + 1;  // odd: pass 3's lanes read distinct banks
  auto request = [&](int t0, int buf) {
    copy_steps<K, KS>(U + (size_t)t0 * K, H, n, min(T, H - t0), vec, sm + buf * C * row, row);
  };
  float total = 0.f;
  for (int mdl = 0; mdl < models; ++mdl) {
    request(0, 0);
    for (int q = lane; q < n * K; q += 32) {
      const int c = q / K, k = q - c * K;
      float gain = 1.f;
      if (a.dr_mode != MTP_DR_NONE) {
        const bool shared = a.dr_mode == MTP_DR_SHARED;
        const uint32_t w = draw(a.key, shared ? (uint32_t)mdl : (uint32_t)(a.row0 + r0 + c), (uint32_t)k, iter,
                                shared ? kTagParamModel : kTagParamSample);
        gain = fmaf(a.dr_hi - a.dr_lo, unit24(w), a.dr_lo);
      }
      G[q] = gain * dt;
      X[q] = a.x0[k];
      V[q] = a.x0[K + k];
      if (STATES) {
        a.X[k] = a.x0[k];
        a.X[K + k] = a.x0[K + k];
      }
    }
    KahanSum J;
    for (int t0 = 0, buf = 0; t0 < H; t0 += T, buf ^= 1) {
      float* const tile = sm + buf * C * row;
      const int steps = min(T, H - t0);
      copy_async_wait_all();
      __syncwarp();  // this chunk is there, and the other buffer's has been used
      if (t0 + T < H) request(t0 + T, buf ^ 1);
      // the lanes' (candidate, step) pairs, 32 further along at every turn
      const int pairs = n * steps;
      const int c_first = lane / steps, t_first = lane - c_first * steps;
      const int dc = 32 / steps, ds = 32 - dc * steps;
      auto next = [&](int& c, int& t) {
        c += dc;
        t += ds;
        if (t >= steps) {
          t -= steps;
          ++c;
        }
      };
      // |u|^2 of the chunk's controls, which the positions then replace
      {
        int c = c_first, t = t_first;
        for (int e = lane; e < pairs; e += 32) {
          float u[K], uu = 0.f;
          load_steps<K>(tile + c * row + t * KS, u);
#pragma unroll
          for (int k = 0; k < K; ++k) uu = fmaf(u[k], u[k], uu);
          cst[c * ld + t] = uu;
          next(c, t);
        }
      }
      __syncwarp();
      for (int q = lane; q < n * K; q += 32) {
        const int c = q / K, k = q - c * K;
        float* s = tile + c * row + k;
        const float g = G[q];
        float v = V[q], x = X[q];
#pragma unroll 8
        for (int t = 0; t < steps; ++t) {
          const float u = s[t * KS];
          s[t * KS] = x;
          v = fmaf(g, u, v);
          x = fmaf(dt, v, x);
          if (STATES) {
            float* xo = a.X + (size_t)(t0 + t + 1) * 2 * K;
            xo[k] = x;
            xo[K + k] = v;
          }
        }
        V[q] = v;
        X[q] = x;
      }
      __syncwarp();
      {
        int c = c_first, t = t_first;
        int e = lane;
        auto stage = [&](auto PP) {
          constexpr int p_n = decltype(PP)::value;
          float p[p_n][K], state[p_n];
          int slot[p_n];
#pragma unroll
          for (int j = 0; j < p_n; ++j) {
            slot[j] = c * ld + t;
            load_steps<K>(tile + c * row + t * KS, p[j]);
            next(c, t);
          }
          pm_state_costs<K, p_n>(pm, p, state);
#pragma unroll
          for (int j = 0; j < p_n; ++j) cst[slot[j]] = fmaf(w_ctrl, cst[slot[j]], state[j]);
        };
        for (; e - lane + 32 * P <= pairs; e += 32 * P) stage(IC<P>{});
        for (; e < pairs; e += 32) stage(IC<1>{});
      }
      __syncwarp();
      if (lane < n) {
        const float* s = cst + lane * ld;
        if (a.kahan) {
#pragma unroll 4
          for (int t = 0; t < steps; ++t) J.add(s[t], true);
        } else {
#pragma unroll 4
          for (int t = 0; t < steps; ++t) J.add(s[t], false);
        }
      }
    }
    if (lane < n) {
      float p[1][K], state[1];
#pragma unroll
      for (int k = 0; k < K; ++k) p[0][k] = X[lane * K + k];
      pm_state_costs<K, 1>(pm, p, state);
      J.add(__fmul_rn(pm.w_term, state[0]), a.kahan);
      total += J.s;
    }
    __syncwarp();  // the next model rewrites the tile
  }
  if (lane < n) {
    float cost = total / (float)models;
    if (!isfinite(cost)) cost = __int_as_float(0x7f800000);
    a.cost[r0 + lane] = cost;
  }
}

// One instance: warp w of the launch takes candidates w C .. w C + C - 1.
template <int K, bool STATES>
__global__ void __launch_bounds__(kPmThreads) k_rollout_pm(const __grid_constant__ RolloutArgs a,
                                                           const __grid_constant__ PointMassModel pm, int C, int T,
                                                           int row, int warp_floats) {
  extern __shared__ __align__(16) float pm_smem[];
  __shared__ PointMassModel models[kPmThreads / 32];
  const int warp = threadIdx.x >> 5;
  const int r0 = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * C;
  if (r0 >= a.rows) return;
  load_pm_model(models[warp], pm);
  rollout_pm_tile<K, STATES>(a, models[warp], r0, C, T, row, pm_smem + warp * warp_floats);
}

// The same, a lane per candidate (rows of whole 16-byte pieces).
template <int K>
__global__ void __launch_bounds__(kPmThreads) k_rollout_pm_lanes(const __grid_constant__ RolloutArgs a,
                                                                 const __grid_constant__ PointMassModel pm) {
  extern __shared__ __align__(16) float pm_smem[];
  __shared__ PointMassModel models[kPmThreads / 32];
  const int warp = threadIdx.x >> 5;
  const int r0 = (int)(blockIdx.x * blockDim.x + threadIdx.x) & ~31;
  if (r0 >= a.rows) return;
  load_pm_model(models[warp], pm);
  using L = PmLane<K>;
  rollout_pm_lanes<K, L::P, L::T>(a, models[warp], r0, pm_smem + warp * L::floats);
}

// The same, a candidate per thread, one step at a time.  Every obstacle slot is
// evaluated, with no branch: one basic block, so the obstacles' SFU latencies
// overlap, and every model index is a constant (those past n_obs have radius 0 and
// add exactly +0).  (Its parameters are not __grid_constant__: that form took up to
// 20 % longer, 8 axes above all.)
template <int K>
__global__ void __launch_bounds__(kPmThreads) k_rollout_pm_direct(const RolloutArgs a, const PointMassModel pm) {
  const int r = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (r >= a.rows) return;
  const uint32_t iter = a.d_iter ? *a.d_iter : a.iter;
  const int models = (a.dr_mode == MTP_DR_SHARED) ? a.R : 1;
  const float dt = a.dt;
  auto state_cost = [&](const float (&p)[K]) {
    float dist2 = 0.f, pen = 0.f;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const float e = p[k] - pm.target[k];
      dist2 = fmaf(e, e, dist2);
    }
#pragma unroll
    for (int o = 0; o < MTP_MAX_OBSTACLES; ++o) {
      float d2 = 0.f;
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const float e = p[k] - pm.obs_c[o][k];
        d2 = fmaf(e, e, d2);
      }
      pen += fmaxf(pm.obs_r[o] - __fmul_rn(d2, rsqrt_normal(fmaxf(d2, kMinNormal))), 0.f);
    }
    return fmaf(pm.w_target, dist2, pm.w_obs * pen);
  };
  float total = 0.f;
  for (int mdl = 0; mdl < models; ++mdl) {
    float gain[K], x[K], v[K];
    dr_scales<K>(a, iter, (a.dr_mode == MTP_DR_SHARED) ? (uint32_t)mdl : (uint32_t)(a.row0 + r), gain);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      gain[k] *= dt;
      x[k] = a.x0[k];
      v[k] = a.x0[K + k];
    }
    KahanSum J;
    for_each_step<K, kPrefetchAlone, 0>(a.U + (size_t)r * a.H * K, a.H, nullptr, [&](int, const float (&u)[K]) {
      float uu = 0.f;
#pragma unroll
      for (int k = 0; k < K; ++k) uu = fmaf(u[k], u[k], uu);
      J.add(fmaf(pm.w_ctrl, uu, state_cost(x)), a.kahan);
#pragma unroll
      for (int k = 0; k < K; ++k) {
        v[k] = fmaf(gain[k], u[k], v[k]);
        x[k] = fmaf(dt, v[k], x[k]);
      }
    });
    J.add(__fmul_rn(pm.w_term, state_cost(x)), a.kahan);
    total += J.s;
  }
  float cost = total / (float)models;
  if (!isfinite(cost)) cost = __int_as_float(0x7f800000);
  a.cost[r] = cost;
}

// Which body a lone instance's costs take.  A tile evaluates more than a lane of
// its own does and pays for its passes in barriers; what it gains is warps, and
// loads that are coalesced and ahead of their use.  So: not for horizons of a few
// steps, and while the tiles are resident at once, in `wave`, or in up to four times
// as many where a lane's direct loads are at their worst (rows whole cache lines
// apart, whose lines fall on the same few sets of the L1, and 12 or 16 axes).  Past
// that many candidates the lanes' own form, staged if the rows can be.  The lines
// were drawn through 3646 sizes (1 to 16 axes, 500 to 300000 candidates, 8 to 256
// steps), where this choice is within 5 % of the faster of the tile and the direct
// form or better, but for a few; us tile / lanes / direct: 7 axes of 33 steps, 4096
// candidates 8.5 / - / 18.2, 30000 candidates 34.5 / - / 20.5; 12 axes of 64 steps,
// 4096 candidates 11.9 / 30.5 / 41.7, 32768 candidates 58.9 / 38.6 / 102.9; 2 axes of
// 9 steps, 8192 candidates 5.7 / - / 4.4.
enum class PmBody { kTile, kLanes, kDirect };

// Candidates whose full tiles an SM holds at once: blocks of four warps.
template <int K>
constexpr int pm_wave_rows() {
  using Shape = PmTileShape<K>;
  const int C = pm_tile_most(K);
  int i = Shape::kLengths - 1;
  while (i > 0 && Shape::floats(C, i) > kPmTileFloats) --i;
  const int bytes = 4 * (Shape::floats(C, i) * (int)sizeof(float) + (int)sizeof(PointMassModel)) + 1024;
  return std::min(16, 228 * 1024 / bytes) * 4 * C;
}

template <int K>
PmBody pm_body(long long rows, int H, bool pieces) {
  const PmBody many = pieces && H >= (K % 4 == 0 ? 20 : 32) && rows >= 118LL * device_sms() ? PmBody::kLanes : PmBody::kDirect;
  if (H < (K > 4 ? 12 : 16)) return many;
  // percent of a wave up to which the tile is taken
  const bool worst = (K > 8 && K % 4 == 0) || (long long)H * K % 32 == 0;
  int most;
  if (H < 32) most = K > 8 && K % 4 == 0 && H >= 20 ? 170 : 90 * H / 32;
  else if (worst && (K > 4 || H >= 48)) most = 400;
  else if (H >= 200) most = 300;
  else if (pieces && H >= 48) most = 200;
  else if (H >= 96) most = 140;
  else most = 100;
  if (K == 1) most = std::min(most, H < 48 ? 50 : 100);
  return 100 * rows <= (long long)most * pm_wave_rows<K>() * device_sms() ? PmBody::kTile : many;
}

}  // namespace
}  // namespace mtp
