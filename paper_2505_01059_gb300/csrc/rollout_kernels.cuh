// rollout_kernels.cuh -- Alg. 2 batch rollout fused with the cost reduction
// (Eq. 2) for the planar serial chain: the device body and kernels,
// instantiated by rollout_chain.cu, rollout_chain_batch.cu and
// rollout_persist.cu.
//
// One thread per candidate keeps the whole state in registers for all H
// steps and accumulates c(x_t, u_t) with compensated FP32 sums; only the
// final cost leaves the SM.  The loop bodies are fully unrolled over the
// compile-time link count, so the per-step linear algebra lives in registers.
// The controls reach a thread either by direct loads a few steps ahead (T = 0)
// or staged through shared memory a horizon chunk of T steps at a time (see
// StagedRows), picked per launch shape by the batch autotuner.
//
// Planar chain: the dynamics are evaluated in absolute link angles phi_j
// (phi_j = q_1 + ... + q_j).  For uniform thin rods the Lagrangian gives the
// mass matrix A_jk = D_jk cos(phi_j - phi_k) with constant D (from the link
// masses and lengths), velocity terms D_jk sin(phi_j - phi_k) w_k^2, gravity
// g l_j beta_j cos(phi_j) and generalised forces tau_j - tau_{j+1}; the
// SPD system is solved by an unrolled Cholesky.  Semi-implicit Euler in
// (phi, w) equals semi-implicit Euler in the relative joint coordinates.
#pragma once

#include "rollout_common.cuh"

namespace mtp {
namespace {

constexpr int kThreads = 128;
// Chains of at least this many links solve their mass matrix by the O(NL)
// semiseparable Cholesky, shorter ones by the dense factor.  At 7 links the
// dense factor is the faster of the two: as fast in a batch, and 99 -> 79 us
// for a lone 4096-candidate arm, whose one warp per SM sub-partition runs
// the step's serial chain (the recursion's is longer).
#ifndef MTP_SEMISEP_LINKS
#define MTP_SEMISEP_LINKS 8
#endif
constexpr int kSemisepLinks = MTP_SEMISEP_LINKS;

// Whether a chain of NL links takes its angles' whole turns by rintf (the same
// value).  The shorter way off the SFU is the faster one for most link counts (lone:
// 3 links 24.4 against 25.5 us, 9 links 85.5 / 87.1, 12 links 98.4 / 101.8, 128
// steps) but not where the step is one short chain of instructions (batches of one
// link, 101 steps: 22.7 against 13.1 us) and not for five links alone, 128 steps of
// which took 46.2 against 36.4 us (in batches 44 / 45).  Nor in direct rollouts of
// so many lone candidates that the issue slots bound them (turns_by_sfu): 40000 of
// 36 steps, off the SFU over on it, 2 1.02, 6 1.02, 9 1.02, 10 1.02, 12 1.04, 4, 7, 8
// and 11 links 1.00 to 1.01; 16384 of 36: 0.96 to 1.00.
template <int NL, int PF>
constexpr bool kSfuTurns = NL == 1 || (NL == 5 && PF == kPrefetchAlone);
inline bool turns_by_sfu(int rows) { return rows > 192 * device_sms(); }

// Direct loads two steps ahead, or staged ones?  Alone a warp waits for its longest
// chain of instructions either way, and which form's code is the shorter one differs
// by link count; the direct loads get worse where the rows are whole cache lines
// apart, whose lines fall on the same few sets of the L1, the more so the more warps
// share an SM.  Staged over direct time, 32 to 256 steps, by link count:
//   rows of whole lines, up to 8192 candidates: 1 0.97, 2 0.87, 3 0.77, 4 1.09, 5
//   1.16, 6 0.93, 7 1.09, 8 0.77, 9 1.02, 10 0.82, 11 0.89, 12 0.90; 16384 and 40000:
//   0.5 to 0.9 for all;
//   other rows, up to 8192 candidates: 2 0.98, 3 0.83, 4 1.12, 5 1.22, 6 0.98, 7
//   1.11, 9 1.13, 10 0.92, 11 1.02, 12 0.97; 40000: 0.9 to 1.09, and shared models
//   of one link 1.09 on any rows.
// Shared models walk the same rows again, which direct loads then find in the L1.
// Staged over direct time with four of them, other rows, 24 to 100 steps: 32 to 8192
// candidates, 2 links 0.99 to 1.02, 3 0.94 to 1.00, 6 1.03 to 1.06, 8 0.94 to 1.01, 10
// 0.98 to 1.07, 12 1.04 to 1.11; 16384: 2 1.02, 3 0.97, 6 1.06, 10 0.96, 12 0.89.
inline bool stages_alone(int links, int H, int rows, bool shared = false) {
  const bool lines = (long long)H * links % 32 == 0;
  if (links == 1 || links == 4 || links == 5 || links == 7 || links == 9) return lines && rows > 96 * device_sms();
  if (lines || links == 11 || rows > 192 * device_sms()) return lines;
  return !shared || links == 3 || links == 8 || (links >= 10 && rows > 96 * device_sms());
}

// Dynamic shared memory of a rollout block of `block` threads staging K
// controls per step T steps at a time (0 for direct loads).
template <int K, int T>
constexpr size_t staged_smem(int block) {
  if constexpr (T == 0) return 0;
  else return (size_t)(block / 32) * StageShape<K, T>::kWarpBytes;
}

// This warp's staging area in the block's dynamic shared memory.
__device__ __forceinline__ float* warp_stage_area(size_t warp_bytes) {
  extern __shared__ __align__(16) unsigned char rollout_dyn_smem[];
  return reinterpret_cast<float*>(rollout_dyn_smem + (threadIdx.x >> 5) * warp_bytes);
}

// ---------------------------------------------------------------------------
// Planar serial chain under joint torques.
// ---------------------------------------------------------------------------
template <int NL>
__device__ __forceinline__ void chain_tip(const float (&len)[NL], const float (&c)[NL],
                                          const float (&s)[NL], float& x, float& y) {
  x = 0.f;
  y = 0.f;
#pragma unroll
  for (int j = 0; j < NL; ++j) {
    x = fmaf(len[j], c[j], x);
    y = fmaf(len[j], s[j], y);
  }
}

template <int NL, int PF, int T, bool SFU = kSfuTurns<NL, PF>>
__device__ __forceinline__ void rollout_chain_body(const RolloutArgs& a, const ChainModel& cm,
                                                   int r, bool live, const StagedRows<NL, T>* st) {
  const int b = a.row0 + r;
  const uint32_t iter = a.d_iter ? *a.d_iter : a.iter;
  const float* Ub = a.U + (size_t)r * a.H * NL;
  const int models = (a.dr_mode == MTP_DR_SHARED) ? a.R : 1;
  const float dt = a.dt;
  float len[NL];
#pragma unroll
  for (int j = 0; j < NL; ++j) len[j] = cm.length[j];
  float total = 0.f;
  for (int mdl = 0; mdl < models; ++mdl) {
    const uint32_t unit = (a.dr_mode == MTP_DR_SHARED) ? (uint32_t)mdl : (uint32_t)b;
    // Lagrangian constants: beta_j = m_j/2 + sum_{i>j} m_i, lb_j = l_j beta_j,
    // D_jj = l_j^2 (m_j/3 + sum_{i>j} m_i), G_j = g l_j beta_j.
    float lb[NL], Dd[NL], G[NL];
    {
      float mass[NL];
      dr_scales<NL>(a, iter, unit, mass);
#pragma unroll
      for (int j = 0; j < NL; ++j) mass[j] *= cm.mass[j];
      float outer = 0.f;
#pragma unroll
      for (int j = NL - 1; j >= 0; --j) {
        const float beta = fmaf(0.5f, mass[j], outer);
        lb[j] = len[j] * beta;
        Dd[j] = len[j] * len[j] * fmaf(mass[j], 1.f / 3.f, outer);
        G[j] = cm.gravity * lb[j];
        outer += mass[j];
      }
    }
    float phi[NL], w[NL];
    {
      float ph = 0.f, om = 0.f;
#pragma unroll
      for (int j = 0; j < NL; ++j) {
        ph += a.x0[j];
        om += a.x0[NL + j];
        phi[j] = ph;
        w[j] = om;
      }
    }
    if (a.X) {
#pragma unroll
      for (int j = 0; j < NL; ++j) {
        a.X[j] = a.x0[j];
        a.X[NL + j] = a.x0[NL + j];
      }
    }
    KahanSum J;
    for_each_step<NL, PF, T>(Ub, a.H, st, [&](int t, const float (&u)[NL]) {
      float c[NL], s[NL], tau[NL];
#pragma unroll
      for (int j = 0; j < NL; ++j) {
        tau[j] = u[j];
        sincos_reduced<SFU>(phi[j], &s[j], &c[j]);
      }
      // stage cost c(x_t, u_t): reach error of the tip and torque penalty
      {
        float x, y;
        chain_tip<NL>(len, c, s, x, y);
        const float ex = x - cm.target[0], ey = y - cm.target[1];
        float tt = 0.f;
#pragma unroll
        for (int j = 0; j < NL; ++j) tt = fmaf(tau[j], tau[j], tt);
        J.add(fmaf(cm.w_target, fmaf(ex, ex, ey * ey), cm.w_ctrl * tt), a.kahan);
      }
      // right-hand side: generalised forces and gravity
      float rhs[NL];
#pragma unroll
      for (int j = 0; j < NL; ++j) {
        const float q_next = (j + 1 < NL) ? tau[j + 1] : 0.f;
        rhs[j] = fmaf(-G[j], c[j], tau[j] - q_next);
      }
      // the dense mass matrix (lower triangle) of the shorter chains, built
      // before the velocity terms so that its independent products overlap
      // their prefix sums: A_jk = D_jk cos(phi_j - phi_k) with D_jk = l_k lb_j
      // below the diagonal
      using Tr = Tri<NL>;
      float A[Tr::size];
      if constexpr (NL < kSemisepLinks) {
#pragma unroll
        for (int j = 0; j < NL; ++j) A[Tr::at(j, j)] = Dd[j];
        Unroll<1, NL>::run([&](auto J) {
          constexpr int j = decltype(J)::value;
          Unroll<0, j>::run([&](auto K) {
            constexpr int k = decltype(K)::value;
            A[Tr::at(j, k)] = (len[k] * lb[j]) * fmaf(c[j], c[k], s[j] * s[k]);  // cos(phi_j - phi_k)
          });
        });
      }
      // velocity terms sum_k D_jk sin(phi_j - phi_k) w_k^2 in O(NL): with
      // a_k = c_k w_k^2, b_k = s_k w_k^2 the sum is
      // s_j (lb_j Pa_j + l_j Sa_j) - c_j (lb_j Pb_j + l_j Sb_j), where P sums
      // l_k (.)_k over k < j and S sums lb_k (.)_k over k > j
      {
        float wa[NL], wb[NL];
#pragma unroll
        for (int k = 0; k < NL; ++k) {
          const float w2 = w[k] * w[k];
          wa[k] = c[k] * w2;
          wb[k] = s[k] * w2;
        }
        float Pa = 0.f, Pb = 0.f;
        float Sa[NL], Sb[NL];
        Sa[NL - 1] = 0.f;
        Sb[NL - 1] = 0.f;
#pragma unroll
        for (int k = NL - 2; k >= 0; --k) {
          Sa[k] = fmaf(lb[k + 1], wa[k + 1], Sa[k + 1]);
          Sb[k] = fmaf(lb[k + 1], wb[k + 1], Sb[k + 1]);
        }
#pragma unroll
        for (int j = 0; j < NL; ++j) {
          const float ca = fmaf(lb[j], Pa, len[j] * Sa[j]);
          const float cb = fmaf(lb[j], Pb, len[j] * Sb[j]);
          rhs[j] = rhs[j] - fmaf(s[j], ca, -c[j] * cb);
          Pa = fmaf(len[j], wa[j], Pa);
          Pb = fmaf(len[j], wb[j], Pb);
        }
      }
      if constexpr (NL >= kSemisepLinks) {
        // Below the diagonal A_jk = u_j . v_k with u_j = lb_j (cos phi_j,
        // sin phi_j) and v_k = l_k (cos phi_k, sin phi_k): a rank-2
        // semiseparable matrix plus its diagonal Dd.  Its Cholesky factor
        // has the same form, L_jk = u_j . w_k, built link by link with the
        // running 2 x 2 matrix M = sum_{i<k} w_i w_i^T:
        //   d_k^2 = Dd_k - u_k^T M u_k,  w_k = (v_k - M u_k) / d_k,  M += w_k w_k^T;
        // then L y = rhs and L^T phi'' = y with running 2-vectors: O(NL)
        // work and registers, against O(NL^3) work and O(NL^2) registers
        // for the dense factor.
        float u1[NL], u2[NL], w1[NL], w2[NL], dinv[NL];
        float m11 = 0.f, m12 = 0.f, m22 = 0.f;
#pragma unroll
        for (int k = 0; k < NL; ++k) {
          u1[k] = lb[k] * c[k];
          u2[k] = lb[k] * s[k];
          const float mu1 = fmaf(m11, u1[k], m12 * u2[k]);
          const float mu2 = fmaf(m12, u1[k], m22 * u2[k]);
          const float inv = rsqrtf(Dd[k] - fmaf(u1[k], mu1, u2[k] * mu2));
          dinv[k] = inv;
          w1[k] = fmaf(len[k], c[k], -mu1) * inv;
          w2[k] = fmaf(len[k], s[k], -mu2) * inv;
          m11 = fmaf(w1[k], w1[k], m11);
          m12 = fmaf(w1[k], w2[k], m12);
          m22 = fmaf(w2[k], w2[k], m22);
        }
        float z1 = 0.f, z2 = 0.f;
#pragma unroll
        for (int j = 0; j < NL; ++j) {
          rhs[j] = (rhs[j] - fmaf(u1[j], z1, u2[j] * z2)) * dinv[j];
          z1 = fmaf(w1[j], rhs[j], z1);
          z2 = fmaf(w2[j], rhs[j], z2);
        }
        float r1 = 0.f, r2 = 0.f;
#pragma unroll
        for (int k = NL - 1; k >= 0; --k) {
          rhs[k] = (rhs[k] - fmaf(w1[k], r1, w2[k] * r2)) * dinv[k];
          r1 = fmaf(u1[k], rhs[k], r1);
          r2 = fmaf(u2[k], rhs[k], r2);
        }
      } else {
        float inv[NL];
        // Cholesky A = L L^T in place (inv holds 1 / L_jj), then the two
        // triangular solves
        Unroll<0, NL>::run([&](auto J) {
          constexpr int j = decltype(J)::value;
          float d = A[Tr::at(j, j)];
          Unroll<0, j>::run([&](auto K) {
            constexpr int k = decltype(K)::value;
            d = fmaf(-A[Tr::at(j, k)], A[Tr::at(j, k)], d);
          });
          inv[j] = rsqrtf(d);
          Unroll<j + 1, NL>::run([&](auto I) {
            constexpr int i = decltype(I)::value;
            float v = A[Tr::at(i, j)];
            Unroll<0, j>::run([&](auto K) {
              constexpr int k = decltype(K)::value;
              v = fmaf(-A[Tr::at(i, k)], A[Tr::at(j, k)], v);
            });
            A[Tr::at(i, j)] = v * inv[j];
          });
        });
        Unroll<0, NL>::run([&](auto I) {
          constexpr int i = decltype(I)::value;
          float v = rhs[i];
          Unroll<0, i>::run([&](auto K) {
            constexpr int k = decltype(K)::value;
            v = fmaf(-A[Tr::at(i, k)], rhs[k], v);
          });
          rhs[i] = v * inv[i];
        });
        Unroll<0, NL>::run([&](auto I) {
          constexpr int i = NL - 1 - decltype(I)::value;
          float v = rhs[i];
          Unroll<i + 1, NL>::run([&](auto K) {
            constexpr int k = decltype(K)::value;
            v = fmaf(-A[Tr::at(k, i)], rhs[k], v);
          });
          rhs[i] = v * inv[i];
        });
      }
      // semi-implicit Euler in absolute coordinates
#pragma unroll
      for (int j = 0; j < NL; ++j) {
        w[j] = fmaf(dt, rhs[j], w[j]);
        phi[j] = fmaf(dt, w[j], phi[j]);
      }
      if (a.X) {
        float* xo = a.X + (size_t)(t + 1) * 2 * NL;
#pragma unroll
        for (int j = 0; j < NL; ++j) {
          xo[j] = phi[j] - (j ? phi[j - 1] : 0.f);
          xo[NL + j] = w[j] - (j ? w[j - 1] : 0.f);
        }
      }
    });
    {
      float c[NL], s[NL], x, y;
#pragma unroll
      for (int j = 0; j < NL; ++j) sincos_reduced<SFU>(phi[j], &s[j], &c[j]);
      chain_tip<NL>(len, c, s, x, y);
      const float ex = x - cm.target[0], ey = y - cm.target[1];
      J.add(cm.w_term * cm.w_target * fmaf(ex, ex, ey * ey), a.kahan);
    }
    total += J.s;
  }
  if (!live) return;
  float cst = total / (float)models;
  if (!isfinite(cst)) cst = __int_as_float(0x7f800000);
  a.cost[r] = cst;
}

// Standalone launches: one thread per candidate row.  Direct loads (T = 0)
// let threads past the last row leave at once; staged loads keep every lane
// of a warp in the warp's copy protocol.
template <int NL, int T, bool SFU>
__global__ void __launch_bounds__(kThreads) k_rollout_chain(const RolloutArgs a,
                                                            const ChainModel cm) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if constexpr (T == 0) {
    if (r >= a.rows) return;
    rollout_chain_body<NL, kPrefetchAlone, 0, SFU>(a, cm, r, true, nullptr);
  } else {
    if (__all_sync(0xffffffffu, r >= a.rows)) return;
    const int r0 = r & ~31;
    const StagedRows<NL, T> st{a.U + (size_t)r0 * a.H * NL, min(32, a.rows - r0),
                               warp_stage_area(StageShape<NL, T>::kWarpBytes)};
    rollout_chain_body<NL, kPrefetchAlone, T, SFU>(a, cm, r, r < a.rows, &st);
  }
}

template <int NL, int T>
__global__ void __launch_bounds__(kThreads) k_rollout_chain_batch(const RolloutArgs* __restrict__ ra,
                                                                  const ChainModel* __restrict__ cms,
                                                                  const int* __restrict__ row_start,
                                                                  int count) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= __ldg(row_start + count)) return;
  const int i = batch_instance(row_start, count, g);
  const RolloutArgs a = ra[i];
  const ChainModel cm = cms[i];
  const int r = g - __ldg(row_start + i);
  const bool live = r < a.rows;
  if constexpr (T == 0) {
    if (!live) return;
    rollout_chain_body<NL, kPrefetchBatch, 0>(a, cm, r, true, nullptr);
  } else {
    const int r0 = r & ~31;  // rows are padded to whole warps
    const StagedRows<NL, T> st{a.U + (size_t)r0 * a.H * NL, min(32, a.rows - r0),
                               warp_stage_area(StageShape<NL, T>::kWarpBytes)};
    rollout_chain_body<NL, kPrefetchBatch, T>(a, cm, r, live, &st);
  }
}

}  // namespace
}  // namespace mtp
