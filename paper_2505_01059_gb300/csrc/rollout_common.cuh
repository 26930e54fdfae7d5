// rollout_common.cuh -- helpers shared by the rollout kernels: compile-time
// loops, packed lower-triangle indexing, the per-model randomisation scales,
// reduced-range sine / cosine and the batch row -> instance lookup.
#pragma once

#include "mtp_device.cuh"

namespace mtp {
namespace {

// Threads per block: fill as many SMs as the batch allows (one thread per
// candidate; small batches get one warp per block).
inline int rollout_block(int rows) {
  const int sms = device_sms();
  int bd = 128;
  while (bd > 32 && (rows + bd - 1) / bd < sms) bd >>= 1;
  return bd;
}

// Control steps requested ahead of use by rollouts that load directly.
// Measured on GB300 (depths 1 / 2 / 3 / 4): a lone instance, which has one
// warp per SM sub-partition at most, is fastest at 2 (7-link arm 118 / 105 /
// 105 / 109 us per step); a batch, where registers set how many warps are
// resident, at 1 (256 instances 4.06 / 4.16 / 4.25 / 4.37 ms per iteration).
constexpr int kPrefetchAlone = 2;
constexpr int kPrefetchBatch = 1;

// Compile-time loop: calls f(IC<i>) for i in [B, E), so every array index
// derived from i is a constant and the arrays stay in registers.
template <int V>
struct IC {
  static constexpr int value = V;
};
template <int B, int E>
struct Unroll {
  template <class F>
  static __device__ __forceinline__ void run(F&& f) {
    if constexpr (B < E) {
      f(IC<B>{});
      Unroll<B + 1, E>::run(f);
    }
  }
};

// Model scales of slots 0..S-1 for one model unit, four slots per generator
// call (the same words draw() returns one at a time).
template <int S>
__device__ __forceinline__ void dr_scales(const RolloutArgs& a, uint32_t iter, uint32_t unit,
                                          float (&out)[S]) {
  if (a.dr_mode == MTP_DR_NONE) {
#pragma unroll
    for (int j = 0; j < S; ++j) out[j] = 1.f;
    return;
  }
  const uint32_t tag = (a.dr_mode == MTP_DR_SHARED) ? kTagParamModel : kTagParamSample;
  const float span = a.dr_hi - a.dr_lo;
#pragma unroll
  for (int g = 0; g < (S + 3) / 4; ++g) {
    const uint4 r = philox(make_uint4(unit, (uint32_t)g, iter, tag), a.key);
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (4 * g + q < S) out[4 * g + q] = fmaf(span, unit24(w[q]), a.dr_lo);
  }
}

// rintf for every x, by adding and taking off 2^23 (from there on x is whole):
// without rintf's place in the SFU's queue (8 cycles per warp and operation, in
// front of the sines and cosines).
__device__ __forceinline__ float round_nearest(float x) {
  const float a = fabsf(x);
  const float r = copysignf(__fadd_rn(__fadd_rn(a, 8388608.f), -8388608.f), x);
  return a < 8388608.f ? r : x;
}

// sin and cos of an absolute link angle: Cody-Waite reduction of x by 2 pi
// (a two-term split of 2 pi) to [-pi, pi], then the SFU sine / cosine, whose
// absolute error on that interval is about 4e-7.  SFU: the whole turns by rintf.
template <bool SFU = false>
__device__ __forceinline__ void sincos_reduced(float x, float* s, float* c) {
  const float turns = __fmul_rn(x, 0.15915494309189535f);
  const float k = SFU ? rintf(turns) : round_nearest(turns);
  float r = fmaf(-k, 6.28318548202514648f, x);
  r = fmaf(-k, -1.7484556e-07f, r);
  __sincosf(r, s, c);
}

// Asynchronous 4-byte global-to-shared copy (cp.async, cached at L1), its
// commit, and the wait for all of the thread's committed copies.
__device__ __forceinline__ void copy_async_f32(float* smem_dst, const float* gmem_src) {
  const unsigned dst = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void copy_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void copy_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// ---------------------------------------------------------------------------
// Staged control rows.  A rollout thread reads its candidate's controls one
// step after another; a warp's 32 lanes read 32 different rows, H * n floats
// apart, so each direct warp load touches 32 cache lines (measured: 31
// sectors per request and the L1 at 83-93 % of its throughput in the batched
// 7-link and 9-axis rollouts).  Staged instead, the rows pass through shared
// memory a horizon chunk of T steps at a time: the warp copies the next chunk of
// all its rows with asynchronous 16-byte copies, neighbouring lanes on
// neighbouring pieces, into the one of two buffers that it does not read.  The
// host stages only rows whose base is 16-byte aligned and whose length H * K is
// a multiple of 4 floats, with T a multiple of 4, so every chunk is whole
// pieces.  (One bulk copy per lane and an mbarrier per buffer, as before, took
// about 300 instructions of the integer pipe per chunk in the protocol and its
// bounded wait.)  The row stride in shared memory is a multiple of 4 floats with
// an odd quotient, so that the lanes' 16-byte row starts fall in distinct bank
// quads (a scalar read is then a 4-way conflict, against 32 lines per direct
// warp load).
// ---------------------------------------------------------------------------
template <int K, int T>
struct StageShape {
  static_assert(T % 4 == 0, "chunks must be whole 16-byte units");
  static constexpr int kQuads = (T * K + 3) / 4;
  static constexpr int kStride = 4 * (kQuads % 2 ? kQuads : kQuads + 1);  // floats
  static constexpr int kBuf = 32 * kStride;                               // floats per buffer
  static constexpr size_t kWarpBytes = 2 * kBuf * sizeof(float);
};

__device__ __forceinline__ void copy_async_16(float* smem_dst, const float* gmem_src) {
  const unsigned dst = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(gmem_src) : "memory");
}

// Asynchronous copies, by one warp, of n candidates' next `steps` steps of
// controls (src, H K floats apart) into rows `row` floats apart: in 16-byte
// pieces (vec: every piece is aligned) or by single floats.
template <int K>
__device__ __forceinline__ void copy_controls(const float* src, int H, int n, int steps, bool vec, float* dst, int row) {
  const int lane = threadIdx.x & 31;
  const int len = vec ? steps * K / 4 : steps * K;  // pieces per candidate
  int i = lane / len, o = lane - i * len;
  const int di = 32 / len, dlen = 32 - di * len;
  while (i < n) {
    if (vec) copy_async_16(dst + i * row + 4 * o, src + (size_t)i * H * K + 4 * o);
    else copy_async_f32(dst + i * row + o, src + (size_t)i * H * K + o);
    i += di;
    o += dlen;
    if (o >= len) {
      o -= len;
      ++i;
    }
  }
  copy_async_commit();
}

// The rows of a warp's candidates (the first one's, and how many there are) and
// its two buffers.
template <int K, int T>
struct StagedRows {
  using Shape = StageShape<K, T>;
  const float* rows;
  int n;
  float* buf;
  // steps t0 .. t0 + T - 1 (those below H) into buffer b; every lane calls it
  __device__ __forceinline__ void request(int t0, int H, int b) const {
    const int lane = threadIdx.x & 31;
    float* const dst = buf + b * Shape::kBuf;
    const float* const src = rows + (size_t)t0 * K;
    if (t0 + T <= H) {
      // a whole chunk: T K / 4 pieces per lane, their rows known but for the
      // lane's first
      constexpr int len = T * K / 4, di = 32 / len, dlen = 32 - di * len;
      int i = lane / len, o = lane - i * len;
#pragma unroll 1
      for (int q = 0; q < len; ++q) {
        if (i < n) copy_async_16(dst + i * Shape::kStride + 4 * o, src + (size_t)i * H * K + 4 * o);
        i += di;
        o += dlen;
        if (o >= len) {
          o -= len;
          ++i;
        }
      }
      copy_async_commit();
    } else {
      copy_controls<K>(src, H, n, H - t0, true, dst, Shape::kStride);
    }
  }
};

// Feeds step(t, u) the K controls of every step t = 0 .. H-1 of this lane's
// candidate row Ub.  T == 0: direct loads PF steps ahead into a rotating
// register buffer (the loop is unrolled by PF so its slots are constants).
// T > 0: the warp's rows staged through shared memory (every lane calls it).
template <int K, int PF, int T, class Step>
__device__ __forceinline__ void for_each_step(const float* Ub, int H, const StagedRows<K, T>* st, Step&& step) {
  if constexpr (T == 0) {
    (void)st;
    float ubuf[PF][K];
#pragma unroll
    for (int q = 0; q < PF; ++q)
#pragma unroll
      for (int k = 0; k < K; ++k) ubuf[q][k] = __ldg(Ub + min(q, H - 1) * K + k);
    for (int t0 = 0; t0 < H; t0 += PF) {
      Unroll<0, PF>::run([&](auto Q) {
        constexpr int q = decltype(Q)::value;
        const int t = t0 + q;
        if (t < H) {
          float u[K];
          const int tn = min(t + PF, H - 1);
#pragma unroll
          for (int k = 0; k < K; ++k) {
            u[k] = ubuf[q][k];
            ubuf[q][k] = __ldg(Ub + tn * K + k);  // PF steps ahead
          }
          step(t, u);
        }
      });
    }
  } else {
    using Shape = StageShape<K, T>;
    const float* const mine = st->buf + (threadIdx.x & 31) * Shape::kStride;
    __syncwarp();  // the warp's previous rows have been used
    st->request(0, H, 0);
    for (int t0 = 0, b = 0; t0 < H; t0 += T, b ^= 1) {
      copy_async_wait_all();
      __syncwarp();  // this chunk is there, and the other buffer's has been used
      if (t0 + T < H) st->request(t0 + T, H, b ^ 1);
      // a rolled loop over the chunk's steps: its reads need no constant
      // slots, and the step body stays one copy
      const float* src = mine + b * Shape::kBuf;
      const int t1 = min(t0 + T, H);
#pragma unroll 1
      for (int t = t0; t < t1; ++t, src += K) {
        float u[K];
#pragma unroll
        for (int k = 0; k < K; ++k) u[k] = src[k];
        step(t, u);
      }
    }
  }
}

template <int NL>
struct Tri {
  static constexpr int size = NL * (NL + 1) / 2;
  static __device__ __forceinline__ constexpr int at(int i, int j) { return i * (i + 1) / 2 + j; }
};

// Instance of global row g in a batch: row_start (count + 1 entries) holds
// each instance's first row, rows padded to whole warps.
__device__ __forceinline__ int batch_instance(const int* __restrict__ row_start, int count, int g) {
  int lo = 0, hi = count;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (__ldg(row_start + mid) <= g) lo = mid;
    else hi = mid;
  }
  return lo;
}

}  // namespace
}  // namespace mtp
