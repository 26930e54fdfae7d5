// bspline_tc.cu -- Def. 2 B-spline interpolation of the graph paths as a
// dense contraction on the 5th-generation tensor cores (tcgen05), for the
// BF16-operand mode (MTP_FLAG_BF16_BASIS).
//
// The graph rows of an iteration are U[b, t, i] = sum_m B[t, m] C[b, m, i]
// (Def. 2 with the basis B_p sampled at the H evaluation times and the
// waypoints C of path b, Alg. 1).  Seen as one GEMM,
// D[(b, i), t] = sum_m W[(b, i), m] B[t, m] with W the gathered waypoints
// (one row per path and control dimension) and B the (H x M) basis table,
// K = M.  A tile is up to 128 (path, dimension) rows by one 128-step slice
// of the horizon: accumulator lanes 32 w .. 32 w + 31 hold floor(32 / n) whole
// paths (rows 32 w + n p + i), so a path never straddles two quarters and the
// rows are dense for any n.  Each CTA (two warpgroups) loops over tiles: its
// threads draw the paths' layer indices (Alg. 1, four layers per generator
// call) and gather their waypoints from the instance's graph (written in
// bfloat16 by the graph launch, copied to shared memory once per instance) into
// the A operand, eight layers of a row per 16-byte store, and one thread issues
// tcgen05.mma.cta_group::1.kind::f16 (BF16 x BF16 -> FP32, M = 128 rows, N = 128
// steps, K = 16 per instruction) into tensor memory.  The B operand comes from
// the handle's table in its shared-memory layout.  The products of two bfloat16 values are exact in FP32; the
// sums are FP32.  In the epilogue warps w and w + 4 take the two halves of
// quarter w's steps, 16 at a time with tcgen05.ld, clamp them to the control box and write them
// through a per-warp shared-memory transpose: for each path, 16 steps x n
// controls are one contiguous block of U, stored with 16-byte vector stores
// whose places in the transpose and in U a lane computes once per instance.
//
// What bounds it: the epilogue's instructions and the latency of a tile's
// serial phases, hence two warpgroups and four CTAs per SM.  On the 16-link
// legged workload (18.9 M elements) it took 44 us with one warpgroup, three CTAs
// per SM, the gather of 8 paths on one warp and a division per stored vector.
//
// Shared-memory operands use the canonical K-major layout without swizzle:
// 8-row x 16-byte core matrices, the two (or more) core matrices of a row
// group along K 128 bytes apart (leading byte offset) and consecutive row
// groups 16 K bytes apart (stride byte offset).  Each CTA allocates 128
// tensor-memory columns (its accumulator) and asks for enough shared memory
// that at most four CTAs share an SM, so their allocations always fit the
// SM's 512 columns.
#include <algorithm>
#include <cstring>
#include <vector>

#include <cuda_bf16.h>

#include "mtp_device.cuh"

namespace mtp {
namespace {

constexpr int kTcThreads = 256;
constexpr int kTcWarps = kTcThreads / 32;
constexpr int kMaxK = 64;            // layers (M) padded to a multiple of 16
constexpr int kMaxSlices = 2;        // 128-step horizon slices (H <= 256)
constexpr int kZsMax = 16384;        // graph elements (M N n) staged in shared memory
constexpr uint32_t kTmemCols = 128;
constexpr size_t kMinSmem = 50 * 1024;  // at most four CTAs per SM (their TMEM fits)
constexpr int kBatchTilesPerCta = 8;

// The fixed part of a CTA's shared memory; what depends on the instance follows
// it: the operands (A: waypoints, row 32 w + n p + i, K-major; B: basis of one
// slice, row t, K-major; 128 K bfloat16 each), the tile's places in the graph
// per path and layer (16 bits: M N n <= 40960), and the instance's graph in
// bfloat16 when it is staged.
struct TcSmem {
  // per warp: 16 steps of its paths' rows, path by path in the order of U
  float stage[kTcWarps][32 * 16];
  float lo[MTP_MAX_CTRL], hi[MTP_MAX_CTRL];
  uint64_t mma_bar;
  uint32_t tmem_base;
  alignas(128) unsigned char rest[];
};
__host__ __device__ constexpr int up16(int bytes) { return (bytes + 15) / 16 * 16; }

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// Byte offset of element (row, k) in a K-major, unswizzled canonical layout
// with K columns: core matrix (row / 8, k / 8), row (row % 8) of 16 bytes.
__host__ __device__ __forceinline__ int kmajor_offset(int row, int k, int K) {
  return (row >> 3) * (16 * K) + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2;
}

// tcgen05 shared-memory matrix descriptor: start address, leading and stride
// byte offsets (all in 16-byte units), the fixed version field (bits 46-48 =
// 0b001), no base offset, no swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1),
// BF16 A and B (bits 7-9, 10-12 = 1), both K-major, N >> 3 at bit 17,
// M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

// Paths per quarter of the accumulator lanes and per tile for n control
// dimensions (n <= 16).
__host__ __device__ constexpr int tc_paths_per_warp(int n) { return 32 / n; }
__host__ __device__ constexpr int tc_paths_per_tile(int n) {
  return 4 * tc_paths_per_warp(n);
}

__host__ __device__ __forceinline__ bool graph_staged(const CandArgs& a) {
  return a.C_in == nullptr && a.dm.M * a.dm.N * a.dm.n <= kZsMax;
}

// One instance as a thread of the CTA sees it: where its data lies, and this
// thread's shares of the gather and of the stores.
struct TcPlan {
  int K, ppw, staged;
  unsigned char *W, *Bs;
  uint16_t* at;
  const __nv_bfloat16* Zs;
  // gather: row tid % 128 of the A operand is dimension i of the tile's path q
  // (q < 0: none); the thread makes one half of its K columns
  int q, i;
  // accumulator lane: path p (of the quarter's ppw) and dimension d
  int p, d;
  // stores of one warp's 16-step chunk: vector z (of at most four: ppw n <= 32
  // rows of 16 steps are at most 128 vectors) belongs to path[z] and lies at
  // from[z] in the transpose (p 16 n + 4 o) and at to[z] in U (p H n + 4 o)
  int path[4], from[4], to[4];
};
__device__ __forceinline__ TcPlan tc_plan(TcSmem& S, const CandArgs& a) {
  TcPlan pl;
  const int n = a.dm.n, Hn = a.dm.H * n, lane = threadIdx.x & 31;
  pl.K = (a.dm.M + 15) / 16 * 16;
  pl.ppw = tc_paths_per_warp(n);
  pl.staged = graph_staged(a);
  pl.W = S.rest;
  pl.Bs = pl.W + 256 * pl.K;
  pl.at = reinterpret_cast<uint16_t*>(pl.Bs + 256 * pl.K);
  pl.Zs = pl.staged ? reinterpret_cast<const __nv_bfloat16*>(pl.Bs + 256 * pl.K + up16(8 * pl.ppw * pl.K))
                    : reinterpret_cast<const __nv_bfloat16*>(a.Z_global);
  pl.p = lane / n;
  pl.d = lane - pl.p * n;
  pl.i = pl.d;  // the row's lane is the thread's
  pl.q = pl.p < pl.ppw ? (int)((threadIdx.x & 127) >> 5) * pl.ppw + pl.p : -1;
  const int q4 = 4 * n;  // vectors of one path in a chunk
#pragma unroll
  for (int z = 0; z < 4; ++z) {
    const int e = 32 * z + lane;
    const int p = e / q4, o = e - p * q4;
    pl.path[z] = p;
    pl.from[z] = 16 * n * p + 4 * o;
    pl.to[z] = Hn * p + 4 * o;
  }
  return pl;
}

// Sixteen accumulator columns of this lane's row.  The load and the wait for it
// are one statement: a register of the load means nothing before the wait, and
// what names the registers in between (a merge with another path's, a hoisted
// use) is the compiler's choice.
__device__ __forceinline__ void tmem_load16(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr)
      : "memory");
}

// Path group g of one instance's graph rows, horizon slice s (the B operand
// holds that slice's basis).  Returns false when the bounded wait for the
// MMA gave up.
__device__ __forceinline__ bool tc_tile(TcSmem& S, const CandArgs& a, const TcPlan& pl, int g, int s, uint32_t iter,
                                        uint32_t& phase) {
  const Dims dm = a.dm;
  const int H = dm.H, n = dm.n, M = dm.M, N = dm.N, K = pl.K;
  const int ppw = pl.ppw;
  const int b0 = g * 4 * ppw;
  const int nb = min(4 * ppw, a.graph_rows - b0);
  // Alg. 1: the places of the tile's waypoints in the graph
  if (a.C_in == nullptr) {
    const int quads = (M + 3) >> 2;
    for (int e = threadIdx.x; e < nb * quads; e += kTcThreads) {
      const int q = e / quads, mq = e - q * quads;
      const uint4 r = philox(make_uint4((uint32_t)(b0 + q), (uint32_t)mq, iter, kTagPath), a.key);
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const int m = 4 * mq + w;
        if (m < M) pl.at[q * K + m] = (uint16_t)((m * N + index_of(pick(r, (uint32_t)w), (uint32_t)N)) * n);
      }
    }
    __syncthreads();
  }
  // the A operand: this thread's row, eight columns (one core matrix row) at a time
  if (pl.q >= 0 && pl.q < nb) {
    const int row = threadIdx.x & 127, half = threadIdx.x >> 7;
    for (int m0 = half * (K / 2); m0 < (half + 1) * (K / 2); m0 += 8) {
      uint32_t pair[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint16_t x[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int m = m0 + 2 * c + h;
          __nv_bfloat16 z = __float2bfloat16_rn(0.f);
          if (m < M)
            z = a.C_in ? __float2bfloat16_rn(a.C_in[((size_t)(b0 + pl.q) * M + m) * n + pl.i])
                       : pl.Zs[pl.at[pl.q * K + m] + pl.i];
          x[h] = __bfloat16_as_ushort(z);
        }
        pair[c] = (uint32_t)x[0] | ((uint32_t)x[1] << 16);
      }
      *reinterpret_cast<uint4*>(pl.W + kmajor_offset(row, m0, K)) = make_uint4(pair[0], pair[1], pair[2], pair[3]);
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t idesc = idesc_bf16(128, 128);
    const uint32_t sbo = 16u * (uint32_t)K;
    const uint32_t d_tmem = S.tmem_base;
    for (int ks = 0; ks < K / 16; ++ks) {
      const uint64_t ad = smem_desc(smem_u32(pl.W) + 256u * ks, 128u, sbo);
      const uint64_t bd = smem_desc(smem_u32(pl.Bs) + 256u * ks, 128u, sbo);
      const uint32_t acc = ks > 0 ? 1u : 0u;
      asm volatile(
          "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
          " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
          "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
          : "memory");
    }
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(&S.mma_bar))
                 : "memory");
  }
  const bool ok = mbar_wait_bounded(&S.mma_bar, phase);
  phase ^= 1u;
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (!__syncthreads_and(ok)) return false;
  // epilogue: warps w and w + 4 read accumulator lanes 32 (w % 4) .. + 31,
  // steps 64 (w / 4) .. + 63 of the slice, 16 steps (columns) at a time; lane l
  // holds row (path l / n, dimension l % n) of the quarter's paths.  Clamped
  // values go to the warp's staging area in the order of U (path-major, then
  // step, then dimension), from which each path's 16 n contiguous floats of U
  // are written.
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int w = warp & 3;
  const int p = pl.p, i = pl.d;
  const int wb0 = b0 + w * ppw;                          // the quarter's first path
  const int wpaths = max(0, min(ppw, a.graph_rows - wb0));  // its paths in this tile
  const float lo = i < n ? S.lo[i] : 0.f, hi = i < n ? S.hi[i] : 0.f;
  const size_t Hn = (size_t)H * n;
  const bool vec = ((reinterpret_cast<uintptr_t>(a.U_graph) & 15) == 0) && (Hn & 3) == 0;
  const int t_first = 128 * s + 64 * (warp >> 2);
  const int t_end = min(t_first + 64, H);
  float* st = S.stage[warp];
  float* mine = st + p * 16 * n + i;
  float* out = a.U_graph + (size_t)wb0 * Hn + (size_t)t_first * n;
  const uint32_t taddr = S.tmem_base + ((uint32_t)(32 * w) << 16) + (uint32_t)(64 * (warp >> 2));
  for (int t0 = t_first; t0 < t_end; t0 += 16, out += 16 * n) {
    uint32_t v[16];
    tmem_load16(taddr + (uint32_t)(t0 - t_first), v);
    const int steps = min(16, H - t0);  // steps of this chunk inside the horizon
    __syncwarp();                        // the previous chunk's reads of st are done
    if (p < wpaths) {
#pragma unroll
      for (int tt = 0; tt < 16; ++tt) mine[tt * n] = clamp_box(__uint_as_float(v[tt]), lo, hi);
    }
    __syncwarp();
    if (vec && steps == 16) {
#pragma unroll
      for (int z = 0; z < 4; ++z)
        if (pl.path[z] < wpaths)
          *reinterpret_cast<float4*>(out + pl.to[z]) = *reinterpret_cast<const float4*>(st + pl.from[z]);
    } else {
      // flat over the quarter's pieces; the piece index e / len is taken as
      // (e + 1/2) * (1 / len) rounded down, exact here (e < 2^12, len <= 256:
      // the product's rounding error stays far below the 1/(2 len) margin)
      const int piece = steps * n;  // floats of one path in this chunk
      const float inv = 1.f / (float)piece;
      for (int e = lane; e < wpaths * piece; e += 32) {
        const int pp = __float2int_rz(((float)e + 0.5f) * inv), o = e - pp * piece;
        out[pp * Hn + o] = st[pp * 16 * n + o];
      }
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  return true;
}

// Copies `bytes` (a multiple of 16, from 16-byte aligned global memory) into
// shared memory by the whole CTA, asynchronously.
__device__ __forceinline__ void copy_in(void* dst, const void* src, int bytes) {
  const unsigned d = smem_u32(dst);
  for (int o = 16 * threadIdx.x; o < bytes; o += 16 * kTcThreads)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d + o),
                 "l"(reinterpret_cast<const unsigned char*>(src) + o)
                 : "memory");
}

// The B operand of horizon slice s, and with `instance` what a CTA keeps of the
// instance: the box and its graph (when it fits).
__device__ void tc_load(TcSmem& S, const CandArgs& a, const TcPlan& pl, int s, bool instance) {
  __syncthreads();  // the previous instance's or slice's readers are done
  if (instance) {
    for (int i = threadIdx.x; i < a.dm.n; i += blockDim.x) {
      S.lo[i] = a.umin[i];
      S.hi[i] = a.umax[i];
    }
    if (pl.staged)
      copy_in(const_cast<__nv_bfloat16*>(pl.Zs), a.Z_global, up16(a.dm.M * a.dm.N * a.dm.n * (int)sizeof(__nv_bfloat16)));
  }
  copy_in(pl.Bs, a.basis_tc + (size_t)s * 128 * pl.K, 256 * pl.K);
  asm volatile("cp.async.commit_group;\ncp.async.wait_all;\n" ::: "memory");
  __syncthreads();
}

__device__ void tc_begin(TcSmem& S) {
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&S.tmem_base)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&S.mma_bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Releases the tensor memory.  After a failed wait, first waits (bounded)
// for the MMA still in flight.
__device__ void tc_end(TcSmem& S, bool failed, uint32_t phase, uint32_t* status) {
  if (failed) {
    mbar_wait_bounded(&S.mma_bar, phase ^ 1u);
    if (threadIdx.x == 0 && status) atomicOr(status, kStatusTcTimeout);
  }
  __syncthreads();
  if (threadIdx.x < 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(S.tmem_base),
                 "r"(kTmemCols)
                 : "memory");
}

__device__ __forceinline__ TcSmem& tc_smem() {
  extern __shared__ __align__(1024) unsigned char tc_dyn_smem[];
  return *reinterpret_cast<TcSmem*>(tc_dyn_smem);
}

// One instance: CTAs loop over its tiles, slice-major (tile = s * groups + g),
// so that a CTA changes slice, and reloads the basis, rarely.
__global__ void __launch_bounds__(kTcThreads, 4) k_bspline_tc(const __grid_constant__ CandArgs a) {
  TcSmem& S = tc_smem();
  const int groups = (a.graph_rows + tc_paths_per_tile(a.dm.n) - 1) / tc_paths_per_tile(a.dm.n);
  const int tiles = groups * ((a.dm.H + 127) / 128);
  const uint32_t iter = (a.d_iter ? *a.d_iter : a.iter) + a.iter_offset;
  tc_begin(S);
  const TcPlan pl = tc_plan(S, a);
  uint32_t phase = 0;
  bool failed = false;
  int cur_s = -1;
  for (int tile = blockIdx.x; tile < tiles && !failed; tile += gridDim.x) {
    const int s = tile / groups, g = tile - s * groups;
    if (s != cur_s) tc_load(S, a, pl, s, cur_s < 0);
    cur_s = s;
    failed = !tc_tile(S, a, pl, g, s, iter, phase);
  }
  tc_end(S, failed, phase, a.status);
}

// Many instances: tile_start (count + 1 entries) numbers each instance's
// first tile; each CTA takes a contiguous range of the global tile list (so
// it changes instance, and reloads its set-up, rarely) and sets up again
// whenever the instance or the slice changes.
__global__ void __launch_bounds__(kTcThreads, 4) k_bspline_tc_batch(const CandArgs* __restrict__ args,
                                                                    const int* __restrict__ tile_start, int count) {
  TcSmem& S = tc_smem();
  __shared__ CandArgs sa;
  tc_begin(S);
  const int total = tile_start[count];
  int cur = -1, cur_s = -1;
  uint32_t iter = 0, phase = 0;
  TcPlan pl{};
  bool failed = false;
  const int per = (total + gridDim.x - 1) / gridDim.x;
  const int g_end = min(total, ((int)blockIdx.x + 1) * per);
  for (int g = (int)blockIdx.x * per; g < g_end && !failed; ++g) {
    int lo = 0, hi = count;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (tile_start[mid] <= g) lo = mid;
      else hi = mid;
    }
    const bool instance = lo != cur;
    if (instance) {
      __syncthreads();
      const int* src = reinterpret_cast<const int*>(args + lo);
      int* dst = reinterpret_cast<int*>(&sa);
      for (int q = threadIdx.x; q < (int)(sizeof(CandArgs) / sizeof(int)); q += blockDim.x) dst[q] = src[q];
      __syncthreads();
      cur = lo;
      iter = (sa.d_iter ? *sa.d_iter : sa.iter) + sa.iter_offset;
      pl = tc_plan(S, sa);
    }
    // the instance's tiles slice-major, as in the single-instance kernel
    const int groups = (sa.graph_rows + tc_paths_per_tile(sa.dm.n) - 1) / tc_paths_per_tile(sa.dm.n);
    const int tile = g - tile_start[lo];
    const int s = tile / groups, pg = tile - s * groups;
    if (instance || s != cur_s) tc_load(S, sa, pl, s, instance);
    cur_s = s;
    failed = !tc_tile(S, sa, pl, pg, s, iter, phase);
  }
  tc_end(S, failed, phase, cur >= 0 ? sa.status : nullptr);
}

}  // namespace

// The basis (row t, M columns, already rounded) as the B operands of the
// horizon's slices: [slice][128 K] bfloat16 in the K-major layout, zero past H
// and past M.
std::vector<uint16_t> bspline_tc_basis(const float* basis, int H, int M) {
  const int K = (M + 15) / 16 * 16, slices = (H + 127) / 128;
  std::vector<uint16_t> out((size_t)slices * 128 * K, 0);
  for (int t = 0; t < H; ++t)
    for (int m = 0; m < M; ++m) {
      uint32_t bits;
      std::memcpy(&bits, basis + (size_t)t * M + m, 4);
      out[(size_t)(t / 128) * 128 * K + kmajor_offset(t % 128, m, K) / 2] = (uint16_t)(bits >> 16);
    }
  return out;
}

// Shared memory of a CTA working on one instance.
size_t bspline_tc_smem(const CandArgs& a) {
  const size_t K = (size_t)(a.dm.M + 15) / 16 * 16;
  const size_t at = up16(8 * tc_paths_per_warp(a.dm.n) * (int)K);
  const size_t zs = graph_staged(a) ? up16(a.dm.M * a.dm.N * a.dm.n * (int)sizeof(__nv_bfloat16)) : 0;
  return std::max(sizeof(TcSmem) + 512 * K + at + zs, kMinSmem);
}

bool bspline_tc_eligible(const CandArgs& a) {
  return a.bf16 && a.interp == MTP_INTERP_BSPLINE && a.dm.H <= 128 * kMaxSlices &&
         a.dm.M <= kMaxK && a.dm.n <= 16 && a.graph_rows > 0;
}

int bspline_tc_tiles(const CandArgs& a) {
  const int per = tc_paths_per_tile(a.dm.n);
  return ((a.graph_rows + per - 1) / per) * ((a.dm.H + 127) / 128);
}

// Shared memory of an SM, and what a CTA takes besides its dynamic part (set
// with the kernels' attributes): from them the CTAs resident on one SM (the
// occupancy query answered 1 for these kernels, while ncu's launch statistics,
// with the maximum carveout, showed room for more).
static size_t g_tc_smem_sm = 0, g_tc_smem_fixed = 0;

static int tc_blocks_per_sm(size_t smem) {
  return std::max(1, std::min((int)(g_tc_smem_sm / (smem + g_tc_smem_fixed)), 4));
}

cudaError_t init_bspline_tc_attributes() {
  // the largest any instance takes: 64 layers, one dimension, a full staged graph
  const int most = (int)(sizeof(TcSmem) + 512 * kMaxK + up16(8 * 32 * kMaxK) + kZsMax * sizeof(__nv_bfloat16));
  cudaError_t e;
  for (const void* k : {(const void*)k_bspline_tc, (const void*)k_bspline_tc_batch}) {
    // and the largest shared-memory carveout, so that several CTAs fit an SM
    if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, most)) ||
        (e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared)))
      return e;
  }
  int dev = 0, smem_sm = 0, reserved = 0;
  if ((e = cudaGetDevice(&dev)) ||
      (e = cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev)) ||
      (e = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev)))
    return e;
  cudaFuncAttributes fa{};
  if ((e = cudaFuncGetAttributes(&fa, k_bspline_tc_batch))) return e;
  g_tc_smem_sm = (size_t)smem_sm;
  g_tc_smem_fixed = fa.sharedSizeBytes + (size_t)reserved;
  return cudaSuccess;
}

cudaError_t launch_bspline_tc(const CandArgs& a, cudaStream_t s) {
  const int tiles = bspline_tc_tiles(a);
  if (tiles <= 0) return cudaSuccess;
  const size_t smem = bspline_tc_smem(a);
  const int grid = std::min(tiles, tc_blocks_per_sm(smem) * device_sms());
  k_bspline_tc<<<grid, kTcThreads, smem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_bspline_tc_batch(const CandArgs* d_args, const int* d_tile_start, int count,
                                    int total_tiles, size_t smem, cudaStream_t s) {
  if (total_tiles <= 0) return cudaSuccess;
  // at least kBatchTilesPerCta tiles per CTA: in a batch the launches of
  // other groups run beside this one, and each CTA's set-up (tensor memory,
  // operands) is paid once for its whole range
  const int grid = std::min((total_tiles + kBatchTilesPerCta - 1) / kBatchTilesPerCta,
                            tc_blocks_per_sm(smem) * device_sms());
  k_bspline_tc_batch<<<grid, kTcThreads, smem, s>>>(d_args, d_tile_start, count);
  return cudaGetLastError();
}

}  // namespace mtp
