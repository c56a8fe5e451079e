// LM-head greedy argmax that allocates nothing (oos_lm_head_argmax_static).
//
// For callers that cannot allocate device memory at all -- code that runs
// inside a CUDA graph being captured by someone else, under a memory pool or
// allocator they do not own, or in a process whose allocator is locked -- this
// entry point needs no workspace: its per-block partial results live in a
// fixed file-scope device array that every call shares.
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace oos {

constexpr int kStaticBlocks = 512;   // vocabulary blocks per call (grid size)
constexpr int kStaticMaxT = 128;     // rows of `hidden` per call
constexpr int kStaticThreads = 256;

// Shared by every call on a device: [block][row] partial top-2 states, then the
// arrival counter (zero at load; the last block of a call sets it back to zero).
struct StaticScratch {
  Top2 part[kStaticBlocks][kStaticMaxT];
  int arrived;
};
static __device__ __align__(256) StaticScratch g_argmax_scratch;

// A task is `R` vocabulary rows by `TT` hidden rows, one warp.  The lanes split
// the hidden dimension (VEC consecutive elements each in turn), so that every
// logit is 32 short fp32 chains added as a tree; the R x TT products of the
// loaded elements are formed in registers.
//
// What bounds it is the weight stream for a few hidden rows (T = 1: 230 us for the
// 1.24 GB of 151936 x 4096 bf16) and, from about 6 on, FMA issue behind loads of
// hidden rows that L1 does not hold: per VEC elements a lane loads R + 2 TT 16-byte
// words for R * TT * VEC FMAs.  R = 8 (bf16) or 4 (fp32) and TT <= 8 keep the sums
// and the loaded weights in registers.  The warps of a block take the token groups
// of a row group side by side, so a row group comes from HBM once and from L1 after
// that.  17 rows: 9051 us with one FMA per load, 765 now (303 of FMAs).
template <typename E>
struct StaticRows {
  static constexpr int v = sizeof(E) == 2 ? 8 : 4;
};
// blocks an SM holds: from 6 tokens a task the sums and unpacked weights want
// more than 128 registers
constexpr int static_blocks_per_sm(int tt) { return tt >= 6 ? 1 : 2; }

template <typename E, int VEC>
struct StaticVec;   // VEC consecutive weights as loaded, and as floats
template <>
struct StaticVec<__nv_bfloat16, 8> {
  uint4 u;
  OOS_DEV void load(const __nv_bfloat16* p) { u = __ldg(reinterpret_cast<const uint4*>(p)); }
  OOS_DEV float get(int i) const {
    const uint32_t w = i < 2 ? u.x : i < 4 ? u.y : i < 6 ? u.z : u.w;
    return __uint_as_float((i & 1) ? (w & 0xffff0000u) : (w << 16));
  }
};
template <>
struct StaticVec<float, 8> {
  float4 a, b;
  OOS_DEV void load(const float* p) {
    a = __ldg(reinterpret_cast<const float4*>(p));
    b = __ldg(reinterpret_cast<const float4*>(p) + 1);
  }
  OOS_DEV float get(int i) const {
    const float4 v = i < 4 ? a : b;
    return (i & 3) == 0 ? v.x : (i & 3) == 1 ? v.y : (i & 3) == 2 ? v.z : v.w;
  }
};
template <typename E>
struct StaticVec<E, 1> {
  float v;
  OOS_DEV void load(const E* p) { v = to_f32(*p); }
  OOS_DEV float get(int) const { return v; }
};

// Block b scans vocabulary rows [b*rows, (b+1)*rows) in tasks (row group, token
// group), one warp each; every logit updates that warp's running top-2.  The
// last block to finish merges all blocks' states, in block order.
template <typename E, int TT, int VEC>
__global__ void __launch_bounds__(kStaticThreads, static_blocks_per_sm(TT))
    k_lm_argmax_static(const E* __restrict__ W, int V, int H, int rows_per_block, const float* __restrict__ hidden, int T,
                       StaticScratch* sc, int32_t* out_argmax, float* out_top1, float* out_top2) {
  constexpr int R = StaticRows<E>::v, WARPS = kStaticThreads / 32;
  __shared__ Top2 st[WARPS][kStaticMaxT];
  __shared__ float lg[WARPS][R * TT];
  __shared__ int s_last;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int t = lane; t < T; t += 32) st[warp][t] = Top2{-INFINITY, 0x7fffffff, -INFINITY};
  __syncwarp();
  const int r_begin = blockIdx.x * rows_per_block;
  const int r_end = V - r_begin > rows_per_block ? r_begin + rows_per_block : V;
  const int groups = (T + TT - 1) / TT;
  const int tasks = r_begin < r_end ? (r_end - r_begin + R - 1) / R * groups : 0;
  const int chunks = H / VEC;
  for (int task = warp; task < tasks; task += WARPS) {
    const int r0 = r_begin + task / groups * R, t0 = task % groups * TT;
    float acc[R * TT];
#pragma unroll
    for (int i = 0; i < R * TT; ++i) acc[i] = 0.f;
    const E* w0 = W + (size_t)r0 * H;
    const float* h0 = hidden + (size_t)t0 * H;
    const int nr = min(R, r_end - r0), nt = min(TT, T - t0);   // rows past the end repeat the last one
    // element offsets from the group's first rows: 32 bits (launch_static), and kept as
    // indexes, so that they do not take the registers of R + TT pointers
    using Off = std::conditional_t<VEC == 1, size_t, uint32_t>;
#pragma unroll 1
    for (int c = lane; c < chunks; c += 32) {
      StaticVec<E, VEC> w[R];
#pragma unroll
      for (int r = 0; r < R; ++r) w[r].load(w0 + ((Off)min(r, nr - 1) * (Off)H + (Off)(c * VEC)));
#pragma unroll
      for (int t = 0; t < TT; ++t) {
        StaticVec<float, VEC> h;
        h.load(h0 + ((Off)min(t, nt - 1) * (Off)H + (Off)(c * VEC)));
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
          for (int i = 0; i < VEC; ++i) acc[r * TT + t] = fmaf(w[r].get(i), h.get(i), acc[r * TT + t]);
      }
    }
    int base, n;
    warp_sums(acc, base, n);
#pragma unroll
    for (int i = 0; i < R * TT; ++i)
      if (i < n) lg[warp][base + i] = acc[i];
    __syncwarp();
    if (lane < nt) {
      Top2 s = st[warp][t0 + lane];
      for (int r = 0; r < nr; ++r) s = top2_merge(s, Top2{lg[warp][r * TT + lane], r0 + r, -INFINITY});
      st[warp][t0 + lane] = s;
    }
    __syncwarp();
  }
  __syncthreads();
  for (int t = threadIdx.x; t < T; t += blockDim.x) {
    Top2 r = st[0][t];
    for (int w = 1; w < WARPS; ++w) r = top2_merge(r, st[w][t]);
    sc->part[blockIdx.x][t] = r;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const int old = atomicAdd(&sc->arrived, 1);
    s_last = old == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  for (int t = threadIdx.x; t < T; t += blockDim.x) {
    Top2 r{-INFINITY, 0x7fffffff, -INFINITY};
    for (int b = 0; b < (int)gridDim.x; ++b) {
      const Top2 p{__ldcg(&sc->part[b][t].v1), __ldcg(&sc->part[b][t].i1), __ldcg(&sc->part[b][t].v2)};
      r = top2_merge(r, p);
    }
    out_argmax[t] = r.i1;
    out_top1[t] = r.v1;
    out_top2[t] = r.v2;
  }
  if (threadIdx.x == 0) sc->arrived = 0;   // the next call starts from zero
}

// Device address of the scratch array.  In host code g_argmax_scratch names a
// host-side stand-in, not device memory, so the kernel is given the address
// cudaGetSymbolAddress returns for the current device.  Outside stream
// capture it is looked up on every call (cheap, and right again after a
// cudaDeviceReset reloads the module); a call made while its stream is being
// captured uses the address cached by the last uncaptured call on the device.
static std::mutex g_scratch_mu;
static StaticScratch* g_scratch_ptr[64];

static StaticScratch* scratch_for_current_device(cudaStream_t st) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) return nullptr;
  std::lock_guard<std::mutex> lock(g_scratch_mu);
  if (cs == cudaStreamCaptureStatusNone) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_argmax_scratch) != cudaSuccess) return nullptr;
    g_scratch_ptr[dev] = static_cast<StaticScratch*>(p);
  }
  return g_scratch_ptr[dev];
}

struct StaticCall {
  const void* w;
  int V, H;
  const float* hidden;
  int T;
  StaticScratch* sc;
  int32_t* argmax;
  float *top1, *top2;
  cudaStream_t st;
};

template <typename E, int TT, int VEC>
static bool launch_static_tt(const StaticCall& c) {
  // one wave; a block's rows are whole row groups
  constexpr int R = StaticRows<E>::v;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return false;
  const int fit = static_blocks_per_sm(TT) * sms;
  const int most = fit < kStaticBlocks ? fit : kStaticBlocks;
  const int groups = c.V / R + (c.V % R != 0);
  const int rows = (groups + most - 1) / most * R;
  const int blocks = c.V / rows + (c.V % rows != 0);
  k_lm_argmax_static<E, TT, VEC><<<blocks, kStaticThreads, 0, c.st>>>((const E*)c.w, c.V, c.H, rows, c.hidden, c.T, c.sc,
                                                                     c.argmax, c.top1, c.top2);
  return cudaGetLastError() == cudaSuccess;
}

template <typename E>
static bool launch_static(const StaticCall& c) {
  // 16-byte loads where every row of both matrices starts on a 16-byte
  // boundary and a row group's offsets fit 32 bits (8 rows of up to 2^29 elements);
  // any other shape or address goes element by element, in 64 bits.
  if (c.H % 8 == 0 && c.H <= 1 << 29 && (((uintptr_t)c.w | (uintptr_t)c.hidden) & 15) == 0) {
    const int groups = (c.T + 7) / 8, tt = (c.T + groups - 1) / groups;   // the fewest groups, evenly filled
    if (tt <= 1) return launch_static_tt<E, 1, 8>(c);
    if (tt <= 2) return launch_static_tt<E, 2, 8>(c);
    if (tt <= 4) return launch_static_tt<E, 4, 8>(c);
    if (tt <= 6) return launch_static_tt<E, 6, 8>(c);
    return launch_static_tt<E, 8, 8>(c);
  }
  return launch_static_tt<E, 8, 1>(c);
}

}  // namespace oos

using namespace oos;

extern "C" int oos_lm_head_argmax_static(int32_t dtype, int32_t vocab, int32_t hidden_dim, const void* lm_head,
                                         const float* hidden, int32_t T, int32_t* out_argmax, float* out_top1,
                                         float* out_top2, void* stream) {
  if (!lm_head || !hidden || !out_argmax || !out_top1 || !out_top2) return OOS_EINVAL;
  if (dtype != OOS_DTYPE_F32 && dtype != OOS_DTYPE_BF16) return OOS_EINVAL;
  if (vocab < 1 || hidden_dim < 1) return OOS_EINVAL;
  if (T < 1 || T > kStaticMaxT) return OOS_EINVAL;   // the scratch array holds kStaticMaxT rows
  cudaStream_t st = (cudaStream_t)stream;
  StaticScratch* sc = scratch_for_current_device(st);
  if (!sc) return OOS_ECUDA;
  StaticCall c{lm_head, vocab, hidden_dim, hidden, T, sc, out_argmax, out_top1, out_top2, st};
  if (dtype == OOS_DTYPE_BF16) return launch_static<__nv_bfloat16>(c) ? OOS_OK : OOS_ECUDA;
  return launch_static<float>(c) ? OOS_OK : OOS_ECUDA;
}
