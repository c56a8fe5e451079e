// Weight-streaming GEMMs of the verify step.
//
// bf16 path (tcgen05): D[f, t] = sum_k W[f, k] * X[t, k] with the weight rows
// f in the MMA's M = 128 slot and the T tree nodes in N ("swap-AB": T <= 128
// is far too small for M).  Weights are the only large operand; each is read
// from HBM exactly once per step.  Per CTA: one TMA producer thread streams
// weight tiles of 64 k and the matching 64-wide slice of X through a
// shared-memory ring; one thread issues tcgen05.mma into a TMEM accumulator;
// eight epilogue warps drain TMEM with tcgen05.ld.
// The layer's elementwise steps run in the GEMM epilogues (see below); the LM
// head keeps a per-node running (max, argmax, second max) so logits never
// reach memory.
#include <string.h>

#include "common.cuh"
#include "internal.h"

// Step timeline (built only with -DOOS_TIMELINE, see timeline.py): per GEMM
// launch of a step and per CTA, the globaltimer at entry (0), at the end of the
// dependency wait (1), when the last accumulator is ready (2), when it is
// staged for the cluster (4), when every split's is (5) and at exit (3).  One
// slot per (layer, GEMM).
#ifdef OOS_TIMELINE
namespace oos {
__device__ unsigned long long g_tl_gemm[1024][160][6];
}
#define TL_GEMM(ev)                                                                   \
  do {                                                                                \
    if (!ARGMAX && blockIdx.x < 160)                                                  \
      oos::g_tl_gemm[a.tl_slot & 1023][blockIdx.x][ev] = oos::globaltimer();          \
  } while (0)
#else
#define TL_GEMM(ev) \
  do {              \
  } while (0)
#endif

namespace oos {

// Epilogues fused into the weight GEMMs (bf16 path):
//   EPI_QKV   : input RMSNorm scale, bias, per-head q/k RMSNorm, RoPE at
//               ctx + depth; q (hi/lo bf16) to the query buffer, k/v to cache
//               slot ctx + t.
//   EPI_RESID : x += W.a (O- and down-projections), then y = g (.) x for the
//               next RMSNorm (hi/lo bf16) and per-tile sums of x^2.
//   EPI_SILU  : a tile holds the same rows of gate and up; act = silu(r g) * (r u).
//   EPI_ARGMAX: LM head -- logits scaled by the final RMSNorm factor and folded
//               into a per-node running top-2.
// A prefill chunk too small for the tiles of prefill.cu runs through the same
// kernels in token tiles (CHUNK) of 128, or 64 for gate/up: the token tiles of a
// weight tile are separate clusters (or CTAs).  So does gate/up of a narrow model's
// tree of more than 64 nodes.
//
// RMSNorm is split across kernels by linearity: a producer stores y = g (.) x
// and sum(x^2) per feature tile; the consumer GEMM computes W.y and multiplies
// column t by r_t = rsqrt(sum x_t^2 / H + eps) in its epilogue.
//
// Work split.  Every matrix is cut into tiles of `rows` weight rows (a multiple
// of 8 up to the MMA's 128; the accumulator lanes past it hold sums of whatever
// follows in shared memory and are never read), see plan_cluster and plan_rows:
//   QKV, RESID: a thread-block cluster of `split` CTAs shares a tile, each CTA
//     one k-range of it.  Each stages its fp32 sums in its own shared memory
//     (over the ring, idle by then); after a cluster barrier CTA i pulls every
//     split's rows of its share of the tokens, adds them in split order (so the
//     result is the same from run to run) and finishes them.  Everything else
//     the epilogue reads (residual, rotary factors, norm sums) is loaded while
//     the weights stream.
//   SILU, ARGMAX: whole-K tiles, dealt round-robin (the weights of the next tile
//     stream while one is finished).  Above 64 tokens SILU runs in pairs of CTAs
//     (cta_group::2): two neighbouring tiles share one MMA, each CTA staging its
//     own weights and one activation half, hi or lo.  A CTA alone would be bound by
//     its shared memory there: per k-block its MMAs read 128 KB of operands and TMA
//     writes 56 (96 rows), against ~128 bytes a clock; in pairs 64 and 40.  Gate/up of
//     the 14336 x 4096 shape at T = 128: last accumulator 57 -> 50 us after the start.
//     Up to 64 tokens HBM is the bound (5.2 TB/s at 12288 x 4096, T = 64) and a pair's
//     setup costs more than it gives (8B step 4026 -> 4053 us, 0.6B 1277 -> 1304).
//     A narrow model's gate/up goes in tiles of 64 tokens instead (launch_gemm_gu).
enum { EPI_QKV = 0, EPI_RESID = 1, EPI_SILU = 2, EPI_ARGMAX = 3 };

// A work tile is SUB weight subtiles that share every staged activation slice:
// gate and up rows, or 2 x 128 rows of the LM head.
template <int EPI>
struct EpiOf {
  static constexpr int sub = (EPI == EPI_SILU || EPI == EPI_ARGMAX) ? 2 : 1;
  static constexpr bool cluster = EPI == EPI_QKV || EPI == EPI_RESID;
};

struct GemmArgs {
  int seg_tiles[3];   // EPI_QKV: cumulative tile counts of the q, k, v matrices
  int rows;           // weight rows per subtile
  int n_work, kbt;    // work tiles, k-blocks per tile
  int split;          // CTAs sharing a tile (cluster size)
  int chain;          // CHUNK: most k-blocks an accumulator collects (see k_chain)
  int stages;         // ring depth
  int N;              // output rows (features / vocab; intermediate rows for EPI_SILU)
  int T;              // valid columns (tree nodes; all token tiles together)
  int ldr;            // CHUNK: token rows the activation buffers are laid out for (else kMaxT)
  int tl_slot;        // timeline slot (layer * 4 + kind)
  uint32_t* status;
  // RMSNorm scale of the GEMM input (EPI_QKV, EPI_SILU, EPI_ARGMAX)
  const float* ss_in;   // [chunk][ldr]
  int ss_chunks;
  float inv_dim, eps;
  // EPI_QKV
  int nq, nkv;
  const __nv_bfloat16 *bq, *bk, *bv, *gq, *gk;
  const float2* rope;   // [ldr][64] (cos, sin) of the step's positions
  __nv_bfloat16 *q_out, *kc, *vc;
  const int32_t* ctx;   // committed length of the step (device; K/V of node t go to slot *ctx + t)
  int kv_f16;           // the KV cache (and so q) are binary16 instead of bf16
  // EPI_RESID
  float* x;
  const __nv_bfloat16* gain;
  __nv_bfloat16* y_out;
  float* ss_out;
  // EPI_SILU
  __nv_bfloat16* act_out;
  // EPI_ARGMAX
  float* am_v1;
  int32_t* am_i;
  float* am_v2;
};

// token rows of the activation buffers; the lo halves follow them
template <bool CHUNK>
OOS_DEV int ldr(const GemmArgs& a) { return CHUNK ? a.ldr : kMaxT; }

constexpr int kEpiWarps = 8;
constexpr int kEpiThreads = kEpiWarps * 32;
constexpr int kGemmThreads = 64 + kEpiThreads;
constexpr int kMaxStages = 12;
constexpr int kGemmSmemMax = 227 * 1024;

template <int BN, int EPI>
struct TcCfg {
  static constexpr int kSub = EpiOf<EPI>::sub;
  static constexpr int B_BYTES = BN * kBK * 2;                 // one activation half (hi or lo)
  static constexpr int BAR_BYTES = 256;
  static constexpr int EPI_BYTES = kMaxT * 4;                  // input RMSNorm factors
  static constexpr int RED_BYTES = EPI == EPI_ARGMAX ? 5 * BN * 12 : 0;   // argmax cross-warp scratch + running state
  static constexpr int HEAD = (BAR_BYTES + EPI_BYTES + RED_BYTES + 1023) / 1024 * 1024;   // what precedes the ring
  static constexpr int FIXED = 1024 /*align slack*/ + HEAD;
  // The hi and lo activation halves sit in one slot, hi rows then lo rows, so
  // one MMA with N = 2 BN multiplies both ("paired": half the MMAs, the weight
  // subtile read from shared memory once); the accumulator then holds the hi
  // products in columns [0, BN) and the lo products in [BN, 2 BN).  Paired
  // when the accumulator buffers then fit the 512 TMEM columns.
  static constexpr bool PAIR = EPI == EPI_SILU && BN == 128;
  static constexpr int BUFS = PAIR && 2 * kSub * 2 * BN > 512 ? 1 : 2;
  static constexpr bool PAIRED = BUFS * kSub * 2 * BN <= 512;
  static_assert(!PAIR || PAIRED, "a pair of CTAs splits the hi and lo halves");
  static constexpr int SUB_COLS = PAIRED ? 2 * BN : BN;        // accumulator columns per subtile
  static constexpr int NCOLS = BUFS * kSub * SUB_COLS < 32 ? 32 : BUFS * kSub * SUB_COLS;
  // k-segments of a tile with an accumulator each, added in fp32 by the
  // epilogue: the tensor core truncates every addition to its accumulator, an
  // error that grows with the chain, so the chains are kept short (one segment
  // where both buffers do not fit: 256 MMAs at K = 4096, hi and lo apart)
  static constexpr int SEGS = EPI == EPI_ARGMAX ? 1 : BUFS;
  // 16-token column chunks of an epilogue warp (`half`, `half` + 2, ...)
  static constexpr int CHUNKS = BN >= 32 ? BN / 32 : 1;
  static constexpr int X_BYTES = PAIR ? B_BYTES : 2 * B_BYTES;   // activations of a stage in this CTA
  static __host__ __device__ int stage_bytes(int rows) { return kSub * rows * kBK * 2 + X_BYTES; }
  static int stages(int rows) {
    const int s = (kGemmSmemMax - FIXED) / stage_bytes(rows);
    return s > kMaxStages ? kMaxStages : s;
  }
  // ring, or what the MMAs touch past the last weight subtile, or the staged tile
  static int smem(int rows) {
    const int s = stages(rows);
    int ring = s * stage_bytes(rows);
    const int reach = (s * kSub - 1) * rows * kBK * 2 + kTile * kBK * 2;
    if (ring < reach) ring = reach;
    if (EpiOf<EPI>::cluster && ring < BN * kTile * 4) ring = BN * kTile * 4;
    return FIXED + ring;
  }
};

OOS_DEV void epi_bar() { asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory"); }

OOS_DEV float4 f4_add(float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
OOS_DEV float4 ld_cluster_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}

OOS_DEV float4 bf16x4(const __nv_bfloat16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  const __nv_bfloat16* h = reinterpret_cast<const __nv_bfloat16*>(&u);
  return make_float4(__bfloat162float(h[0]), __bfloat162float(h[1]), __bfloat162float(h[2]), __bfloat162float(h[3]));
}

// RMSNorm factors of tokens [tb, te) of the token tile at tok0 into rms[], by the
// epilogue warps (w of kEpiWarps): lanes take the chunk sums, four tokens of a
// warp in flight.
template <bool CHUNK>
OOS_DEV void input_rms(const GemmArgs& a, float* rms, int tok0, int tb, int te, int w) {
  const int l = threadIdx.x & 31;
  for (int t0 = tb + 4 * w; t0 < te; t0 += 4 * kEpiWarps) {
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    for (int c = l; c < a.ss_chunks; c += 32) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (t0 + k < te) s[k] += __ldcg(a.ss_in + (size_t)c * ldr<CHUNK>(a) + tok0 + t0 + k);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) s[k] = warp_sum(s[k]);
    if (l == 0) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (t0 + k < te) rms[t0 + k] = rsqrtf(s[k] * a.inv_dim + a.eps);
    }
  }
}

// Finishing a tile of QKV or RESID: warp w of the eight epilogue warps owns
// token rows t = t0 + w + 8k, k < kFinRows, of a pass, lane l the four features
// 4l..4l+3 of the tile, so a token's features sit in one warp (RMSNorm sums,
// q/k norm and the RoPE pair exchange are warp shuffles).
constexpr int kFinRows = 4;
constexpr int kFinPass = kFinRows * kEpiWarps;

// acc[k] = sum over the cluster's CTAs, in rank order, of their staged row of
// token t0 + w + 8k (peer[s]: shared-memory address of CTA s's stage), SB CTAs' rows
// in flight
template <int SB>
OOS_DEV void pull_rows(float4 (&acc)[kFinRows], const uint32_t (&peer)[kMaxSplit], int split, int t0, int te, int w,
                       bool live) {
  const uint32_t off = (uint32_t)(threadIdx.x & 31) * 16;
#pragma unroll
  for (int k = 0; k < kFinRows; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int s0 = 0; s0 < kMaxSplit; s0 += SB) {
    if (s0 >= split) break;
    float4 v[SB][kFinRows];
#pragma unroll
    for (int s = 0; s < SB; ++s)
#pragma unroll
      for (int k = 0; k < kFinRows; ++k) {
        const int t = t0 + w + kEpiWarps * k;
        v[s][k] = (s0 + s < split && t < te && live) ? ld_cluster_f4(peer[s0 + s] + (uint32_t)t * (kTile * 4) + off)
                                                     : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
    for (int s = 0; s < SB; ++s)
#pragma unroll
      for (int k = 0; k < kFinRows; ++k) acc[k] = f4_add(acc[k], v[s][k]);
  }
}

// what a finishing pass of RESID reads from global memory
struct ResidRows {
  float4 x[kFinRows];
};
template <bool CHUNK>
OOS_DEV void resid_load(const GemmArgs& a, ResidRows& r, int f, bool live, int tok0, int t0, int te, int w) {
#pragma unroll
  for (int k = 0; k < kFinRows; ++k) {
    const int t = t0 + w + kEpiWarps * k;
    r.x[k] = (t < te && live) ? __ldcg(reinterpret_cast<const float4*>(a.x + (size_t)(tok0 + t) * a.N + f))
                              : make_float4(0.f, 0.f, 0.f, 0.f);
  }
}
// x += W.a; y = g (.) x; per-tile sums of x^2
template <bool CHUNK>
OOS_DEV void resid_finish(const GemmArgs& a, const ResidRows& r, const float4 (&acc)[kFinRows], float4 g, int tile, int f,
                          bool live, bool st, int tok0, int t0, int te, int w) {
  const int l = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < kFinRows; ++k) {
    const int t = t0 + w + kEpiWarps * k;
    if (t >= te) break;
    const float4 xv = f4_add(r.x[k], acc[k]);
    if (live && st) {
      *reinterpret_cast<float4*>(a.x + (size_t)(tok0 + t) * a.N + f) = xv;
      store_act4(a.y_out, (size_t)(tok0 + t) * a.N + f, (size_t)ldr<CHUNK>(a) * a.N,
                 make_float4(g.x * xv.x, g.y * xv.y, g.z * xv.z, g.w * xv.w));
    }
    const float sq = warp_sum(live ? xv.x * xv.x + xv.y * xv.y + xv.z * xv.z + xv.w * xv.w : 0.f);
    if (l == 0 && st) a.ss_out[(size_t)tile * ldr<CHUNK>(a) + tok0 + t] = sq;
  }
}

// what a finishing pass of QKV reads from global memory: the rotary factors
struct QkvRows {
  float2 cs[kFinRows][4];
};
template <bool CHUNK>
OOS_DEV void qkv_load(const GemmArgs& a, QkvRows& r, int kind, int tok0, int t0, int te, int w) {
  const int m0 = 4 * (threadIdx.x & 15);   // rotary frequency index of this lane's first feature
#pragma unroll
  for (int k = 0; k < kFinRows; ++k) {
    const int t = t0 + w + kEpiWarps * k;
    const bool ok = kind < 2 && t < te;
    const float4* p = reinterpret_cast<const float4*>(a.rope + (size_t)(tok0 + t) * (kTile / 2) + m0);
    const float4 u = ok ? __ldcg(p) : make_float4(1.f, 0.f, 1.f, 0.f);
    const float4 v = ok ? __ldcg(p + 1) : make_float4(1.f, 0.f, 1.f, 0.f);
    r.cs[k][0] = make_float2(u.x, u.y);
    r.cs[k][1] = make_float2(u.z, u.w);
    r.cs[k][2] = make_float2(v.x, v.y);
    r.cs[k][3] = make_float2(v.z, v.w);
  }
}
// one head (kind 0: q, 1: k, 2: v) of the tokens of a pass
template <bool CHUNK>
OOS_DEV void qkv_finish(const GemmArgs& a, const QkvRows& r, const float4 (&acc)[kFinRows], float4 b4, bool norm,
                        float4 g4, int kind, int h, int ctx, const float* rms, bool st, int tok0, int t0, int te, int w) {
  const int l = threadIdx.x & 31;
  const bool first_half = l < 16;   // features 0..63 pair with 64..127 held by lane ^ 16
#pragma unroll
  for (int k = 0; k < kFinRows; ++k) {
    const int t = t0 + w + kEpiWarps * k;
    if (t >= te) break;
    const float rt = rms[t];
    float v[4] = {acc[k].x * rt + b4.x, acc[k].y * rt + b4.y, acc[k].z * rt + b4.z, acc[k].w * rt + b4.w};
    if (norm) {   // per-head RMSNorm over the head's 128 features
      const float ss = warp_sum(v[0] * v[0] + v[1] * v[1] + v[2] * v[2] + v[3] * v[3]);
      const float rn = rsqrtf(ss * (1.f / kTile) + a.eps);
      v[0] *= rn * g4.x;
      v[1] *= rn * g4.y;
      v[2] *= rn * g4.z;
      v[3] *= rn * g4.w;
    }
    if (kind < 2) {   // rotate-half RoPE at position ctx + depth(t)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float other = __shfl_xor_sync(0xffffffffu, v[c], 16);
        v[c] = first_half ? v[c] * r.cs[k][c].x - other * r.cs[k][c].y : v[c] * r.cs[k][c].x + other * r.cs[k][c].y;
      }
    }
    if (!st) {
      asm volatile("" ::"f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]));
    } else if (kind == 0) {   // q as hi/lo halves in the cache's 16-bit format: the attention product sees ~16-bit q
      const size_t qi = ((size_t)(tok0 + t) * a.nq + h) * kTile + 4 * l, lo_off = (size_t)ldr<CHUNK>(a) * a.nq * kTile;
      if (a.kv_f16) store_act4_h(reinterpret_cast<__half*>(a.q_out), qi, lo_off, make_float4(v[0], v[1], v[2], v[3]));
      else store_act4(a.q_out, qi, lo_off, make_float4(v[0], v[1], v[2], v[3]));
    } else {           // K/V in the cache's format (bf16, or binary16)
      __nv_bfloat16* dst = (kind == 1 ? a.kc : a.vc) + ((size_t)(ctx + tok0 + t) * a.nkv + h) * kTile;
      uint2 o;
      if (a.kv_f16) {
        __half hv[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) hv[c] = __float2half_rn(v[c]);
        o = *reinterpret_cast<const uint2*>(hv);
      } else {
        __nv_bfloat16 bv[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) bv[c] = __float2bfloat16_rn(v[c]);
        o = *reinterpret_cast<const uint2*>(bv);
      }
      *reinterpret_cast<uint2*>(dst + 4 * l) = o;
    }
  }
}

template <int BN, int EPI, bool CHUNK>
__global__ void __launch_bounds__(kGemmThreads, 1)
    k_gemm_tc(const __grid_constant__ CUtensorMap wm0, const __grid_constant__ CUtensorMap wm1,
              const __grid_constant__ CUtensorMap wm2, const __grid_constant__ CUtensorMap am,
              const __grid_constant__ GemmArgs a) {
  using C = TcCfg<BN, EPI>;
  constexpr int kSub = C::kSub;
  constexpr bool ARGMAX = EPI == EPI_ARGMAX;
  constexpr bool CLUSTER = EpiOf<EPI>::cluster;
  constexpr bool PAIR = C::PAIR;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  // [barriers | RMSNorm factors | argmax state], then from `ring` on the weight
  // subtiles of every stage and after them the activation slices (hi, lo)
  const int S = a.stages;
  const int a_bytes = a.rows * kBK * 2;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem);
  uint64_t* empty = full + kMaxStages;
  uint64_t* accf = empty + kMaxStages;
  uint64_t* acce = accf + 2;
  uint64_t* drain = acce + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  static_assert((2 * kMaxStages + 5) * 8 + 12 <= C::BAR_BYTES, "barrier block");
  float* rms = reinterpret_cast<float*>(smem + C::BAR_BYTES);                                  // [kMaxT]
  Top2* red = reinterpret_cast<Top2*>(smem + C::BAR_BYTES + C::EPI_BYTES);                   // [4][BN]
  Top2* run = red + 4 * BN;                                                                   // [BN]
  unsigned char* ring = smem + C::HEAD;
  unsigned char* ring_x = ring + S * kSub * a_bytes;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // which use of its buffer the n-th accumulator is
  auto uses = [](uint32_t n) { return C::BUFS > 1 ? n >> 1 : n; };
  if (threadIdx.x == 0) TL_GEMM(0);

  // this CTA's work: k-blocks [kb0, kb0 + n_units) of tile `first` (cluster), or
  // all k-blocks of tiles first, first + step, ...
  int first, step, kb0, nkb, n_units, tok0 = 0;
  uint32_t rank = 0;
  if (CLUSTER) {
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    first = blockIdx.x / a.split;
    step = 0;
    if (CHUNK) {
      tok0 = first / a.n_work * BN;
      first %= a.n_work;
    }
    kb0 = a.kbt * (int)rank / a.split;
    nkb = n_units = a.kbt * ((int)rank + 1) / a.split - kb0;
  } else {
    if (PAIR) asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    first = blockIdx.x;
    step = gridDim.x;
    kb0 = 0;
    nkb = a.kbt;
    if (CHUNK) {   // one tile per CTA
      tok0 = first / a.n_work * BN;
      first %= a.n_work;
      n_units = a.kbt;
    } else {
      n_units = first < a.n_work ? (a.n_work - first + step - 1) / step * a.kbt : 0;
    }
  }
  const int T = CHUNK ? min(a.T - tok0, BN) : a.T;   // tokens of this CTA's tiles
  // k-segments of a tile: as many as it has accumulators, or (CHUNK) as the longest
  // chain makes, the accumulators taken in turn
  const int segs = CHUNK ? (nkb + a.chain - 1) / a.chain : nkb < C::SEGS ? 1 : C::SEGS;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], PAIR ? 2 * kEpiWarps : kEpiWarps);
    }
    mbar_init(drain, 1);
    abort_flag[0] = 0;
    abort_flag[1] = 0;
    mbar_fence_init();
  }
  if (warp == 2) {
    if (PAIR) tmem_alloc_pair(tmem_slot, C::NCOLS);
    else tmem_alloc(tmem_slot, C::NCOLS);
  }
  if (ARGMAX && threadIdx.x >= 64) {
    for (int e = threadIdx.x - 64; e < BN; e += kEpiThreads) run[e] = Top2{-INFINITY, 0x7fffffff, -INFINITY};
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (PAIR) {   // the other CTA's barriers are set up before anything arrives on them
    cluster_arrive_release();
    cluster_wait_acquire();
  }
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      tma_prefetch_desc(&wm0);
      tma_prefetch_desc(&am);
      const uint64_t pol_w = policy_evict_first();
      const uint64_t pol_a = policy_evict_last();
      const uint32_t stage_bytes = (uint32_t)(kSub * a_bytes + C::X_BYTES);
      // a pair's copies all complete on rank 0's barriers, which expect both CTAs' bytes
      const uint32_t full0 = PAIR ? dsmem_addr(full, 0) : 0u;
      auto load = [&](void* dst, const CUtensorMap* map, int stage, int x, int y, uint64_t pol) {
        if (PAIR) tma_load_2d_pair(dst, map, full0 + (uint32_t)stage * 8u, x, y, pol);
        else tma_load_2d(dst, map, &full[stage], x, y, pol);
      };
      auto expect = [&](int stage) {
        if (!PAIR) mbar_arrive_expect_tx(&full[stage], stage_bytes);
        else if (rank == 0) mbar_arrive_expect_tx(&full[stage], 2 * stage_bytes);
      };
      // weights of the unit at (tile, kb) into `stage`; rows past the matrix
      // read zeros (TMA out-of-bounds fill)
      auto load_sub = [&](const CUtensorMap* wm, unsigned char* dst, int kb, int row, int stage) {
        load(dst, wm, stage, kb * kBK, row, pol_w);
        if (CHUNK)   // the chunk's boxes are 64 rows high
          load(dst + 64 * kBK * 2, wm, stage, kb * kBK, row + 64, pol_w);
      };
      auto load_w = [&](int tile, int kb, int stage) {
        unsigned char* dst = ring + stage * kSub * a_bytes;
        if (EPI == EPI_SILU) {
          load_sub(&wm0, dst, kb, tile * a.rows, stage);
          load_sub(&wm1, dst + a_bytes, kb, tile * a.rows, stage);
        } else if (EPI == EPI_QKV) {
          const CUtensorMap* wm = tile < a.seg_tiles[0] ? &wm0 : tile < a.seg_tiles[1] ? &wm1 : &wm2;
          const int base = tile < a.seg_tiles[0] ? 0 : tile < a.seg_tiles[1] ? a.seg_tiles[0] : a.seg_tiles[1];
          load_sub(wm, dst, kb, (tile - base) * a.rows, stage);
        } else {
#pragma unroll
          for (int sub = 0; sub < kSub; ++sub)
            load_sub(&wm0, dst + sub * a_bytes, kb, (tile * kSub + sub) * a.rows, stage);
        }
      };
      auto load_x = [&](int kb, int stage) {
        unsigned char* dst = ring_x + stage * C::X_BYTES;
        if (!PAIR || rank == 0) load(dst, &am, stage, kb * kBK, tok0, pol_a);   // hi rows
        if (!PAIR || rank == 1)                                                // lo rows
          load(PAIR ? dst : dst + C::B_BYTES, &am, stage, kb * kBK, ldr<CHUNK>(a) + tok0, pol_a);
      };
      // weights do not depend on the previous kernel: start streaming them
      // before waiting for it (programmatic dependent launch)
      const int n_pre = n_units < S ? n_units : S;
      {
        int tile = first, kb = 0;
        for (int j = 0; j < n_pre; ++j) {
          expect(j);
          load_w(tile, kb0 + kb, j);
          if (++kb == nkb) {
            kb = 0;
            tile += step;
          }
        }
      }
      pdl_wait();
      pdl_trigger();
      TL_GEMM(1);
      int tile = first, kb = 0;
      auto advance = [&]() {
        if (++kb == nkb) {
          kb = 0;
          tile += step;
        }
      };
      for (int j = 0; j < n_pre; ++j) {
        load_x(kb0 + kb, j);
        advance();
      }
      int stage = n_pre % S;
      uint32_t phase = (n_pre == S) ? 1u : 0u;
      int issued = n_pre;
      for (int j = n_pre; j < n_units; ++j) {
        if (!mbar_wait(&empty[stage], phase ^ 1u, abort_flag, a.status)) break;
        expect(stage);
        load_w(tile, kb0 + kb, stage);
        load_x(kb0 + kb, stage);
        advance();
        ++issued;
        if (++stage == S) {
          stage = 0;
          phase ^= 1u;
        }
      }
      if (!PAIR || rank == 0) {
        // every copy this thread issued has landed before the CTA can exit,
        // whoever gave up (immediate on the normal path, where all were consumed;
        // after an abort of one CTA of a pair a phase may stay short of the
        // other's bytes, so the whole wait is bounded, well above a copy's time)
        const unsigned long long t0 = globaltimer(), most = PAIR ? 10000000ull : kWaitLimitNs;
        for (int j = issued - S > 0 ? issued - S : 0; j < issued; ++j) {
          while (!mbar_test(smem_addr(&full[j % S]), (uint32_t)((j / S) & 1)) && globaltimer() - t0 < most) {
          }
        }
      } else if (issued < n_units) {
        // rank 1 gave up: its last copies complete on rank 0's barriers, which may
        // never have expected them; they land long before this ends
        const unsigned long long t0 = globaltimer();
        while (globaltimer() - t0 < 200000ull) {
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0 && (!PAIR || rank == 0)) {
      constexpr uint32_t idesc = idesc_bf16_f32(PAIR ? 2 * kTile : kTile, C::PAIRED ? 2 * BN : BN);
      auto commit = [&](uint64_t* bar) {
        if (PAIR) tc_commit_pair(bar);
        else tc_commit(bar);
      };
      int stage = 0;
      uint32_t phase = 0;
      int acc = 0;
      uint32_t use = 0;   // accumulators handed over so far (two buffers in turn)
      bool ok = true;
      for (int j = 0; j < n_units && ok; j += nkb) {
        for (int sg = 0; sg < segs && ok; ++sg) {
          if (!mbar_wait(&acce[acc], (uses(use) & 1u) ^ 1u, abort_flag, a.status)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d0 = tmem_base + (uint32_t)(acc * kSub * C::SUB_COLS);
          const int n = nkb * (sg + 1) / segs - nkb * sg / segs;
          for (int jj = 0; jj < n; ++jj) {
            if (!mbar_wait(&full[stage], phase, abort_flag, a.status)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t wbase = smem_addr(ring + stage * kSub * a_bytes);
            const uint32_t xbase = smem_addr(ring_x + stage * C::X_BYTES);
            const uint64_t bh = smem_desc_sw128(xbase);
#pragma unroll
            for (int k = 0; k < kBK / 16; ++k) {
#pragma unroll
              for (int sub = 0; sub < kSub; ++sub) {
                const uint64_t ad = smem_desc_sw128(wbase + (uint32_t)(sub * a_bytes));
                const uint32_t d = d0 + (uint32_t)(sub * C::SUB_COLS);
                if (PAIR) tc_mma_bf16_pair(d, ad + 2 * k, bh + 2 * k, idesc, (jj > 0 || k > 0) ? 1u : 0u);
                else tc_mma_bf16(d, ad + 2 * k, bh + 2 * k, idesc, (jj > 0 || k > 0) ? 1u : 0u);
                if (!C::PAIRED) tc_mma_bf16(d, ad + 2 * k, smem_desc_sw128(xbase + C::B_BYTES) + 2 * k, idesc, 1u);
              }
            }
            commit(&empty[stage]);
            if (++stage == S) {
              stage = 0;
              phase ^= 1u;
            }
          }
          if (!ok) break;
          commit(&accf[acc]);
          ++use;
          if (C::BUFS > 1) acc ^= 1;
        }
      }
      // all issued MMAs complete before TMEM is released
      commit(drain);
      const unsigned long long t0 = globaltimer();
      while (!mbar_test(smem_addr(drain), 0) && globaltimer() - t0 < kWaitLimitNs) {
      }
    }
    __syncwarp();
  }

  // -------------------------------------------------------------- epilogue (warps 2..9)
  const int ew = warp - 2;              // epilogue warp 0..7
  const int q = warp & 3;               // TMEM lane quarter this warp may access
  const int half = ew >> 2;             // 16-token column chunks half, half + 2, ...
  const int row = q * 32 + lane;        // weight row of the tile
  const uint32_t lane_base = tmem_base + ((uint32_t)(q * 32) << 16);
  // 16 accumulator columns (tokens) starting at column `col`: paired hi + lo products
  auto acc16 = [&](uint32_t col, float (&v)[16]) {
    if (C::PAIRED) {
      float lo[16];
      tmem_ld16_nowait(lane_base + col, v);
      tmem_ld16_nowait(lane_base + col + BN, lo);
      tmem_wait_ld();
      reg_fence(v);
      reg_fence(lo);
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] += lo[i];
    } else {
      tmem_ld16(lane_base + col, v);
    }
  };

  // CHUNK: the k-segments before the last, added up in registers while the
  // MMAs of the next run: part[c][sub] is chunk c of this warp.  `use` counts the
  // accumulators taken.  False when a wait gave up.
  auto take_early = [&](float (&part)[C::CHUNKS][kSub][16], uint32_t& use) {
    for (int sg = 0; sg + 1 < segs; ++sg, ++use) {
      const uint32_t b = use & 1u;
      if (!__all_sync(0xffffffffu, mbar_wait(&accf[b], uses(use) & 1u, abort_flag, a.status))) return false;
      tc_fence_after();
#pragma unroll
      for (int c = 0; c < C::CHUNKS; ++c) {
        const int cc = half + 2 * c;
        if (cc * 16 >= T) continue;   // warp-uniform
#pragma unroll
        for (int sub = 0; sub < kSub; ++sub) {
          float v[16];
          acc16(b * (uint32_t)(kSub * C::SUB_COLS) + (uint32_t)(sub * C::SUB_COLS + cc * 16), v);
#pragma unroll
          for (int i = 0; i < 16; ++i) part[c][sub][i] = sg == 0 ? v[i] : part[c][sub][i] + v[i];
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acce[b]);
    }
    return true;
  };
  // chunk 0 of the sums leaves and the others move up: a window over registers in a
  // loop that is not unrolled
  auto next_chunk = [&](float (&part)[C::CHUNKS][kSub][16]) {
#pragma unroll
    for (int c = 0; c + 1 < C::CHUNKS; ++c)
#pragma unroll
      for (int sub = 0; sub < kSub; ++sub)
#pragma unroll
        for (int i = 0; i < 16; ++i) part[c][sub][i] = part[c + 1][sub][i];
  };

  if (CLUSTER && warp >= 2) {
    const int tile = first;
    // tokens [tb, te) are finished here
    const int tb = T * (int)rank / a.split, te = T * ((int)rank + 1) / a.split;
    const int f = EPI == EPI_RESID ? tile * a.rows + 4 * lane : 4 * lane;
    const bool live = 4 * lane < a.rows && (EPI != EPI_RESID || f < a.N);
    const bool two = nkb >= 2;   // one accumulator per k-segment, both read at the end
    int kind = 0, h = 0, ctx = 0;
    bool norm = false, have = false;
    float4 b4 = make_float4(0.f, 0.f, 0.f, 0.f), g4 = make_float4(1.f, 1.f, 1.f, 1.f);
    ResidRows rr;
    QkvRows qr;
    float* stage = reinterpret_cast<float*>(ring);   // [token][kTile]
    if (EPI == EPI_RESID) {
      if (live) g4 = bf16x4(a.gain + f);
    } else {
      if (tile < a.nq) { kind = 0; h = tile; }
      else if (tile < a.nq + a.nkv) { kind = 1; h = tile - a.nq; }
      else { kind = 2; h = tile - a.nq - a.nkv; }
      const __nv_bfloat16* bias = kind == 0 ? a.bq : kind == 1 ? a.bk : a.bv;
      const __nv_bfloat16* gn = kind == 0 ? a.gq : kind == 1 ? a.gk : nullptr;
      if (bias) b4 = bf16x4(bias + h * kTile + f);
      if (gn) g4 = bf16x4(gn + f);
      norm = gn != nullptr;
    }
    if (CHUNK) {
      pdl_wait();
      pdl_trigger();
      uint32_t use = 0;
      float part[C::CHUNKS][kSub][16];
      have = take_early(part, use);
      if (EPI == EPI_QKV) {
        ctx = *a.ctx;
        input_rms<CHUNK>(a, rms, tok0, tb, te, ew);
      }
      have = have && mbar_wait(&accf[use & 1u], uses(use) & 1u, abort_flag, a.status);
      have = __all_sync(0xffffffffu, have);
      tc_fence_after();
      // every MMA has read its operands: the ring is free for the sums
#pragma unroll 1
      for (int cc = half; cc < BN / 16; cc += 2) {
        if (cc * 16 >= T) break;
        float v[16];
        acc16((use & 1u) * (uint32_t)C::SUB_COLS + (uint32_t)(cc * 16), v);
        if (segs > 1) {
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] += part[0][0][i];
          next_chunk(part);
        }
        if (have && row < a.rows) {
#pragma unroll
          for (int i = 0; i < 16; ++i) stage[(cc * 16 + i) * kTile + row] = v[i];
        }
      }
      auto load = [&](int t0) {   // what a finishing pass reads
        if (EPI == EPI_RESID) resid_load<CHUNK>(a, rr, f, live, tok0, t0, te, ew);
        else qkv_load<CHUNK>(a, qr, kind, tok0, t0, te, ew);
      };
      load(tb);
      cluster_arrive_release();   // twice, as below
      __syncwarp();
      cluster_wait_acquire();
      uint32_t peer[kMaxSplit];
#pragma unroll
      for (int s = 0; s < kMaxSplit; ++s) peer[s] = dsmem_addr(stage, (uint32_t)(s < a.split ? s : 0));
#pragma unroll 1
      for (int t0 = tb;; t0 += kFinPass) {
        const bool last = t0 + kFinPass >= te;
        float4 acc[kFinRows];
        pull_rows<2>(acc, peer, a.split, t0, te, ew, live);
        if (last) cluster_arrive_release();
        if (EPI == EPI_RESID) resid_finish<CHUNK>(a, rr, acc, g4, tile, f, live, have, tok0, t0, te, ew);
        else qkv_finish<CHUNK>(a, qr, acc, b4, norm, g4, kind, h, ctx, rms, have, tok0, t0, te, ew);
        if (last) break;
        load(t0 + kFinPass);
      }
    }
    // Pass -1 is a dry run of the whole epilogue before the dependency wait:
    // no wait, barrier or store, values discarded.  The epilogue runs once per
    // launch, and the step's other kernels have evicted its code from the SM's
    // instruction caches since the previous layer; this fetches it while the
    // warps have nothing else to do.
#pragma unroll 1
    for (int pass = -1; !CHUNK; ++pass) {
      asm volatile("" : "+r"(pass));   // one copy of the body for every pass
      const bool dry = pass < 0;
      const int t0 = dry ? tb : tb + pass * kFinPass;
      if (pass > 0 && t0 >= te) break;
      if (pass == 0) {
        pdl_wait();
        pdl_trigger();
      }
      // what the finishing reads, while the weights stream
      if (EPI == EPI_RESID) {
        resid_load<CHUNK>(a, rr, f, live, tok0, t0, te, ew);
      } else {
        qkv_load<CHUNK>(a, qr, kind, tok0, t0, te, ew);
        if (pass <= 0) {
          ctx = *a.ctx;
          input_rms<CHUNK>(a, rms, tok0, tb, te, ew);
        }
      }
      if (pass <= 0) {
        if (!dry) {
          have = mbar_wait(&accf[0], 0, abort_flag, a.status) && (!two || mbar_wait(&accf[1], 0, abort_flag, a.status));
          have = __all_sync(0xffffffffu, have);
          if (threadIdx.x == 64) TL_GEMM(2);
          tc_fence_after();
        }
        // every MMA has read its operands: the ring is free for the sums
        const bool put = have && row < a.rows;
#pragma unroll 1
        for (int cc = half; cc < BN / 16; cc += 2) {
          if (cc * 16 >= T) break;
          float v[16];
          acc16((uint32_t)(cc * 16), v);
          if (two) {
            float v1[16];
            acc16((uint32_t)(C::SUB_COLS + cc * 16), v1);
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] += v1[i];
          }
          if (put) {
#pragma unroll
            for (int i = 0; i < 16; ++i) stage[(cc * 16 + i) * kTile + row] = v[i];
          }
        }
        if (!dry) {
          if (threadIdx.x == 64) TL_GEMM(4);
          // Every thread of the cluster arrives twice, whatever happened before:
          // when its sums are staged, and when it has pulled its share (a CTA's
          // stage must outlive its readers).
          cluster_arrive_release();
          __syncwarp();
          cluster_wait_acquire();
          if (threadIdx.x == 64) TL_GEMM(5);
        }
      }
      uint32_t peer[kMaxSplit];   // the dry run reads its own stage: the peers may not run yet
#pragma unroll
      for (int s = 0; s < kMaxSplit; ++s) peer[s] = dsmem_addr(stage, dry ? rank : (uint32_t)(s < a.split ? s : 0));
      float4 acc[kFinRows];
      pull_rows<4>(acc, peer, a.split, t0, te, ew, live);
      // the last pull: before this pass's stores, which the barrier then need not await
      if (!dry && t0 + kFinPass >= te) cluster_arrive_release();
      if (EPI == EPI_RESID) resid_finish<CHUNK>(a, rr, acc, g4, tile, f, live, have, tok0, t0, te, ew);
      else qkv_finish<CHUNK>(a, qr, acc, b4, norm, g4, kind, h, ctx, rms, have, tok0, t0, te, ew);
    }
    __syncwarp();
    cluster_wait_acquire();
  } else if (CLUSTER) {   // the producer's and the issuer's warps: their two arrivals
    cluster_arrive_release();
    __syncwarp();
    cluster_wait_acquire();
    cluster_arrive_release();
    __syncwarp();
    cluster_wait_acquire();
  } else if (!ARGMAX && warp >= 2) {
    // Gate and up of one row sit in the same lane, so act is formed in
    // registers.  Tile -1 is a dry run, as above.
    const bool two = !CHUNK && C::SEGS > 1 && nkb >= 2;
    const bool odd = lane & 1;
    const uint32_t acce0 = PAIR ? dsmem_addr(acce, 0) : 0u;   // rank 0's, where the issuer waits
    uint32_t use = 0;   // tiles drained
    uint32_t acc0 = 0;  // buffer of the tile's first k-segment (the second's is the other one)
#pragma unroll 1
    for (int it = CHUNK ? 0 : -1;; ++it) {
      asm volatile("" : "+r"(it));
      const bool dry = it < 0;
      const int tile = first + (dry ? 0 : it) * step;
      if (it == 0) {
        pdl_wait();
        pdl_trigger();
      }
      if (it <= 0) {
        input_rms<CHUNK>(a, rms, tok0, 0, T, ew);
        epi_bar();
      }
      float part[C::CHUNKS][kSub][16];
      if (CHUNK && !dry) {   // one tile a CTA
        if (it > 0 || !take_early(part, use) ||
            !__all_sync(0xffffffffu, mbar_wait(&accf[use & 1u], uses(use) & 1u, abort_flag, a.status)))
          break;
        tc_fence_after();
        acc0 = use & 1u;
      } else if (!dry) {
        if (it * nkb >= n_units) break;
        const bool ok = two ? mbar_wait(&accf[0], use & 1u, abort_flag, a.status) &&
                                  mbar_wait(&accf[1], use & 1u, abort_flag, a.status)
                            : mbar_wait(&accf[acc0], uses(use) & 1u, abort_flag, a.status);
        if (!__all_sync(0xffffffffu, ok)) break;
        if (threadIdx.x == 64 && (it + 1) * nkb >= n_units) TL_GEMM(2);
        tc_fence_after();
      }
      const uint32_t col0 = acc0 * (uint32_t)(kSub * C::SUB_COLS), col1 = (acc0 ^ 1u) * (uint32_t)(kSub * C::SUB_COLS);
      const int fi = tile * a.rows + (row & ~1);
      const bool live = row < a.rows && fi < a.N && !dry;
#pragma unroll 1
      for (int cc = half; cc < BN / 16; cc += 2) {
        if (cc * 16 >= T) break;
        float g[16], u[16];
        acc16(col0 + cc * 16, g);
        acc16(col0 + C::SUB_COLS + cc * 16, u);
        if (CHUNK && !dry && segs > 1) {
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            g[i] += part[0][0][i];
            u[i] += part[0][kSub - 1][i];
          }
          next_chunk(part);
        }
        if (two) {
          float v[16];
          acc16(col1 + cc * 16, v);
#pragma unroll
          for (int i = 0; i < 16; ++i) g[i] += v[i];
          acc16(col1 + C::SUB_COLS + cc * 16, v);
#pragma unroll
          for (int i = 0; i < 16; ++i) u[i] += v[i];
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float r = rms[cc * 16 + i];
          u[i] = silu(g[i] * r) * (u[i] * r);
        }
        // lane pairs swap tokens so that a store covers two neighbouring features
#pragma unroll
        for (int i = 0; i < 16; i += 2) {
          const float mine = odd ? u[i + 1] : u[i];
          const float other = __shfl_xor_sync(0xffffffffu, odd ? u[i] : u[i + 1], 1);
          const float v0 = odd ? other : mine, v1 = odd ? mine : other;   // features row & ~1, row | 1
          const int t = cc * 16 + i + (odd ? 1 : 0);
          const __nv_bfloat162 hi = __floats2bfloat162_rn(v0, v1);
          const __nv_bfloat162 lo = __floats2bfloat162_rn(v0 - __low2float(hi), v1 - __high2float(hi));
          if (live && t < T) {
            __nv_bfloat16* dst = a.act_out + (size_t)(tok0 + t) * a.N + fi;
            *reinterpret_cast<__nv_bfloat162*>(dst) = hi;
            *reinterpret_cast<__nv_bfloat162*>(dst + (size_t)ldr<CHUNK>(a) * a.N) = lo;
          }
        }
      }
      if (!dry && !CHUNK) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          for (uint32_t b = acc0;; b ^= 1u) {
            if (PAIR) mbar_arrive_remote(acce0 + 8u * b);
            else mbar_arrive(&acce[b]);
            if (!two || b != acc0) break;
          }
        }
        ++use;
        if (!two && C::BUFS > 1) acc0 ^= 1u;
      }
    }
  } else if (warp >= 2) {
    pdl_wait();
    pdl_trigger();
    const int e = threadIdx.x - 64;       // 0..kEpiThreads-1
    input_rms<CHUNK>(a, rms, tok0, 0, T, ew);
    epi_bar();
    int acc = 0;
    uint32_t use = 0;
    for (int j = 0, tile = first; j < n_units; j += nkb, tile += step) {
      mbar_wait(&accf[acc], (use >> 1) & 1u, abort_flag, a.status);
      // the barriers below need every epilogue warp on one path: all of them
      // leave on one sample of the flag
      epi_bar();
      if (e == 0) abort_flag[1] = abort_flag[0];
      epi_bar();
      if (abort_flag[1]) break;
      tc_fence_after();
      const uint32_t col0 = (uint32_t)(acc * kSub * C::SUB_COLS);
#pragma unroll 1
      for (int sub = 0; sub < kSub; ++sub) {
        const int f = (tile * kSub + sub) * kTile + row;
#pragma unroll 1
        for (int cc = half; cc < BN / 16; cc += 2) {
          if (cc * 16 >= T) break;
          float v[16];
          acc16(col0 + sub * C::SUB_COLS + cc * 16, v);
          // Top 2 over the warp's 32 rows, the 16 tokens folded over the lanes: each
          // exchange halves the tokens a lane still holds, 16 merges.  With every lane
          // reducing every token (80) the epilogue of the last tile, and at T = 128 that
          // of every tile, was what the weights waited for: 151936 x 4096 at T = 1 / 64
          // 182.7 / 193.2 -> 177.4 / 182.5 us, 128256 x 4096 at T = 128 234 -> 205.
          Top2 s[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) s[i] = Top2{f < a.N ? v[i] * rms[cc * 16 + i] : -INFINITY, f, -INFINITY};
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            const bool up = lane & o;
            const int n = o / 2;   // tokens kept (0: the last one, by both lanes)
#pragma unroll
            for (int i = 0; i < (n ? n : 1); ++i) {
              const Top2 give = n && !up ? s[i + n] : s[i];
              const Top2 keep = n && up ? s[i + n] : s[i];
              Top2 y;
              y.v1 = __shfl_xor_sync(0xffffffffu, give.v1, o);
              y.i1 = __shfl_xor_sync(0xffffffffu, give.i1, o);
              y.v2 = __shfl_xor_sync(0xffffffffu, give.v2, o);
              s[i] = top2_merge(keep, y);
            }
          }
          if (!(lane & 1)) {
            Top2* slot = &red[q * BN + cc * 16 + lane / 2];
            *slot = sub == 0 ? s[0] : top2_merge(*slot, s[0]);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acce[acc]);
      epi_bar();
      if (e < T) {
        Top2 r = run[e];
#pragma unroll
        for (int w = 0; w < 4; ++w) r = top2_merge(r, red[w * BN + e]);
        run[e] = r;
      }
      epi_bar();
      ++use;
      acc ^= 1;
    }
    if (e < T) {
      const Top2 r = run[e];
      a.am_v1[(size_t)blockIdx.x * kMaxT + e] = r.v1;
      a.am_i[(size_t)blockIdx.x * kMaxT + e] = r.i1;
      a.am_v2[(size_t)blockIdx.x * kMaxT + e] = r.v2;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0) TL_GEMM(3);
  if (PAIR) {   // neither CTA leaves while the other's MMAs, copies or arrivals may reach it
    cluster_arrive_release();
    cluster_wait_acquire();
  }
  if (warp == 2) {
    tc_fence_after();
    if (PAIR) tmem_dealloc_pair(tmem_base, C::NCOLS);
    else tmem_dealloc(tmem_base, C::NCOLS);
  }
}

// ------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn get_encode() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

static bool encode_2d(CUtensorMap* map, const void* ptr, int rows, int K, int box_rows) {
  EncodeTiledFn enc = get_encode();
  if (!enc) return false;
  memset(map, 0, sizeof(*map));
  cuuint64_t gdim[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  cuuint64_t gstride[1] = {(cuuint64_t)K * 2};
  cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), gdim, gstride, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

bool encode_bf16_map(CUtensorMap* map, const void* ptr, int rank, const uint64_t* dims, const uint64_t* strides,
                     const uint32_t* box, bool f16) {
  EncodeTiledFn enc = get_encode();
  if (!enc || rank < 1 || rank > 5) return false;
  memset(map, 0, sizeof(*map));
  cuuint64_t gdim[5], gstride[4];
  cuuint32_t bx[5], estr[5];
  for (int i = 0; i < rank; ++i) {
    gdim[i] = dims[i];
    bx[i] = box[i];
    estr[i] = 1;
    if (i + 1 < rank) gstride[i] = strides[i];
  }
  CUresult r = enc(map, f16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank,
                   const_cast<void*>(ptr), gdim, gstride, bx,
                   estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

bool encode_rows_map(CUtensorMap* map, const void* ptr, int rows, int K, int box_rows) {
  return encode_2d(map, ptr, rows, K, box_rows);
}
bool encode_act_map(CUtensorMap* map, const void* ptr, int K, int box_rows) {
  return encode_2d(map, ptr, 2 * kMaxT, K, box_rows);   // hi rows [0, 128), lo rows [128, 256)
}

int bn_index(int T) { return T <= 16 ? 0 : T <= 32 ? 1 : T <= 64 ? 2 : 3; }

template <int BN, int EPI, bool CHUNK = false>
static cudaError_t set_smem() {
  // the depth of the ring, and so the size, depends on the plan's tile rows:
  // allow the most any plan takes
  return cudaFuncSetAttribute(k_gemm_tc<BN, EPI, CHUNK>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGemmSmemMax);
}

template <int BN>
static cudaError_t set_smem_all() {
  cudaError_t e = set_smem<BN, EPI_QKV>();
  if (e == cudaSuccess) e = set_smem<BN, EPI_RESID>();
  if (e == cudaSuccess) e = set_smem<BN, EPI_SILU>();
  if (e == cudaSuccess) e = set_smem<BN, EPI_ARGMAX>();
  return e;
}

cudaError_t gemm_setup() {
  cudaError_t e = set_smem_all<16>();
  if (e == cudaSuccess) e = set_smem_all<32>();
  if (e == cudaSuccess) e = set_smem_all<64>();
  if (e == cudaSuccess) e = set_smem_all<128>();
  if (e == cudaSuccess) e = set_smem<128, EPI_QKV, true>();
  if (e == cudaSuccess) e = set_smem<128, EPI_RESID, true>();
  if (e == cudaSuccess) e = set_smem<64, EPI_SILU, true>();
  return e;
}

// Clusters of `c` GEMM CTAs resident at once (one CTA per SM).  Not every place the
// occupancy query counts is free when the clusters arrive (odd sizes leave SM
// pairs half used, and the previous kernel's CTAs go one by one), and a cluster
// left over runs after all the others: 46 clusters of 3 took 98 us where 43 take
// 55, so a margin is kept.
int gemm_fit(int c) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(c);
  lc.blockDim = dim3(kGemmThreads);
  lc.dynamicSmemBytes = kGemmSmemMax;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = c;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  lc.attrs = attr;
  lc.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, (const void*)k_gemm_tc<64, EPI_RESID, false>, &lc) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  if (c > 1) n -= (c & 1) ? (n + 11) / 12 : 1;
  return n;
}

// k-blocks that one accumulator may collect where K goes in segments (CHUNK, prefill.cu).  The tensor core
// truncates every addition to its accumulator, an error that grows with the chain of
// MMAs, so K goes in chains no longer than the pieces that an even deal of the matrix's
// k-blocks over the SMs would cut (8B shape: q/k/v 15, O 11, down 33, gate/up 24; 0.6B:
// two each), added in fp32 registers.  A small matrix has short chains, which its
// latency mostly hides.  Four MMAs a k-block where the hi and lo products have columns
// of their own.  Error of the first layer's V (mostly bf16 values rounded the other
// way) of 2048 tokens with the 0.6B / 8B shape: 1.1e-4 / 1.0e-4 in chains of 128 MMAs,
// 2.4e-5 / 7.2e-5 so.  One layer of the 0.6B shape, 333 tokens: 77 -> 86 us.
int k_chain(int rows, int K, int n_sms) {
  const int tiles = (rows + kTile - 1) / kTile, kbt = K / kBK;
  const int kb = tiles * kbt / (tiles + n_sms);
  return kb < 2 ? 2 : kb;
}

// Tile rows and k-split of a QKV (rows fixed at one head) or RESID GEMM: of the
// splits whose clusters fit the GPU, the one whose CTAs move the fewest bytes in
// sequence, weights and activations (for 64 nodes) together, with a charge per
// split for the sums it pulls and one per extra wave for a second prologue and
// epilogue (~8 us at ~80 KB/us).  Tiles are cut below the MMA's 128 rows only when
// every cluster that fits then has one of at least kMinCut: a CTA stages the whole
// activation slice however few its rows.  O and down of the 0.6B shape as 32 rows x 4
// splits and 48 x 6 took 2.8 / 2.5 / 2.1 / 8.5 us more per layer at T = 1 / 32 / 64 / 128
// than as 128 x 8; 4096 rows as 120 x 4 take 0.7 us less than as 128 x 4 (T = 64).
constexpr int kMinCut = 112;   // 7/8 of the MMA's rows
GemmPlan plan_cluster(int N, int K, bool whole_heads) {
  GemmPlan best = {};
  long long best_cost = -1;
  const int kbt = K / kBK;
  for (int c = 1; c <= kMaxSplit && c <= kbt; ++c) {
    const int fit = gemm_fit(c);
    if (fit < 1) continue;
    const int even = ((N + fit - 1) / fit + 7) / 8 * 8;   // rows that give every cluster a tile
    const int rows = !whole_heads && even >= kMinCut && even < kTile ? even : kTile;
    const int n_work = (N + rows - 1) / rows;
    const long long waves = (n_work + fit - 1) / fit;
    const long long cost = waves * ((kbt + c - 1) / c) * (rows * 128 + 16384) + (long long)c * 16384 +
                           (waves - 1) * 640 * 1024;
    if (best_cost < 0 || cost < best_cost) {
      best_cost = cost;
      best = GemmPlan{rows, n_work, kbt, c, n_work * c};
    }
  }
  return best;
}

// Whole-K tiles (gate/up: `rows` of each matrix per tile), an even number, since they
// go to pairs of CTAs; the last may lie past the matrix (zeros).  Tiles of 128 rows
// where one round of them takes up to half the SMs (a short stream: the fewer CTAs
// stage the activations, and the next kernel's CTAs start on the SMs left) or at least
// 7 in 10 (enough to draw the full bandwidth).  Else tiles of equal rows that fill
// the SMs in as few rounds as 128 rows allow.  Per layer, 128 rows against the even
// cut at T = 1 / 32 / 64 / 128: 3072 rows (24 tiles against 128) -1.3 / -2.8 / -5.0 /
// -10.8 us, 9728 (76, 152) -1.0 / -1.8 / -2.2 / -1.6, 14336 (112, 150) 0 / -2.6 / -1.0 /
// -1.3; between the lines, 12288 (96, 140), +1.6 / +1.0 / -0.2 / -1.3.
GemmPlan plan_rows(int N, int K, int n_sms) {
  n_sms &= ~1;
  const int rounds = (N + kTile * n_sms - 1) / (kTile * n_sms), full = (N + kTile - 1) / kTile;
  int rows = kTile;
  if (rounds > 1 || (2 * full > n_sms && 10 * full < 7 * n_sms))
    rows = ((N + rounds * n_sms - 1) / (rounds * n_sms) + 7) / 8 * 8;
  const int n_work = ((N + rows - 1) / rows + 1) & ~1;
  return GemmPlan{rows, n_work, K / kBK, 1, n_work < n_sms ? n_work : n_sms};
}

// grid: CTAs, `split` times the tiles for the cluster GEMMs
template <int BN, int EPI, bool CHUNK = false>
static cudaError_t launch_tc(Model& m, const GemmW& g, const CUtensorMap& amap, int grid, GemmArgs& a, cudaStream_t st) {
  using C = TcCfg<BN, EPI>;
  a.stages = C::stages(a.rows);
  const CUtensorMap* maps = CHUNK ? g.pf_map : g.map;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(grid);
  lc.blockDim = dim3(kGemmThreads);
  lc.dynamicSmemBytes = (size_t)C::smem(a.rows);
  lc.stream = st;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (EpiOf<EPI>::cluster || C::PAIR) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = C::PAIR ? 2 : a.split;
    attr[n].val.clusterDim.y = 1;
    attr[n].val.clusterDim.z = 1;
    ++n;
  }
  if (m.pdl) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  lc.attrs = attr;
  lc.numAttrs = n;
  const CUtensorMap& w1 = g.n_seg > 1 ? maps[1] : maps[0];
  const CUtensorMap& w2 = g.n_seg > 2 ? maps[2] : maps[0];
  return cudaLaunchKernelEx(&lc, k_gemm_tc<BN, EPI, CHUNK>, maps[0], w1, w2, amap, a);
}

template <int EPI>
static cudaError_t dispatch_tc(Model& m, const GemmW& g, const CUtensorMap* amaps, int T, GemmArgs& a,
                               cudaStream_t st) {
  switch (bn_index(T)) {
    case 0: return launch_tc<16, EPI>(m, g, amaps[0], g.plan.grid, a, st);
    case 1: return launch_tc<32, EPI>(m, g, amaps[1], g.plan.grid, a, st);
    case 2: return launch_tc<64, EPI>(m, g, amaps[2], g.plan.grid, a, st);
    default: return launch_tc<128, EPI>(m, g, amaps[3], g.plan.grid, a, st);
  }
}

static GemmArgs base_args(Model& m, const GemmW& g, int T, int slot) {
  GemmArgs a;
  memset(&a, 0, sizeof(a));
  a.rows = g.plan.rows;
  a.n_work = g.plan.n_work;
  a.kbt = g.plan.kbt;
  a.split = g.plan.split;
  a.chain = g.chain;
  a.N = g.N;
  a.T = T;
  a.tl_slot = slot;
  a.status = m.ws.status;
  a.ss_in = m.ws.ss;
  a.inv_dim = 1.0f / (float)m.cfg.hidden;
  a.eps = m.cfg.rms_eps;
  return a;
}

// number of sum-of-squares chunks the input of layer `layer`'s attention block
// comes with (layer n_layers: the final norm's): the embedding writes one per
// 128 features, a down projection one per tile
int norm_chunks(const Model& m, int layer) {
  return layer == 0 ? (m.cfg.hidden + kTile - 1) / kTile : m.g_down[layer - 1].plan.n_work;
}

static GemmArgs qkv_args(Model& m, int layer, void* kc, void* vc, int T) {
  const auto& c = m.cfg;
  const oos_layer_weights& L = m.layers[layer];
  GemmArgs a = base_args(m, m.g_qkv[layer], T, layer * 4);
  a.seg_tiles[0] = c.n_q_heads;
  a.seg_tiles[1] = c.n_q_heads + c.n_kv_heads;
  a.seg_tiles[2] = c.n_q_heads + 2 * c.n_kv_heads;
  a.ss_chunks = norm_chunks(m, layer);
  a.nq = c.n_q_heads;
  a.nkv = c.n_kv_heads;
  a.bq = (const __nv_bfloat16*)(c.qkv_bias ? L.b_q : nullptr);
  a.bk = (const __nv_bfloat16*)(c.qkv_bias ? L.b_k : nullptr);
  a.bv = (const __nv_bfloat16*)(c.qkv_bias ? L.b_v : nullptr);
  a.gq = (const __nv_bfloat16*)(c.qk_norm ? L.q_norm : nullptr);
  a.gk = (const __nv_bfloat16*)(c.qk_norm ? L.k_norm : nullptr);
  a.rope = m.ws.rope;
  a.q_out = (__nv_bfloat16*)m.ws.q;
  a.kc = (__nv_bfloat16*)kc;
  a.vc = (__nv_bfloat16*)vc;
  a.ctx = m.ws.ctx;
  a.kv_f16 = c.kv_f16 ? 1 : 0;
  return a;
}

cudaError_t launch_gemm_qkv(Model& m, int layer, void* kc, void* vc, int T, cudaStream_t st) {
  GemmArgs a = qkv_args(m, layer, kc, vc, T);
  return dispatch_tc<EPI_QKV>(m, m.g_qkv[layer], m.amap_xn, T, a, st);
}

static cudaError_t launch_resid(Model& m, const GemmW& g, const CUtensorMap* amaps, const void* gain, int slot, int T,
                                cudaStream_t st) {
  GemmArgs a = base_args(m, g, T, slot);
  a.x = m.ws.x;
  a.gain = (const __nv_bfloat16*)gain;
  a.y_out = (__nv_bfloat16*)m.ws.xn;
  a.ss_out = m.ws.ss;
  return dispatch_tc<EPI_RESID>(m, g, amaps, T, a, st);
}

cudaError_t launch_gemm_o(Model& m, int layer, int T, cudaStream_t st) {
  return launch_resid(m, m.g_o[layer], m.amap_attn, m.layers[layer].mlp_norm, layer * 4 + 1, T, st);
}

cudaError_t launch_gemm_down(Model& m, int layer, int T, cudaStream_t st) {
  const void* gain = layer + 1 < m.cfg.n_layers ? m.layers[layer + 1].attn_norm : m.w.final_norm;
  return launch_resid(m, m.g_down[layer], m.amap_act, gain, layer * 4 + 3, T, st);
}

cudaError_t launch_gemm_gu(Model& m, int layer, int T, cudaStream_t st) {
  GemmArgs a = base_args(m, m.g_gu[layer], T, layer * 4 + 2);
  a.ss_chunks = m.g_o[layer].plan.n_work;
  a.act_out = (__nv_bfloat16*)m.ws.act;
  // Above 64 tokens, where tiles of 64 tokens x 128 rows leave SMs free: chains of
  // k_chain, where a pair's single accumulator collects all of K (an MLP's error, its
  // attention off: 2048 x 6144 6.3e-6 in pairs, 5.6e-6 so, 5.7e-6 in trees of 64; from 76
  // tiles on the pairs' is no larger than the even deal's would be).  A layer at T = 65 / 128:
  // 6144 rows 69.3 -> 67.2 / 82.4 -> 79.9 us, 3072 52.7 -> 54.3 / 64.1 -> 64.4.
  const int tiles = a.N / kTile;
  if (T > 64 && 2 * tiles < m.num_sms) {
    a.rows = kTile;
    a.n_work = tiles;
    a.ldr = kMaxT;
    return launch_tc<64, EPI_SILU, true>(m, m.g_gu[layer], m.amap_xn[2], 2 * tiles, a, st);
  }
  return dispatch_tc<EPI_SILU>(m, m.g_gu[layer], m.amap_xn, T, a, st);
}

// ---- a prefill chunk in token tiles (prefill.cu chooses between these and its own
// tiles): 128 weight rows a tile, buffers of kPfTokens rows, norm sums per 128
// features as prefill.cu writes them
static void chunk_args(Model& m, GemmArgs& a, int n_work, int split) {
  a.rows = kTile;
  a.n_work = n_work;
  a.split = split;
  a.ldr = kPfTokens;
  a.ss_in = m.ws.pf_ss;
  a.ss_chunks = m.cfg.hidden / kTile;
}
static int chunk_tiles(const GemmArgs& a, int tokens) { return a.n_work * ((a.T + tokens - 1) / tokens); }
cudaError_t launch_chunk_qkv(Model& m, int layer, void* kc, void* vc, int T, int split, cudaStream_t st) {
  GemmArgs a = qkv_args(m, layer, kc, vc, T);
  chunk_args(m, a, m.cfg.n_q_heads + 2 * m.cfg.n_kv_heads, split);
  a.rope = m.ws.pf_rope;
  a.q_out = (__nv_bfloat16*)m.ws.pf_q;
  return launch_tc<128, EPI_QKV, true>(m, m.g_qkv[layer], m.pf_xn_map, chunk_tiles(a, 128) * split, a, st);
}
cudaError_t launch_chunk_resid(Model& m, int layer, bool down, const void* gain, int T, int split, cudaStream_t st) {
  const GemmW& g = down ? m.g_down[layer] : m.g_o[layer];
  GemmArgs a = base_args(m, g, T, layer * 4 + (down ? 3 : 1));
  chunk_args(m, a, g.N / kTile, split);
  a.x = m.ws.pf_x;
  a.gain = (const __nv_bfloat16*)gain;
  a.y_out = (__nv_bfloat16*)m.ws.pf_xn;
  a.ss_out = m.ws.pf_ss;
  return launch_tc<128, EPI_RESID, true>(m, g, down ? m.pf_act_map : m.pf_attn_map, chunk_tiles(a, 128) * split, a, st);
}
// 64 tokens a tile: the registers hold the segments' sums of gate and up
cudaError_t launch_chunk_gu(Model& m, int layer, int T, cudaStream_t st) {
  const GemmW& g = m.g_gu[layer];
  GemmArgs a = base_args(m, g, T, layer * 4 + 2);
  chunk_args(m, a, g.N / kTile, 1);
  a.act_out = (__nv_bfloat16*)m.ws.pf_act;
  return launch_tc<64, EPI_SILU, true>(m, g, m.pf_xn64_map, chunk_tiles(a, 64), a, st);
}

cudaError_t launch_lm_head_tc(Model& m, int T, cudaStream_t st) {
  GemmArgs a = base_args(m, m.g_lm, T, 0);
  a.ss_chunks = norm_chunks(m, m.cfg.n_layers);
  a.am_v1 = m.ws.lm_v1;
  a.am_i = m.ws.lm_i;
  a.am_v2 = m.ws.lm_v2;
  return dispatch_tc<EPI_ARGMAX>(m, m.g_lm, m.amap_xn, T, a, st);
}

}  // namespace oos

#ifdef OOS_TIMELINE
// timeline accessors (the OOS_TIMELINE library only)
extern "C" int oos_timeline_gemm_read(void* out, size_t bytes) {
  return cudaMemcpyFromSymbol(out, oos::g_tl_gemm, bytes < sizeof(oos::g_tl_gemm) ? bytes : sizeof(oos::g_tl_gemm)) ==
                 cudaSuccess
             ? 0
             : OOS_ECUDA;
}
extern "C" int oos_timeline_gemm_clear() {
  void* p = nullptr;
  if (cudaGetSymbolAddress(&p, oos::g_tl_gemm) != cudaSuccess) return OOS_ECUDA;
  return cudaMemset(p, 0, sizeof(oos::g_tl_gemm)) == cudaSuccess ? 0 : OOS_ECUDA;
}
#endif
