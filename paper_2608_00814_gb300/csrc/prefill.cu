// Target prefill of the bf16 path: chunks of up to kPfTokens prompt tokens
// through the decoder, causal attention over the cache and the chunk.
//
// A chunk of a thousand tokens has the arithmetic intensity the verify step
// lacks, so its GEMMs are compute-bound and tiled the ordinary way: tokens in the
// MMA's M, 256 weight rows in N.  The activations keep their two bf16 halves,
// so every k-step is two MMAs on the same weights.  The tensor core truncates each
// addition to its accumulator, an error that grows with the chain, so K goes in
// segments whose sums the epilogue warps add in fp32 registers, as long as k_chain
// (gemm.cu) has them.  A segment costs 0.6 us: four layers of the 8B shape, 2048
// tokens, take 4714 us in segments of 16 k-blocks (128 MMAs) and 4802 so (64 MMAs for
// q/k/v, 48 for O).
// A tile goes to a pair of CTAs (cta_group::2): 256 tokens, each CTA staging its 128
// and half the weight rows.  A CTA alone would stage 64 KB per k-block and read 96 KB
// of MMA operands in the 1024 clocks of its MMAs, more than its shared memory and its
// share of L2 give; in a pair 48 and 64 (four layers of the 8B shape, 2048 tokens:
// 5138 us in single CTAs, 4666 in pairs).
// Persistent pairs, one CTA per SM: one TMA producer thread, one MMA issuer, eight
// epilogue warps; two accumulators in tensor memory, so a segment is drained, and a
// tile finished, under the next one's MMAs.
//
// With tokens in M a token is one TMEM lane, so a thread holds a token's 128
// features of a head or residual tile: the q/k norm, the rotary pairs and the
// RMSNorm sums need no exchange between threads.  The epilogues are those of the
// verify GEMMs (gemm.cu): bias, q/k norm, RoPE and the cache format; residual add,
// next norm's gain and sums; SwiGLU.
#include <string.h>

#include "common.cuh"
#include "internal.h"

namespace oos {

constexpr int kPfRows = 128;                      // tokens per tile
constexpr int kPfHalf = kPfRows * kBK * 2;        // bytes of one activation half per stage
constexpr int kPfEpiWarps = 8;
constexpr int kPfThreads = 128 + 32 * kPfEpiWarps;   // a warp group for the producer and the issuer
// registers a thread keeps in each role (setmaxnreg): 128 * 56 + 256 * 224 of the
// 384 * 168 the block is launched with
constexpr int kPfRegsIssue = 56, kPfRegsEpi = 224, kPfRegsLaunch = 168;
static_assert(128 * kPfRegsIssue + 32 * kPfEpiWarps * kPfRegsEpi <= kPfThreads * kPfRegsLaunch, "register split");

constexpr int kPfCols = 256;                      // weight rows per tile
constexpr int kPfStage = 2 * kPfHalf + kPfCols / 2 * kBK * 2;   // a CTA's activations and half the weight rows
constexpr int kPfStages = (227 * 1024 - 2048) / kPfStage;
constexpr int kPfSmem = 2048 + kPfStages * kPfStage;   // alignment slack + barriers
constexpr int kPfTmem = 512;                      // two accumulators

enum { PF_QKV = 0, PF_RESID = 1, PF_SILU = 2 };

struct PfArgs {
  int T;              // tokens of the chunk
  int kbt;            // k-blocks
  int segs;           // segments of them, an accumulator each
  int m_tiles, n_tiles;   // token tiles (of 256 for a pair), weight tiles
  int N;              // output features (PF_SILU: intermediate size; PF_QKV: heads * 128)
  uint32_t* status;
  const float* ss_in;   // [chunk][kPfTokens]
  int ss_chunks;
  float inv_dim, eps;
  // PF_QKV
  int nq, nkv, kv_f16;
  const __nv_bfloat16 *bq, *bk, *bv, *gq, *gk;
  const float2* rope;   // [kPfTokens][64]
  __nv_bfloat16 *q_out, *kc, *vc;
  const int32_t* ctx;
  // PF_RESID
  float* x;
  const __nv_bfloat16* gain;
  float* ss_out;
  // PF_RESID, PF_SILU: hi rows, lo rows lo_off elements further
  __nv_bfloat16* out;
  size_t lo_off;
};

// 16 consecutive values as 16-bit words, one 32-byte run
template <typename H2>
OOS_DEV void store16(void* dst, const H2 (&h)[8]) {
  const uint4* s = reinterpret_cast<const uint4*>(h);
  reinterpret_cast<uint4*>(dst)[0] = s[0];
  reinterpret_cast<uint4*>(dst)[1] = s[1];
}
OOS_DEV void pack16(const float* v, __nv_bfloat162 (&hi)[8], __nv_bfloat162 (&lo)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    hi[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    lo[i] = __floats2bfloat162_rn(v[2 * i] - __low2float(hi[i]), v[2 * i + 1] - __high2float(hi[i]));
  }
}
OOS_DEV void pack16(const float* v, __half2 (&hi)[8], __half2 (&lo)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    hi[i] = __floats2half2_rn(v[2 * i], v[2 * i + 1]);
    lo[i] = __floats2half2_rn(v[2 * i] - __low2float(hi[i]), v[2 * i + 1] - __high2float(hi[i]));
  }
}
template <typename H2>
OOS_DEV void store16_hilo(void* hi_dst, void* lo_dst, const float* v) {
  H2 hi[8], lo[8];
  pack16(v, hi, lo);
  store16(hi_dst, hi);
  store16(lo_dst, lo);
}
template <typename H2>
OOS_DEV void store16_one(void* dst, const float* v) {
  H2 hi[8], lo[8];
  pack16(v, hi, lo);
  store16(dst, hi);
}
// norm gains and biases: 8 bytes at a time, the alignment the verify GEMMs ask of them too
OOS_DEV void load16(const __nv_bfloat16* p, float (&v)[16]) {
  const uint2* q = reinterpret_cast<const uint2*>(p);
  const uint2 u[4] = {__ldg(q), __ldg(q + 1), __ldg(q + 2), __ldg(q + 3)};
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(u);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    v[2 * i] = __low2float(h[i]);
    v[2 * i + 1] = __high2float(h[i]);
  }
}

template <int EPI>
__global__ void __launch_bounds__(kPfThreads, 1)
    k_pf_gemm(const __grid_constant__ CUtensorMap wm0, const __grid_constant__ CUtensorMap wm1,
              const __grid_constant__ CUtensorMap wm2, const __grid_constant__ CUtensorMap am,
              const __grid_constant__ PfArgs a) {
  constexpr int S = kPfStages;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* ring = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  // stage: [activations hi | activations lo | weights]
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + S * kPfStage);
  uint64_t* empty = full + S;
  uint64_t* accf = empty + S;
  uint64_t* acce = accf + 2;
  uint64_t* drain = acce + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  static_assert((2 * S + 5) * 8 + 8 <= 1024, "barrier block");

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // a pair works on one tile, each CTA (rank) on 128 of its tokens
  const int rank = blockIdx.x & 1, me = blockIdx.x >> 1, G = gridDim.x >> 1;
  const int tiles = a.m_tiles * a.n_tiles;
  const int my_tiles = me < tiles ? (tiles - me + G - 1) / G : 0;
  auto m_of = [&](int tile) { return tile % a.m_tiles * 2 + rank; };   // 128-token tile
  const int n_units = my_tiles * a.kbt;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], 2 * kPfEpiWarps);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 2) tmem_alloc_pair(tmem_slot, kPfTmem);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // the other CTA's barriers are set up before anything arrives on them
  cluster_arrive_release();
  cluster_wait_acquire();
  const uint32_t tmem_base = *tmem_slot;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kPfRegsIssue));
    // ------------------------------------------------------------ TMA producer
    if (warp == 0 && lane == 0) {
      tma_prefetch_desc(&wm0);
      tma_prefetch_desc(&am);
      const uint64_t pol = policy_evict_last();   // every operand is read by many blocks
      // a pair's copies all complete on rank 0's barriers, which expect both CTAs' bytes
      const uint32_t full0 = dsmem_addr(full, 0);
      auto load = [&](void* dst, const CUtensorMap* map, int stage, int x, int y) {
        tma_load_2d_pair(dst, map, full0 + (uint32_t)stage * 8u, x, y, pol);
      };
      auto expect = [&](int stage) {
        if (rank == 0) mbar_arrive_expect_tx(&full[stage], 2 * kPfStage);
      };
      auto load_w = [&](int n, int kb, int stage) {
        unsigned char* dst = ring + stage * kPfStage + 2 * kPfHalf;
#pragma unroll
        for (int j = 0; j < kPfCols / 128; ++j) {   // boxes of 64 weight rows
          const int i = rank * (kPfCols / 128) + j;
          const CUtensorMap* wm = &wm0;
          int row = n * kPfCols + i * 64;          // past the last row: zeros
          if (EPI == PF_SILU) {
            wm = i < 2 ? &wm0 : &wm1;
            row = n * (kPfCols / 2) + (i & 1) * 64;
          } else if (EPI == PF_QKV) {
            int h = n * 2 + i / 2;
            if (h >= a.nq + 2 * a.nkv) h = 0;   // an odd head count's last tile: columns nobody reads
            const int base = h < a.nq ? 0 : h < a.nq + a.nkv ? a.nq : a.nq + a.nkv;
            wm = h < a.nq ? &wm0 : h < a.nq + a.nkv ? &wm1 : &wm2;
            row = (h - base) * 128 + (i & 1) * 64;
          }
          load(dst + j * 64 * kBK * 2, wm, stage, kb * kBK, row);
        }
      };
      auto load_x = [&](int m, int kb, int stage) {
        unsigned char* dst = ring + stage * kPfStage;
        load(dst, &am, stage, kb * kBK, m * kPfRows);
        load(dst + kPfHalf, &am, stage, kb * kBK, kPfTokens + m * kPfRows);
      };
      // the first stages' weights do not depend on the previous kernel
      const int n_pre = n_units < S ? n_units : S;
      int tile = me, kb = 0;
      for (int j = 0; j < n_pre; ++j) {
        expect(j);
        load_w(tile / a.m_tiles, kb, j);
        if (++kb == a.kbt) { kb = 0; tile += G; }
      }
      pdl_wait();
      pdl_trigger();
      tile = me;
      kb = 0;
      int issued = 0;
      for (int j = 0; j < n_units; ++j) {
        const int stage = j % S;
        if (j >= n_pre) {
          if (!mbar_wait(&empty[stage], (uint32_t)(j / S - 1) & 1u, abort_flag, a.status)) break;
          expect(stage);
          load_w(tile / a.m_tiles, kb, stage);
        }
        load_x(m_of(tile), kb, stage);
        ++issued;
        if (++kb == a.kbt) { kb = 0; tile += G; }
      }
      // every copy has landed before the block can exit (immediate on the normal
      // path, where all were consumed; after an abort of one CTA of a pair a phase
      // may stay short of the other's bytes, so the whole wait is bounded)
      const unsigned long long t0 = globaltimer(), most = 10000000ull;
      if (rank == 0) {
        for (int j = issued - S > 0 ? issued - S : 0; j < issued; ++j) {
          while (!mbar_test(smem_addr(&full[j % S]), (uint32_t)((j / S) & 1)) && globaltimer() - t0 < most) {
          }
        }
      } else if (issued < n_units) {   // rank 1 gave up: its last copies land long before this ends
        while (globaltimer() - t0 < 200000ull) {
        }
      }
    }
    // ------------------------------------------------------------ MMA issuer
    if (warp == 1 && lane == 0 && rank == 0) {
      constexpr uint32_t idesc = idesc_bf16_f32(2 * kPfRows, kPfCols);
      int j = 0;
      bool ok = true;
      uint32_t sg = 0;   // segments handed over; they use the two accumulators in turn
      for (int it = 0; it < my_tiles && ok; ++it) {
        for (int i = 0; i < a.segs && ok; ++i, ++sg) {
          const uint32_t b = sg & 1u;
          if (!mbar_wait(&acce[b], ((sg >> 1) & 1u) ^ 1u, abort_flag, a.status)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d = tmem_base + b * kPfCols;
          const int n = a.kbt * (i + 1) / a.segs - a.kbt * i / a.segs;
          for (int kb = 0; kb < n; ++kb, ++j) {
            const int stage = j % S;
            if (!mbar_wait(&full[stage], (uint32_t)(j / S) & 1u, abort_flag, a.status)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t base = smem_addr(ring + stage * kPfStage);
            const uint64_t xh = smem_desc_sw128(base), xl = smem_desc_sw128(base + kPfHalf);
            const uint64_t w = smem_desc_sw128(base + 2 * kPfHalf);
            // lo first: the accumulator is small then, and so is what an addition truncates
#pragma unroll
            for (int k = 0; k < kBK / 16; ++k)
              tc_mma_bf16_pair(d, xl + 2 * k, w + 2 * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
#pragma unroll
            for (int k = 0; k < kBK / 16; ++k) tc_mma_bf16_pair(d, xh + 2 * k, w + 2 * k, idesc, 1u);
            tc_commit_pair(&empty[stage]);
          }
          if (ok) tc_commit_pair(&accf[b]);
        }
      }
      // all issued MMAs complete before TMEM is released
      tc_commit_pair(drain);
      const unsigned long long t0 = globaltimer();
      while (!mbar_test(smem_addr(drain), 0) && globaltimer() - t0 < kWaitLimitNs) {
      }
    }
    __syncwarp();
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kPfRegsEpi));
    // ------------------------------------------------------------ epilogue (warps 4..11)
    pdl_wait();
    pdl_trigger();
    const int q = warp & 3, grp = (warp - 4) >> 2;
    const uint32_t lane_base = tmem_base + ((uint32_t)(q * 32) << 16);
    const int ctx = EPI == PF_QKV ? *a.ctx : 0;
    const uint32_t acce0 = dsmem_addr(acce, 0);   // rank 0's, where the issuer waits
    uint32_t sg = 0;
    for (int it = 0; it < my_tiles; ++it) {
      const int tile = me + it * G;
      const int n = tile / a.m_tiles, t = m_of(tile) * kPfRows + q * 32 + lane;
      const bool live = t < a.T;
      float r = 0.f;
      if (EPI != PF_RESID && live) {   // the input's RMSNorm factor
        float s = 0.f;
#pragma unroll 8
        for (int c = 0; c < a.ss_chunks; ++c) s += a.ss_in[(size_t)c * kPfTokens + t];
        r = rsqrtf(s * a.inv_dim + a.eps);
      }
      // this thread's 128 sums: a head, 128 features, or 64 gate and 64 up rows
      float acc[128];
      bool ok = true;
      for (int i = 0; i < a.segs; ++i, ++sg) {
        const uint32_t b = sg & 1u;
        ok = __all_sync(0xffffffffu, mbar_wait(&accf[b], (sg >> 1) & 1u, abort_flag, a.status));
        if (!ok) break;
        tc_fence_after();
        const uint32_t base = lane_base + b * kPfCols;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const uint32_t col = EPI == PF_SILU ? base + (c < 4 ? 0 : kPfCols / 2) + grp * 64 + (c & 3) * 16
                                              : base + grp * 128 + c * 16;
          float v[16];
          tmem_ld16_nowait(col, v);
          tmem_wait_ld();
          reg_fence(v);
#pragma unroll
          for (int k = 0; k < 16; ++k) acc[c * 16 + k] = i == 0 ? v[k] : acc[c * 16 + k] + v[k];
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_remote(acce0 + 8u * b);
      }
      if (!ok) break;
      auto finish = [&]() {
        const int unit = n * 2 + grp;   // head, or 128-feature block
        if (EPI == PF_QKV) {
          if (unit >= a.nq + 2 * a.nkv) return;
          const int kind = unit < a.nq ? 0 : unit < a.nq + a.nkv ? 1 : 2;
          const int h = kind == 0 ? unit : kind == 1 ? unit - a.nq : unit - a.nq - a.nkv;
          const __nv_bfloat16* bias = kind == 0 ? a.bq : kind == 1 ? a.bk : a.bv;
          const __nv_bfloat16* gn = kind == 0 ? a.gq : kind == 1 ? a.gk : nullptr;
#pragma unroll
          for (int c = 0; c < 128; ++c) acc[c] *= r;
          if (bias) {
#pragma unroll
            for (int c = 0; c < 128; c += 16) {
              float bv[16];
              load16(bias + h * 128 + c, bv);
#pragma unroll
              for (int i = 0; i < 16; ++i) acc[c + i] += bv[i];
            }
          }
          if (gn) {   // per-head RMSNorm
            float ss[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int c = 0; c < 128; ++c) ss[c & 3] += acc[c] * acc[c];
            const float rn = rsqrtf(((ss[0] + ss[1]) + (ss[2] + ss[3])) * (1.f / 128.f) + a.eps);
#pragma unroll
            for (int c = 0; c < 128; c += 16) {
              float g[16];
              load16(gn + c, g);
#pragma unroll
              for (int i = 0; i < 16; ++i) acc[c + i] *= rn * g[i];
            }
          }
          if (kind < 2) {   // rotary pairs c and 64 + c
            const float4* rp = reinterpret_cast<const float4*>(a.rope + (size_t)t * 64);
#pragma unroll
            for (int c = 0; c < 64; c += 2) {
              const float4 cs = __ldg(rp + c / 2);
              const float p0 = acc[c], p1 = acc[64 + c], q0 = acc[c + 1], q1 = acc[65 + c];
              acc[c] = p0 * cs.x - p1 * cs.y;
              acc[64 + c] = p1 * cs.x + p0 * cs.y;
              acc[c + 1] = q0 * cs.z - q1 * cs.w;
              acc[65 + c] = q1 * cs.z + q0 * cs.w;
            }
          }
          if (kind == 0) {
            __nv_bfloat16* dst = a.q_out + ((size_t)t * a.nq + h) * 128;
            const size_t lo = (size_t)kPfTokens * a.nq * 128;
#pragma unroll
            for (int c = 0; c < 128; c += 16) {
              if (a.kv_f16) store16_hilo<__half2>(dst + c, dst + lo + c, acc + c);
              else store16_hilo<__nv_bfloat162>(dst + c, dst + lo + c, acc + c);
            }
          } else {
            __nv_bfloat16* dst = (kind == 1 ? a.kc : a.vc) + ((size_t)(ctx + t) * a.nkv + h) * 128;
#pragma unroll
            for (int c = 0; c < 128; c += 16) {
              if (a.kv_f16) store16_one<__half2>(dst + c, acc + c);
              else store16_one<__nv_bfloat162>(dst + c, acc + c);
            }
          }
        } else if (EPI == PF_RESID) {
          const int f0 = unit * 128;
          if (f0 >= a.N) return;
          float ss = 0.f;
#pragma unroll
          for (int c = 0; c < 128; c += 16) {
            float g[16];
            float4 xv[4];
            float4* xp = reinterpret_cast<float4*>(a.x + (size_t)t * a.N + f0 + c);
#pragma unroll
            for (int i = 0; i < 4; ++i) xv[i] = xp[i];
            load16(a.gain + f0 + c, g);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              float* v = acc + c + 4 * i;
              xv[i].x += v[0];
              xv[i].y += v[1];
              xv[i].z += v[2];
              xv[i].w += v[3];
              xp[i] = xv[i];
              ss += xv[i].x * xv[i].x + xv[i].y * xv[i].y + xv[i].z * xv[i].z + xv[i].w * xv[i].w;
              v[0] = g[4 * i] * xv[i].x;
              v[1] = g[4 * i + 1] * xv[i].y;
              v[2] = g[4 * i + 2] * xv[i].z;
              v[3] = g[4 * i + 3] * xv[i].w;
            }
            __nv_bfloat16* y = a.out + (size_t)t * a.N + f0 + c;
            store16_hilo<__nv_bfloat162>(y, y + a.lo_off, acc + c);
          }
          a.ss_out[(size_t)unit * kPfTokens + t] = ss;
        } else {
          const int i0 = n * (kPfCols / 2) + grp * 64;
          if (i0 >= a.N) return;
#pragma unroll
          for (int c = 0; c < 64; c += 16) {
#pragma unroll
            for (int i = c; i < c + 16; ++i) acc[i] = silu(acc[i] * r) * (acc[64 + i] * r);
            __nv_bfloat16* y = a.out + (size_t)t * a.N + i0 + c;
            store16_hilo<__nv_bfloat162>(y, y + a.lo_off, acc + c);
          }
        }
      };
      if (live) finish();
      __syncwarp();
    }
  }
  tc_fence_before();
  __syncthreads();
  // neither CTA leaves while the other's MMAs, copies or arrivals may reach it
  cluster_arrive_release();
  cluster_wait_acquire();
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, kPfTmem);
  }
}

// ------------------------------------------------------------ chunk preparation
// Validates the chunk's tokens and publishes its committed length.  The first
// chunk of a prompt clears the status words, later ones only add to them.
__global__ void __launch_bounds__(1024) k_pf_prep(const int32_t* __restrict__ tokens, int T, int ctx, int first, int vocab,
                                                  uint32_t* status, int32_t* ctx_out) {
  pdl_wait();
  pdl_trigger();
  bool bad = false;
  for (int i = threadIdx.x; i < T; i += blockDim.x) bad |= tokens[i] < 0 || tokens[i] >= vocab;
  const bool any = __syncthreads_or(bad);
  if (threadIdx.x == 0) {
    *ctx_out = ctx;
    *status = (first ? 0u : *status) | (any ? ST_TREE : 0u);
  }
  if (first && threadIdx.x >= 1 && threadIdx.x < 8) status[threadIdx.x] = 0u;
}

// The last token's final-norm input as row 0 of the verify step's buffers, for
// the LM head: its two halves, and its sum of squares as the first of `chunks`.
__global__ void __launch_bounds__(256) k_pf_last(const __nv_bfloat16* __restrict__ y, size_t lo_off,
                                                 const float* __restrict__ ss, int in_chunks, int t, int H,
                                                 __nv_bfloat16* __restrict__ y_out, float* __restrict__ ss_out,
                                                 int chunks) {
  __shared__ float red[32];
  pdl_wait();
  pdl_trigger();
  for (int f = threadIdx.x; f < H; f += blockDim.x) {
    y_out[f] = y[(size_t)t * H + f];
    y_out[(size_t)kMaxT * H + f] = y[lo_off + (size_t)t * H + f];
  }
  float s = 0.f;
  for (int c = threadIdx.x; c < in_chunks; c += blockDim.x) s += ss[(size_t)c * kPfTokens + t];
  s = block_sum(s, red);
  for (int c = threadIdx.x; c < chunks; c += blockDim.x) ss_out[(size_t)c * kMaxT] = c == 0 ? s : 0.f;
}

// ------------------------------------------------------------ host side
template <int EPI>
static cudaError_t pf_smem() {
  const cudaError_t e = cudaFuncSetAttribute(k_pf_gemm<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPfSmem);
  return e == cudaSuccess ? check_launch_regs((const void*)k_pf_gemm<EPI>, kPfRegsLaunch) : e;
}
cudaError_t prefill_setup() {
  cudaError_t e = pf_smem<PF_QKV>();
  if (e == cudaSuccess) e = pf_smem<PF_RESID>();
  return e == cudaSuccess ? pf_smem<PF_SILU>() : e;
}

bool prefill_encode(Model& m) {
  const auto& c = m.cfg;
  const int qd = c.n_q_heads * c.head_dim;
  return encode_rows_map(&m.pf_xn_map, m.ws.pf_xn, 2 * kPfTokens, c.hidden, kPfRows) &&
         encode_rows_map(&m.pf_xn64_map, m.ws.pf_xn, 2 * kPfTokens, c.hidden, 64) &&
         encode_rows_map(&m.pf_attn_map, m.ws.pf_attn, 2 * kPfTokens, qd, kPfRows) &&
         encode_rows_map(&m.pf_act_map, m.ws.pf_act, 2 * kPfTokens, c.intermediate, kPfRows);
}

// Segments of a GEMM in pairs' tiles: their hi and lo products share an accumulator,
// eight MMAs a k-block, so the k-blocks are half of k_chain's.  Not gate/up's: the MLP's
// share of the next layer's K/V error shows no difference (hidden 1024 .. 5120).
static int pf_segs(const GemmW& g, int epi) {
  const int kbt = g.K / kBK, chain = epi == PF_SILU ? g.chain : (g.chain + 1) / 2;
  return (kbt + chain - 1) / chain;
}

// How one GEMM of a chunk runs: 0 as pairs' tiles of 256 tokens x 256 weight rows
// here, c >= 1 as the verify GEMM's tiles of 128 x 128, k split over clusters of c
// (gate/up: unsplit, 64 tokens x 128 rows of each).
//
// Estimates in microseconds of work in line, one wave after the other: a k-block of
// a pair's tile takes 0.5, a segment 0.6 and a tile's turnover 10, a k-block of a
// verify tile 0.4 and its turnover 8.5, each rank of a cluster 0.9 for the sums it
// pulls; the residual's tiles cost 24 more here (64 or fewer pairs hide neither the
// first loads nor the rows of x they read and write), gate/up's 5.  Against timings of
// each choice in turn at 8 chunk lengths of 136..2048 tokens in 6 shapes (hidden
// 256..5120), the choice is the fastest or within 4 us of it in 180 of 192, and within
// 10 in all.  Both ways, one layer's down GEMM: 512 tokens of the 8B shape 45 us less
// in verify tiles, 2048 tokens of the 2048 x 6144 shape 6 us less in pairs.
static int pf_split(const Model& m, const GemmW& g, int rows, int T, int epi) {
  const int kbt = g.K / kBK;
  const int mt = (T + kPfRows - 1) / kPfRows;
  auto waves = [](long long tiles, int fit) { return (double)((tiles + fit - 1) / fit); };
  const long long tiles = epi == PF_SILU ? (long long)((T + 63) / 64) * ((rows + 255) / 256)
                                         : (long long)mt * ((rows + 127) / 128);
  double best = waves((long long)((mt + 1) / 2) * ((rows + kPfCols - 1) / kPfCols), m.num_sms / 2) *
                    (kbt * 0.5 + pf_segs(g, epi) * 0.6 + 10) +
                (epi == PF_RESID ? 24 : epi == PF_SILU ? 5 : 0);
  int split = 0;
  for (int c = 1; c <= (epi == PF_SILU ? 1 : kMaxSplit) && c <= kbt; ++c) {
    if (m.fit[c] < 1) continue;
    const double t = waves(tiles, m.fit[c]) * ((kbt + c - 1) / c * 0.4 + 8.5) + 0.9 * c;
    if (t < best) {
      best = t;
      split = c;
    }
  }
  return split;
}

template <int EPI>
static cudaError_t launch_pf(Model& m, const GemmW& g, const CUtensorMap& am, PfArgs& a, int rows, cudaStream_t st) {
  // rows: stacked weight rows of the GEMM
  const auto& c = m.cfg;
  a.kbt = g.K / kBK;
  a.segs = pf_segs(g, EPI);
  a.m_tiles = (a.T + 2 * kPfRows - 1) / (2 * kPfRows);
  a.n_tiles = (rows + kPfCols - 1) / kPfCols;
  a.status = m.ws.status;
  a.ss_in = m.ws.pf_ss;
  a.ss_chunks = c.hidden / kTile;
  a.inv_dim = 1.0f / (float)c.hidden;
  a.eps = c.rms_eps;
  const CUtensorMap& w1 = g.n_seg > 1 ? g.pf_map[1] : g.pf_map[0];
  const CUtensorMap& w2 = g.n_seg > 2 ? g.pf_map[2] : g.pf_map[0];
  const long long tiles = (long long)a.m_tiles * a.n_tiles;
  const int pairs = (int)(tiles < m.num_sms / 2 ? tiles : m.num_sms / 2);
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(2 * pairs);
  lc.blockDim = dim3(kPfThreads);
  lc.dynamicSmemBytes = (size_t)kPfSmem;
  lc.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = attr;
  lc.numAttrs = m.pdl ? 2 : 1;
  return cudaLaunchKernelEx(&lc, k_pf_gemm<EPI>, g.pf_map[0], w1, w2, am, a);
}

static PfArgs pf_args(int T) {
  PfArgs a;
  memset(&a, 0, sizeof(a));
  a.T = T;
  return a;
}

static cudaError_t launch_pf_resid(Model& m, int layer, bool down, const void* gain, int T, cudaStream_t st) {
  const GemmW& g = down ? m.g_down[layer] : m.g_o[layer];
  const int split = pf_split(m, g, m.cfg.hidden, T, PF_RESID);
  if (split) return launch_chunk_resid(m, layer, down, gain, T, split, st);
  PfArgs a = pf_args(T);
  a.N = m.cfg.hidden;
  a.x = m.ws.pf_x;
  a.gain = (const __nv_bfloat16*)gain;
  a.out = (__nv_bfloat16*)m.ws.pf_xn;
  a.lo_off = (size_t)kPfTokens * m.cfg.hidden;
  a.ss_out = m.ws.pf_ss;
  return launch_pf<PF_RESID>(m, g, down ? m.pf_act_map : m.pf_attn_map, a, a.N, st);
}

static cudaError_t launch_pf_qkv(Model& m, int layer, void* kc, void* vc, int T, cudaStream_t st) {
  const auto& c = m.cfg;
  const oos_layer_weights& L = m.layers[layer];
  const int rows = (c.n_q_heads + 2 * c.n_kv_heads) * c.head_dim;
  const int split = pf_split(m, m.g_qkv[layer], rows, T, PF_QKV);
  if (split) return launch_chunk_qkv(m, layer, kc, vc, T, split, st);
  PfArgs a = pf_args(T);
  a.N = rows;
  a.nq = c.n_q_heads;
  a.nkv = c.n_kv_heads;
  a.kv_f16 = c.kv_f16 ? 1 : 0;
  a.bq = (const __nv_bfloat16*)(c.qkv_bias ? L.b_q : nullptr);
  a.bk = (const __nv_bfloat16*)(c.qkv_bias ? L.b_k : nullptr);
  a.bv = (const __nv_bfloat16*)(c.qkv_bias ? L.b_v : nullptr);
  a.gq = (const __nv_bfloat16*)(c.qk_norm ? L.q_norm : nullptr);
  a.gk = (const __nv_bfloat16*)(c.qk_norm ? L.k_norm : nullptr);
  a.rope = m.ws.pf_rope;
  a.q_out = (__nv_bfloat16*)m.ws.pf_q;
  a.kc = (__nv_bfloat16*)kc;
  a.vc = (__nv_bfloat16*)vc;
  a.ctx = m.ws.ctx;
  return launch_pf<PF_QKV>(m, m.g_qkv[layer], m.pf_xn_map, a, rows, st);
}

static cudaError_t launch_pf_gu(Model& m, int layer, int T, cudaStream_t st) {
  const auto& c = m.cfg;
  if (pf_split(m, m.g_gu[layer], 2 * c.intermediate, T, PF_SILU)) return launch_chunk_gu(m, layer, T, st);
  PfArgs a = pf_args(T);
  a.N = c.intermediate;
  a.out = (__nv_bfloat16*)m.ws.pf_act;
  a.lo_off = (size_t)kPfTokens * c.intermediate;
  return launch_pf<PF_SILU>(m, m.g_gu[layer], m.pf_xn_map, a, 2 * a.N, st);
}

// Every layer of one chunk of T tokens (128 < T <= kPfTokens) at cache position
// ctx: K/V into slots ctx.., the final norm's input in pf_xn / pf_ss.
cudaError_t prefill_chunk(Model& m, const oos_kv_cache* kv, int ctx, const int32_t* tokens, int T, bool first,
                          cudaStream_t st) {
  const auto& c = m.cfg;
  cudaError_t e = launch(false, k_pf_prep, dim3(1), dim3(1024), 0, st, tokens, T, ctx, first ? 1 : 0, c.vocab,
                         m.ws.status, m.ws.ctx);
  if (e == cudaSuccess) e = launch_embed_pf(m, tokens, T, st);
  for (int l = 0; l < c.n_layers && e == cudaSuccess; ++l) {
    const void* gain = l + 1 < c.n_layers ? m.layers[l + 1].attn_norm : m.w.final_norm;
    e = launch_pf_qkv(m, l, kv->k[l], kv->v[l], T, st);
    if (e == cudaSuccess) e = launch_attention_pf(m, l, kv->k[l], kv->v[l], kv->capacity, ctx, T, st);
    if (e == cudaSuccess) e = launch_pf_resid(m, l, false, m.layers[l].mlp_norm, T, st);
    if (e == cudaSuccess) e = launch_pf_gu(m, l, T, st);
    if (e == cudaSuccess) e = launch_pf_resid(m, l, true, gain, T, st);
  }
  return e;
}

// pf_split of one GEMM of a chunk of T tokens: what the tests of the tiles ask, so that
// they know which ones they reach
static int pf_choice(const Model& m, int layer, int stage, int T) {
  const auto& c = m.cfg;
  switch (stage) {
    case OOS_STAGE_QKV:
      return pf_split(m, m.g_qkv[layer], (c.n_q_heads + 2 * c.n_kv_heads) * c.head_dim, T, PF_QKV);
    case OOS_STAGE_O: return pf_split(m, m.g_o[layer], c.hidden, T, PF_RESID);
    case OOS_STAGE_GATE_UP: return pf_split(m, m.g_gu[layer], 2 * c.intermediate, T, PF_SILU);
    default: return pf_split(m, m.g_down[layer], c.hidden, T, PF_RESID);
  }
}

// the chunk's last token into row 0 of the verify buffers the LM head reads
cudaError_t prefill_last(Model& m, int T, cudaStream_t st) {
  const auto& c = m.cfg;
  return launch(m.pdl, k_pf_last, dim3(1), dim3(256), 0, st, (const __nv_bfloat16*)m.ws.pf_xn,
                (size_t)kPfTokens * c.hidden, (const float*)m.ws.pf_ss, c.hidden / kTile, T - 1, c.hidden,
                (__nv_bfloat16*)m.ws.xn, m.ws.ss, norm_chunks(m, c.n_layers));
}

}  // namespace oos

// not part of the C ABI: 0 pairs' tiles, c >= 1 the verify GEMM's in clusters of c, -1
// no chunk of T tokens or no such GEMM
extern "C" int oos_prefill_tiles(const oos_model* m, int32_t layer, int32_t stage, int32_t T) {
  if (!m || m->cfg.dtype != OOS_DTYPE_BF16 || layer < 0 || layer >= m->cfg.n_layers || T <= oos::kMaxT ||
      T > oos::kPfTokens || stage < OOS_STAGE_QKV || stage > OOS_STAGE_DOWN)
    return -1;
  return oos::pf_choice(*m, layer, stage, T);
}
