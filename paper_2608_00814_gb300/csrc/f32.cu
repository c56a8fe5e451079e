// The fp32 path: small models on the CUDA cores.
//
// A step of such a model is bound by launch and load latency, not by bytes (6 MB
// for the 2-layer, 256-wide decoder), so the kernels are few -- five per layer, the
// elementwise steps in the projections -- and every one forms all the dot products
// it can from one round of loads: a warp takes R weight rows and TOK tokens at a
// time, the lanes split the reduction, and the R TOK sums are reduced together.
// TOK is 8, or 4, 2 or 1 for a tree that has no more nodes: a wide model's weights
// would otherwise wait for arithmetic that nobody reads (2 layers of the
// 2048-wide shape at T = 1 / 2 / 8: 671 / 624 / 370 us with 8 always, 208 / 239 / 322 so).
// RMSNorm needs no kernel of its own: a projection reads the whole input rows, so
// it sums their squares alongside and scales its products by the row's factor.
// The 2-layer decoder's step (T = 8, 128 cached positions): 176 us with a kernel
// per elementwise step and a loop over tokens, 62 us with these.
#include <math.h>

#include "common.cuh"
#include "internal.h"

namespace oos {

constexpr int kF32Tok = 8;        // most tokens a warp takes at a time
constexpr int kF32Warps = 4;      // warps per block, but for the q/k/v projection

// V consecutive floats (V = 4: from a 16-byte boundary)
template <int V>
struct F32Vec {
  float v[V];
  OOS_DEV void load(const float* p) {
    if (V == 4) {
      const float4 u = __ldg(reinterpret_cast<const float4*>(p));
      v[0] = u.x;
      v[V > 1 ? 1 : 0] = u.y;
      v[V > 2 ? 2 : 0] = u.z;
      v[V > 3 ? 3 : 0] = u.w;
    } else {
      v[0] = *p;
    }
  }
};

// Number of values a call of f32_dots leaves in buf: R rows x TOK tokens, then the
// TOK sums of squares when NORM.
template <int R, bool NORM, int TOK>
constexpr int kDots = R * TOK + (NORM ? TOK : 0);

// buf[r * TOK + t] = w[r] . (gain (.) x[t]), buf[R * TOK + t] = |x[t]|^2, by one warp.
// x: nt <= TOK rows of K floats, FULL: TOK of them; plain loads, since the previous
// kernel wrote them.
template <int R, int V, bool NORM, int TOK, bool FULL>
OOS_DEV void f32_dots_of(const float* const (&w)[R], const float* x, const float* __restrict__ gain, int K, int nt,
                         float* buf) {
  const int lane = threadIdx.x & 31;
  float acc[kDots<R, NORM, TOK>];
#pragma unroll
  for (int i = 0; i < kDots<R, NORM, TOK>; ++i) acc[i] = 0.f;
#pragma unroll(TOK <= 2 ? 16 / V : 2)
  for (int k = lane * V; k < K; k += 32 * V) {
    F32Vec<V> wv[R], g;
#pragma unroll
    for (int r = 0; r < R; ++r) wv[r].load(w[r] + k);
    if (NORM) g.load(gain + k);
#pragma unroll
    for (int t = 0; t < TOK; ++t) {
      const float* p = x + (size_t)t * K + k;
      float xv[V];
      if (!FULL && t >= nt) {
#pragma unroll
        for (int c = 0; c < V; ++c) xv[c] = 0.f;
      } else if (V == 4) {
        const float4 u = __ldcg(reinterpret_cast<const float4*>(p));
        xv[0] = u.x;
        xv[V > 1 ? 1 : 0] = u.y;
        xv[V > 2 ? 2 : 0] = u.z;
        xv[V > 3 ? 3 : 0] = u.w;
      } else {
        xv[0] = __ldcg(p);
      }
#pragma unroll
      for (int c = 0; c < V; ++c) {
        const float xg = NORM ? xv[c] * g.v[c] : xv[c];
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r * TOK + t] = fmaf(wv[r].v[c], xg, acc[r * TOK + t]);
        if (NORM) acc[R * TOK + t] = fmaf(xv[c], xv[c], acc[R * TOK + t]);
      }
    }
  }
  int base, n;
  warp_sums(acc, base, n);
#pragma unroll
  for (int i = 0; i < kDots<R, NORM, TOK>; ++i)
    if (i < n) buf[base + i] = acc[i];
  __syncwarp();
}

template <int R, int V, bool NORM, int TOK>
OOS_DEV void f32_dots(const float* const (&w)[R], const float* x, const float* __restrict__ gain, int K, int nt,
                      float* buf) {
  if (nt == TOK) f32_dots_of<R, V, NORM, TOK, true>(w, x, gain, K, nt, buf);
  else f32_dots_of<R, V, NORM, TOK, false>(w, x, gain, K, nt, buf);
}

// ------------------------------------------------------------ embedding, rotary table
// x[t] = E[token_t]; block t also fills its row of the step's RoPE table: cos/sin of
// pos[t] * theta^(-2m/d), the angle reduced to [-pi, pi] in fp64.
__global__ void __launch_bounds__(256) k_f32_embed(const int32_t* __restrict__ tokens, const float* __restrict__ emb,
                                                   int H, int vocab, float* __restrict__ x, const int32_t* pos,
                                                   const double* __restrict__ inv_freq, int half_d,
                                                   float2* __restrict__ rope) {
  pdl_wait();
  pdl_trigger();
  const int t = blockIdx.x;
  if (threadIdx.x < half_d) {
    const double two_pi = 6.283185307179586476925286766559;
    const double ang = (double)pos[t] * inv_freq[threadIdx.x];
    float sn, cs;
    sincosf((float)(ang - two_pi * rint(ang / two_pi)), &sn, &cs);
    rope[t * half_d + threadIdx.x] = make_float2(cs, sn);
  }
  int tok = tokens[t];
  tok = tok < 0 ? 0 : (tok >= vocab ? vocab - 1 : tok);   // invalid trees are flagged by tree_prep
  for (int f = threadIdx.x; f < H; f += blockDim.x) x[(size_t)t * H + f] = emb[(size_t)tok * H + f];
}

// ------------------------------------------------------------ q/k/v
// Block (head slot, token group): the d rows of one q, k or v head for TOK tokens,
// kQkvWarps warps of 4 rows at a time; then a warp per token: bias, q/k RMSNorm,
// RoPE; q to the query buffer, k and v to cache slots *ctx + t (skipped when the
// cache pointers are null).
constexpr int kQkvWarps = 16;

struct F32QkvArgs {
  const float *wq, *wk, *wv, *bq, *bk, *bv, *gq, *gk, *gain, *x;
  const float2* rope;
  float *q, *kc, *vc;
  const int32_t* ctx;
  int H, nq, nkv, d, T;
  float eps;
};

template <int V, int TOK>
__global__ void __launch_bounds__(32 * kQkvWarps) k_f32_qkv(F32QkvArgs a) {
  __shared__ float s_out[TOK][128];
  __shared__ float s_buf[kQkvWarps][kDots<4, true, TOK>];
  pdl_wait();
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int hs = blockIdx.x, t0 = blockIdx.y * TOK, nt = min(TOK, a.T - t0);
  const int kind = hs < a.nq ? 0 : hs < a.nq + a.nkv ? 1 : 2;
  const int h = kind == 0 ? hs : kind == 1 ? hs - a.nq : hs - a.nq - a.nkv;
  const float* W = (kind == 0 ? a.wq : kind == 1 ? a.wk : a.wv) + (size_t)h * a.d * a.H;
  for (int r0 = warp * 4; r0 < a.d; r0 += kQkvWarps * 4) {
    const float* w[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) w[r] = W + (size_t)min(r0 + r, a.d - 1) * a.H;
    f32_dots<4, V, true, TOK>(w, a.x + (size_t)t0 * a.H, a.gain, a.H, nt, s_buf[warp]);
    // lane = (row, token)
    const int r = lane / TOK, t = lane % TOK;
    if (r < 4 && r0 + r < a.d)
      s_out[t][r0 + r] = s_buf[warp][lane] * rsqrtf(s_buf[warp][4 * TOK + t] / (float)a.H + a.eps);
    __syncwarp();
  }
  __syncthreads();
  const int t = warp, half = a.d / 2;
  if (t >= nt) return;
  const float* bias = kind == 0 ? a.bq : kind == 1 ? a.bk : a.bv;
  const float* g = kind == 0 ? a.gq : kind == 1 ? a.gk : nullptr;
  float* v = s_out[t];
  float ss = 0.f;
  for (int j = lane; j < a.d; j += 32) {
    if (bias) v[j] += bias[h * a.d + j];
    ss += v[j] * v[j];
  }
  const float rn = g ? rsqrtf(warp_sum(ss) / (float)a.d + a.eps) : 1.f;
  __syncwarp();
  float* dst;
  if (kind == 0) {
    dst = a.q + ((size_t)(t0 + t) * a.nq + h) * a.d;
  } else {
    float* c = kind == 1 ? a.kc : a.vc;
    if (!c) return;
    dst = c + ((size_t)(*a.ctx + t0 + t) * a.nkv + h) * a.d;
  }
  for (int j = lane; j < half; j += 32) {   // the rotate-half pair (j, j + d/2)
    float v0 = v[j], v1 = v[j + half];
    if (g) {
      v0 *= rn * g[j];
      v1 *= rn * g[j + half];
    }
    if (kind < 2) {
      const float2 cs = a.rope[(size_t)(t0 + t) * half + j];
      const float o0 = v0 * cs.x - v1 * cs.y;
      v1 = v1 * cs.x + v0 * cs.y;
      v0 = o0;
    }
    dst[j] = v0;
    dst[j + half] = v1;
  }
}

// ------------------------------------------------------------ attention
// Block per (node, head).  Per tile of 256 keys: a thread scores one key (16-byte
// loads where d allows), then the threads take (output dim, key share) and add
// their share's weighted values; the shares meet in shared memory at the end.
constexpr int kF32Keys = 256;
__global__ void __launch_bounds__(kF32Keys) k_f32_attn(const float* __restrict__ q, const float* kc, const float* vc,
                                                       const unsigned long long* __restrict__ anc, int T, int nq, int nkv,
                                                       int d, int vec, const int32_t* __restrict__ ctx_dev, float scale,
                                                       float* __restrict__ out) {
  __shared__ __align__(16) float qs[128];
  __shared__ float ps[kF32Keys];
  __shared__ float red[32];
  __shared__ float s_acc[kF32Keys];
  pdl_wait();
  pdl_trigger();
  const int ctx = *ctx_dev;
  const int i = blockIdx.x, h = blockIdx.y, g = h / (nq / nkv), tid = threadIdx.x;
  if (tid < d) qs[tid] = __ldcg(q + ((size_t)i * nq + h) * d + tid);
  const unsigned long long w0 = anc[2 * i], w1 = anc[2 * i + 1];
  __syncthreads();
  const int shares = kF32Keys / d, share = tid / d, dim = tid - share * d;   // 2 or more shares (d <= 128)
  float m = -INFINITY, l = 0.f, acc = 0.f;
  const int n_keys = ctx + T;
  for (int base = 0; base < n_keys; base += kF32Keys) {
    const int kk = base + tid;
    bool valid = kk < n_keys;
    if (valid && kk >= ctx) {
      const int j = kk - ctx;
      valid = ((j < 64 ? (w0 >> j) : (w1 >> (j - 64))) & 1ull) != 0;
    }
    float sc = -INFINITY;
    if (valid) {
      const float* kr = kc + ((size_t)kk * nkv + g) * d;
      float dot[4] = {0.f, 0.f, 0.f, 0.f};
      if (vec) {
#pragma unroll 8
        for (int c = 0; c < d; c += 4) {
          const float4 k4 = __ldcg(reinterpret_cast<const float4*>(kr + c));
          const float4 q4 = *reinterpret_cast<const float4*>(qs + c);
          dot[0] = fmaf(q4.x, k4.x, dot[0]);
          dot[1] = fmaf(q4.y, k4.y, dot[1]);
          dot[2] = fmaf(q4.z, k4.z, dot[2]);
          dot[3] = fmaf(q4.w, k4.w, dot[3]);
        }
      } else {
#pragma unroll 8
        for (int c = 0; c < d; ++c) dot[0] = fmaf(qs[c], __ldcg(kr + c), dot[0]);
      }
      sc = ((dot[0] + dot[1]) + (dot[2] + dot[3])) * scale;
    }
    const float mn = fmaxf(m, block_max(sc, red));
    const float p = valid ? expf(sc - mn) : 0.f;
    const float corr = (m == -INFINITY) ? 0.f : expf(m - mn);   // nothing is valid before the first valid key
    ps[tid] = p;
    l = l * corr + block_sum(p, red);   // (its barriers publish ps)
    acc *= corr;
    if (share < shares) {
      const int nk = min(kF32Keys, n_keys - base);
      const float* vr = vc + ((size_t)base * nkv + g) * d + dim;
      int k = share;
      // a weight of 0 drops its value: slots of other branches may hold anything
      for (; k + 7 * shares < nk; k += 8 * shares) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = __ldcg(vr + (size_t)(k + u * shares) * nkv * d);
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (ps[k + u * shares] != 0.f) acc = fmaf(ps[k + u * shares], v[u], acc);
      }
      for (; k < nk; k += shares)
        if (ps[k] != 0.f) acc = fmaf(ps[k], __ldcg(vr + (size_t)k * nkv * d), acc);
    }
    m = mn;
    __syncthreads();
  }
  s_acc[tid] = share < shares ? acc : 0.f;
  __syncthreads();
  if (tid < d) {
    float s = 0.f;
    for (int u = 0; u < shares; ++u) s += s_acc[u * d + tid];
    out[(size_t)i * nq * d + (size_t)h * d + tid] = s / l;
  }
}

// ------------------------------------------------------------ O and down: x[t][f] += W[f] . in[t]
// a warp per output row and TOK tokens
template <int V, int TOK>
__global__ void __launch_bounds__(32 * kF32Warps) k_f32_resid(const float* __restrict__ W, int N, int K, const float* in,
                                                              int T, float* x) {
  __shared__ float s_buf[kF32Warps][kDots<1, false, TOK>];
  pdl_wait();
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int f = blockIdx.x * kF32Warps + warp, t0 = blockIdx.y * TOK, nt = min(TOK, T - t0);
  if (f >= N) return;
  const float* w[1] = {W + (size_t)f * K};
  const float old = lane < nt ? __ldcg(x + (size_t)(t0 + lane) * N + f) : 0.f;
  f32_dots<1, V, false, TOK>(w, in + (size_t)t0 * K, nullptr, K, nt, s_buf[warp]);
  if (lane < nt) x[(size_t)(t0 + lane) * N + f] = old + s_buf[warp][lane];
}

// ------------------------------------------------------------ gate/up: act = silu(gate) * up
// a warp per intermediate row (its gate and its up row) and TOK tokens
template <int V, int TOK>
__global__ void __launch_bounds__(32 * kF32Warps) k_f32_gu(const float* __restrict__ Wg, const float* __restrict__ Wu, int I,
                                                           int K, const float* x, const float* __restrict__ gain, float eps,
                                                           int T, float* __restrict__ act) {
  __shared__ float s_buf[kF32Warps][kDots<2, true, TOK>];
  pdl_wait();
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * kF32Warps + warp, t0 = blockIdx.y * TOK, nt = min(TOK, T - t0);
  if (i >= I) return;
  const float* w[2] = {Wg + (size_t)i * K, Wu + (size_t)i * K};
  float* b = s_buf[warp];
  f32_dots<2, V, true, TOK>(w, x + (size_t)t0 * K, gain, K, nt, b);
  if (lane < nt) {
    const float r = rsqrtf(b[2 * TOK + lane] / (float)K + eps);
    const float g = b[lane] * r, u = b[TOK + lane] * r;
    act[(size_t)(t0 + lane) * I + i] = g / (1.f + expf(-g)) * u;
  }
}

// ------------------------------------------------------------ LM head
// Block b scans vocabulary rows [b*rows, (b+1)*rows), four rows of a warp at a time;
// each warp keeps a running top-2 per node, merged at the end.
template <int V, int TOK>
__global__ void __launch_bounds__(32 * kF32Warps) k_f32_lm_head(const float* __restrict__ W, int vocab, int H,
                                                                int rows_per_block, const float* x,
                                                                const float* __restrict__ gain, float eps, int T,
                                                                float* am_v1, int32_t* am_i, float* am_v2) {
  __shared__ Top2 st[kF32Warps][kMaxT];
  __shared__ float s_buf[kF32Warps][kDots<4, true, TOK>];
  pdl_wait();
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int t = lane; t < T; t += 32) st[warp][t] = Top2{-INFINITY, 0x7fffffff, -INFINITY};
  __syncwarp();
  const int r_begin = blockIdx.x * rows_per_block;
  const int r_end = min(vocab, r_begin + rows_per_block);
  float* b = s_buf[warp];
  for (int r0 = r_begin + 4 * warp; r0 < r_end; r0 += 4 * kF32Warps) {
    const float* w[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) w[r] = W + (size_t)min(r0 + r, r_end - 1) * H;
    for (int t0 = 0; t0 < T; t0 += TOK) {
      const int nt = min(TOK, T - t0);
      f32_dots<4, V, true, TOK>(w, x + (size_t)t0 * H, gain, H, nt, b);
      if (lane < nt) {
        const float rt = rsqrtf(b[4 * TOK + lane] / (float)H + eps);
        Top2 s = st[warp][t0 + lane];
        for (int r = 0; r < 4 && r0 + r < r_end; ++r)
          s = top2_merge(s, Top2{b[r * TOK + lane] * rt, r0 + r, -INFINITY});
        st[warp][t0 + lane] = s;
      }
      __syncwarp();
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < T; t += blockDim.x) {
    Top2 r = st[0][t];
    for (int w = 1; w < kF32Warps; ++w) r = top2_merge(r, st[w][t]);
    am_v1[(size_t)blockIdx.x * kMaxT + t] = r.v1;
    am_i[(size_t)blockIdx.x * kMaxT + t] = r.i1;
    am_v2[(size_t)blockIdx.x * kMaxT + t] = r.v2;
  }
}

// checking output only: hidden[t] = x[t] * rsqrt(mean(x[t]^2) + eps) * g
__global__ void __launch_bounds__(256) k_f32_hidden(const float* x, const float* __restrict__ gain, int H, float eps,
                                                    float* __restrict__ hidden) {
  __shared__ float red[32];
  pdl_wait();
  pdl_trigger();
  const float* xr = x + (size_t)blockIdx.x * H;
  float ss = 0.f;
  for (int f = threadIdx.x; f < H; f += blockDim.x) ss += xr[f] * xr[f];
  const float r = rsqrtf(block_sum(ss, red) / (float)H + eps);
  for (int f = threadIdx.x; f < H; f += blockDim.x) hidden[(size_t)blockIdx.x * H + f] = xr[f] * r * gain[f];
}

// ------------------------------------------------------------ host side
static const float* fp(const void* p) { return (const float*)p; }
// 16-byte loads of rows of K floats: every row of every matrix on a 16-byte
// boundary (the workspace's buffers are), else element by element
static bool rows16(int K, const void* a, const void* b = nullptr, const void* c = nullptr, const void* d = nullptr) {
  return K % 4 == 0 && (((uintptr_t)a | (uintptr_t)b | (uintptr_t)c | (uintptr_t)d) & 15) == 0;
}
template <int N>
struct Tok {
  static constexpr int value = N;
};
// f(tokens a warp takes) for a tree of T nodes
template <typename F>
static cudaError_t by_tokens(int T, F f) {
  if (T == 1) return f(Tok<1>{});
  if (T == 2) return f(Tok<2>{});
  return T <= 4 ? f(Tok<4>{}) : f(Tok<kF32Tok>{});
}
// f(floats a load, tokens a warp takes)
template <typename F>
static cudaError_t by_form(bool rows_16, int T, F f) {
  return by_tokens(T, [&](auto tok) { return rows_16 ? f(Tok<4>{}, tok) : f(Tok<1>{}, tok); });
}

cudaError_t launch_f32_embed(Model& m, const int32_t* tokens, int T, cudaStream_t st) {
  const auto& c = m.cfg;
  return launch(m.pdl, k_f32_embed, dim3(T), dim3(256), 0, st, tokens, fp(m.w.embed), c.hidden, c.vocab, m.ws.x,
                (const int32_t*)m.ws.pos, (const double*)m.ws.inv_freq, c.head_dim / 2, m.ws.rope);
}

cudaError_t launch_f32_qkv(Model& m, int layer, void* kc, void* vc, int T, cudaStream_t st) {
  const auto& c = m.cfg;
  const oos_layer_weights& L = m.layers[layer];
  F32QkvArgs a;
  a.wq = fp(L.w_q);
  a.wk = fp(L.w_k);
  a.wv = fp(L.w_v);
  a.bq = fp(c.qkv_bias ? L.b_q : nullptr);
  a.bk = fp(c.qkv_bias ? L.b_k : nullptr);
  a.bv = fp(c.qkv_bias ? L.b_v : nullptr);
  a.gq = fp(c.qk_norm ? L.q_norm : nullptr);
  a.gk = fp(c.qk_norm ? L.k_norm : nullptr);
  a.gain = fp(L.attn_norm);
  a.x = m.ws.x;
  a.rope = m.ws.rope;
  a.q = (float*)m.ws.q;
  a.kc = (float*)kc;
  a.vc = (float*)vc;
  a.ctx = m.ws.ctx;
  a.H = c.hidden;
  a.nq = c.n_q_heads;
  a.nkv = c.n_kv_heads;
  a.d = c.head_dim;
  a.T = T;
  a.eps = c.rms_eps;
  return by_form(rows16(c.hidden, L.w_q, L.w_k, L.w_v, L.attn_norm), T, [&](auto v, auto tok) {
    constexpr int V = decltype(v)::value, TOK = decltype(tok)::value;
    return launch(m.pdl, k_f32_qkv<V, TOK>, dim3(c.n_q_heads + 2 * c.n_kv_heads, (T + TOK - 1) / TOK),
                  dim3(32 * kQkvWarps), 0, st, a);
  });
}

cudaError_t launch_f32_attention(Model& m, const void* kc, const void* vc, int T, cudaStream_t st) {
  const auto& c = m.cfg;
  const int vec = rows16(c.head_dim, kc) ? 1 : 0;
  return launch(m.pdl, k_f32_attn, dim3(T, c.n_q_heads), dim3(kF32Keys), 0, st, fp(m.ws.q), fp(kc), fp(vc),
                (const unsigned long long*)m.ws.anc, T, c.n_q_heads, c.n_kv_heads, c.head_dim, vec,
                (const int32_t*)m.ws.ctx, 1.0f / sqrtf((float)c.head_dim), (float*)m.ws.attn);
}

static cudaError_t launch_f32_resid(Model& m, const void* W, int K, const void* in, int T, cudaStream_t st) {
  const int H = m.cfg.hidden;
  return by_form(rows16(K, W), T, [&](auto v, auto tok) {
    constexpr int V = decltype(v)::value, TOK = decltype(tok)::value;
    return launch(m.pdl, k_f32_resid<V, TOK>, dim3((H + kF32Warps - 1) / kF32Warps, (T + TOK - 1) / TOK),
                  dim3(32 * kF32Warps), 0, st, fp(W), H, K, fp(in), T, m.ws.x);
  });
}
cudaError_t launch_f32_o(Model& m, int layer, int T, cudaStream_t st) {
  return launch_f32_resid(m, m.layers[layer].w_o, m.cfg.n_q_heads * m.cfg.head_dim, m.ws.attn, T, st);
}
cudaError_t launch_f32_down(Model& m, int layer, int T, cudaStream_t st) {
  return launch_f32_resid(m, m.layers[layer].w_down, m.cfg.intermediate, m.ws.act, T, st);
}

cudaError_t launch_f32_gu(Model& m, int layer, int T, cudaStream_t st) {
  const auto& c = m.cfg;
  const oos_layer_weights& L = m.layers[layer];
  return by_form(rows16(c.hidden, L.w_gate, L.w_up, L.mlp_norm), T, [&](auto v, auto tok) {
    constexpr int V = decltype(v)::value, TOK = decltype(tok)::value;
    return launch(m.pdl, k_f32_gu<V, TOK>, dim3((c.intermediate + kF32Warps - 1) / kF32Warps, (T + TOK - 1) / TOK),
                  dim3(32 * kF32Warps), 0, st, fp(L.w_gate), fp(L.w_up), c.intermediate, c.hidden, (const float*)m.ws.x,
                  fp(L.mlp_norm), c.rms_eps, T, (float*)m.ws.act);
  });
}

cudaError_t launch_f32_lm_head(Model& m, int T, cudaStream_t st) {
  const auto& c = m.cfg;
  const int rows = (c.vocab + m.lm_grid - 1) / m.lm_grid;
  return by_form(rows16(c.hidden, m.w.lm_head, m.w.final_norm), T, [&](auto v, auto tok) {
    constexpr int V = decltype(v)::value, TOK = decltype(tok)::value;
    return launch(m.pdl, k_f32_lm_head<V, TOK>, dim3(m.lm_grid), dim3(32 * kF32Warps), 0, st, fp(m.w.lm_head), c.vocab,
                  c.hidden, rows, (const float*)m.ws.x, fp(m.w.final_norm), c.rms_eps, T, m.ws.lm_v1, m.ws.lm_i,
                  m.ws.lm_v2);
  });
}

cudaError_t launch_f32_hidden(Model& m, float* hidden, int T, cudaStream_t st) {
  const auto& c = m.cfg;
  return launch(m.pdl, k_f32_hidden, dim3(T), dim3(256), 0, st, (const float*)m.ws.x, fp(m.w.final_norm), c.hidden,
                c.rms_eps, hidden);
}

}  // namespace oos
