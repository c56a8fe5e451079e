// Small kernels of the verify step: tree preparation, embedding, the argmax
// merge with the greedy-acceptance walk, and KV compaction.
#include <math.h>

#include <vector>

#include "common.cuh"
#include "internal.h"

namespace oos {

// ============================================================ tree preparation
// Tree encoding: parents-first numbering (parent[0] = -1, parent[i] < i).  Node
// i attends to the committed cache and its ancestors (itself included); its
// RoPE position is ctx + depth(i).  Ancestor sets are 128-bit masks.
// ctx: the committed length, from the host (ctx_in == nullptr) or from device
// memory; written to ctx_out, where every later kernel of the step reads it.
// first: the call starts here; a later tree of a prompt adds to the status words that
// the chunks before it left.
__global__ void __launch_bounds__(kMaxT) k_tree_prep(const int32_t* __restrict__ tokens,
                                                     const int32_t* __restrict__ parent, int T, int ctx,
                                                     const int32_t* __restrict__ ctx_in, int32_t* ctx_out,
                                                     int first, int vocab, uint32_t* status, int32_t* depth_out,
                                                     int32_t* pos_out, unsigned long long* anc_out) {
  __shared__ int s_parent[kMaxT];
  __shared__ int s_bad;
  pdl_wait();
  pdl_trigger();
  if (ctx_in) ctx = *ctx_in;
  const int i = threadIdx.x;
  if (i == 0) *ctx_out = ctx;
  if (i == 0) s_bad = 0;
  __syncthreads();
  if (i < T) {
    const int p = parent[i];
    const int tok = tokens[i];
    const bool ok = (i == 0 ? p == -1 : (p >= 0 && p < i)) && tok >= 0 && tok < vocab;
    s_parent[i] = p;
    if (!ok) atomicOr(&s_bad, 1);
  }
  __syncthreads();
  if (i == 0) *status = (first ? 0u : *status) | (s_bad ? ST_TREE : 0u);
  if (first && i >= 1 && i < 8) status[i] = 0u;   // where a pipeline wait gave up (see common.cuh)
  if (i < T) {
    int d = 0;
    unsigned long long lo = 0, hi = 0;
    if (!s_bad) {
      for (int a = i; a >= 0; a = (a == 0 ? -1 : s_parent[a])) {
        if (a < 64) lo |= 1ull << a; else hi |= 1ull << (a - 64);
        if (a != i) ++d;
      }
    } else {
      if (i < 64) lo = 1ull << i; else hi = 1ull << (i - 64);
    }
    depth_out[i] = d;
    pos_out[i] = ctx + d;
    anc_out[2 * i] = lo;
    anc_out[2 * i + 1] = hi;
  }
}

// The first kernel of a step is launched without programmatic serialisation:
// it starts only after all earlier work on the stream (the previous step's
// compaction, the caller's cache writes) has completed.  Every kernel of the
// step lets its dependents launch only after its own dependency wait, so a
// kernel that starts finds the kernel two launches back, and all before it,
// complete: later kernels may read cache positions < ctx, and ctx itself,
// before their own dependency wait.
cudaError_t launch_tree_prep(Model& m, const int32_t* tokens, const int32_t* parent, int T, int ctx,
                             const int32_t* ctx_dev, bool first, cudaStream_t st) {
  return launch(false, k_tree_prep, dim3(1), dim3(kMaxT), 0, st, tokens, parent, T, ctx, ctx_dev, m.ws.ctx,
                first ? 1 : 0, m.cfg.vocab, m.ws.status, m.ws.depth, m.ws.pos, m.ws.anc);
}

cudaGraphNode_t find_tree_prep_node(cudaGraph_t g) {
  size_t n = 0;
  if (cudaGraphGetNodes(g, nullptr, &n) != cudaSuccess || n == 0) return nullptr;
  std::vector<cudaGraphNode_t> nodes(n);
  if (cudaGraphGetNodes(g, nodes.data(), &n) != cudaSuccess) return nullptr;
  for (size_t i = 0; i < n; ++i) {
    cudaGraphNodeType t;
    if (cudaGraphNodeGetType(nodes[i], &t) != cudaSuccess || t != cudaGraphNodeTypeKernel) continue;
    cudaKernelNodeParams p;
    if (cudaGraphKernelNodeGetParams(nodes[i], &p) != cudaSuccess) continue;
    if (p.func == (void*)k_tree_prep) return nodes[i];
  }
  return nullptr;
}

// the same arguments launch_tree_prep passes, with another committed length
cudaError_t set_tree_prep_ctx(Model& m, cudaGraphExec_t ex, cudaGraphNode_t node, const int32_t* tokens,
                              const int32_t* parent, int T, int ctx) {
  const int32_t* ctx_in = nullptr;
  int32_t* ctx_out = m.ws.ctx;
  int first = 1;
  int vocab = m.cfg.vocab;
  uint32_t* status = m.ws.status;
  int32_t* depth = m.ws.depth;
  int32_t* pos = m.ws.pos;
  unsigned long long* anc = m.ws.anc;
  void* args[] = {&tokens, &parent, &T, &ctx, &ctx_in, &ctx_out, &first, &vocab, &status, &depth, &pos, &anc};
  cudaKernelNodeParams p = {};
  p.func = (void*)k_tree_prep;
  p.gridDim = dim3(1);
  p.blockDim = dim3(kMaxT);
  p.sharedMemBytes = 0;
  p.kernelParams = args;
  return cudaGraphExecKernelNodeSetParams(ex, node, &p);
}

// ============================================================ embedding
// bf16 path: the first RMSNorm is folded into the QKV GEMM.  Block (t, chunk)
// writes x = E[token] (fp32 residual), y = g (.) x (hi/lo bf16 GEMM input) and
// the chunk's sum of x^2 (the GEMM epilogue turns the chunk sums into
// rsqrt(mean(x^2) + eps)).
// Block (t, 0) also fills the step's RoPE table: cos/sin of pos[t] * theta^(-2m/d)
// for m < d/2, the angle formed and reduced to [-pi, pi] in fp64 once per step
// (every layer reuses it).  `rows`: token rows the buffers are laid out for (the
// lo halves lie rows * H elements further, the sums rows apart).  pos: the nodes'
// positions, or nullptr for consecutive tokens from *ctx (a prefill chunk).
__global__ void __launch_bounds__(128) k_embed_tc(const int32_t* __restrict__ tokens, const __nv_bfloat16* __restrict__ emb,
                                                  const __nv_bfloat16* __restrict__ gain, int H, int vocab,
                                                  float* __restrict__ x, __nv_bfloat16* __restrict__ y, int rows,
                                                  float* __restrict__ ss, const int32_t* __restrict__ pos,
                                                  const int32_t* __restrict__ ctx,
                                                  const double* __restrict__ inv_freq, int half_d,
                                                  float2* __restrict__ rope) {
  __shared__ float red[32];
  pdl_wait();
  pdl_trigger();
  const int t = blockIdx.x, f = blockIdx.y * 128 + threadIdx.x;
  if (blockIdx.y == 0 && threadIdx.x < half_d) {
    const double two_pi = 6.283185307179586476925286766559;
    const double ang = (double)(pos ? pos[t] : *ctx + t) * inv_freq[threadIdx.x];
    float sn, cs;
    sincosf((float)(ang - two_pi * rint(ang / two_pi)), &sn, &cs);
    rope[t * half_d + threadIdx.x] = make_float2(cs, sn);
  }
  int tok = tokens[t];
  tok = tok < 0 ? 0 : (tok >= vocab ? vocab - 1 : tok);   // invalid trees are flagged by tree_prep
  float v = 0.f;
  if (f < H) {
    v = __bfloat162float(emb[(size_t)tok * H + f]);
    x[(size_t)t * H + f] = v;
    store_act(y, (size_t)t * H + f, (size_t)rows * H, v * __bfloat162float(gain[f]));
  }
  const float s = block_sum(v * v, red);
  if (threadIdx.x == 0) ss[(size_t)blockIdx.y * rows + t] = s;
}

cudaError_t launch_embed_tc(Model& m, const int32_t* tokens, int T, cudaStream_t st) {
  const auto& c = m.cfg;
  return launch(m.pdl, k_embed_tc, dim3(T, (c.hidden + 127) / 128), dim3(128), 0, st, tokens,
                (const __nv_bfloat16*)m.w.embed, (const __nv_bfloat16*)m.layers[0].attn_norm, c.hidden, c.vocab,
                m.ws.x, (__nv_bfloat16*)m.ws.xn, kMaxT, m.ws.ss, (const int32_t*)m.ws.pos, (const int32_t*)nullptr,
                (const double*)m.ws.inv_freq, c.head_dim / 2, m.ws.rope);
}
cudaError_t launch_embed_pf(Model& m, const int32_t* tokens, int T, cudaStream_t st) {
  const auto& c = m.cfg;
  return launch(m.pdl, k_embed_tc, dim3(T, (c.hidden + 127) / 128), dim3(128), 0, st, tokens,
                (const __nv_bfloat16*)m.w.embed, (const __nv_bfloat16*)m.layers[0].attn_norm, c.hidden, c.vocab,
                m.ws.pf_x, (__nv_bfloat16*)m.ws.pf_xn, kPfTokens, m.ws.pf_ss, (const int32_t*)nullptr,
                (const int32_t*)m.ws.ctx, (const double*)m.ws.inv_freq, c.head_dim / 2, m.ws.pf_rope);
}

// bf16 path, checking output only: the final RMSNorm output in fp32,
// hidden[t] = x[t] * rsqrt(mean(x[t]^2) + eps) * g.
__global__ void __launch_bounds__(256) k_final_hidden(const float* __restrict__ x, const float* __restrict__ ss,
                                                      int chunks, const __nv_bfloat16* __restrict__ gain, int H,
                                                      float eps, float* __restrict__ hidden) {
  pdl_wait();
  pdl_trigger();
  const int t = blockIdx.x;
  float s = 0.f;
  for (int c = 0; c < chunks; ++c) s += ss[(size_t)c * kMaxT + t];
  const float r = rsqrtf(s / (float)H + eps);
  for (int f = threadIdx.x; f < H; f += blockDim.x)
    hidden[(size_t)t * H + f] = x[(size_t)t * H + f] * r * __bfloat162float(gain[f]);
}

cudaError_t launch_final_hidden(Model& m, float* hidden, int T, cudaStream_t st) {
  const auto& c = m.cfg;
  return launch(m.pdl, k_final_hidden, dim3(T), dim3(256), 0, st, (const float*)m.ws.x, (const float*)m.ws.ss,
                norm_chunks(m, c.n_layers), (const __nv_bfloat16*)m.w.final_norm, c.hidden, c.rms_eps, hidden);
}

// ============================================================ argmax merge + acceptance walk
// Greedy longest-prefix acceptance (Eq. 1; "Verify and commit") by one warp.
// ok(0) = 1; ok(i) = ok(parent) and token_i == argmax(parent).  The committed
// path ends at the deepest ok node (lowest id on ties); bonus = its argmax.
// Nodes at or past n_valid are padding of a fixed-size tree and never ok.
OOS_DEV void accept_walk_warp(const int32_t* tokens, const int32_t* parent, const int32_t* depth,
                              const int32_t* argmax, int T, int n_valid, bool bad, int32_t* len_out,
                              int32_t* nodes_out, int32_t* toks_out, int32_t* bonus_out) {
  const int lane = threadIdx.x & 31;
  if (bad) {
    for (int i = lane; i < T; i += 32) {
      nodes_out[i] = -1;
      toks_out[i] = -1;
    }
    if (lane == 0) {
      *len_out = 0;
      *bonus_out = -1;
    }
    return;
  }
  int best_key = 0x7fffffff;  // key = (kMaxT - depth) * 256 + node: min = deepest, then lowest id
  for (int i = lane; i < T; i += 32) {
    bool ok = i < n_valid;
    for (int a = i; ok && a != 0; a = parent[a]) {
      const int p = parent[a];
      if (tokens[a] != argmax[p]) {
        ok = false;
        break;
      }
    }
    if (ok) {
      const int key = (kMaxT - depth[i]) * 256 + i;
      best_key = key < best_key ? key : best_key;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const int other = __shfl_xor_sync(0xffffffffu, best_key, o);
    best_key = other < best_key ? other : best_key;
  }
  const int deepest = best_key & 255;
  const int len = depth[deepest] + 1;
  for (int j = len + lane; j < T; j += 32) {
    nodes_out[j] = -1;
    toks_out[j] = -1;
  }
  if (lane == 0) {
    for (int a = deepest; a >= 0; a = (a == 0 ? -1 : parent[a])) {
      nodes_out[depth[a]] = a;
      toks_out[depth[a]] = tokens[a];
    }
    *len_out = len;
    *bonus_out = argmax[deepest];
  }
}

__global__ void __launch_bounds__(1024) k_argmax_accept(const float* __restrict__ v1, const int32_t* __restrict__ i1,
                                                         const float* __restrict__ v2, int n_parts,
                                                         const int32_t* __restrict__ tokens,
                                                         const int32_t* __restrict__ parent,
                                                         const int32_t* __restrict__ depth, const uint32_t* status,
                                                         int T, const int32_t* __restrict__ n_valid_dev,
                                                         int32_t* argmax_ws, float* top1_ws, float* top2_ws,
                                                         int32_t* len, int32_t* nodes, int32_t* toks, int32_t* bonus,
                                                         int32_t* dbg_argmax, float* dbg_top1, float* dbg_top2) {
  __shared__ int32_t s_tok[kMaxT], s_par[kMaxT], s_dep[kMaxT], s_arg[kMaxT];
  __shared__ Top2 s_top[1024];   // [CTA states' share][node]
  pdl_wait();
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  // The merge is order independent (max with lowest-id ties, multiset second max).
  // One SM's loads bound this kernel, so a warp reads 32 neighbouring nodes of a CTA's
  // states at a time, its share of the CTAs; then a warp per node merges the shares.
  // A lane per CTA instead fetched 32 bytes for every 4 it used: the Llama step at T =
  // 128 took 18 us more (5064 against 5046), the 0.6B one at T = 32 1 us.
  const int groups = (T + 31) / 32, shares = nw / groups;
  const int share = warp / groups, node = warp % groups * 32 + lane;
  if (share < shares && node < T) {
    Top2 r{-INFINITY, 0x7fffffff, -INFINITY};
#pragma unroll 4
    for (int c = share; c < n_parts; c += shares) {
      const size_t k = (size_t)c * kMaxT + node;
      r = top2_merge(r, Top2{v1[k], i1[k], v2[k]});
    }
    s_top[share * T + node] = r;
  }
  __syncthreads();
  for (int t = warp; t < T; t += nw) {
    Top2 r{-INFINITY, 0x7fffffff, -INFINITY};
    if (lane < shares) r = s_top[lane * T + t];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      Top2 y{__shfl_xor_sync(0xffffffffu, r.v1, o), __shfl_xor_sync(0xffffffffu, r.i1, o),
             __shfl_xor_sync(0xffffffffu, r.v2, o)};
      r = top2_merge(r, y);
    }
    if (lane == 0) {
      argmax_ws[t] = r.i1;
      top1_ws[t] = r.v1;
      top2_ws[t] = r.v2;
      if (dbg_argmax) dbg_argmax[t] = r.i1;
      if (dbg_top1) dbg_top1[t] = r.v1;
      if (dbg_top2) dbg_top2[t] = r.v2;
      s_arg[t] = r.i1;
    }
  }
  const int i = threadIdx.x;
  if (i < T) {
    s_tok[i] = tokens[i];
    s_par[i] = parent[i];
    s_dep[i] = depth[i];
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    int n_valid = n_valid_dev ? *n_valid_dev : T;
    n_valid = n_valid < 1 ? 1 : (n_valid > T ? T : n_valid);
    // a malformed tree or a pipeline wait that gave up: no accepted path
    accept_walk_warp(s_tok, s_par, s_dep, s_arg, T, n_valid, (*status & (ST_TREE | ST_TIMEOUT)) != 0, len, nodes,
                     toks, bonus);
  }
}

cudaError_t launch_argmax_accept(Model& m, const int32_t* tokens, const int32_t* parent, int T, const int32_t* n_valid,
                                 int n_parts, int32_t* len, int32_t* nodes, int32_t* toks, int32_t* bonus,
                                 int32_t* dbg_argmax, float* dbg_top1, float* dbg_top2, cudaStream_t st) {
  return launch(m.pdl, k_argmax_accept, dim3(1), dim3(1024), 0, st, (const float*)m.ws.lm_v1,
                (const int32_t*)m.ws.lm_i, (const float*)m.ws.lm_v2, n_parts, tokens, parent,
                (const int32_t*)m.ws.depth, (const uint32_t*)m.ws.status, T, n_valid, m.ws.argmax, m.ws.top1,
                m.ws.top2, len, nodes, toks, bonus, dbg_argmax, dbg_top1, dbg_top2);
}

// standalone walk: validates the tree itself
__global__ void k_accept_walk(const int32_t* tokens, const int32_t* parent, const int32_t* argmax, int T,
                              int32_t* len, int32_t* nodes, int32_t* toks, int32_t* bonus, int32_t* status) {
  __shared__ int32_t s_tok[kMaxT], s_par[kMaxT], s_dep[kMaxT], s_arg[kMaxT];
  __shared__ int s_bad;
  const int i = threadIdx.x;
  if (i == 0) s_bad = 0;
  __syncthreads();
  if (i < T) {
    s_tok[i] = tokens[i];
    s_par[i] = parent[i];
    s_arg[i] = argmax[i];
    const bool ok = i == 0 ? s_par[i] == -1 : (s_par[i] >= 0 && s_par[i] < i);
    if (!ok) atomicOr(&s_bad, 1);
  }
  __syncthreads();
  if (i < T) {
    int d = 0;
    if (!s_bad)
      for (int a = i; a != 0; a = s_par[a]) ++d;
    s_dep[i] = d;
  }
  __syncthreads();
  if (i < 32) accept_walk_warp(s_tok, s_par, s_dep, s_arg, T, T, s_bad != 0, len, nodes, toks, bonus);
  if (i == 0) *status = s_bad ? OOS_ETREE : OOS_OK;
}

cudaError_t launch_accept_walk(const int32_t* tokens, const int32_t* parent, const int32_t* argmax, int T,
                               int32_t* len, int32_t* nodes, int32_t* toks, int32_t* bonus, int32_t* status,
                               cudaStream_t st) {
  k_accept_walk<<<1, kMaxT, 0, st>>>(tokens, parent, argmax, T, len, nodes, toks, bonus, status);
  return cudaGetLastError();
}

// ============================================================ KV compaction
// Slot ctx + j <- slot ctx + nodes[j] for j < len, per layer, for K and V.
// One block per (layer, K|V, kv head): all sources are staged in shared
// memory before any destination is written, so a source that is also a later
// destination is read before it is overwritten.
struct KvPtrs {
  void* k[kMaxLayers];
  void* v[kMaxLayers];
};

template <typename E>
__global__ void k_kv_compact(KvPtrs p, int nkv, int d, int ctx, const int32_t* __restrict__ ctx_dev,
                             const int32_t* __restrict__ nodes, const int32_t* __restrict__ len_ptr, int max_len) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  E* buf = reinterpret_cast<E*>(smem_raw);
  pdl_wait();
  pdl_trigger();
  if (ctx_dev) ctx = *ctx_dev;
  const int layer = blockIdx.x, which = blockIdx.y, g = blockIdx.z;
  E* base = (E*)(which == 0 ? p.k[layer] : p.v[layer]);
  int len = *len_ptr;
  len = len < 0 ? 0 : (len > max_len ? max_len : len);
  for (int e = threadIdx.x; e < len * d; e += blockDim.x) {
    const int j = e / d, c = e % d;
    const int src = nodes[j];
    if (src >= 0 && src < max_len) buf[e] = base[((size_t)(ctx + src) * nkv + g) * d + c];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < len * d; e += blockDim.x) {
    const int j = e / d, c = e % d;
    const int src = nodes[j];
    if (src >= 0 && src < max_len) base[((size_t)(ctx + j) * nkv + g) * d + c] = buf[e];
  }
}

cudaError_t compact_setup() {
  cudaError_t e = cudaFuncSetAttribute(k_kv_compact<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kMaxT * 128 * 4);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_kv_compact<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              kMaxT * 128 * 2);
}

cudaError_t launch_kv_compact(Model& m, const oos_kv_cache& kv, int ctx, const int32_t* ctx_dev, const int32_t* nodes,
                              const int32_t* len, int max_len, cudaStream_t st) {
  const auto& c = m.cfg;
  KvPtrs p;
  for (int l = 0; l < c.n_layers; ++l) {
    p.k[l] = kv.k[l];
    p.v[l] = kv.v[l];
  }
  dim3 grid(c.n_layers, 2, c.n_kv_heads);
  const size_t smem = (size_t)max_len * c.head_dim * m.esize;
  if (c.dtype == OOS_DTYPE_BF16)
    return launch(m.pdl, k_kv_compact<__nv_bfloat16>, grid, dim3(256), smem, st, p, c.n_kv_heads, c.head_dim, ctx,
                  ctx_dev, nodes, len, max_len);
  return launch(m.pdl, k_kv_compact<float>, grid, dim3(256), smem, st, p, c.n_kv_heads, c.head_dim, ctx, ctx_dev,
                nodes, len, max_len);
}

}  // namespace oos
